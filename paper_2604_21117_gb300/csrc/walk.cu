// The walk index: its construction on the device and the search of a batch
// as given through it (walk.cuh describes the index).
#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>

#include "walk.cuh"

namespace btgb {

// --------------------------------------------------------- construction

// Where the key of rank i lies in the tree image's leaves.
struct LeafView {
    const void *keys, *vals;
    uint64_t base, rem;  // keys per leaf, leaves with one more
    uint32_t m;
};

__device__ __forceinline__ uint64_t leaf_slot(const LeafView &lv, uint64_t i)
{
    uint64_t leaf, slot;
    rank_to_leaf(i, lv.base, lv.rem, leaf, slot);
    return leaf * lv.m + slot;
}

template <typename K>
__device__ __forceinline__ typename WalkWord<K>::type walk_word(const LeafView &lv, uint64_t i, int p0)
{
    const K k = static_cast<const K *>(lv.keys)[leaf_slot(lv, i)];
    if constexpr (sizeof(K) > 8)
        return key32_window(k, p0);
    else
        return k;
}

// One thread per key slot of the entries.
template <typename K, typename V>
__global__ void k_walk_entries(LeafView lv, uint64_t n, uint64_t slots, unsigned char *__restrict__ entries)
{
    constexpr uint32_t G = walk_group(sizeof(K), sizeof(V));
    for (uint64_t i = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x; i < slots;
         i += static_cast<uint64_t>(gridDim.x) * blockDim.x) {
        unsigned char *p = entries + i / G * 64u;
        K *k = reinterpret_cast<K *>(p) + i % G;
        V *v = reinterpret_cast<V *>(p + 32) + i % G;
        if (i < n) {
            const uint64_t s = leaf_slot(lv, i);
            *k = static_cast<const K *>(lv.keys)[s];
            *v = static_cast<const V *>(lv.vals)[s];
        } else {
            *k = KeyOps<K>::ones();
            *v = static_cast<V>(~static_cast<V>(0));
        }
    }
}

// One thread per separator of a level whose nodes' children span `span`
// entries each (E entries of G keys in all).
template <typename K>
__global__ void k_walk_nodes(LeafView lv, uint64_t nodes, uint64_t span, uint64_t E, uint32_t G, int p0,
                             typename WalkWord<K>::type *__restrict__ out)
{
    using W = typename WalkWord<K>::type;
    constexpr uint32_t SEP = 32 / sizeof(W);
    for (uint64_t i = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x; i < nodes * SEP;
         i += static_cast<uint64_t>(gridDim.x) * blockDim.x) {
        const uint64_t end = (i / SEP * (SEP + 1) + i % SEP + 1) * span;  // entries up to this child's last
        out[i] = end < E ? walk_word<K>(lv, end * G - 1, p0) : static_cast<W>(~static_cast<W>(0));
    }
}

// The binary tree over the segments' largest keys (all but the last
// segment's): position k at depth d holds the separator of sorted rank
// ((2 (k - 2^d) + 1) << (bits - 1 - d)) - 1.
template <typename K>
__global__ void k_walk_top(LeafView lv, int bits, uint64_t span, uint64_t E, uint32_t G, int p0,
                           typename WalkWord<K>::type *__restrict__ out)
{
    using W = typename WalkWord<K>::type;
    const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= (1u << bits)) return;
    W v = static_cast<W>(~static_cast<W>(0));
    if (k > 0) {
        const int d = 31 - __clz(k);
        const uint64_t rank = (static_cast<uint64_t>(2u * (k - (1u << d)) + 1u) << (bits - 1 - d)) - 1;
        const uint64_t end = (rank + 1) * span;
        if (end < E) v = walk_word<K>(lv, end * G - 1, p0);
    }
    out[k] = v;
}

static unsigned fill_grid(uint64_t items)
{
    const uint64_t g = (items + 255) / 256;
    return static_cast<unsigned>(g < 65536 ? (g > 0 ? g : 1) : 65536);
}

template <typename K>
static cudaError_t build_levels(WalkDev &w, const LeafView &lv, uint64_t E, uint32_t G, const uint64_t *count,
                                unsigned char *top, unsigned char *nodes, cudaStream_t s)
{
    using W = typename WalkWord<K>::type;
    constexpr uint64_t F = 32 / sizeof(W) + 1;
    uint64_t span = 1;
    for (int l = w.levels - 1; l >= 0; --l) {
        k_walk_nodes<K><<<fill_grid(count[l] * (F - 1)), 256, 0, s>>>(lv, count[l], span, E, G, w.p0,
                                                                     reinterpret_cast<W *>(nodes + w.off[l]));
        span *= F;
    }
    if (w.top_bits)
        k_walk_top<K><<<(1u << w.top_bits) / 256 + 1, 256, 0, s>>>(lv, w.top_bits, span, E, G, w.p0,
                                                                  reinterpret_cast<W *>(top));
    return cudaGetLastError();
}

template <typename K, typename V>
static cudaError_t build_entries(const LeafView &lv, uint64_t n, uint64_t E, uint32_t G, unsigned char *entries,
                                 cudaStream_t s)
{
    k_walk_entries<K, V><<<fill_grid(E * G), 256, 0, s>>>(lv, n, E * G, entries);
    return cudaGetLastError();
}

cudaError_t walk_build(bt_tree *t, cudaStream_t s)
{
    const DevTree &d = t->dev;
    const uint64_t n = t->info.n;
    if (n == 0) return cudaSuccess;
    const int kb = d.key_bytes, vb = d.val_bytes, wb = kb > 8 ? 8 : kb;
    const uint32_t G = walk_group(kb, vb);
    const uint64_t F = walk_fan(kb), E = (n + G - 1) / G;
    if (E >= (1ull << 32)) return cudaSuccess;  // node and entry numbers are 32-bit
    WalkDev w;
    memset(&w, 0, sizeof(w));
    w.n = n;
    w.p0 = d.split_p0;
    memcpy(w.kmin32, d.kmin32, sizeof(w.kmin32));
    memcpy(w.kmax32, d.kmax32, sizeof(w.kmax32));
    // as few levels of nodes as leave at most 2^walk_top_bits segments
    uint64_t segs = E, count[kWalkLevels];
    while (segs > (1ull << walk_top_bits(kb))) {
        segs = (segs + F - 1) / F;
        ++w.levels;
    }
    uint64_t c = E;
    for (int l = w.levels - 1; l >= 0; --l) {
        c = (c + F - 1) / F;
        count[l] = c;
    }
    if (segs > 1) {
        w.top_bits = 2;  // whole 16-byte pieces for the bulk copy
        while ((1ull << w.top_bits) < segs) ++w.top_bits;
        w.top_bytes = static_cast<uint32_t>(wb) << w.top_bits;
    }
    uint64_t bytes = (static_cast<uint64_t>(w.top_bytes) + 255) & ~255ull;
    const uint64_t node_off = bytes;
    for (int l = 0; l < w.levels; ++l) {
        w.off[l] = bytes - node_off;
        bytes += count[l] * 32;
    }
    bytes = (bytes + 255) & ~255ull;
    const uint64_t ent_off = bytes;
    bytes += E * 64;
    size_t free_b = 0, total_b = 0;
    cudaError_t e = cudaMemGetInfo(&free_b, &total_b);
    if (e != cudaSuccess) return e;
    if (bytes > free_b / 4) return cudaSuccess;
    e = cudaMalloc(&t->d_walk, bytes);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();  // searched by the descent, as without this index
        t->d_walk = nullptr;
        return cudaSuccess;
    }
    if (e != cudaSuccess) return e;
    unsigned char *base = static_cast<unsigned char *>(t->d_walk);
    w.top = base;
    w.nodes = base + node_off;
    w.entries = base + ent_off;
    const int leaf = d.height - 1;
    const LeafView lv{d.keys[leaf], d.vals, d.cbase[leaf], d.crem[leaf], static_cast<uint32_t>(d.m)};
    unsigned char *nodes = base + node_off, *ent = base + ent_off;
    if (kb == 32) {
        e = build_levels<Key32>(w, lv, E, G, count, base, nodes, s);
        if (e == cudaSuccess)
            e = vb == 8 ? build_entries<Key32, uint64_t>(lv, n, E, G, ent, s)
                        : build_entries<Key32, uint32_t>(lv, n, E, G, ent, s);
    } else if (kb == 8) {
        e = build_levels<uint64_t>(w, lv, E, G, count, base, nodes, s);
        if (e == cudaSuccess)
            e = vb == 8 ? build_entries<uint64_t, uint64_t>(lv, n, E, G, ent, s)
                        : build_entries<uint64_t, uint32_t>(lv, n, E, G, ent, s);
    } else {
        e = build_levels<uint32_t>(w, lv, E, G, count, base, nodes, s);
        if (e == cudaSuccess)
            e = vb == 8 ? build_entries<uint32_t, uint64_t>(lv, n, E, G, ent, s)
                        : build_entries<uint32_t, uint32_t>(lv, n, E, G, ent, s);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    t->walk = w;
    return e;
}

// --------------------------------------------------------------- search

template <int MODEL>
constexpr int walk_threads()
{
    return MODEL == kModelMLP ? 512 : 1024;  // the network's hidden layer stays in registers
}

// A model and what turns its window of leaves into one of segments.
struct WalkModel {
    ModelDev md;
    uint64_t leaf_base, leaf_rem;  // keys per leaf, leaves with one more
    uint32_t span;                 // entries per segment
};

// One query per lane, one block per SM; every block takes a contiguous run
// of 32-query chunks of the batch, its warps chunk by chunk in turn, the
// next chunk's queries loaded while the present one walks.  The top is
// copied once per block by one bulk copy, before the wait for the previous
// kernel of the stream.
//
// What bounds it: divergent sectors.  A warp's 32-lane read of one sector
// per lane occupies an SM for 34 cycles when it comes from the L2 and 20
// when it hits L1; an 8-byte probe of the top in shared memory for 6 (5-ary
// nodes in shared memory: 30 per level, so the top is binary).  Over 2^24
// uint64 keys a query is 13 probes, four nodes and an entry of two sectors,
// about 290 cycles per warp, 30 us for 2^20 queries; measured 41.1 us with
// three trees in turn (38.7 for one), against 92.4 us for the partition and
// the level-wise descent.  1024 threads on one SM: with two blocks of 768 or
// 512 the two copies of the top take the L1 the nodes want (42-67 us).
// The kernel does not trigger the launch of its successor: blocks started
// early pair up on the SMs that drain first, and the batch then waits for
// those (300,007 uint32 queries: 15.0 us with the trigger, 8.6 without).
//
// MODEL: the learned search.  The model's window of leaves, as a range of
// segments, takes the place of the top's binary search where the separators
// around it prove it; the walk below is the same.
template <typename K, typename V, int MODEL>
__global__ void __launch_bounds__(walk_threads<MODEL>())
    k_walk(const WalkDev w, const WalkModel m, const RawOf<K> *__restrict__ q, uint32_t nq, V *__restrict__ out_v,
           uint8_t *__restrict__ out_f, uint32_t wait_polls)
{
    using W = typename WalkWord<K>::type;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) uint64_t bar;
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (threadIdx.x == 0) {
        mbar_init(&bar);
        mbar_arrive_expect_tx(&bar, w.top_bytes);
        if (w.top_bytes) bulk_g2s(smem, w.top, w.top_bytes, &bar);
    }
    ModelView mv{};
    if constexpr (MODEL != kModelNone) mv = model_to_smem<MODEL>(m.md, smem + w.top_bytes);
    pdl_wait();
    const uint32_t chunks = (nq + 31) / 32;
    const uint32_t c1 = static_cast<uint32_t>(static_cast<uint64_t>(chunks) * (blockIdx.x + 1) / gridDim.x);
    uint32_t c = static_cast<uint32_t>(static_cast<uint64_t>(chunks) * blockIdx.x / gridDim.x) + warp;
    // lanes past the end follow the last query (no traffic of their own)
    auto load = [&](uint32_t chunk) {
        const uint32_t i = chunk * 32 + lane;
        return KeyOps<K>::load(q, i < nq ? i : nq - 1);
    };
    K next = KeyOps<K>::ones();
    if (c < c1) next = load(c);
    __syncthreads();  // the barrier is initialised, the model copied
    if (!mbar_wait_warp(&bar, 0, wait_polls)) {
        mbar_give_up(&bar, 0, static_cast<int>(lane));
        return;
    }
    for (; c < c1; c += nw) {
        K key = next;
        if (c + nw < c1) next = load(c + nw);
        bool in = true;
        W word;
        if constexpr (sizeof(K) > 8) {
            // outside [smallest, largest] the word says nothing: walk the
            // smallest key, and miss
            const Key32 lo{{w.kmin32[0], w.kmin32[1], w.kmin32[2], w.kmin32[3]}};
            const Key32 hi{{w.kmax32[0], w.kmax32[1], w.kmax32[2], w.kmax32[3]}};
            in = !(key < lo) && !(hi < key);
            if (!in) key = lo;
            word = key32_window(key, w.p0);
        } else {
            word = key;
        }
        const W *top = reinterpret_cast<const W *>(smem);
        uint32_t seg;
        if constexpr (MODEL == kModelNone) {
            seg = walk_segment<W>(top, w.top_bits, word);
        } else {
            constexpr uint32_t G = walk_group(sizeof(K), sizeof(V));
            uint32_t lo, hi;
            model_window<MODEL>(m.md, mv, static_cast<uint64_t>(key), lo, hi);
            // first key of leaf lo, last key of leaf hi, as entries, as segments
            const uint64_t r0 = lo * m.leaf_base + (lo < m.leaf_rem ? lo : m.leaf_rem);
            const uint64_t r1 = (hi + 1ull) * m.leaf_base + (hi + 1ull < m.leaf_rem ? hi + 1ull : m.leaf_rem) - 1;
            seg = walk_segment_in<W>(top, w.top_bits, static_cast<uint32_t>(r0 / G) / m.span,
                                     static_cast<uint32_t>(r1 / G) / m.span, word);
        }
        V val;
        bool hit = walk_lookup<K, V>(w, walk_entry<W>(w, seg, word), key, val);
        if (!in) {
            hit = false;
            val = static_cast<V>(~static_cast<V>(0));
        }
        const uint32_t i = c * 32 + lane;
        if (i < nq) {
            out_v[i] = val;
            out_f[i] = hit ? 1 : 0;
        }
    }
}

template <typename K, typename V, int MODEL>
static cudaError_t walk_launch(const bt_tree *t, const ModelDev *md, const void *q, uint64_t nq, void *out_v,
                               uint8_t *out_f, cudaStream_t s)
{
    auto kern = k_walk<K, V, MODEL>;
    const WalkDev &w = t->walk;
    constexpr int kMaxTop = static_cast<int>(sizeof(typename WalkWord<K>::type)) << walk_top_bits(sizeof(K));
    constexpr int kMaxModel = MODEL == kModelNone ? 0 : static_cast<int>(kModelSmemSegments) * 20;
    int sms = 0;
    cudaError_t e = dev_sm_count(&sms);
    if (e == cudaSuccess) e = ensure_dyn_smem(reinterpret_cast<const void *>(kern), kMaxTop + kMaxModel);
    if (e != cudaSuccess) return e;
    WalkModel m;
    memset(&m, 0, sizeof(m));
    if (MODEL != kModelNone) {
        const int leaf = t->dev.height - 1;
        m.md = *md;
        m.leaf_base = t->dev.cbase[leaf];
        m.leaf_rem = t->dev.crem[leaf];
        m.span = 1;
        for (int l = 0; l < w.levels; ++l) m.span *= walk_fan(static_cast<int>(sizeof(K)));
    }
    // one block per SM with as many warps as its share of the chunks
    constexpr uint64_t kWarps = walk_threads<MODEL>() / 32;
    const uint64_t chunks = (nq + 31) / 32, n = static_cast<uint64_t>(sms > 0 ? sms : 1);
    const uint64_t per_sm = (chunks + n - 1) / n;
    const uint64_t warps = per_sm < kWarps ? per_sm : kWarps;
    const uint64_t grid = (chunks + warps - 1) / warps < n ? (chunks + warps - 1) / warps : n;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(static_cast<unsigned>(grid));
    cfg.blockDim = dim3(static_cast<unsigned>(warps * 32));
    cfg.dynamicSmemBytes = w.top_bytes + (MODEL == kModelNone ? 0u : model_smem_bytes(m.md));
    cfg.stream = s;
    cudaLaunchAttribute attr;
    memset(&attr, 0, sizeof(attr));
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, w, m, static_cast<const RawOf<K> *>(q), static_cast<uint32_t>(nq),
                              static_cast<V *>(out_v), out_f, first_wait_polls());
}

template <typename K, typename V>
static cudaError_t walk_model(const bt_tree *t, const ModelDev *md, const void *q, uint64_t nq, void *out_v,
                              uint8_t *out_f, cudaStream_t s)
{
    if constexpr (sizeof(K) <= 8) {
        if (md && md->kind == kModelPL) return walk_launch<K, V, kModelPL>(t, md, q, nq, out_v, out_f, s);
        if (md) return walk_launch<K, V, kModelMLP>(t, md, q, nq, out_v, out_f, s);
    }
    return walk_launch<K, V, kModelNone>(t, md, q, nq, out_v, out_f, s);
}

cudaError_t walk_search(const bt_tree *t, const void *q, uint64_t nq, void *out_v, uint8_t *out_f, cudaStream_t s,
                        const ModelDev *md)
{
    const int kb = t->dev.key_bytes;
    const bool v8 = t->dev.val_bytes == 8;
    if (kb == 32)
        return v8 ? walk_model<Key32, uint64_t>(t, md, q, nq, out_v, out_f, s)
                  : walk_model<Key32, uint32_t>(t, md, q, nq, out_v, out_f, s);
    if (kb == 8)
        return v8 ? walk_model<uint64_t, uint64_t>(t, md, q, nq, out_v, out_f, s)
                  : walk_model<uint64_t, uint32_t>(t, md, q, nq, out_v, out_f, s);
    return v8 ? walk_model<uint32_t, uint64_t>(t, md, q, nq, out_v, out_f, s)
              : walk_model<uint32_t, uint32_t>(t, md, q, nq, out_v, out_f, s);
}

cudaError_t take_wait_counters_walk(unsigned *timeouts, unsigned *pending)
{
    return take_wait_counters(timeouts, pending);
}

}  // namespace btgb
