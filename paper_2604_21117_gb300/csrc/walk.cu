// The walk index: its construction on the device and the search of a batch
// as given through it (walk.cuh describes the index).
#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>
#include <vector>

#include "walk.cuh"

namespace btgb {

// --------------------------------------------------------- construction

constexpr uint64_t kWalkAskBytes = 32ull << 20;  // larger indexes are held to a share of the free memory

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
        constexpr uint32_t B = walk_entry_bytes(sizeof(K));
        unsigned char *p = entries + i / G * B;
        K *k = reinterpret_cast<K *>(p) + i % G;
        V *v = reinterpret_cast<V *>(p + B / 2) + i % G;
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

// The words that bound the keys of coded node `root`, which spans `span`
// entries: (lo, hi].
template <typename K>
__device__ __forceinline__ void root_bounds(const LeafView &lv, uint64_t root, uint64_t span, uint64_t n, uint32_t G,
                                            int p0, typename WalkWord<K>::type &lo, typename WalkWord<K>::type &hi)
{
    const uint64_t first = root * span * G, end = first + span * G;
    lo = walk_word<K>(lv, first ? first - 1 : 0, p0);
    hi = walk_word<K>(lv, (end < n ? end : n) - 1, p0);
}

// One thread per code of a coded level whose nodes' children span `span`
// entries, under roots of `root_span` entries.
template <typename K>
__global__ void k_walk_codes(LeafView lv, uint64_t nodes, uint64_t span, uint64_t root_span, uint64_t n, uint64_t E,
                             uint32_t G, int p0, uint16_t *__restrict__ out)
{
    using W = typename WalkWord<K>::type;
    constexpr uint32_t SEP = kCodeFan - 1;
    for (uint64_t i = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x; i < nodes * SEP;
         i += static_cast<uint64_t>(gridDim.x) * blockDim.x) {
        const uint64_t end = (i / SEP * kCodeFan + i % SEP + 1) * span;  // entries up to this child's last
        uint32_t code = 0xFFFFu;
        if (end < E) {
            W lo, hi;
            root_bounds<K>(lv, (end - 1) / root_span, root_span, n, G, p0, lo, hi);
            code = walk_code<W>(walk_word<K>(lv, end * G - 1, p0), lo, hi);
        }
        out[i] = static_cast<uint16_t>(code);
    }
}

// Neighbouring entries under one root whose largest keys' codes tie.
template <typename K>
__global__ void k_walk_ties(LeafView lv, uint64_t root_span, uint64_t n, uint64_t E, uint32_t G, int p0,
                            unsigned long long *__restrict__ ties)
{
    using W = typename WalkWord<K>::type;
    unsigned long long mine = 0;
    for (uint64_t i = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x; i + 1 < E;
         i += static_cast<uint64_t>(gridDim.x) * blockDim.x) {
        if (i / root_span != (i + 1) / root_span) continue;
        W lo, hi;
        root_bounds<K>(lv, i / root_span, root_span, n, G, p0, lo, hi);
        const uint64_t next = (i + 2) * G;
        if (walk_code<W>(walk_word<K>(lv, (i + 1) * G - 1, p0), lo, hi) ==
            walk_code<W>(walk_word<K>(lv, (next < n ? next : n) - 1, p0), lo, hi))
            ++mine;
    }
    if (mine) atomicAdd(ties, mine);
}

static unsigned fill_grid(uint64_t items)
{
    const uint64_t g = (items + 255) / 256;
    return static_cast<unsigned>(g < 65536 ? (g > 0 ? g : 1) : 65536);
}

// Sum over the keys of the probes that a search for each needs to come from
// the first key with its word to itself (two per doubling of the distance).
__global__ void k_walk_runs(LeafView lv, uint64_t n, int p0, unsigned long long *__restrict__ probes)
{
    unsigned long long mine = 0;
    for (uint64_t i = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x; i < n;
         i += static_cast<uint64_t>(gridDim.x) * blockDim.x) {
        const uint64_t word = walk_word<Key32>(lv, i, p0);
        if (i == 0 || walk_word<Key32>(lv, i - 1, p0) != word) continue;
        uint64_t lo = 0, hi = i;  // the first key whose word is not below
        while (lo < hi) {
            const uint64_t mid = (lo + hi) / 2;
            if (walk_word<Key32>(lv, mid, p0) < word)
                lo = mid + 1;
            else
                hi = mid;
        }
        mine += 2u * static_cast<unsigned>(64 - __clzll(static_cast<long long>(i - lo)));
    }
    if (mine) atomicAdd(probes, mine);
}

template <typename K>
static cudaError_t build_levels(const WalkDev &w, const LeafView &lv, uint64_t E, uint32_t G, const uint64_t *count,
                                unsigned char *nodes, cudaStream_t s)
{
    using W = typename WalkWord<K>::type;
    constexpr uint64_t F = 32 / sizeof(W) + 1;
    uint64_t span = 1, root_span = 1;
    for (int l = 0; l < w.coded; ++l) root_span *= kCodeFan;
    for (int l = w.levels - 1; l >= 0; --l) {
        if (l >= w.levels - w.coded) {
            k_walk_codes<K><<<fill_grid(count[l] * (kCodeFan - 1)), 256, 0, s>>>(
                lv, count[l], span, root_span, w.n, E, G, w.p0, reinterpret_cast<uint16_t *>(nodes + w.off[l]));
            span *= kCodeFan;
        } else {
            k_walk_nodes<K><<<fill_grid(count[l] * (F - 1)), 256, 0, s>>>(lv, count[l], span, E, G, w.p0,
                                                                         reinterpret_cast<W *>(nodes + w.off[l]));
            span *= F;
        }
    }
    return cudaGetLastError();
}

// Whether codes of `coded` levels would tie for more than one entry in 256.
// Every query of a tied run goes on from the run's first entry: 2^20 queries
// over 2^23 uniform keys, with one key in 1000 / 200 / 100 / 50 of them in
// dense runs of 40 (a tenth, half, one and two percent of the entries tie):
// 30.1 / 31.7 / 33.3 / 36.0 us through codes, 31.9 through full words at any
// share (27.9 and 31.9 without runs).
// *skip: 32-byte keys whose words tie in runs so long that walking on from
// the first of one costs more than the descent, on average 16 probes (2^20
// keys in runs of 30 / 200 / 5000, 2^20 lookups: 70 / 97 / 145 us, by the
// partition and descent 114 / 131 / 130; 1000 lookups: 6.9 / 8.6 / 11.4 us
// against 9.0 / 9.4 / 9.8).
template <typename K>
static cudaError_t codes_tie(const LeafView &lv, int coded, uint64_t n, uint64_t E, uint32_t G, int p0, bool *tie,
                             bool *skip, unsigned char *d_room, cudaStream_t s)
{
    uint64_t root_span = 1;
    for (int l = 0; l < coded; ++l) root_span *= kCodeFan;
    unsigned long long *d = reinterpret_cast<unsigned long long *>(d_room), h[2] = {0, 0};
    cudaError_t e = d ? cudaSuccess : cudaMalloc(&d, sizeof(h));
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(d, 0, sizeof(h), s);
    if (e == cudaSuccess) {
        if (coded) k_walk_ties<K><<<fill_grid(E), 256, 0, s>>>(lv, root_span, n, E, G, p0, d);
        if constexpr (sizeof(K) > 8) k_walk_runs<<<fill_grid(n), 256, 0, s>>>(lv, n, p0, d + 1);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(h, d, sizeof(h), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (!d_room) cudaFree(d);
    *tie = h[0] > E / 256;
    *skip = h[1] > 16 * n;
    return e;
}

template <typename K, typename V>
static cudaError_t build_entries(const LeafView &lv, uint64_t n, uint64_t E, uint32_t G, unsigned char *entries,
                                 cudaStream_t s)
{
    k_walk_entries<K, V><<<fill_grid(E * G), 256, 0, s>>>(lv, n, E * G, entries);
    return cudaGetLastError();
}

// The word of the key of rank i in the caller's array.
static uint64_t host_word(const void *h_keys, uint64_t i, int kb, int p0)
{
    if (kb == 8) return static_cast<const uint64_t *>(h_keys)[i];
    if (kb == 4) return static_cast<const uint32_t *>(h_keys)[i];
    const unsigned char *b = static_cast<const unsigned char *>(h_keys) + i * 32 + p0;
    uint64_t v = 0;
    for (int j = 0; j < 8; ++j) v = v << 8 | b[j];
    return v;
}

// The top: separators (the last one the largest word), bins, octaves.
template <typename W>
static std::vector<unsigned char> build_top(WalkDev &w, const std::vector<uint64_t> &sep)
{
    uint32_t held[64] = {};
    std::vector<uint32_t> oct(sep.size());
    std::vector<uint64_t> x(sep.size());
    for (size_t i = 0; i + 1 < sep.size(); ++i) {
        oct[i] = walk_octave<W>(w, static_cast<W>(sep[i]), x[i]);
        ++held[oct[i]];
    }
    WalkOctave table[64];
    uint32_t bins = 0;
    for (int o = 0; o < 64; ++o) {
        int bits = 0;
        while (bits < o && (2u << bits) <= held[o]) ++bits;
        table[o] = WalkOctave{bins, static_cast<uint32_t>(o - bits)};
        bins += 1u << bits;
    }
    w.bin_off = static_cast<uint32_t>((sep.size() * sizeof(W) + 15) / 16 * 16);
    w.oct_off = static_cast<uint32_t>((w.bin_off + (bins + 1) * 2 + 15) / 16 * 16);
    w.top_bytes = w.oct_off + static_cast<uint32_t>(sizeof(table));
    std::vector<unsigned char> top(w.top_bytes, 0);
    W *s = reinterpret_cast<W *>(top.data());
    uint16_t *first = reinterpret_cast<uint16_t *>(top.data() + w.bin_off);
    size_t at = 0;
    for (size_t i = 0; i < sep.size(); ++i) {
        s[i] = static_cast<W>(sep[i]);
        if (i + 1 == sep.size()) break;
        const uint32_t bin = table[oct[i]].base + static_cast<uint32_t>(x[i] >> table[oct[i]].shift);
        while (at <= bin) first[at++] = static_cast<uint16_t>(i);
    }
    while (at <= bins) first[at++] = static_cast<uint16_t>(sep.size() - 1);
    memcpy(top.data() + w.oct_off, table, sizeof(table));
    return top;
}

// Up to 8 MB of entries share the image's allocation: one cudaMalloc and one
// cudaFree less (247,326 uint64 keys: bt_build 0.95 -> 0.78 ms, 0.74 without
// an index, bt_free 95 -> 67 us; 50,000 32-byte keys, whose check for ties
// then needs no allocation either: 0.79 -> 0.63 and 0.55 ms).  The most the
// index can take: the largest top, full-word nodes (a fifth of the entries,
// and again), the entries.
uint64_t walk_room(uint64_t n, int key_bytes, int val_bytes)
{
    const uint64_t G = walk_group(key_bytes, val_bytes), E = (n + G - 1) / G;
    const uint64_t entries = E * walk_entry_bytes(key_bytes);
    if (n == 0 || entries > (8ull << 20)) return 0;
    const uint64_t segs = E < walk_max_segs(key_bytes) ? E : walk_max_segs(key_bytes);
    const uint64_t top = segs * ((key_bytes == 4 ? 4u : 8u) + 2u) + 64 * 2 + 64 * 8 + 64;
    const uint64_t nodes = E > kWalkSegs ? (E / 4 + kWalkLevels) * 32 : 0;
    return top + nodes + entries + 3 * 256;
}

cudaError_t walk_build(bt_tree *t, const void *h_keys, unsigned char *d_room, uint64_t room, cudaStream_t s)
{
    const DevTree &d = t->dev;
    const uint64_t n = t->info.n;
    if (n == 0) return cudaSuccess;
    const int kb = d.key_bytes, vb = d.val_bytes;
    const uint32_t G = walk_group(kb, vb);
    const uint64_t F = walk_fan(kb), E = (n + G - 1) / G;
    if (E >= (1ull << 32)) return cudaSuccess;  // node and entry numbers are 32-bit
    // what an earlier call left in the runtime (and has reported) is not these
    // launches' error: before the index a build launched nothing and never asked
    cudaGetLastError();
    WalkDev w;
    memset(&w, 0, sizeof(w));
    w.n = n;
    w.p0 = d.split_p0;
    memcpy(w.kmin32, d.kmin32, sizeof(w.kmin32));
    memcpy(w.kmax32, d.kmax32, sizeof(w.kmax32));
    w.wmin = host_word(h_keys, 0, kb, w.p0);
    w.wmax = host_word(h_keys, n - 1, kb, w.p0);
    const int leaf = d.height - 1;
    const LeafView lv{d.keys[leaf], d.vals, d.cbase[leaf], d.crem[leaf], static_cast<uint32_t>(d.m)};
    cudaError_t e = cudaSuccess;
    // coded levels: one where it leaves at most kWalkSegs segments, else two;
    // none where codes tie; then levels of full words down to walk_max_segs
    // (without codes half of it)
    uint64_t segs = E, span = 1, count[kWalkLevels];
    if (E > kWalkSegs) w.coded = (E + kCodeFan - 1) / kCodeFan <= kWalkSegs ? 1 : 2;
    if (w.coded || kb == 32) {
        bool tie = false, skip = false;
        e = kb == 32 ? codes_tie<Key32>(lv, w.coded, n, E, G, w.p0, &tie, &skip, d_room, s)
            : kb == 8 ? codes_tie<uint64_t>(lv, w.coded, n, E, G, w.p0, &tie, &skip, d_room, s)
                      : codes_tie<uint32_t>(lv, w.coded, n, E, G, w.p0, &tie, &skip, d_room, s);
        if (e == cudaErrorMemoryAllocation) {
            cudaGetLastError();  // no room for an index then
            return cudaSuccess;
        }
        if (e != cudaSuccess) return e;
        if (skip) return cudaSuccess;
        if (tie) w.coded = 0;
    }
    for (int l = 0; l < w.coded; ++l) {
        segs = (segs + kCodeFan - 1) / kCodeFan;
        span *= kCodeFan;
    }
    w.levels = w.coded;
    while (segs > (w.coded ? walk_max_segs(kb) : walk_max_segs(kb) / 2)) {
        segs = (segs + F - 1) / F;
        span *= F;
        ++w.levels;
    }
    uint64_t c = E;
    for (int l = w.levels - 1; l >= 0; --l) {
        const uint64_t fan = l >= w.levels - w.coded ? kCodeFan : F;
        c = (c + fan - 1) / fan;
        count[l] = c;
    }
    w.segs = static_cast<uint32_t>(segs);
    w.span = static_cast<uint32_t>(span);
    std::vector<uint64_t> sep(segs);
    for (uint64_t i = 0; i < segs; ++i) {
        const uint64_t end = (i + 1) * span * G;
        sep[i] = host_word(h_keys, (end < n ? end : n) - 1, kb, w.p0);
    }
    std::vector<unsigned char> top;
    if (segs > 1) top = kb == 4 ? build_top<uint32_t>(w, sep) : build_top<uint64_t>(w, sep);
    uint64_t bytes = (static_cast<uint64_t>(w.top_bytes) + 255) & ~255ull;
    const uint64_t node_off = bytes;
    for (int l = 0; l < w.levels; ++l) {
        w.off[l] = bytes - node_off;
        bytes += count[l] * 32;
    }
    bytes = (bytes + 255) & ~255ull;
    const uint64_t ent_off = bytes;
    bytes += E * walk_entry_bytes(kb);
    // At most a quarter of what is free.  Only a large index asks how much
    // that is: the answer takes 18 us (bt_build of 1000 uint64 keys: 182 us
    // with it, 163 without).
    if (bytes > kWalkAskBytes) {
        size_t free_b = 0, total_b = 0;
        e = cudaMemGetInfo(&free_b, &total_b);
        if (e != cudaSuccess) return e;
        if (bytes > free_b / 4) return cudaSuccess;
    }
    t->walk_own = bytes > room;
    if (t->walk_own)
        e = cudaMalloc(&t->d_walk, bytes);
    else
        t->d_walk = d_room;
    if (t->walk_own && e == cudaSuccess) t->walk_bytes += bytes;
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
    unsigned char *nodes = base + node_off, *ent = base + ent_off;
    if (w.top_bytes) e = cudaMemcpyAsync(base, top.data(), top.size(), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return e;
    if (kb == 32) {
        e = build_levels<Key32>(w, lv, E, G, count, nodes, s);
        if (e == cudaSuccess)
            e = vb == 8 ? build_entries<Key32, uint64_t>(lv, n, E, G, ent, s)
                        : build_entries<Key32, uint32_t>(lv, n, E, G, ent, s);
    } else if (kb == 8) {
        e = build_levels<uint64_t>(w, lv, E, G, count, nodes, s);
        if (e == cudaSuccess)
            e = vb == 8 ? build_entries<uint64_t, uint64_t>(lv, n, E, G, ent, s)
                        : build_entries<uint64_t, uint32_t>(lv, n, E, G, ent, s);
    } else {
        e = build_levels<uint32_t>(w, lv, E, G, count, nodes, s);
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
    uint32_t span_inv;             // floor((2^32 - 1) / entries per segment)
};

// The model's parameters in shared memory behind the top, each array rounded
// up to whole 16-byte pieces (the model's allocation pads them).  The error
// bounds last: a lane reads one of 256, and L1 is full of entries (2^20
// lookups over 2^24 lognormal keys by 256 segments 38.7 -> 38.2 us, 1024 by
// the MLP 7.48 -> 7.41).
__host__ __device__ inline uint32_t walk_model_bytes(const ModelDev &m)
{
    if (m.kind == kModelPL)
        return m.segments <= kModelSmemSegments
                   ? (m.segments * 8u + 15u) / 16u * 16u + 3u * ((m.segments * 4u + 15u) / 16u * 16u) + kErrRanges * 4u
                   : 0u;
    if (m.kind == kModelMLP) return kMlpStage1 * 12u + (kMlpParams * 4u + 15u) / 16u * 16u + kErrRanges * 4u;
    return 0u;
}

// Where the parameters lie behind the top, and (one thread, `bar` given) the
// bulk copies that bring them there.
template <int MODEL>
__device__ __forceinline__ ModelView walk_model(const ModelDev &md, unsigned char *msm, uint64_t *bar = nullptr)
{
    auto put = [&](const void *src, uint32_t bytes) {
        const uint32_t padded = (bytes + 15u) / 16u * 16u;
        unsigned char *dst = msm;
        if (bar) bulk_g2s(dst, src, padded, bar);
        msm += padded;
        return dst;
    };
    ModelView v{};
    const uint32_t S = MODEL == kModelPL ? md.segments : kMlpStage1;
    v.b = reinterpret_cast<const uint64_t *>(put(md.b, S * 8u));
    v.inv_w = reinterpret_cast<const float *>(put(md.inv_w, S * 4u));
    if constexpr (MODEL == kModelPL) {
        v.slope = reinterpret_cast<const float *>(put(md.slope, S * 4u));
        v.icpt = reinterpret_cast<const float *>(put(md.icpt, S * 4u));
    } else {
        v.mlp = reinterpret_cast<const float *>(put(md.mlp, kMlpParams * 4u));
    }
    v.errs = reinterpret_cast<const uint32_t *>(put(md.errs, kErrRanges * 4u));
    return v;
}

// One query per lane, one block per SM; every block takes a contiguous run
// of 32-query chunks of the batch, its warps chunk by chunk in turn, the
// next chunk's queries loaded while the present one walks.  The top is
// copied once per block by one bulk copy, before the wait for the previous
// kernel of the stream.
//
// What bounds it: divergent reads.  A warp's read of one sector per lane
// occupies an SM for 34 cycles when it comes from the L2 and 20 when it hits
// L1, whatever part of the sector is used (about 4.7 us per 2^20 queries); a
// probe of the top in shared memory for 6; and 2^20 reads of random entries
// take 18 us from memory by themselves.  Over 2^24 uint64 keys a query is
// about six probes, three nodes and an entry: 32.7 us for 2^20 queries with
// three trees in turn (30.2 for one).  Before the walk, the partition and
// the level-wise descent: 92.4 us; with four nodes of full words under a top
// searched by bisection (13 probes) and entries of 64 bytes: 41.6; with the
// top's tables 41.2; with coded nodes 33.4.  For 32-byte keys (2^20 keys) 113,
// 38.6, 36.9, now 32.3 us; over 10^6 uint64 keys 61, 25.1, -, now 17.5.
// 1024 threads on one SM: two blocks (of 1024, 768 or 512) hold two copies
// of the top and gain nothing from the additional warps (2^20 queries over
// 2^24 keys, full-word nodes: 42.3, 43.5 and 51.4 us against 40.4).
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
        mbar_arrive_expect_tx(&bar, w.top_bytes + (MODEL == kModelNone ? 0u : walk_model_bytes(m.md)));
        if (w.top_bytes) bulk_g2s(smem, w.top, w.top_bytes, &bar);
        if constexpr (MODEL != kModelNone)
            if (walk_model_bytes(m.md)) walk_model<MODEL>(m.md, smem + w.top_bytes, &bar);
    }
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
    __syncthreads();  // the barrier is initialised
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
        uint32_t seg;
        if constexpr (MODEL == kModelNone) {
            seg = walk_segment<W>(w, smem, word);
        } else {
            constexpr uint32_t G = walk_group(sizeof(K), sizeof(V));
            const W *sep = reinterpret_cast<const W *>(smem);
            uint32_t lo, hi;
            // (two calls, so that each reads the parameters by their own address space)
            if (MODEL == kModelMLP || walk_model_bytes(m.md))
                model_window<MODEL>(m.md, walk_model<MODEL>(m.md, smem + w.top_bytes), static_cast<uint64_t>(key), lo,
                                    hi);
            else
                model_window<MODEL>(m.md, ModelView{m.md.b, m.md.inv_w, m.md.slope, m.md.icpt, m.md.mlp, nullptr},
                                    static_cast<uint64_t>(key), lo, hi);
            // first key of leaf lo, last key of leaf hi, as entries, as segments
            const uint64_t r0 = lo * m.leaf_base + (lo < m.leaf_rem ? lo : m.leaf_rem);
            const uint64_t r1 = (hi + 1ull) * m.leaf_base + (hi + 1ull < m.leaf_rem ? hi + 1ull : m.leaf_rem) - 1;
            const uint32_t s0 = div_by(static_cast<uint32_t>(r0 / G), w.span, m.span_inv);
            const uint32_t s1 = div_by(static_cast<uint32_t>(r1 / G), w.span, m.span_inv);
            // proven by the separators on both sides, else the whole top searched
            if ((s0 == 0 || sep[s0 - 1] < word) && (s1 + 1 >= w.segs || !(sep[s1] < word)))
                seg = walk_segment_in<W>(sep, s0, s1, word);
            else
                seg = walk_segment<W>(w, smem, word);
        }
        V val;
        bool hit = walk_lookup<K, V>(w, walk_entry<W>(w, smem, seg, word), key, val);
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
    constexpr int kMaxTop = walk_max_top(sizeof(K));
    constexpr int kMaxModel =
        MODEL == kModelNone ? 0 : static_cast<int>(kModelSmemSegments) * 20 + 64 + static_cast<int>(kErrRanges) * 4;
    int sms = 0;
    cudaError_t e = dev_sm_count(&sms);
    if (e == cudaSuccess) e = ensure_dyn_smem(reinterpret_cast<const void *>(kern), kMaxTop + kMaxModel, kWalkCarveout);
    if (e != cudaSuccess) return e;
    WalkModel m;
    memset(&m, 0, sizeof(m));
    if (MODEL != kModelNone) {
        const int leaf = t->dev.height - 1;
        m.md = *md;
        m.leaf_base = t->dev.cbase[leaf];
        m.leaf_rem = t->dev.crem[leaf];
        m.span_inv = ~0u / w.span;
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
    cfg.dynamicSmemBytes = w.top_bytes + (MODEL == kModelNone ? 0u : walk_model_bytes(m.md));
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
static cudaError_t walk_any(const bt_tree *t, const ModelDev *md, const void *q, uint64_t nq, void *out_v,
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
        return v8 ? walk_any<Key32, uint64_t>(t, md, q, nq, out_v, out_f, s)
                  : walk_any<Key32, uint32_t>(t, md, q, nq, out_v, out_f, s);
    if (kb == 8)
        return v8 ? walk_any<uint64_t, uint64_t>(t, md, q, nq, out_v, out_f, s)
                  : walk_any<uint64_t, uint32_t>(t, md, q, nq, out_v, out_f, s);
    return v8 ? walk_any<uint32_t, uint64_t>(t, md, q, nq, out_v, out_f, s)
              : walk_any<uint32_t, uint32_t>(t, md, q, nq, out_v, out_f, s);
}

cudaError_t take_wait_counters_walk(unsigned *timeouts, unsigned *pending)
{
    return take_wait_counters(timeouts, pending);
}

}  // namespace btgb
