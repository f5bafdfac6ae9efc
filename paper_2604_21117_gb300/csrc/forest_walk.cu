// Many batches over several trees in one launch, every tree searched through
// its walk index (walk.cuh): the kernel of forests whose trees all have one
// and no learned model; forest.cu holds the others.
//
// A batch's queries are cut into chunks of 32, one query per lane, and the
// chunks of the whole list are dealt out to the blocks in contiguous runs of
// equal cost, each block's to its warps likewise.  A chunk costs what its
// tree's walk does (ForestWalk::cost): over trees of 10^3 to 2 * 10^7 keys
// runs of equal length left warps idle for a quarter of the launch.  Where a
// run starts is found without a plan kernel: every block adds up the list
// itself, a row of 32 work-list entries per warp and step, and scans the row
// totals in shared memory (a list of 10,000 entries is 160 KB from the L2
// for every block, about 2 us, against about 20 us for a one-block plan
// kernel and its launch).  A warp then holds the row its run is in, one entry
// per lane, and moves on to the next row as the run does.
#include <cuda_runtime.h>

#include <cstring>

#include "forest.h"
#include "walk.cuh"

namespace btgb {

__device__ unsigned long long g_bt_bad_walk_batches;

constexpr uint32_t kWalkForestThreads = 1024;

// A position in the list is a cost: entry after entry, each as many chunks as
// it has times the cost of one.
struct Entry {
    bt_batch_desc bd;
    uint32_t chunks, cost;  // cost of one chunk
};

// An entry's chunks; a rejected one keeps one chunk so that it is seen and
// counted.  unit: every chunk costs 1 (the host's chunk offsets).
__device__ __forceinline__ Entry list_entry(const bt_batch_desc *batches, uint32_t i, uint32_t nb,
                                            const ForestWalk *tab, uint32_t ntrees, uint64_t nq, bool unit)
{
    Entry e{{0, 0, 0}, 0, 1};
    if (i < nb) {
        e.bd = batches[i];
        const bool ok = forest_desc_ok(e.bd, ntrees, nq);
        e.chunks = ok ? (e.bd.count + 31u) / 32u : 1u;
        if (ok && !unit) e.cost = tab[e.bd.tree].cost;
    }
    return e;
}

__device__ __forceinline__ uint64_t warp_incl_scan(uint64_t x, uint32_t lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t y = __shfl_up_sync(0xffffffffu, static_cast<unsigned long long>(x), o);
        if (lane >= static_cast<uint32_t>(o)) x += y;
    }
    return x;
}

// Shared memory: the tops that have a place (top_total bytes), the table, then
// (lists without chunk offsets) the positions of the list's rows.
template <typename K, typename V>
__global__ void __launch_bounds__(kWalkForestThreads)
    k_forest_walk(const ForestWalk *__restrict__ gtab, uint32_t ntrees, uint32_t top_total,
                  const bt_batch_desc *__restrict__ batches, uint32_t nb, const uint32_t *__restrict__ chunk_start,
                  const K *__restrict__ q, uint64_t nq, V *__restrict__ out_v, uint8_t *__restrict__ out_f,
                  ForestDone done, uint32_t wait_polls)
{
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint64_t s_scan[32];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    ForestWalk *tab = reinterpret_cast<ForestWalk *>(smem + top_total);
    uint64_t *rows = reinterpret_cast<uint64_t *>(tab + ntrees);
    const uint32_t nrows = (nb + 31) / 32;
    if (threadIdx.x == 0) {
        mbar_init(&bar);
        mbar_arrive_expect_tx(&bar, top_total);
        for (uint32_t i = 0; i < ntrees && top_total; ++i)
            if (gtab[i].top_off != kNoTop && gtab[i].w.top_bytes)
                bulk_g2s(smem + gtab[i].top_off, gtab[i].w.top, gtab[i].w.top_bytes, &bar);
    }
    for (uint32_t i = threadIdx.x; i < ntrees * sizeof(ForestWalk) / 8; i += blockDim.x)
        reinterpret_cast<uint64_t *>(tab)[i] = reinterpret_cast<const uint64_t *>(gtab)[i];
    __syncthreads();
    // the work list, the queries and the outputs belong to the previous
    // kernel of the stream until it is done
    pdl_wait();
    const bool unit = chunk_start != nullptr;
    if (!unit) {
        // row totals (several rows' entries in flight per warp), then their
        // exclusive scan in place (rows[nrows] = the whole list)
        constexpr int U = 10;
        for (uint32_t r0 = warp; r0 < nrows; r0 += nw * U) {
            Entry e[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                e[u] = list_entry(batches, (r0 + u * nw) * 32 + lane, nb, tab, ntrees, nq, false);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                // at most 2^27 chunks of a cost below 2^12: two sums below 2^32
                const uint64_t x = static_cast<uint64_t>(e[u].chunks) * e[u].cost;
                const uint32_t lo = __reduce_add_sync(0xffffffffu, static_cast<uint32_t>(x) & 0xFFFFFu);
                const uint32_t hi = __reduce_add_sync(0xffffffffu, static_cast<uint32_t>(x >> 20));
                if (lane == 0 && r0 + u * nw < nrows) rows[r0 + u * nw] = lo + (static_cast<uint64_t>(hi) << 20);
            }
        }
        __syncthreads();
        const uint32_t per = (nrows + blockDim.x - 1) / blockDim.x, r0 = threadIdx.x * per;
        uint64_t sum = 0;
        for (uint32_t k = 0; k < per; ++k) sum += r0 + k < nrows ? rows[r0 + k] : 0u;
        const uint64_t x = warp_incl_scan(sum, lane);
        if (lane == 31) s_scan[warp] = x;
        __syncthreads();
        uint64_t run = x - sum;
        for (uint32_t k = 0; k < warp; ++k) run += s_scan[k];
        for (uint32_t k = 0; k < per; ++k)
            if (r0 + k < nrows) {
                const uint64_t c = rows[r0 + k];
                rows[r0 + k] = run;
                run += c;
            }
        if (threadIdx.x == blockDim.x - 1) rows[nrows] = run;
    }
    __syncthreads();
    // A warp whose wait gives up is counted and reads every top through L1, as
    // those without a place: the completion signal below says that the whole
    // list has been searched, and whoever polls it reads no other word.
    bool tops_here = true;
    if (top_total && !mbar_wait_warp(&bar, 0, wait_polls)) {
        mbar_give_up(&bar, 0, static_cast<int>(lane));
        tops_here = false;
    }
    auto row_pos = [&](uint32_t r) -> uint64_t { return unit ? chunk_start[r * 32] : rows[r]; };
    const uint64_t total = unit ? chunk_start[nb] : rows[nrows];
    // the chunks that start in [p, p1) are this warp's: an equal share of the
    // block's equal share of the list
    const uint64_t b0 = total / gridDim.x * blockIdx.x + total % gridDim.x * blockIdx.x / gridDim.x;
    const uint64_t b1 = total / gridDim.x * (blockIdx.x + 1) + total % gridDim.x * (blockIdx.x + 1) / gridDim.x;
    const uint64_t p = b0 + (b1 - b0) * warp / nw, p1 = b0 + (b1 - b0) * (warp + 1) / nw;
    if (p < p1) {
        uint32_t lo = 0, hi = nrows - 1;  // the last row that starts at or before p
        while (lo < hi) {
            const uint32_t mid = (lo + hi + 1) / 2;
            if (row_pos(mid) <= p)
                lo = mid;
            else
                hi = mid - 1;
        }
        // The row, an entry per lane, and in `todo` the entries of it that are
        // left; the entry at hand, the same in every lane.
        uint32_t row = lo;
        Entry mine;
        uint64_t first;  // position of this lane's entry
        auto load_row = [&](uint64_t start) {
            mine = list_entry(batches, row * 32 + lane, nb, tab, ntrees, nq, unit);
            const uint64_t x = static_cast<uint64_t>(mine.chunks) * mine.cost;
            const uint64_t end = start + warp_incl_scan(x, lane);
            first = end - x;
            return end;
        };
        uint64_t end = load_row(row_pos(row));
        unsigned todo = __ballot_sync(0xffffffffu, mine.chunks && end > p);
        Entry e{{0, 0, 0}, 0, 1};
        uint32_t k = 0;  // the entry's next chunk
        uint64_t at = 0; // its position
        bool good = false;
        auto advance = [&]() -> bool {
            while (todo == 0) {
                if (++row >= nrows) return false;
                end = load_row(__shfl_sync(0xffffffffu, static_cast<unsigned long long>(end), 31));
                todo = __ballot_sync(0xffffffffu, mine.chunks != 0);
            }
            const int src = __ffs(todo) - 1;
            todo &= todo - 1;
            e.bd.tree = __shfl_sync(0xffffffffu, mine.bd.tree, src);
            e.bd.count = __shfl_sync(0xffffffffu, mine.bd.count, src);
            e.bd.offset = __shfl_sync(0xffffffffu, static_cast<unsigned long long>(mine.bd.offset), src);
            e.chunks = __shfl_sync(0xffffffffu, mine.chunks, src);
            e.cost = __shfl_sync(0xffffffffu, mine.cost, src);
            at = __shfl_sync(0xffffffffu, static_cast<unsigned long long>(first), src);
            k = 0;
            good = forest_desc_ok(e.bd, ntrees, nq);
            if (at < p) {  // the run starts inside this entry
                k = static_cast<uint32_t>((p - at + e.cost - 1) / e.cost);
                at += static_cast<uint64_t>(k) * e.cost;
            }
            return true;
        };
        // A chunk's queries, loaded while the chunk before it walks; lanes
        // past the batch's end follow its first query and write nothing.
        struct Chunk {
            uint32_t tree;
            bool live, valid;
            uint64_t pos;
            K key;
        };
        // the next chunk of the run, or false past its end
        auto fetch = [&](Chunk &n) -> bool {
            while (k >= e.chunks)
                if (!advance()) return false;
            if (at >= p1) return false;
            n.live = good;
            n.tree = e.bd.tree;
            const uint32_t j0 = k * 32u, j = j0 + lane;
            ++k;
            at += e.cost;
            if (!good) {
                if (lane == 0) atomicAdd(&g_bt_bad_walk_batches, 1ull);
                return true;
            }
            n.valid = j < e.bd.count;
            n.pos = e.bd.offset + (n.valid ? j : j0);
            n.key = q[n.pos];
            return true;
        };
        Chunk next{0, false, false, 0, KeyOps<K>::ones()};
        bool more = fetch(next);
        while (more) {
            const Chunk now = next;
            more = fetch(next);
            if (!now.live) continue;
            const ForestWalk &F = tab[now.tree];
            V val = static_cast<V>(~static_cast<V>(0));
            bool hit = false;
            if (F.w.n) {
                // (two calls, so that each reads the top by its own address space)
                uint32_t entry;
                if (tops_here && F.top_off != kNoTop) {
                    const unsigned char *top = smem + F.top_off;
                    entry = walk_entry<K>(F.w, top, walk_segment<K>(F.w, top, now.key), now.key);
                } else {
                    entry = walk_entry<K>(F.w, F.w.top, walk_segment<K>(F.w, F.w.top, now.key), now.key);
                }
                hit = walk_lookup<K, V>(F.w, entry, now.key, val);
            }
            if (now.valid) {
                out_v[now.pos] = val;
                out_f[now.pos] = hit ? 1 : 0;
            }
        }
    }
    if (done.counter) {
        // every thread's results visible system-wide, then one arrival per block;
        // the last block to arrive resets the counter and raises the flag
        __threadfence_system();
        __syncthreads();
        if (threadIdx.x == 0) {
            const unsigned prev = atomicAdd(done.counter, 1u);
            if (prev == gridDim.x - 1) {
                *done.counter = 0u;
                __threadfence_system();
                asm volatile("st.release.sys.u64 [%0], %1;" ::"l"(done.flag), "l"(done.seq) : "memory");
            }
        }
    }
}

template <typename K, typename V>
static cudaError_t walk_forest_launch(const ForestWalk *tab, uint32_t ntrees, uint32_t top_total,
                                      const bt_batch_desc *b, uint32_t nb, const uint32_t *cs, uint32_t host_chunks,
                                      const void *q, uint64_t nq, void *ov, uint8_t *of, cudaStream_t s,
                                      ForestDone done)
{
    auto kern = k_forest_walk<K, V>;
    int sms = 0;
    cudaError_t e = dev_sm_count(&sms);
    if (e == cudaSuccess) e = ensure_dyn_smem(reinterpret_cast<const void *>(kern), 220 * 1024, kWalkCarveout);
    if (e != cudaSuccess) return e;
    const uint32_t smem = top_total + ntrees * static_cast<uint32_t>(sizeof(ForestWalk)) +
                          (cs ? 0u : ((nb + 31u) / 32u + 1u) * 8u);
    // as many warps per SM as the list has chunks for (a device list: at most
    // as many as batches that do not overlap can have), up to 32
    const uint64_t n = static_cast<uint64_t>(sms > 0 ? sms : 1);
    const uint64_t chunks = cs ? host_chunks : nb + nq / 32;
    uint64_t warps = (chunks + n - 1) / n;
    warps = warps < 1 ? 1 : warps > kWalkForestThreads / 32 ? kWalkForestThreads / 32 : warps;
    uint64_t grid = (chunks + warps - 1) / warps;
    grid = grid < 1 ? 1 : grid > n ? n : grid;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(static_cast<unsigned>(grid));
    cfg.blockDim = dim3(static_cast<unsigned>(warps * 32));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr;
    memset(&attr, 0, sizeof(attr));
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, tab, ntrees, top_total, b, nb, cs, static_cast<const K *>(q), nq,
                              static_cast<V *>(ov), of, done, first_wait_polls());
}

cudaError_t forest_walk_run(const ForestWalk *tab, uint32_t ntrees, uint32_t top_total, int kb, int vb,
                            const bt_batch_desc *b, uint32_t nb, const uint32_t *cs, uint32_t host_chunks,
                            const void *q, uint64_t nq, void *ov, uint8_t *of, cudaStream_t s, ForestDone done)
{
    auto launch = kb == 8 ? (vb == 8 ? walk_forest_launch<uint64_t, uint64_t> : walk_forest_launch<uint64_t, uint32_t>)
                          : (vb == 8 ? walk_forest_launch<uint32_t, uint64_t> : walk_forest_launch<uint32_t, uint32_t>);
    return launch(tab, ntrees, top_total, b, nb, cs, host_chunks, q, nq, ov, of, s, done);
}

cudaError_t take_wait_counters_forest(unsigned *timeouts, unsigned *pending)
{
    return take_wait_counters(timeouts, pending);
}

cudaError_t forest_walk_take_bad(unsigned long long *bad)
{
    unsigned long long v = 0;
    cudaError_t e = cudaMemcpyFromSymbol(&v, g_bt_bad_walk_batches, sizeof(v));
    if (e == cudaSuccess && v) {
        const unsigned long long zero = 0;
        e = cudaMemcpyToSymbol(g_bt_bad_walk_batches, &zero, sizeof(zero));
    }
    *bad += v;
    return e;
}

}  // namespace btgb
