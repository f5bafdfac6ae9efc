// Search of a batch as given (no partition) through a tree's walk index.
//
// The level-wise descent reads a whole node block per level: 256 bytes at
// fanout 32 and 64-bit keys.  Over a partitioned batch a warp shares those
// blocks; over a batch as given every lane needs its own, and what bounds
// the search is the bytes (in 32-byte sectors) that cross from the L2 to the
// SMs.  The walk index holds the same keys and values a second time in the
// form that costs the fewest sectors per query:
//
//   top      the largest keys of up to 2^13 segments of equal length (2^14
//            for 32-bit keys), as an implicit binary tree in breadth-first
//            order (children of k at 2k and 2k + 1, root at 1), all-ones
//            where there is no segment; copied to shared memory by every
//            block, where a probe costs a third of a sector from L1;
//   nodes    one 32-byte sector each: SEP = 32 / word separators (4 of 64
//            bits, 8 of 32), FAN = SEP + 1 children; node i of a level has the
//            children FAN i .. FAN i + SEP of the next level, separator j the
//            largest key under child j, all-ones where child j + 1 does not
//            exist.  Level 0 has one node per segment; levels lie one after
//            the other;
//   entries  64 bytes each, the children of the last level.  Integer keys: G
//            consecutive keys (bytes 0..31, unused slots all-ones) and their
//            values (bytes 32..63), G = 32 / max(key, value bytes); the keys
//            are packed densely, entry e holding ranks G e .. G e + G - 1.
//            Memory is read 64 bytes at a time, so a query costs one such
//            access for its key and its value together.
//            32-byte keys: one key (four words, as Key32) and its value.
//
// 32-byte keys are walked by one 64-bit word, the 8 bytes after the bytes all
// keys share: a query between the smallest and the largest key shares those
// bytes too, so the word orders it among the keys up to ties, and the entry
// found is the first whose word is not below the query's.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "descent.cuh"

namespace btgb {

// Words the top and the nodes hold: the keys, or for 32-byte keys one 64-bit
// word of each.
template <typename K>
struct WalkWord {
    using type = K;
};
template <>
struct WalkWord<Key32> {
    using type = uint64_t;
};

constexpr uint32_t walk_fan(int key_bytes) { return key_bytes == 4 ? 9u : 5u; }
constexpr int walk_top_bits(int key_bytes) { return key_bytes == 4 ? 14 : 13; }

// Keys per entry.
__host__ __device__ constexpr uint32_t walk_group(int key_bytes, int val_bytes)
{
    return key_bytes > 8 ? 1u : 32u / static_cast<uint32_t>(key_bytes > val_bytes ? key_bytes : val_bytes);
}

// One 32-byte sector as words.
template <typename W>
struct Sector {
    W w[32 / sizeof(W)];
};

// One aligned sector in one load, through L1 for nodes and entries alike:
// keeping entries out of L1 gained 4-8% on uniform queries (2^20 over 2^24
// keys: 39.5 against 41.1 us) and lost a third on skewed ones, whose hot
// entries then all come from one L2 slice (Zipf(1.1) over 10^6 keys: 37.0
// against 25.6 us; 2^20 queries of a 1000-key tree: 34.6 against 11.7 us).
template <typename W>
__device__ __forceinline__ Sector<W> ld_sector(const void *p)
{
    uint64_t v[4];
    asm volatile("ld.global.nc.v4.u64 {%0, %1, %2, %3}, [%4];"
                 : "=l"(v[0]), "=l"(v[1]), "=l"(v[2]), "=l"(v[3])
                 : "l"(p));
    Sector<W> s;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if constexpr (sizeof(W) == 8) {
            s.w[i] = v[i];
        } else {
            s.w[2 * i] = static_cast<W>(v[i]);
            s.w[2 * i + 1] = static_cast<W>(v[i] >> 32);
        }
    }
    return s;
}

// Separators of a node below the query: the child to take.
template <typename W>
__device__ __forceinline__ uint32_t sector_rank(const Sector<W> &s, W q)
{
    uint32_t r = 0;
#pragma unroll
    for (int j = 0; j < static_cast<int>(32 / sizeof(W)); ++j) r += s.w[j] < q ? 1u : 0u;
    return r;
}

// The segment of q: the first whose largest key is not below q, or the last
// padded position.  top: the implicit binary tree of depth `bits`.
template <typename W>
__device__ __forceinline__ uint32_t walk_segment(const W *top, int bits, W q)
{
    uint32_t k = 1;
    for (int i = 0; i < bits; ++i) k = 2u * k + (top[k] < q ? 1u : 0u);
    return k - (1u << bits);
}

// Separator of sorted rank r of the top (all-ones from the last segment on).
template <typename W>
__device__ __forceinline__ W walk_top_at(const W *top, int bits, uint32_t r)
{
    const int t = __ffs(static_cast<int>(r + 1)) - 1;  // the node's height over the bottom
    return top[(1u << (bits - 1 - t)) + ((r + 1) >> (t + 1))];
}

// The same segment when [s0, s1] is believed to hold it: proven by the
// separators on both sides and searched inside, else the whole top searched.
template <typename W>
__device__ __forceinline__ uint32_t walk_segment_in(const W *top, int bits, uint32_t s0, uint32_t s1, W q)
{
    const uint32_t last = (1u << bits) - 1;  // position behind the separators
    if ((s0 > 0 && !(walk_top_at(top, bits, s0 - 1) < q)) || (s1 < last && walk_top_at(top, bits, s1) < q))
        return walk_segment(top, bits, q);
    while (s0 < s1) {
        const uint32_t mid = (s0 + s1) / 2;
        if (walk_top_at(top, bits, mid) < q)
            s0 = mid + 1;
        else
            s1 = mid;
    }
    return s0;
}

// The same from the top in global memory, through L1.
template <typename W>
__device__ __forceinline__ uint32_t walk_segment_l1(const unsigned char *top, int bits, W q)
{
    uint32_t k = 1;
    for (int i = 0; i < bits; ++i) k = 2u * k + (ld_key(reinterpret_cast<const W *>(top) + k) < q ? 1u : 0u);
    return k - (1u << bits);
}

// The entry of q from its segment: the first entry whose largest key (32-byte
// keys: word) is not below q, or the last one.
template <typename W>
__device__ __forceinline__ uint32_t walk_entry(const WalkDev &w, uint32_t node, W q)
{
    for (int l = 0; l < w.levels; ++l)
        node = node * (32u / sizeof(W) + 1u) +
               sector_rank<W>(ld_sector<W>(w.nodes + w.off[l] + static_cast<uint64_t>(node) * 32u), q);
    return node;
}

// Key and value of q in entry e.
template <typename K, typename V>
__device__ __forceinline__ bool walk_lookup(const WalkDev &w, uint32_t e, const K &q, V &val)
{
    constexpr uint32_t G = walk_group(sizeof(K), sizeof(V));
    const unsigned char *p = w.entries + static_cast<uint64_t>(e) * 64u;
    bool hit = false;
    val = static_cast<V>(~static_cast<V>(0));
    if constexpr (sizeof(K) <= 8) {
        const Sector<K> k = ld_sector<K>(p);
        const Sector<V> v = ld_sector<V>(p + 32);
        // the last entry's unused slots hold all-ones, which may be the query
        const uint64_t left = w.n - static_cast<uint64_t>(e) * G;
#pragma unroll
        for (uint32_t j = 0; j < G; ++j)
            if (k.w[j] == q && j < left) {
                hit = true;
                val = v.w[j];
            }
    } else {
        const Sector<uint64_t> k = ld_sector<uint64_t>(p);
        const Sector<V> v = ld_sector<V>(p + 32);
        const Key32 key{{k.w[0], k.w[1], k.w[2], k.w[3]}};
        hit = key == q;
        if (hit) val = v.w[0];
        if (!hit && key < q) {
            // keys that share the word: gallop right over the full keys to the
            // first that is not below q
            auto at = [&](uint64_t i) {
                const Sector<uint64_t> s = ld_sector<uint64_t>(w.entries + i * 64u);
                return Key32{{s.w[0], s.w[1], s.w[2], s.w[3]}};
            };
            uint64_t lo = static_cast<uint64_t>(e) + 1, step = 1;
            while (lo + step <= w.n && at(lo + step - 1) < q) {
                lo += step;
                step *= 2;
            }
            uint64_t hi = lo + step - 1 < w.n ? lo + step - 1 : w.n;
            while (lo < hi) {
                const uint64_t mid = (lo + hi) / 2;
                if (at(mid) < q)
                    lo = mid + 1;
                else
                    hi = mid;
            }
            if (lo < w.n && at(lo) == q) {
                hit = true;
                val = ld_sector<V>(w.entries + lo * 64u + 32).w[0];
            }
        }
    }
    return hit;
}

}  // namespace btgb
