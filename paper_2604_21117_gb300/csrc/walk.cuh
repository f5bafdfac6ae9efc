// Search of a batch as given (no partition) through a tree's walk index.
//
// The level-wise descent reads a whole node block per level: 256 bytes at
// fanout 32 and 64-bit keys.  Over a partitioned batch a warp shares those
// blocks; over a batch as given every lane needs its own, and what bounds
// the search is the bytes (in 32-byte sectors) that cross from the L2 to the
// SMs.  The walk index holds the same keys and values a second time in the
// form that costs the fewest sectors per query:
//
//   top      the largest keys of up to 2^14 segments of equal length,
//            ascending, and two tables that narrow the search
//            among them to a few: the octave of x = key - smallest key (its
//            leading one) gives a range of bins, as many as the octave has
//            separators (rounded down to a power of two), the bits after the
//            leading one a bin of them, and the bin the separators in it.  For
//            uniform keys the upper octaves' bins hold one or two separators
//            each, for a lognormal mixture every octave's do; keys crowded in
//            a small part of an octave cost the binary search they would have
//            cost.  Copied to shared memory by every block, where a probe
//            costs a third of a sector from L1;
//   nodes    one 32-byte sector each, levels one after the other, level 0
//            with one node per segment.  The bottom one or two levels are
//            coded: 16 separators of 16 bits, 17 children.  A code is the
//            distance of a key from the last key before the (upper) coded
//            node, shifted so that the node's last key fits; a query takes
//            its own code once for both levels.  Codes order keys up to ties:
//            the entry found is the first whose largest key's code is not
//            below the query's, and a query above that entry's keys goes on
//            from it.  Levels above (and all levels of a tree whose keys
//            crowd so that codes would often tie) hold full words: SEP = 32 /
//            word separators (4 of 64 bits, 8 of 32), FAN = SEP + 1 children.
//            Node i has the children FAN i .. FAN i + SEP of the next level
//            (17 i .. 17 i + 16), separator j stands for the largest key under
//            child j, all-ones where child j + 1 does not exist;
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
constexpr uint32_t kCodeFan = 17;
// Segments at most: above 2^12 a second coded level is cheaper than the
// larger top (its copy, and the room it takes from L1), and a level of full
// words dearer than a top of up to 2^14.
constexpr uint32_t kWalkSegs = 4096, kWalkMaxSegs = 16384;
// Bytes of the largest top: separators, at most one bin each and one per
// octave besides, the octaves, padding.
constexpr int walk_max_top(int key_bytes)
{
    return static_cast<int>(kWalkMaxSegs) * ((key_bytes == 4 ? 4 : 8) + 2) + 64 * 2 + 64 * 8 + 64;
}

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

// The same for a coded node (two codes per word, the earlier in the low half)
// and a query's code.
__device__ __forceinline__ uint32_t coded_rank(const Sector<uint32_t> &s, uint32_t code)
{
    const uint32_t c = code << 16;  // against the high half the low one does not matter
    uint32_t r = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) r += ((s.w[j] << 16) < c ? 1u : 0u) + (s.w[j] < c ? 1u : 0u);
    return r;
}

// Code of word q under a coded node whose keys lie in (lo, hi].
template <typename W>
__device__ __forceinline__ uint32_t walk_code(W q, W lo, W hi)
{
    const W width = hi - lo, d = q > lo ? q - lo : 0;
    const int bits = sizeof(W) == 8 ? 64 - __clzll(static_cast<long long>(width)) : 32 - __clz(static_cast<int>(width));
    const W c = d >> (bits > 16 ? bits - 16 : 0);
    return c < 0xFFFFu ? static_cast<uint32_t>(c) : 0xFFFFu;
}

// Bins of one octave: the first, and the shift that makes a bin of the bits
// after the leading one.
struct WalkOctave {
    uint32_t base, shift;
};

// The bin of word q (host and device: the build fills the table by it).
template <typename W>
__host__ __device__ __forceinline__ uint32_t walk_octave(const WalkDev &w, W q, uint64_t &x)
{
    uint64_t y = q > static_cast<W>(w.wmin) ? static_cast<uint64_t>(q) - w.wmin : 0;
    const uint64_t range = w.wmax - w.wmin;
    y = (y < range ? y : range) | 1u;
#ifdef __CUDA_ARCH__
    const int o = 63 - __clzll(static_cast<long long>(y));
#else
    const int o = 63 - __builtin_clzll(y);
#endif
    x = y - (1ull << o);
    return static_cast<uint32_t>(o);
}

// The segment of q among the segments [lo, hi]: the first whose largest key
// is not below q (the last one when none is known to be).
template <typename W>
__device__ __forceinline__ uint32_t walk_segment_in(const W *sep, uint32_t lo, uint32_t hi, W q)
{
    while (lo < hi) {
        const uint32_t mid = (lo + hi) / 2;
        if (sep[mid] < q)
            lo = mid + 1;
        else
            hi = mid;
    }
    return lo;
}

// The segment of q: the first whose largest key is not below q, or the last.
// top: the top in shared or global memory.
template <typename W>
__device__ __forceinline__ uint32_t walk_segment(const WalkDev &w, const unsigned char *top, W q)
{
    if (w.segs == 1) return 0;
    uint64_t x;
    const uint32_t o = walk_octave<W>(w, q, x);
    const WalkOctave oct = reinterpret_cast<const WalkOctave *>(top + w.oct_off)[o];
    const uint16_t *bins = reinterpret_cast<const uint16_t *>(top + w.bin_off) + oct.base + static_cast<uint32_t>(x >> oct.shift);
    return walk_segment_in<W>(reinterpret_cast<const W *>(top), bins[0], bins[1], q);
}

// The entry of q from its segment: the first entry whose largest key
// (32-byte keys: word), or that key's code, is not below q, or the last one.
// top: as walk_segment.
template <typename W>
__device__ __forceinline__ uint32_t walk_entry(const WalkDev &w, const unsigned char *top, uint32_t node, W q)
{
    constexpr uint32_t SEP = 32u / sizeof(W);
    const W *sep = reinterpret_cast<const W *>(top);
    // the keys below lie in (lo, hi]
    W lo = static_cast<W>(w.wmin), hi = static_cast<W>(w.wmax);
    if (w.coded) {
        if (node) lo = sep[node - 1];
        hi = sep[node];
    }
    int l = 0;
    for (; l < w.levels - w.coded; ++l) {
        const Sector<W> s = ld_sector<W>(w.nodes + w.off[l] + static_cast<uint64_t>(node) * 32u);
        uint32_t r = 0;
#pragma unroll
        for (uint32_t j = 0; j < SEP; ++j) {
            const bool below = s.w[j] < q;
            r += below ? 1u : 0u;
            if (below) lo = s.w[j];
        }
#pragma unroll
        for (uint32_t j = SEP; j-- > 0;)
            if (!(s.w[j] < q) && s.w[j] != KeyOps<W>::ones()) hi = s.w[j];
        node = node * (SEP + 1) + r;
    }
    if (w.coded) {
        const uint32_t code = walk_code<W>(q, lo, hi);
        for (; l < w.levels; ++l)
            node = node * kCodeFan +
                   coded_rank(ld_sector<uint32_t>(w.nodes + w.off[l] + static_cast<uint64_t>(node) * 32u), code);
    }
    return node;
}

// An entry's keys as loaded, whether its largest lies below q, and q's place
// among them (G: not there).
template <typename K>
struct EntryKeys {
    Sector<typename WalkWord<K>::type> s;
    __device__ __forceinline__ explicit EntryKeys(const unsigned char *p) : s(ld_sector<typename WalkWord<K>::type>(p))
    {
    }
    __device__ __forceinline__ Key32 key32() const { return Key32{{s.w[0], s.w[1], s.w[2], s.w[3]}}; }
    template <uint32_t G>
    __device__ __forceinline__ bool below(const K &q) const
    {
        if constexpr (sizeof(K) > 8)
            return key32() < q;
        else
            return s.w[G - 1] < q;
    }
    template <uint32_t G>
    __device__ __forceinline__ uint32_t find(const K &q) const
    {
        uint32_t at = G;
        if constexpr (sizeof(K) > 8) {
            if (key32() == q) at = 0;
        } else {
#pragma unroll
            for (uint32_t j = G; j-- > 0;)
                if (s.w[j] == q) at = j;
        }
        return at;
    }
};

// Key and value of q, whose entry is e or, when e's keys all lie below q (32-byte
// keys that share the word, or codes that tie), one after it.
template <typename K, typename V>
__device__ __forceinline__ bool walk_lookup(const WalkDev &w, uint32_t e, const K &q, V &val)
{
    constexpr uint32_t G = walk_group(sizeof(K), sizeof(V));
    const unsigned char *p = w.entries + static_cast<uint64_t>(e) * 64u;
    const EntryKeys<K> k(p);
    val = static_cast<V>(~static_cast<V>(0));
    uint32_t at = k.template find<G>(q);
    if (at < G) {
        // the last entry's unused slots hold all-ones, which may be the query
        if (static_cast<uint64_t>(e) * G + at >= w.n) return false;
        // read only now that its place is known, although the entry's two
        // sectors could be asked for together: the keys' read has brought
        // both to the L2, and a second read that waits for memory costs more
        // than one that hits (2^20 over 2^24 keys: 34.5 us together, 33.6 so)
        val = ld_key(reinterpret_cast<const V *>(p + 32) + at);
        return true;
    }
    if (!k.template below<G>(q)) return false;
    // gallop to the first entry that is not below q
    const uint64_t E = (w.n + G - 1) / G;
    uint64_t lo = static_cast<uint64_t>(e) + 1, step = 1;
    while (lo + step <= E && EntryKeys<K>(w.entries + (lo + step - 1) * 64u).template below<G>(q)) {
        lo += step;
        step *= 2;
    }
    uint64_t hi = lo + step - 1 < E ? lo + step - 1 : E;
    while (lo < hi) {
        const uint64_t mid = (lo + hi) / 2;
        if (EntryKeys<K>(w.entries + mid * 64u).template below<G>(q))
            lo = mid + 1;
        else
            hi = mid;
    }
    if (lo >= E) return false;
    p = w.entries + lo * 64u;
    at = EntryKeys<K>(p).template find<G>(q);
    if (at == G || lo * G + at >= w.n) return false;
    val = ld_key(reinterpret_cast<const V *>(p + 32) + at);
    return true;
}

}  // namespace btgb
