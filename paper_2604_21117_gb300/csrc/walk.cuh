// Search of a batch as given (no partition) through a tree's walk index.
//
// The level-wise descent reads a whole node block per level: 256 bytes at
// fanout 32 and 64-bit keys.  Over a partitioned batch a warp shares those
// blocks; over a batch as given every lane needs its own, and what bounds
// the search is the bytes (in 32-byte sectors) that cross from the L2 to the
// SMs.  The walk index holds the same keys and values a second time in the
// form that costs the fewest sectors per query:
//
//   top      the largest keys of up to 15360 segments of equal length (25600
//            for 32-bit keys), ascending, and two tables that narrow the
//            search among them to a few: the octave of x = key - smallest key
//            (its leading one) gives a range of bins, as many as the octave has
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
//   entries  the children of the last level.  Integer keys: one sector, G =
//            32 / (key + value bytes) consecutive keys (bytes 0..15, unused
//            slots all-ones) and their values (bytes 16..31), so that one read
//            brings a query's key and its value; the keys are packed densely,
//            entry e holding ranks G e .. G e + G - 1.  32-byte keys: 64
//            bytes, one key (four words, as Key32) and its value.
//
// 32-byte keys are walked by one 64-bit word, the 8 bytes after the bytes all
// keys share: a query between the smallest and the largest key shares those
// bytes too, so the word orders it among the keys up to ties, and the entry
// found is the first whose word is not below the query's.  A tree whose words
// tie in long runs gets no walk index.
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
// words dearer than a top of up to 160 KB (2^20 queries of 2^23 uint64 keys,
// 148 KB of top: 23.5 us, with a level instead and a 29 KB top 25.4).
constexpr uint32_t kWalkSegs = 4096;
constexpr uint32_t walk_max_segs(int key_bytes) { return key_bytes == 4 ? 25600 : 15360; }
// Bytes of the largest top: separators, at most one bin each and one per
// octave besides, the octaves, padding.
constexpr int walk_max_top(int key_bytes)
{
    return static_cast<int>(walk_max_segs(key_bytes)) * ((key_bytes == 4 ? 4 : 8) + 2) + 64 * 2 + 64 * 8 + 64;
}

// Keys and bytes per entry.
__host__ __device__ constexpr uint32_t walk_group(int key_bytes, int val_bytes)
{
    return key_bytes > 8 ? 1u : 32u / static_cast<uint32_t>(key_bytes + val_bytes);
}
__host__ __device__ constexpr uint32_t walk_entry_bytes(int key_bytes) { return key_bytes > 8 ? 64u : 32u; }

// The walk kernels ask for no more shared memory on an SM than their one
// block needs: misses in flight are held in L1 lines, so L1 is what bounds
// them.  Left to the runtime, which makes room for as many blocks as the SM
// could hold, a top of 100 to 114 KB (two blocks fit) left 28 KB of L1, and
// 2^20 uniform queries of 2 * 10^7 uint32 keys took 51 us instead of 22; with
// 228 / 196 / 164 / 132 / 100 KB of shared memory for the 58 KB top of 2^24
// uint64 keys 2^20 queries take 72 / - / 42.0 / 35.5 / 33.3 us, with as much
// as needed 32.7.
constexpr int kWalkCarveout = 0;  // cudaSharedmemCarveoutMaxL1

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
    const uint32_t bin = oct.base + static_cast<uint32_t>(x >> oct.shift);
    const uint16_t *bins = reinterpret_cast<const uint16_t *>(top + w.bin_off) + bin;
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

// An entry as loaded: whether its keys all lie below q, q's place among them
// (G: not there), and the value there (integer keys).
template <typename K, typename V>
struct WalkEntry {
    static constexpr uint32_t G = walk_group(sizeof(K), sizeof(V));
    Sector<uint32_t> s;
    __device__ __forceinline__ WalkEntry(const WalkDev &w, uint64_t e)
        : s(ld_sector<uint32_t>(w.entries + e * walk_entry_bytes(sizeof(K))))
    {
    }
    __device__ __forceinline__ uint64_t word(uint32_t i) const
    {
        return s.w[2 * i] | static_cast<uint64_t>(s.w[2 * i + 1]) << 32;
    }
    __device__ __forceinline__ K key(uint32_t j) const
    {
        if constexpr (sizeof(K) > 8)
            return Key32{{word(0), word(1), word(2), word(3)}};
        else if constexpr (sizeof(K) == 8)
            return word(j);
        else
            return s.w[j];
    }
    __device__ __forceinline__ bool below(const K &q) const { return key(G - 1) < q; }
    __device__ __forceinline__ uint32_t find(const K &q) const
    {
        uint32_t at = G;
#pragma unroll
        for (uint32_t j = G; j-- > 0;)
            if (key(j) == q) at = j;
        return at;
    }
    __device__ __forceinline__ V value(uint32_t at) const
    {
        V v = 0;
#pragma unroll
        for (uint32_t j = 0; j < G; ++j)
            if (at == j) {
                if constexpr (sizeof(V) == 8)
                    v = word(2 + j);
                else
                    v = s.w[4 + j];
            }
        return v;
    }
};

// Key and value of q, whose entry is e or, when e's keys all lie below q (32-byte
// keys that share the word, or codes that tie), one after it.
template <typename K, typename V>
__device__ __forceinline__ bool walk_lookup(const WalkDev &w, uint32_t e, const K &q, V &val)
{
    using Entry = WalkEntry<K, V>;
    constexpr uint32_t G = Entry::G;
    val = static_cast<V>(~static_cast<V>(0));
    uint64_t at_e = e;
    const Entry x(w, e);
    uint32_t at = x.find(q);
    if (at < G) {
        if constexpr (sizeof(K) <= 8) val = x.value(at);
    } else {
        if (!x.below(q)) return false;
        // gallop to the first entry that is not below q
        const uint64_t E = (w.n + G - 1) / G;
        uint64_t lo = at_e + 1, step = 1;
        while (lo + step <= E && Entry(w, lo + step - 1).below(q)) {
            lo += step;
            step *= 2;
        }
        uint64_t hi = lo + step - 1 < E ? lo + step - 1 : E;
        while (lo < hi) {
            const uint64_t mid = (lo + hi) / 2;
            if (Entry(w, mid).below(q))
                lo = mid + 1;
            else
                hi = mid;
        }
        if (lo >= E) return false;
        const Entry y(w, lo);
        at = y.find(q);
        if (at == G) return false;
        if constexpr (sizeof(K) <= 8) val = y.value(at);
        at_e = lo;
    }
    // the last entry's unused slots hold all-ones, which may be the query
    if (at_e * G + at >= w.n) {
        val = static_cast<V>(~static_cast<V>(0));
        return false;
    }
    // a 32-byte key's value is read only now: the key's read has brought the
    // entry's other sector to the L2 too, and a second read that waits for
    // memory costs more than one that hits (2^20 keys: 32.5 us both at once,
    // 31.4 so)
    if constexpr (sizeof(K) > 8) val = ld_key(reinterpret_cast<const V *>(w.entries + at_e * 64u + 32));
    return true;
}

}  // namespace btgb
