// Insertion by key ranges on sm_103a: the windows of a call are brought
// together by key before anything is counted, so that the countBF sees each
// distinct K-mer once, with its multiplicity, instead of every window.
// Saturating increments commute (Algorithm 3 read per counter), so adding a
// key's multiplicity to its counters at once gives the countBF of adding one
// per window.
//
//   1. pack_kernel: the bases as 2-bit codes and one bit per base that starts
//      a window to be counted; nothing reads the caller's buffers after it.
//   2. sample_kernel, rank_kernel: keys of random windows and their ranks; the
//      ones at even ranks cut the key space into ranges that hold about
//      equally many windows.
//      extract_kernel: per chunk of window starts, every window's canonical
//      key (rolled from base to base); the chunk's keys are grouped by range
//      in shared memory and leave as one contiguous piece, with the piece's
//      range starts in a table.  No key moves by a global atomic.
//   3. large calls, a second level: the pieces of one range are gathered tile
//      by tile (row_prefix_kernel, tile_map_kernel say where a tile begins),
//      cut again by splitters sampled inside the range, and written as tiles
//      grouped by the finer ranges (refine_kernel).
//   4. dedup_kernel: one block per final range gathers its windows, finds the
//      distinct keys and their multiplicities with a shared-memory hash set,
//      and sorts them.  The ranges are in key order, so the distinct keys
//      come out in ascending order with nothing left to sort.
//   5. scan_counts_kernel, then emit_kernel (codes for the partitioned update)
//      or emit_atomic_kernel: the increments of the distinct keys, and the
//      distinct list.
//
// A range is cut by splitters taken from the data itself, so skewed
// compositions only move the splitters.  A key held by very many windows is
// more than one splitter: the last of them becomes the next key, so that the
// range before it holds this key alone and is counted by the lengths of its
// runs.  A range with more distinct keys than fit is handled in several rounds
// over sub-ranges of it.
//
// Keys are cut by their prefix (their top 64 bits), two-word keys whose prefixes
// are equal by their low word: reads with a common beginning of 32 bases and
// more would else all meet in one range, which is one block's.
#include "kmerco_dedup.cuh"
#include "kmerco_stage.cuh"

#include <string.h>

#include <algorithm>

namespace countbf {
namespace {

template <int KW>
struct Key {
    uint64_t lo, hi;   // hi is 0 for one-word keys
    __device__ __forceinline__ bool operator==(const Key &o) const {
        return lo == o.lo && (KW == 1 || hi == o.hi);
    }
    __device__ __forceinline__ bool operator<(const Key &o) const {
        if (KW == 1) return lo < o.lo;
        return hi < o.hi || (hi == o.hi && lo < o.lo);
    }
};

template <int KW>
__device__ __forceinline__ Key<KW> load_key(const uint64_t *p, uint64_t i) {
    Key<KW> k;
    if (KW == 1) {
        k.lo = p[i];
        k.hi = 0;
    } else {
        const ulonglong2 v = ((const ulonglong2 *)p)[i];
        k.lo = v.x;
        k.hi = v.y;
    }
    return k;
}

template <int KW>
__device__ __forceinline__ void store_key(uint64_t *p, uint64_t i, const Key<KW> &k) {
    if (KW == 1) {
        p[i] = k.lo;
    } else {
        ulonglong2 v;
        v.x = k.lo;
        v.y = k.hi;
        ((ulonglong2 *)p)[i] = v;
    }
}

// The top min(2K, 64) bits of a key's 2K bits: what ranges are cut by.
template <int KW>
__device__ __forceinline__ uint64_t prefix_of(const Key<KW> &k, int K) {
    if (KW == 1) return k.lo;
    const int s = 2 * K - 64;   // 2..64
    return s == 64 ? k.hi : (k.hi << (64 - s)) | (k.lo >> s);
}

__device__ __forceinline__ int prefix_bits(int K) { return K < 32 ? 2 * K : 64; }

// Bits of x (0 for 0).
__device__ __forceinline__ int bit_len(uint64_t x) { return 64 - __clzll((long long)x); }

// The canonical one of a window's two strands (InsertArgs::canonical).
__device__ __forceinline__ Key<1> canonical_key(const Key<1> &f, const Key<1> &r, int mode) {
    if (mode == 0) return f;
    if (mode == 1) return r.lo < f.lo ? r : f;
    uint64_t hf, hr, t;   // the strand with the smaller H_0
    murmur8(premix8(f.lo), 0u, hf, t);
    murmur8(premix8(r.lo), 0u, hr, t);
    return hf < hr ? f : r;
}
__device__ __forceinline__ Key<2> canonical_key(const Key<2> &f, const Key<2> &r, int mode) {
    if (mode == 0) return f;
    if (mode == 1) return r < f ? r : f;
    uint64_t hf, hr, t;
    murmur16(f.lo, f.hi, 0u, hf, t);
    murmur16(r.lo, r.hi, 0u, hr, t);
    return hf < hr ? f : r;
}

// A place to cut two-word keys at: the prefix, and the low word for keys with
// that prefix.
struct __align__(16) Cut2 {
    uint64_t p, lo;
    __device__ __forceinline__ bool operator<(const Cut2 &o) const {
        return p < o.p || (p == o.p && lo < o.lo);
    }
};

__device__ __forceinline__ uint64_t shfl_xor(uint64_t v, int m) {
    return __shfl_xor_sync(0xffffffffu, v, m);
}
__device__ __forceinline__ Cut2 shfl_xor(const Cut2 &v, int m) {
    return Cut2{shfl_xor(v.p, m), shfl_xor(v.lo, m)};
}

// What samples of keys are sorted by.
template <int KW> struct SampleOf { using T = uint64_t; };
template <> struct SampleOf<2> { using T = Cut2; };
__device__ __forceinline__ uint64_t sample_of(const Key<1> &k, int) { return k.lo; }
__device__ __forceinline__ Cut2 sample_of(const Key<2> &k, int K) {
    return Cut2{prefix_of<2>(k, K), k.lo};
}
__device__ __forceinline__ void largest_sample(uint64_t &v) { v = ~0ull; }
__device__ __forceinline__ void largest_sample(Cut2 &v) { v.p = v.lo = ~0ull; }

// Index of a key among the n ranges of n - 1 sorted splitters: how many of those
// are at or below it.  x is the key's prefix and low its low word; spl has the
// splitters' prefixes, low_of(i) gives the low word of a two-word splitter: 0 where
// no other splitter has the prefix.
// lut[i] = splitters whose (prefix - lo) >> sh is below i, with kMany set when
// more than one falls into cell i, so that one comparison of prefixes decides
// nearly every key without a branch; in the other cells it bisects the cell's
// splitters.  kTies is set where prefixes are equal among them, and only there low
// words are compared (they stay in global memory; comparing them in every such cell made
// refine_kernel 5% slower).  spl is followed by an all-ones value.
constexpr unsigned kMany = 0x8000u, kTies = 0x4000u, kLutIndex = 0x3fffu;
static_assert(kMaxRanges <= kLutIndex, "an index beside the flags");

template <int KW, typename F>
__device__ __forceinline__ unsigned find_range(const uint64_t *spl, F low_of, const uint16_t *lut,
                                               unsigned n, uint64_t lo, int sh, uint64_t x,
                                               uint64_t low) {
    const unsigned c = (unsigned)((x - lo) >> sh), e = lut[c];
    unsigned a = e & kLutIndex;
    a += spl[a] <= x ? 1u : 0u;
    if (e & kMany) {
        a = e & kLutIndex;
        unsigned b = c + 1 < kLutStride ? lut[c + 1] & kLutIndex : n - 1;
        if (KW == 2 && (e & kTies)) {
            while (a < b) {
                const unsigned m = (a + b) / 2;
                const uint64_t s = spl[m];
                if (s < x || (s == x && low_of(m) <= low))
                    a = m + 1;
                else
                    b = m;
            }
        } else {
            while (a < b) {
                const unsigned m = (a + b) / 2;
                const bool at_or_below = spl[m] <= x;
                a = at_or_below ? m + 1 : a;
                b = at_or_below ? b : m;
            }
        }
    }
    return min(a, n - 1);   // an all-ones prefix passes the end
}

// Ascending bitonic sort of 1024 * E values, E consecutive ones to a thread in
// v (1,024 threads); xch: room for 1024 * E values in shared memory.  Strides
// inside a thread are register swaps, inside a warp shuffles; only the 15 steps
// of larger strides go through shared memory (105 of a plain network of 16,384
// values).
template <int E, typename V>
__device__ __forceinline__ void block_sort(V (&v)[E], V *xch) {
    constexpr unsigned P = 1024 * E;
    const unsigned tid = threadIdx.x, i0 = tid * E;
    for (unsigned k = 2; k <= P; k <<= 1) {
        for (unsigned j = k >> 1; j > 0; j >>= 1) {
            if (j >= 32 * E) {   // the partner is in another warp
                __syncthreads();
#pragma unroll
                for (int e = 0; e < E; ++e) xch[e * 1024 + tid] = v[e];
                __syncthreads();
                const unsigned other = tid ^ (j / E);
                const bool lower = (i0 & j) == 0, up = (i0 & k) == 0;
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const V o = xch[e * 1024 + other];
                    v[e] = (lower == up) == (o < v[e]) ? o : v[e];
                }
            } else if (j >= E) {   // in another lane
                const bool lower = (i0 & j) == 0, up = (i0 & k) == 0;
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const V o = shfl_xor(v[e], (int)(j / E));
                    v[e] = (lower == up) == (o < v[e]) ? o : v[e];
                }
            } else {   // in this thread
#pragma unroll
                for (int b = E / 2; b > 0; b >>= 1) {
                    if (b != (int)j) continue;
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        if (e & b) continue;
                        const bool up = ((i0 + e) & k) == 0;
                        const V x = v[e], y = v[e | b];
                        const bool swap = (y < x) == up;
                        v[e] = swap ? y : x;
                        v[e | b] = swap ? x : y;
                    }
                }
            }
        }
    }
}

// The lookup table of n - 1 splitters of the range [lo, last], v the thread's
// prefix (1,024 threads, n <= kMaxRanges), tie: whether another one has it and their
// low words decide; cells: 32 KiB of shared memory.  In two-word keys' last cell a
// key may have the prefix of the unused splitters, all ones: whole keys there too.
template <int KW>
__device__ __forceinline__ void write_lut(unsigned *cells, uint64_t v, bool tie, bool any,
                                          unsigned n, uint64_t lo, uint64_t last, uint16_t *lut) {
    static_assert(kMaxRanges <= 1024, "a splitter a thread");
    constexpr unsigned E = (1u << kLutBits) / 1024;
    const unsigned j = threadIdx.x;
    int sh = bit_len(last - lo) - kLutBits;
    if (sh < 0) sh = 0;
    for (unsigned i = j; i < (1u << kLutBits); i += 1024) cells[i] = 0;
    __syncthreads();
    if (j + 1 < n && any) {   // splitters in every cell of the table
        const uint64_t c = (v - lo) >> sh;
        if (c < (1u << kLutBits)) atomicAdd(cells + c, tie ? 0x10001u : 1u);
    }
    __syncthreads();
    unsigned c[E], sum = 0;
#pragma unroll
    for (unsigned q = 0; q < E; ++q) sum += (c[q] = cells[j * E + q]) & 0xffffu;
    unsigned tot;
    unsigned pre = block_exclusive_scan<unsigned, 1024>(sum, tot);
#pragma unroll
    for (unsigned q = 0; q < E; ++q) {
        unsigned flags = (c[q] & 0xffffu) > 1 ? kMany : 0u;
        if (KW == 2 && (c[q] > 0xffffu || j * E + q == (unsigned)((last - lo) >> sh)))
            flags = kMany | kTies;
        lut[j * E + q] = (uint16_t)(pre | flags);
        pre += c[q] & 0xffffu;
    }
}

// The cut right behind the cut (p, low), when that is a key: whether it is one, and
// not the largest.  A two-word cut whose low word does not go with its prefix (a
// sample that stands for all keys of its prefix has 0 there) is none.
template <int KW>
__device__ __forceinline__ bool next_cut(uint64_t &p, uint64_t &low, int K) {
    if (KW == 1) {
        if (p == ~0ull) return false;
        ++p;
        return true;
    }
    Key<2> k;
    k.hi = p >> (128 - 2 * K);
    k.lo = low;
    if (prefix_of<2>(k, K) != p || (p == ~0ull && low == ~0ull)) return false;
    k.hi += ++k.lo == 0 ? 1 : 0;
    const uint64_t q = prefix_of<2>(k, K);
    low = q == p ? k.lo : 0;   // (q, 0): in front of all keys of the next prefix
    p = q;
    return true;
}

// Splitter j of n, (p, low), where at(i, p, low) reads splitter i: the last one of
// equal splitters moves behind their key, which is held by more windows than a range
// then has.  Whether there are equal ones.
template <int KW, typename F>
__device__ __forceinline__ bool part_equal(F at, unsigned j, unsigned n, uint64_t &p, uint64_t &low,
                                           int K) {
    p = low = ~0ull;
    if (j >= n) return false;
    at(j, p, low);
    const auto as = [&](unsigned i) {
        uint64_t q, r = low;
        at(i, q, r);
        return q == p && (KW == 1 || r == low);
    };
    const bool prev = j && as(j - 1), next = j + 1 < n && as(j + 1);
    if (prev && !next) {
        uint64_t q = p, r = low;
        if (next_cut<KW>(q, r, K)) {
            p = q;
            low = r;
        }
    }
    return prev || next;
}

// Whether a neighbour among the n splitters has the prefix p of thread j's one too
// (seen: shared memory for the prefixes).
__device__ __forceinline__ bool shares_prefix(uint64_t *seen, unsigned j, unsigned n, uint64_t p) {
    __syncthreads();
    if (j < n) seen[j] = p;
    __syncthreads();
    const bool shared = j < n && ((j && seen[j - 1] == p) || (j + 1 < n && seen[j + 1] == p));
    __syncthreads();
    return shared;
}

__device__ __forceinline__ uint64_t mix64(uint64_t x) { return fmix64(x + 0x9E3779B97F4A7C15ull); }

// ---------------------------------------------------------------- 1. pack
// A pass's bases from its first chunk on as 2-bit codes (InsertArgs' window
// starts are positions in it), and per window start a bit when the window
// lies in one read and its K bases are valid.  Bound by the memory it streams:
// a byte read and 3/8 byte written per base.
template <int CHUNK>
__global__ void __launch_bounds__(CHUNK / 16) pack_kernel(InsertArgs a, PackArgs x) {
    constexpr int NT = CHUNK / 16, kPack32 = ChunkDims<CHUNK>::kPack32;
    __shared__ StageSmem<CHUNK> S;
    const int tid = threadIdx.x, K = a.K;
    unsigned long long my_windows = 0, my_skipped = 0;
    const unsigned p = (unsigned)tid * 16;
    const uint64_t *inv64 = (const uint64_t *)S.inv, *brk64 = (const uint64_t *)S.brk;
    // bit i of an OR over `len` bits from i on, for i < 16, by doubling
    const auto any_of = [](uint64_t lo, uint64_t hi, int len) {
        int have = 1;
        while (have < len) {
            const int s = min(have, len - have);   // 1..32
            lo |= (lo >> s) | (hi << (64 - s));
            hi |= hi >> s;
            have += s;
        }
        return (unsigned)lo & 0xffffu;
    };
    for (int i = tid; i < kPack32 / 2; i += NT) S.brk[i] = 0;
    __syncthreads();
    for (uint64_t chunk = x.chunk_begin + blockIdx.x; chunk < x.chunk_end; chunk += gridDim.x) {
        const uint64_t row = chunk - x.chunk0;
        const unsigned nb = stage_chunk<CHUNK, NT>(a, chunk, S);
        __syncthreads();
        unsigned no_window =
            K > 1 ? any_of(bits_at(brk64, p + 1), bits_at(brk64, p + 65), K - 1) : 0u;
        if (p + 16 + (unsigned)K > nb + 1) {   // the span ends inside these windows
            const int left = (int)nb - K - (int)p + 1;   // of the 16, how many fit
            no_window |= left > 0 ? 0xffffu << left : 0xffffu;
        }
        no_window &= 0xffffu;
        const unsigned bad = any_of(bits_at(inv64, p), bits_at(inv64, p + 64), K) | no_window;
        x.valid[row * NT + tid] = (uint16_t)~bad;
        // the codes of the chunk, and of the K - 1 bases and more after the last one
        const unsigned words = chunk + 1 == x.chunk_last ? kPack32 : NT;
        for (unsigned t = tid; t < words; t += NT) x.codes[row * NT + t] = S.pk[t];
        my_windows += 16 - __popc(no_window);
        my_skipped += __popc(bad & ~no_window);
        __syncthreads();
        for (int i = tid; i < kPack32 / 2; i += NT) S.brk[i] = 0;
        __syncthreads();
    }
    // one addition per block: same-address atomics of every warp and chunk
    // took six times as long as the rest of the kernel
    unsigned long long w, k;
    block_exclusive_scan<unsigned long long, NT>(my_windows, w);
    block_exclusive_scan<unsigned long long, NT>(my_skipped, k);
    if (tid == 0 && w) {
        atomicAdd(&a.ctr->windows, w);
        atomicAdd(&a.ctr->skipped, k);
        atomicAdd(&a.ctr->inserted, w - k);
    }
}

// The forward key of the window at position p of the packed codes (two codes
// words to a 64-bit word, first base most significant).
__device__ __forceinline__ void window_at(const uint64_t *codes, uint64_t p, int K, Key<1> &f) {
    const uint64_t w = p >> 5;
    const unsigned s = (unsigned)(p & 31) * 2;
    const uint64_t x0 = codes[w], x1 = codes[w + 1];
    f.lo = (s ? (x0 << s) | (x1 >> (64 - s)) : x0) >> (64 - 2 * K);
    f.hi = 0;
}
__device__ __forceinline__ void window_at(const uint64_t *codes, uint64_t p, int K, Key<2> &f) {
    const uint64_t w = p >> 5;
    const unsigned s = (unsigned)(p & 31) * 2;
    const uint64_t x0 = codes[w], x1 = codes[w + 1], x2 = codes[w + 2];
    const uint64_t t0 = s ? (x0 << s) | (x1 >> (64 - s)) : x0;
    const uint64_t t1 = s ? (x1 << s) | (x2 >> (64 - s)) : x1;
    const int d = 128 - 2 * K;   // 0..62
    f.lo = d ? (t1 >> d) | (t0 << (64 - d)) : t1;
    f.hi = t0 >> d;
}
__device__ __forceinline__ Key<1> revcomp(const Key<1> &f, int K) {
    Key<1> r;
    r.lo = revcomp64(f.lo, K);
    r.hi = 0;
    return r;
}
__device__ __forceinline__ Key<2> revcomp(const Key<2> &f, int K) {
    Key<2> r;
    revcomp128(f.hi, f.lo, K, r.hi, r.lo);
    return r;
}

// ----------------------------------------------------------- 2. splitters
// Equal prefixes among a level's splitters, or a tile's samples, from which on the low
// words of two-word keys decide too.
constexpr unsigned kCrowd = 5;

constexpr unsigned kSampleTile = 1024;   // samples a block sorts

// The keys at n random valid window starts of the pass's `span` bases (a few tries
// each), as sorted tiles of kSampleTile: samples has their prefixes, samples_lo the
// low words of two-word keys (0 in tiles without more than kCrowd samples of a
// prefix); the last tile is filled up with all ones.  Whole prefixes: copies of a
// repeat have long beginnings in common, and cutting by their top 31 bits left more than
// twice as many windows in some ranges (dedup_big_kernel 2.8 instead of 1.8 ms for
// 3.8e8 two-word windows).
template <int KW>
__global__ void __launch_bounds__(1024) sample_kernel(PackArgs x, int K, int canonical,
                                                      uint64_t span, unsigned n,
                                                      uint64_t *samples, uint64_t *samples_lo,
                                                      DedupMeta *meta) {
    __shared__ typename SampleOf<KW>::T xch[kSampleTile];
    const unsigned i = blockIdx.x * kSampleTile + threadIdx.x;
    Key<KW> key;
    bool found = false;
    for (unsigned t = 0; t < 4 && i < n && !found; ++t) {
        // window starts spread evenly over the pass, jittered; then anywhere
        const uint64_t slot = (uint64_t)i * span / n, wide = max(span / n, (uint64_t)1);
        const uint64_t z = mix64((uint64_t)i * 4 + t);
        const uint64_t at = t < 2 ? slot + __umul64hi(z, wide) : __umul64hi(z, span);
        if (!((x.valid[at >> 4] >> (at & 15)) & 1u)) continue;
        Key<KW> f;
        window_at((const uint64_t *)x.codes, at, K, f);
        key = canonical_key(f, revcomp(f, K), canonical);
        found = true;
    }
    const int c = __syncthreads_count(found);
    if (threadIdx.x == 0 && c) atomicAdd(&meta->sampled, (unsigned)c);
    const uint64_t p = found ? prefix_of<KW>(key, K) : ~0ull;
    uint64_t v[1] = {p}, low = 0;
    block_sort<1>(v, (uint64_t *)xch);
    if constexpr (KW == 2) {
        // many equal prefixes in the tile, which is rare: in the order of the whole keys
        uint64_t *const seen = (uint64_t *)xch;
        const unsigned tid = threadIdx.x;
        __syncthreads();
        seen[tid] = v[0];
        __syncthreads();
        const bool same = tid >= kCrowd && v[0] != ~0ull && seen[tid - kCrowd] == v[0];
        if (__syncthreads_or(same)) {
            if (tid == 0) atomicOr(&meta->crowd, 1u << blockIdx.x);
            Cut2 w[1] = {Cut2{p, found ? key.lo : ~0ull}};
            block_sort<1>(w, xch);
            v[0] = w[0].p;
            low = w[0].lo;
        }
        samples_lo[i] = low;
    }
    samples[i] = v[0];
}

// The samples of even ranks among the n of all tiles become the n_ranges - 1
// splitters.  Block b ranks tile b: a sample's place in it, and by bisection its
// places in the other tiles (their prefixes in shared memory; of equal samples the
// ones of earlier tiles come first).  The last block to finish builds the lookup
// table.  One block that sorted all samples took 20 us for 4,096 of them and 80 for
// 16,384, a fifth to a third of a piece of 5e5 windows.
template <int KW>
__global__ void __launch_bounds__(1024) rank_kernel(const uint64_t *samples,
                                                    const uint64_t *samples_lo, unsigned n,
                                                    unsigned n_ranges, int K, uint64_t last,
                                                    DedupMeta *meta, uint64_t *spl,
                                                    uint64_t *spl_lo, uint16_t *lut) {
    extern __shared__ ulonglong2 s2[];
    __shared__ bool is_last;
    uint64_t *const s = (uint64_t *)s2;
    const unsigned tid = threadIdx.x, own = blockIdx.x;
    for (unsigned i = tid; i < n / 2; i += 1024) s2[i] = ((const ulonglong2 *)samples)[i];
    __syncthreads();
    const uint64_t v = s[own * kSampleTile + tid];
    const unsigned crowd = KW == 2 ? meta->crowd : 0;   // without, all low words are 0
    const uint64_t low = (crowd >> own) & 1u ? samples_lo[own * kSampleTile + tid] : 0;
    unsigned rank = tid;
    for (unsigned c = 0; c < n / kSampleTile; ++c) {
        if (c == own) continue;
        const unsigned t0 = c * kSampleTile;
        const bool lows = KW == 2 && ((crowd >> c | crowd >> own) & 1u);
        // samples of the tile in front of v; with low words, those below its prefix
        const bool below = c < own && !lows;   // and its equals of earlier tiles
        unsigned at = 0;
#pragma unroll
        for (unsigned step = kSampleTile / 2; step; step >>= 1) {
            const uint64_t t = s[t0 + at + step - 1];
            if (t < v || (below && t == v)) at += step;
        }
        if (s[t0 + at] < v || (below && s[t0 + at] == v)) ++at;
        if (lows) {   // and those of the same prefix in front
            unsigned hi = kSampleTile;
            while (at < hi) {
                const unsigned m = (at + hi) / 2;
                const uint64_t w = s[t0 + m] == v ? samples_lo[t0 + m] : low;
                if (s[t0 + m] == v && (w < low || (w == low && c < own)))
                    at = m + 1;
                else
                    hi = m;
            }
        }
        rank += at;
    }
    const unsigned valid = meta->sampled;
    if (rank < valid) {   // splitter k - 1 is the sample of rank k * valid / n_ranges
        const uint64_t r = rank;
        for (uint64_t k = (r * n_ranges + valid - 1) / valid;
             k < n_ranges && k * valid / n_ranges == r; ++k)
            if (k) {
                spl[k - 1] = v;
                if (KW == 2 && crowd) spl_lo[k - 1] = low;
            }
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) is_last = atomicAdd(&meta->ranked, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    uint64_t f = ~0ull, f_lo = ~0ull;   // of the last of the n: what find_range stops at
    bool equal = false, tie = false;
    if (KW == 1 || crowd) {
        equal = part_equal<KW>(
            [&](unsigned i, uint64_t &p, uint64_t &low) {
                p = __ldcg(spl + i);
                if (KW == 2) low = __ldcg(spl_lo + i);
            },
            tid, valid ? n_ranges - 1 : 0, f, f_lo, K);
    } else if (valid && tid + 1 < n_ranges) {
        f = __ldcg(spl + tid);
        f_lo = 0;
    }
    __syncthreads();
    if (KW == 2 && valid && crowd) {
        tie = shares_prefix(s, tid, n_ranges - 1, f) || equal;
        if (!tie && tid + 1 < n_ranges) f_lo = 0;
    }
    if (tid < n_ranges) {
        spl[tid] = f;
        if (KW == 2) spl_lo[tid] = f_lo;
    }
    write_lut<KW>((unsigned *)s, f, tie, valid != 0, n_ranges, 0, last, lut);
}

// ------------------------------------------------- grouping keys by range
// Shared memory of a block that groups up to TILE keys by up to kMaxRanges
// ranges.
template <int KW, int TILE>
struct __align__(16) GroupSmem {
    uint64_t keys[TILE * KW];
    uint64_t spl[kMaxRanges];
    uint16_t lut[1 << kLutBits];
    unsigned hist[kMaxRanges + 128];   // zero from the ranges on
    unsigned start[kMaxRanges + 4];
    unsigned base;
};

constexpr unsigned kNoKey = ~0u;

// Exclusive prefix of S.hist[0, n) into S.start (start[n] = the sum), n up to
// kMaxRanges, by the first warp: a scan by all warps took a tenth of the
// kernels' instructions.
template <int KW, int TILE>
__device__ __forceinline__ void scan_ranges(GroupSmem<KW, TILE> &S, unsigned n) {
    if (threadIdx.x >= 32) return;
    const unsigned lane = threadIdx.x, per = (n + 127) / 128 * 4;   // a lane's, four at a time
    unsigned sum = 0;
    for (unsigned j = 0; j < per; j += 4) {
        const uint4 v = *(const uint4 *)(S.hist + lane * per + j);   // zero past n
        sum += v.x + v.y + v.z + v.w;
    }
    unsigned pre = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, pre, o);
        if (lane >= (unsigned)o) pre += y;
    }
    if (lane == 31) S.start[n] = pre;
    pre -= sum;
    for (unsigned j = 0; j < per; j += 4) {
        const unsigned i = lane * per + j;
        const uint4 v = *(const uint4 *)(S.hist + i);
        uint4 o;
        o.x = pre;
        o.y = o.x + v.x;
        o.z = o.y + v.y;
        o.w = o.z + v.z;
        pre = o.w + v.w;
        if (i + 4 <= n) {
            *(uint4 *)(S.start + i) = o;
        } else {
            if (i < n) S.start[i] = o.x;
            if (i + 1 < n) S.start[i + 1] = o.y;
            if (i + 2 < n) S.start[i + 2] = o.z;
        }
    }
}

// Copies the first n keys of S.keys to out (16-byte aligned) as a whole.
template <int KW, int TILE, int NT>
__device__ __forceinline__ void copy_out(const GroupSmem<KW, TILE> &S, unsigned n, uint64_t *out) {
    const uint4 *src = (const uint4 *)S.keys;
    uint4 *dst = (uint4 *)out;
    const unsigned nv = KW == 1 ? (n + 1) / 2 : n;   // an odd last key takes its padding along
    for (unsigned i = threadIdx.x; i < nv; i += NT) __stcs(dst + i, src[i]);
}

// ---------------------------------------------------------------- extract
// Bound by instruction issue and shared-memory traffic (about 45 instructions
// a window); it writes one key a window.  Eight consecutive windows a thread:
// the first key is cut from the packed codes, the others are rolled on by one
// base.
template <int KW, int CHUNK, int CANON>
__global__ void __launch_bounds__(CHUNK / 8, CHUNK >= 4096 ? 2 : 6)
    extract_kernel(int K, ExtractArgs x) {
    constexpr int NT = CHUNK / 8;
    constexpr int PER = 8;
    extern __shared__ __align__(16) unsigned char dyn[];
    GroupSmem<KW, CHUNK> &S = *reinterpret_cast<GroupSmem<KW, CHUNK> *>(dyn);
    const int tid = threadIdx.x;
    const unsigned nr = x.n_ranges;
    for (unsigned i = tid; i < nr; i += NT) S.spl[i] = x.spl[i];
    for (unsigned i = tid; i < kLutStride / 8; i += NT) ((uint4 *)S.lut)[i] = ((const uint4 *)x.lut)[i];
    const int bits = prefix_bits(K);
    const int sh = bits > kLutBits ? bits - kLutBits : 0;
    const uint64_t mask1 = K >= 32 ? ~0ull : (1ull << (2 * K)) - 1;
    const uint64_t mask_hi = KW == 1 || K >= 64 ? ~0ull : (1ull << (2 * K - 64)) - 1;
    const uint64_t *codes = (const uint64_t *)x.codes;
    for (unsigned row = blockIdx.x; row < x.n_chunks; row += gridDim.x) {
        for (unsigned i = tid; i < nr + 128; i += NT) S.hist[i] = 0;
        const uint64_t p = (uint64_t)row * CHUNK + (unsigned)tid * PER;
        const unsigned valid = ((const uint8_t *)x.valid)[p >> 3];
        Key<KW> f;
        window_at(codes, p, K, f);
        Key<KW> r = revcomp(f, K);
        uint64_t next;   // the bases after the first window, the nearest in the top bits
        {
            const uint64_t q = p + (unsigned)K, w = q >> 5;
            const unsigned s = (unsigned)(q & 31) * 2;
            next = s ? (codes[w] << s) | (codes[w + 1] >> (64 - s)) : codes[w];
        }
        __syncthreads();
        Key<KW> key[PER];
        unsigned br[PER];   // range and rank within it
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            key[i] = canonical_key(f, r, CANON);
            br[i] = kNoKey;
            if ((valid >> i) & 1u) {
                const unsigned bin = find_range<KW>(
                    S.spl, [&](unsigned m) { return __ldg(x.spl_lo + m); }, S.lut, nr, 0, sh,
                    prefix_of<KW>(key[i], K), key[i].lo);
                br[i] = (bin << 16) | atomicAdd(&S.hist[bin], 1u);
            }
            const uint64_t c = next >> 62;
            next <<= 2;
            if (KW == 1) {
                f.lo = ((f.lo << 2) | c) & mask1;
                r.lo = (r.lo >> 2) | ((3 - c) << (2 * K - 2));
            } else {
                f.hi = ((f.hi << 2) | (f.lo >> 62)) & mask_hi;
                f.lo = (f.lo << 2) | c;
                r.lo = (r.lo >> 2) | (r.hi << 62);
                r.hi = (r.hi >> 2) | ((3 - c) << (2 * K - 66));
            }
        }
        __syncthreads();
        scan_ranges(S, nr);
        __syncthreads();
        const unsigned n = S.start[nr];
        if (tid == 0) {
            // pieces begin at even keys: 16-byte aligned
            S.base = atomicAdd(&x.meta->cursor, (n + 1) & ~1u);
            x.piece[row] = S.base;
        }
        for (unsigned i = tid; i <= nr; i += NT)
            x.starts[(uint64_t)i * x.n_chunks + row] = (uint16_t)S.start[i];
#pragma unroll
        for (int i = 0; i < PER; ++i)
            if (br[i] != kNoKey)
                store_key<KW>(S.keys, S.start[br[i] >> 16] + (br[i] & 0xffffu), key[i]);
        __syncthreads();
        copy_out<KW, CHUNK, NT>(S, n, x.out + (uint64_t)S.base * KW);
        // S.keys is written again after the next chunk's barriers
    }
}

// ---------------------------------------------------------- runs of keys
// Brings runs of keys together in shared memory.  Run r (r < n) begins at key
// src[r] of `from` and its keys come to positions pos[r], pos[r + 1] - 1 less
// p0 of dst; only positions in [p0, p1) are copied.  Four to sixteen lanes a run,
// so a warp reads several runs of a sector or two at once; the copies are
// asynchronous (cp.async), so that each thread has many in flight.  ref: where
// not null, receives every copied key's place in `from`.
template <int KW>
__device__ __forceinline__ void copy_key_async(uint64_t *dst, const uint64_t *src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if (KW == 1)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}

__device__ __forceinline__ void copies_done() {
    asm volatile("cp.async.wait_all;" ::: "memory");
}

template <int KW, int NT>
__device__ __forceinline__ void gather_runs(const uint64_t *from, const unsigned *src,
                                            const unsigned *pos, unsigned n, unsigned p0,
                                            unsigned p1, uint64_t *dst, unsigned *ref = nullptr) {
    // as many lanes as nearly every run fills
    const unsigned ls = (p1 - p0) < 8 * n ? 2 : (p1 - p0) < 24 * n ? 3 : 4, step = 1u << ls;
    const unsigned sub = threadIdx.x & (step - 1);
    for (unsigned r = threadIdx.x >> ls; r < n; r += NT >> ls) {
        const unsigned b = pos[r], lo = max(b, p0), hi = min(pos[r + 1], p1);
        const uint64_t s0 = src[r];
        for (unsigned q = lo + sub; q < hi; q += step) {
            copy_key_async<KW>(dst + (uint64_t)(q - p0) * KW, from + (s0 + (q - b)) * KW);
            if (ref) ref[q - p0] = (unsigned)(s0 + (q - b));
        }
    }
}

// ------------------------------------------------------ 3. second level
// Row b of the range starts: prefix[b][c] = keys of range b in pieces before
// piece c; totals[b] = all of them.
__global__ void __launch_bounds__(1024) row_prefix_kernel(const uint16_t *starts, unsigned n_chunks,
                                                          uint32_t *prefix, uint32_t *totals) {
    const uint16_t *r0 = starts + (uint64_t)blockIdx.x * n_chunks, *r1 = r0 + n_chunks;
    uint32_t *out = prefix + (uint64_t)blockIdx.x * n_chunks;
    unsigned carry = 0;
    for (unsigned c0 = 0; c0 < n_chunks; c0 += 4096) {
        unsigned v[4], sum = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const unsigned c = c0 + threadIdx.x * 4 + j;
            v[j] = c < n_chunks ? (unsigned)r1[c] - r0[c] : 0u;
            sum += v[j];
        }
        unsigned tot;
        unsigned pre = block_exclusive_scan<unsigned, 1024>(sum, tot) + carry;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const unsigned c = c0 + threadIdx.x * 4 + j;
            if (c < n_chunks) out[c] = pre;
            pre += v[j];
        }
        carry += tot;
    }
    if (threadIdx.x == 0) totals[blockIdx.x] = carry;
}

// Tile t covers kRefineTile consecutive keys of one range; its range, its
// place among the range's tiles and the piece that its first key is in.
__global__ void __launch_bounds__(1024) tile_map_kernel(const uint32_t *totals, unsigned n_ranges,
                                                        const uint32_t *prefix, unsigned n_chunks,
                                                        uint32_t *tile_base, TileMap *map,
                                                        DedupMeta *meta) {
    __shared__ unsigned base[kMaxRanges + 1];
    const unsigned tid = threadIdx.x;
    const unsigned v = tid < n_ranges ? (totals[tid] + kRefineTile - 1) / kRefineTile : 0u;
    unsigned tot;
    const unsigned pre = block_exclusive_scan<unsigned, 1024>(v, tot);
    if (tid < n_ranges) base[tid] = pre;
    if (tid == 0) base[n_ranges] = tot;
    __syncthreads();
    if (blockIdx.x == 0) {
        for (unsigned i = tid; i <= n_ranges; i += 1024) tile_base[i] = base[i];
        if (tid == 0) meta->n_tiles = tot;
    }
    const unsigned t = blockIdx.x * 1024 + tid;
    if (t >= tot) return;
    unsigned lo = 0, hi = n_ranges - 1;   // the last range whose tiles begin at or before t
    while (lo < hi) {
        const unsigned m = (lo + hi + 1) / 2;
        if (base[m] <= t)
            lo = m;
        else
            hi = m - 1;
    }
    const uint32_t *row = prefix + (uint64_t)lo * n_chunks;
    const unsigned p = (t - base[lo]) * kRefineTile;
    unsigned a = 0, b = n_chunks - 1;   // the last piece with prefix <= p holds key p
    while (a < b) {
        const unsigned m = a + (b - a + 1) / 2;
        if (row[m] <= p)
            a = m;
        else
            b = m - 1;
    }
    map[t].range = lo;
    map[t].piece = a;
}

// Splitters of the fine ranges inside range b: keys of random places of
// random pieces' runs.  One block per range.  Prefixes alone, unless kCrowd
// neighbouring splitters are equal: then half as many samples of whole keys, in the
// same shared memory.  (A prefix of fewer ranges' windows is left together, to
// dedup_big_kernel's few rounds: 2.8e8 windows of copied repeats have many of them,
// and sorting whole keys at two equal ones took 910 instead of 500 us there.)
template <int KW, int E>
__global__ void __launch_bounds__(1024) fine_splitters_kernel(RefineArgs x, int K, unsigned n,
                                                              uint64_t last) {
    extern __shared__ ulonglong2 s2[];
    __shared__ unsigned valid;
    uint64_t *const s = (uint64_t *)s2;
    const unsigned b = blockIdx.x, j = threadIdx.x;
    if (j == 0) valid = 0;
    __syncthreads();
    const uint64_t lo = b ? x.spl[b - 1] : 0;
    const uint64_t hi = b + 1 < x.n_ranges ? x.spl[b] : last;
    const auto draw = [&](unsigned i, Key<KW> &k) {
        for (unsigned t = 0; t < 4; ++t) {
            const uint64_t z = mix64(((uint64_t)b << 32) | (i * 4 + t));
            const unsigned c = (unsigned)__umul64hi(z, (uint64_t)x.n_chunks);
            const unsigned s0 = x.starts[(uint64_t)b * x.n_chunks + c];
            const unsigned m = x.starts[(uint64_t)(b + 1) * x.n_chunks + c] - s0;
            if (!m) continue;
            const unsigned o = (unsigned)(((z & 0xffffffffu) * m) >> 32);
            k = load_key<KW>(x.in, (uint64_t)x.piece[c] + s0 + o);
            return 1u;
        }
        return 0u;
    };
    // as many ranges as this one's windows fill, so that only the fine samples
    // spread the sizes; the others stay empty (all-ones splitters)
    const unsigned nf = max(1u, min(x.n_fine, (x.totals[b] + x.target - 1) / x.target));
    uint64_t f = ~0ull, f_lo = ~0ull;
    {
        uint64_t v[E];
        unsigned found = 0;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            Key<KW> k;
            v[e] = ~0ull;
            if (e * 1024 + j < n && draw(e * 1024 + j, k)) {
                v[e] = prefix_of<KW>(k, K);
                ++found;
            }
        }
        if (found) atomicAdd(&valid, found);
        block_sort<E>(v, s);
        __syncthreads();
#pragma unroll
        for (int e = 0; e < E; ++e) s[j * E + e] = v[e];
    }
    __syncthreads();
    const unsigned used = valid ? nf - 1 : 0;   // splitters
    bool tie = false;
    if constexpr (KW == 1) {
        part_equal<1>(
            [&](unsigned i, uint64_t &p, uint64_t &) { p = s[(uint64_t)(i + 1) * valid / nf]; }, j, used,
            f, f_lo, K);
    } else {
        constexpr int E2 = (E < 4 ? 4 : E) / 2;
        bool same = false;
        if (j < used) {
            f = s[(uint64_t)(j + 1) * valid / nf];
            f_lo = 0;
            same = j + kCrowd < nf && f == s[(uint64_t)(j + kCrowd) * valid / nf];
        }
        if (__syncthreads_or(same)) {
            if (j == 0) valid = 0;
            __syncthreads();
            Cut2 v[E2], *const c = (Cut2 *)s2;
            unsigned found = 0;
#pragma unroll
            for (int e = 0; e < E2; ++e) {
                Key<KW> k;
                largest_sample(v[e]);
                if (e * 1024 + j < n && draw(e * 1024 + j, k)) {
                    v[e] = sample_of(k, K);
                    ++found;
                }
            }
            if (found) atomicAdd(&valid, found);
            block_sort<E2>(v, c);
            __syncthreads();
#pragma unroll
            for (int e = 0; e < E2; ++e) c[j * E2 + e] = v[e];
            __syncthreads();
            tie = part_equal<2>(
                [&](unsigned i, uint64_t &p, uint64_t &low) {
                    const Cut2 at = c[(uint64_t)(i + 1) * valid / nf];
                    p = at.p;
                    low = at.lo;
                },
                j, valid ? nf - 1 : 0, f, f_lo, K);
            tie = shares_prefix(s, j, valid ? nf - 1 : 0, f) || tie;
            if (!tie && valid && j + 1 < nf) f_lo = 0;
        }
        if (j < x.n_fine) x.fine_lo[(uint64_t)b * kMaxRanges + j] = f_lo;
    }
    if (j < x.n_fine) x.fine_spl[(uint64_t)b * kMaxRanges + j] = f;
    __syncthreads();
    write_lut<KW>((unsigned *)s, f, tie, valid != 0, nf, lo, hi, x.fine_lut + (uint64_t)b * kLutStride);
}

// One tile of a range: gather its keys from the pieces, group them by fine
// range in shared memory, write them as one contiguous tile with the fine
// ranges' starts in a table.
template <int KW>
struct __align__(16) RefineSmem {
    GroupSmem<KW, kRefineTile> g;
    unsigned src[kRefineThreads];
    unsigned pos[kRefineThreads + 1];
};

template <int KW>
__global__ void __launch_bounds__(kRefineThreads, 2) refine_kernel(RefineArgs x, int K,
                                                                   uint64_t last) {
    constexpr int NT = kRefineThreads;
    constexpr int PER = kRefineTile / NT;
    extern __shared__ __align__(16) unsigned char dyn[];
    RefineSmem<KW> &S = *reinterpret_cast<RefineSmem<KW> *>(dyn);
    __shared__ unsigned more;
    const unsigned tid = threadIdx.x, nf = x.n_fine;
    const unsigned nt = x.meta->n_tiles;
    // consecutive tiles per block, so that a range's splitters are loaded once
    const unsigned t_begin = (unsigned)((uint64_t)nt * blockIdx.x / gridDim.x);
    const unsigned t_end = (unsigned)((uint64_t)nt * (blockIdx.x + 1) / gridDim.x);
    unsigned cur = ~0u;
    uint64_t lo = 0;
    int sh = 0;
    for (unsigned t = t_begin; t < t_end; ++t) {
        const TileMap tm = x.map[t];
        const unsigned b = tm.range;
        if (b != cur) {
            __syncthreads();
            for (unsigned i = tid; i < nf; i += NT)
                S.g.spl[i] = x.fine_spl[(uint64_t)b * kMaxRanges + i];
            for (unsigned i = tid; i < kLutStride / 8; i += NT)
                ((uint4 *)S.g.lut)[i] = ((const uint4 *)(x.fine_lut + (uint64_t)b * kLutStride))[i];
            lo = b ? x.spl[b - 1] : 0;
            sh = bit_len((b + 1 < x.n_ranges ? x.spl[b] : last) - lo) - kLutBits;
            if (sh < 0) sh = 0;
            cur = b;
        }
        const unsigned local = t - x.tile_base[b];
        const unsigned p0 = local * kRefineTile;
        const unsigned n = min((unsigned)kRefineTile, x.totals[b] - p0);
        const uint32_t *row = x.prefix + (uint64_t)b * x.n_chunks;
        const uint16_t *st0 = x.starts + (uint64_t)b * x.n_chunks, *st1 = st0 + x.n_chunks;
        for (unsigned i = tid; i < nf + 128; i += NT) S.g.hist[i] = 0;
        for (unsigned c0 = tm.piece;; c0 += NT) {
            const unsigned c = c0 + tid;
            unsigned p = ~0u, e = ~0u;   // past the last piece: nothing to copy
            if (c < x.n_chunks) {
                const unsigned s0 = st0[c];
                p = row[c];
                e = p + st1[c] - s0;
                S.src[tid] = x.piece[c] + s0;
            }
            S.pos[tid] = p;
            if (tid == NT - 1) {
                S.pos[NT] = e;
                more = e < p0 + n;   // the tile goes on in the next pieces
            }
            __syncthreads();
            const unsigned nr = min((unsigned)NT, x.n_chunks - c0);
            if (tid == 0 && nr < NT) S.pos[nr] = x.totals[b];
            __syncthreads();
            gather_runs<KW, NT>(x.in, S.src, S.pos, nr, p0, p0 + n, S.g.keys);
            const bool again = more != 0;
            __syncthreads();
            if (!again) break;
        }
        copies_done();
        __syncthreads();
        Key<KW> key[PER];
        unsigned br[PER];
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            const unsigned i = q * NT + tid;
            br[q] = kNoKey;
            if (i < n) {
                key[q] = load_key<KW>(S.g.keys, i);
                const unsigned bin = find_range<KW>(
                    S.g.spl, [&](unsigned m) { return __ldg(x.fine_lo + (uint64_t)b * kMaxRanges + m); },
                    S.g.lut, nf, lo, sh, prefix_of<KW>(key[q], K), key[q].lo);
                br[q] = (bin << 16) | atomicAdd(&S.g.hist[bin], 1u);
            }
        }
        __syncthreads();
        scan_ranges(S.g, nf);
        __syncthreads();
        const uint64_t tiles_b = x.tile_base[b + 1] - x.tile_base[b];
        uint16_t *fs = x.fine_starts + (uint64_t)x.tile_base[b] * (nf + 1) + local;
        for (unsigned i = tid; i <= nf; i += NT) fs[i * tiles_b] = (uint16_t)S.g.start[i];
#pragma unroll
        for (int q = 0; q < PER; ++q)
            if (br[q] != kNoKey)
                store_key<KW>(S.g.keys, S.g.start[br[q] >> 16] + (br[q] & 0xffffu), key[q]);
        __syncthreads();
        copy_out<KW, kRefineTile, NT>(S.g, n, x.out + (uint64_t)t * kRefineTile * KW);
        __syncthreads();
    }
}

// -------------------------------------------------------------- 4. dedup
// A final range as its block reads it: its runs, one in every piece (one level)
// or in every tile of its coarse range (two levels), and this thread's run of the
// first NT.
struct RangeRuns {
    const uint16_t *row0;
    unsigned n_runs, first;
    unsigned src, n;

    __device__ __forceinline__ void load_run(const DedupArgs &x, unsigned r) {
        src = n = 0;
        if (r < n_runs) {
            const unsigned s0 = row0[r];
            n = (unsigned)row0[(uint64_t)n_runs + r] - s0;
            src = (x.n_fine ? (first + r) * (unsigned)kRefineTile : x.piece[r]) + s0;
        }
    }
    __device__ __forceinline__ void load(const DedupArgs &x, unsigned g) {
        first = 0;
        if (x.n_fine) {
            const unsigned b = g / x.n_fine, f = g % x.n_fine;
            first = x.tile_base[b];
            n_runs = x.tile_base[b + 1] - first;
            row0 = x.starts + (uint64_t)first * (x.n_fine + 1) + (uint64_t)f * n_runs;
        } else {
            n_runs = x.n_chunks;
            row0 = x.starts + (uint64_t)g * n_runs;
        }
        load_run(x, threadIdx.x);
    }
};

// How a range's keys are cut evenly into kSubBins2: by their prefixes, or by their
// low words where all of them have one prefix.  One thread finds it out and leaves it
// in shared memory while the block gathers the range (every thread waiting for the
// bounds took 4% of dedup_kernel).
struct RangeCut {
    uint64_t base;     // the smallest prefix (or low word) there can be
    int sh;            // kSubBits2 bits of the difference to it make a cut
    uint16_t by_low, pure;   // pure: the range is one key, whose cut is lo, lo2
    uint64_t lo, lo2;
};

template <int KW>
__device__ __forceinline__ RangeCut range_cut(const DedupArgs &x, unsigned g, int K, uint64_t last) {
    // the range's bounds: prefixes, and of two-word keys the low words
    uint64_t lo = 0, hi = last, lo2 = 0, hi2 = ~0ull;
    bool open = false;   // hi is a splitter: the range ends in front of it
    const auto below = [&](const uint64_t *p, const uint64_t *rest, uint64_t i) {
        lo = p[i];
        if (KW == 2) lo2 = rest[i];
    };
    const auto above = [&](const uint64_t *p, const uint64_t *rest, uint64_t i) {
        const uint64_t v = p[i], w = KW == 2 ? rest[i] : 0;
        // unused splitters are all ones: the last range in use ends where its coarse one
        // does (taken for all the key space, its keys fall into one cut and the block
        // sorts them by the whole bitonic network)
        if (v < hi || (KW == 2 && v == hi && w < hi2)) {
            hi = v;
            hi2 = w;
            open = true;
        }
    };
    if (x.n_fine) {
        const unsigned b = g / x.n_fine, f = g % x.n_fine;
        const uint64_t fs = (uint64_t)b * kMaxRanges + f;
        if (f)
            below(x.fine_spl, x.fine_lo, fs - 1);
        else if (b)
            below(x.spl, x.spl_lo, b - 1);
        if (b + 1 < x.n_ranges) above(x.spl, x.spl_lo, b);
        if (f + 1 < x.n_fine) above(x.fine_spl, x.fine_lo, fs);
    } else {
        if (g) below(x.spl, x.spl_lo, g - 1);
        if (g + 1 < x.n_ranges) above(x.spl, x.spl_lo, g);
    }
    RangeCut c;
    c.by_low = KW == 2 && lo == hi ? 1 : 0;
    c.base = c.by_low ? lo2 : lo;
    c.sh = max(bit_len(c.by_low ? hi2 - lo2 : hi - lo) - kSubBits2, 0);
    c.lo = lo;
    c.lo2 = lo2;
    if (open)
        c.pure = next_cut<KW>(lo, lo2, K) && lo == hi && (KW == 1 || lo2 == hi2);
    else
        c.pure = lo == last && (KW == 1 || lo2 == ~0ull);
    return c;
}

template <int KW>
__device__ __forceinline__ unsigned cut_of(const RangeCut &c, const Key<KW> &k, int K) {
    const uint64_t v = KW == 2 && c.by_low ? k.lo : prefix_of<KW>(k, K);
    return min((unsigned)((v - c.base) >> c.sh), (unsigned)kSubBins2 - 1);
}

template <int KW>
__device__ __forceinline__ unsigned key_hash(const Key<KW> &k) {
    uint64_t x = k.lo;
    if (KW == 2) x ^= rotl64(k.hi, 23) * kMurC2;
    return (unsigned)((x * 0x9E3779B97F4A7C15ull) >> 32);
}

constexpr unsigned kRankLimit = 96;     // cuts of up to this many keys are rank sorted

// Exclusive prefix of sub[0, kSubBins2) in place; most: the thread's largest count.
template <int NT>
__device__ __forceinline__ void scan_cuts(unsigned *sub, unsigned &most) {
    constexpr unsigned E = (kSubBins2 + NT - 1) / NT;
    unsigned v[E], sum = 0;
    most = 0;
#pragma unroll
    for (unsigned j = 0; j < E; ++j) {
        const unsigned i = threadIdx.x * E + j;
        v[j] = i < (unsigned)kSubBins2 ? sub[i] : 0u;
        sum += v[j];
        most = max(most, v[j]);
    }
    unsigned tot;
    unsigned pre = block_exclusive_scan<unsigned, NT>(sum, tot);
#pragma unroll
    for (unsigned j = 0; j < E; ++j) {
        const unsigned i = threadIdx.x * E + j;
        if (i < (unsigned)kSubBins2) sub[i] = pre;
        pre += v[j];
    }
}

// Sorts n places (uint16) by the keys key_of gives them: a bitonic network for
// any length (every compare-exchange puts the smaller key first, partners past
// the end are skipped).  For ranges whose keys crowd into few cuts.
template <int NT, typename F>
__device__ __forceinline__ void bitonic_places(uint16_t *ord, unsigned n, F key_of) {
    unsigned P = 2;
    while (P < n) P <<= 1;
    for (unsigned k = 2; k <= P; k <<= 1) {
        for (unsigned j = k >> 1; j > 0; j >>= 1) {
            for (unsigned p = threadIdx.x; p < P / 2; p += NT) {
                unsigned i, y;
                if (j == (k >> 1)) {   // the flip: i against its mirror in the k-block
                    const unsigned blk = p / j, off = p % j;
                    i = blk * k + off;
                    y = blk * k + (k - 1 - off);
                } else {
                    i = (p / j) * 2 * j + (p % j);
                    y = i + j;
                }
                if (y < n) {
                    const uint16_t u = ord[i], v = ord[y];
                    if (key_of(v) < key_of(u)) {
                        ord[i] = v;
                        ord[y] = u;
                    }
                }
            }
            __syncthreads();
        }
    }
}

// A block takes one final range at a time.  The range's windows are gathered
// into shared memory (stage) and equal keys are found without atomics: every
// window writes its place to its key's slot of a table, and after a barrier
// looks whose place is there.  Equal key: that window stands for both, and its
// count goes up.  Another key's: all windows of this key go on to the next free
// slot together, in a further round.  Nearly all settle in the first round,
// whose reads and writes have no chain between them (compare-and-swap probing
// took 1,500 cycles a window and thread, three round trips a probe); the others
// are listed first, so that the rounds take little.  The
// windows that stand for their key are ordered by a counting sort on an even
// cut of the range and ranked inside the cuts; only 16-bit places move.  Four
// blocks share an SM, and the next range's runs are looked up while this one is
// sorted.  Ranges of more windows than the stage, or too many
// unsettled ones, are listed for dedup_big_kernel.
template <int KW>
struct __align__(16) SmallSmem {
    uint64_t stage[kStage<KW> * KW];
    uint16_t table[kTableSlots];     // then the places in key order
    unsigned cnt[kStage<KW>];
    uint16_t list[kStage<KW>];       // places that stand for their keys
    uint16_t left[kMaxLeft], probe[kMaxLeft];   // unsettled places, and their slots
    unsigned sub[kSubBins2];
    unsigned src[kSmallThreads];
    unsigned pos[kSmallThreads + 1];
    unsigned lists, crowded, out0;   // lists: entries of left above, of list below
    RangeCut cut;
};

constexpr unsigned kNoPlace = 0xffffu;

template <int KW>
__global__ void __launch_bounds__(kSmallThreads, 4) dedup_kernel(DedupArgs x, int K) {
    constexpr int NT = kSmallThreads, Q = kStage<KW> / NT;
    static_assert(kStage<KW> % NT == 0 && kStage<KW> < (int)kTableSlots, "whole rounds, free slots");
    extern __shared__ __align__(16) unsigned char dyn[];
    SmallSmem<KW> &S = *reinterpret_cast<SmallSmem<KW> *>(dyn);
    const unsigned tid = threadIdx.x;
    const uint64_t last = K >= 32 ? ~0ull : (1ull << (2 * K)) - 1;
    RangeRuns next;
    if (blockIdx.x < x.n_total) next.load(x, blockIdx.x);
    for (unsigned g = blockIdx.x; g < x.n_total; g += gridDim.x) {
        const RangeRuns cur = next;
        // all windows of the range
        unsigned n = cur.n;
        for (unsigned r = NT + tid; r < cur.n_runs; r += NT)
            n += (unsigned)cur.row0[(uint64_t)cur.n_runs + r] - cur.row0[r];
        unsigned pre = block_exclusive_scan<unsigned, NT>(n, n);
        if (n == 0 || n > (unsigned)kStage<KW>) {
            if (tid == 0) {
                if (n)
                    x.big[atomicAdd(&x.meta->n_big, 1u)] = g;
                else
                    x.counts[g] = 0;
            }
            if (g + gridDim.x < x.n_total) next.load(x, g + gridDim.x);
            continue;
        }
        for (unsigned r0 = 0, m0 = 0; r0 < cur.n_runs; r0 += NT) {
            RangeRuns seg = cur;
            if (cur.n_runs > NT) {
                if (r0) seg.load_run(x, r0 + tid);
                unsigned m;
                pre = m0 + block_exclusive_scan<unsigned, NT>(seg.n, m);
                m0 += m;
            } else {
                m0 = n;
            }
            S.src[tid] = seg.src;
            S.pos[tid] = pre;
            if (tid == 0) S.pos[NT] = m0;
            __syncthreads();
            gather_runs<KW, NT>(x.in, S.src, S.pos, min((unsigned)NT, cur.n_runs - r0), 0u, n, S.stage);
            if (cur.n_runs > NT) __syncthreads();
        }
        {
            const uint4 none = make_uint4(~0u, ~0u, ~0u, ~0u);
            for (unsigned i = tid; i < kTableSlots / 8; i += NT) ((uint4 *)S.table)[i] = none;
            for (unsigned i = tid; i < (unsigned)kSubBins2; i += NT) S.sub[i] = 0;
            if (tid == 0) {
                S.lists = S.crowded = 0;
                if (x.ordered) S.cut = range_cut<KW>(x, g, K, last);
            }
        }
        copies_done();
        __syncthreads();
        unsigned slot[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const unsigned i = q * NT + tid;
            slot[q] = 0;
            if (i < n) {
                slot[q] = __umulhi(key_hash(load_key<KW>(S.stage, i)), kTableSlots);
                S.table[slot[q]] = (uint16_t)i;
                S.cnt[i] = 0;
            }
        }
        __syncthreads();
        unsigned rep = 0, left = 0;   // bit q: window q stands for its key / is not settled
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const unsigned i = q * NT + tid;
            if (i < n) {
                const unsigned w = S.table[slot[q]];
                if (w == i || load_key<KW>(S.stage, w) == load_key<KW>(S.stage, i)) {
                    atomicAdd(&S.cnt[w], 1u);
                    rep |= (w == i ? 1u : 0u) << q;
                } else {
                    left |= 1u << q;
                }
            }
        }
        // the windows that stand for their keys and the unsettled ones, listed: what
        // follows touches no others
        {
            const unsigned mine = __popc(left) << 16 | __popc(rep);
            unsigned upto = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned y = __shfl_up_sync(0xffffffffu, upto, o);
                if ((tid & 31) >= (unsigned)o) upto += y;
            }
            unsigned first = 0;
            if ((tid & 31) == 31) first = atomicAdd(&S.lists, upto);
            first = __shfl_sync(0xffffffffu, first, 31) + upto - mine;
            unsigned a = first & 0xffffu, b = first >> 16;
            for (; rep; rep &= rep - 1) S.list[a++] = (uint16_t)((__ffs(rep) - 1) * NT + tid);
            for (; left && b < kMaxLeft; left &= left - 1, ++b) {
                S.left[b] = (uint16_t)((__ffs(left) - 1) * NT + tid);
                S.probe[b] = kNoPlace;
            }
        }
        __syncthreads();
        const unsigned n_left = S.lists >> 16;
        if (n_left > kMaxLeft) {   // a crowded table: the other kernel's
            if (tid == 0) x.big[atomicAdd(&x.meta->n_big, 1u)] = g;
            if (g + gridDim.x < x.n_total) next.load(x, g + gridDim.x);
            __syncthreads();
            continue;
        }
        for (bool any = n_left != 0; any;) {
            // a further round: every window of a key sees the same table and takes
            // the same free slot
            for (unsigned p = tid; p < n_left; p += NT) {
                const unsigned i = S.left[p];
                if (i == kNoPlace) continue;   // settled
                unsigned t = S.probe[p];
                if (t == kNoPlace) t = __umulhi(key_hash(load_key<KW>(S.stage, i)), kTableSlots);
                do {
                    t = (t + 1) & (kTableSlots - 1);
                } while (S.table[t] != kNoPlace);
                S.probe[p] = (uint16_t)t;
            }
            __syncthreads();
            for (unsigned p = tid; p < n_left; p += NT)
                if (S.left[p] != kNoPlace) S.table[S.probe[p]] = S.left[p];
            __syncthreads();
            bool mine = false;
            for (unsigned p = tid; p < n_left; p += NT) {
                const unsigned i = S.left[p];
                if (i == kNoPlace) continue;
                const unsigned w = S.table[S.probe[p]];
                if (w == i || load_key<KW>(S.stage, w) == load_key<KW>(S.stage, i)) {
                    atomicAdd(&S.cnt[w], 1u);
                    if (w == i) S.list[atomicAdd(&S.lists, 1u) & 0xffffu] = (uint16_t)i;
                    S.left[p] = kNoPlace;
                } else {
                    mine = true;
                }
            }
            any = __syncthreads_or(mine);
        }
        if (g + gridDim.x < x.n_total) next.load(x, g + gridDim.x);
        const unsigned nd = S.lists & 0xffffu;
        if (!x.ordered) {
            if (tid == 0) S.out0 = atomicAdd(&x.meta->out_cursor, nd);
            __syncthreads();
            for (unsigned p = tid; p < nd; p += NT) {
                const unsigned i = S.list[p];
                store_key<KW>(x.out, S.out0 + p, load_key<KW>(S.stage, i));
                x.mult[S.out0 + p] = S.cnt[i];
            }
            __syncthreads();
            continue;
        }
        // their order
        const RangeCut cut = S.cut;
        for (unsigned p = tid; p < nd; p += NT)
            atomicAdd(&S.sub[cut_of(cut, load_key<KW>(S.stage, S.list[p]), K)], 1u);
        if (tid == 0) {
            S.out0 = atomicAdd(&x.meta->out_cursor, nd);
            x.places[g] = S.out0;
            x.counts[g] = nd;
        }
        __syncthreads();
        unsigned most;
        scan_cuts<NT>(S.sub, most);
        if (most > kRankLimit) S.crowded = 1;
        __syncthreads();
        uint16_t *ord = S.table;   // the table is done with
        for (unsigned p = tid; p < nd; p += NT) {
            const unsigned i = S.list[p];
            const unsigned c = cut_of(cut, load_key<KW>(S.stage, i), K);
            ord[atomicAdd(&S.sub[c], 1u)] = (uint16_t)i;
        }
        __syncthreads();
        const uint64_t at = S.out0;
        const bool crowded = S.crowded != 0;
        if (crowded)
            bitonic_places<NT>(ord, nd, [&](unsigned i) { return load_key<KW>(S.stage, i); });
        for (unsigned p = tid; p < nd; p += NT) {
            const unsigned i = ord[p];
            const Key<KW> k = load_key<KW>(S.stage, i);
            unsigned rk = p;
            if (!crowded) {   // a cut's keys end at its cursor and begin at the one before
                const unsigned c = cut_of(cut, k, K);
                const unsigned a0 = c ? S.sub[c - 1] : 0u, a1 = S.sub[c];
                if (a1 - a0 > 1) {
                    rk = a0;
                    for (unsigned j = a0; j < a1; ++j)
                        rk += load_key<KW>(S.stage, ord[j]) < k ? 1u : 0u;
                }
            }
            store_key<KW>(x.out, at + rk, k);
            x.mult[at + rk] = S.cnt[i];
        }
        __syncthreads();
    }
}

// Ranges of any number of windows, batch by batch: every thread puts keys into
// an open-addressing table, which counts them; whoever puts a key there first
// appends its slot to a list, and everything after works on the list.  A range
// with more distinct keys than the table takes is handled in rounds over
// sub-ranges [lo, hi) of it: a round that overflows stops, and begins again up to
// the median of up to 32 of the keys in the table (so it leaves some of them out,
// and the rounds end); a round that succeeds goes on to the bound before.  D keys
// take about 4 D / slots rounds, half of them broken off.
constexpr unsigned kBoundsMax = 16;
template <int KW>
struct __align__(16) DedupSmem {
    static constexpr int SLOTS = kDedupSlots<KW>;
    uint64_t stage[kDedupStage<KW> * KW];   // a batch of windows; then uint16 slots in key order
    uint64_t slot[SLOTS];            // one-word keys: the key; two-word keys: hash and place
    unsigned ref[KW == 2 ? kDedupStage<KW> : 1];   // two-word keys: places of the batch's windows
    unsigned cnt[SLOTS];
    uint16_t list[SLOTS];            // slots in the order they were taken
    unsigned sub[kSubBins2];         // keys per cut, then the cuts' cursors
    unsigned src[kDedupThreads];     // runs: first key
    unsigned pos[kDedupThreads + 1]; // and place among the range's windows
    unsigned nd, over, crowded, ones, out0, cut;
    RangeCut cut_by;
    Key<KW> pivot;
    Key<KW> bounds[kBoundsMax];      // the rounds' ends to come, the nearest last
};
static_assert(kDedupSlots<1> * 2 <= kDedupStage<1> * 8 && kDedupSlots<2> * 2 <= kDedupStage<2> * 16,
              "the slots in key order take the batch's place");

constexpr uint64_t kFree = ~0ull;
constexpr int kProbeMax = 192;          // probes after which the table counts as full

// The key in a slot: of two-word keys, where it stands in the input.
__device__ __forceinline__ Key<1> table_key(const DedupSmem<1> &S, const uint64_t *, unsigned slot) {
    return Key<1>{S.slot[slot], 0};
}
__device__ __forceinline__ Key<2> table_key(const DedupSmem<2> &S, const uint64_t *in, unsigned slot) {
    return load_key<2>(in, (unsigned)S.slot[slot]);
}

// Counts one window's key, key `at` of the input.  One-word keys are claimed
// whole with a 64-bit compare-and-swap.  Two-word keys claim a slot with their
// hash and their place in the input, and are compared there (the range is in
// L1), so that no thread waits for another to finish writing a key.
template <int KW>
__device__ __forceinline__ void table_add(DedupSmem<KW> &S, const Key<KW> &k, const uint64_t *in,
                                          unsigned at) {
    if (KW == 1 && k.lo == kFree) {   // 32-mers of T alone, forward strand
        atomicAdd(&S.ones, 1u);
        return;
    }
    const unsigned h = key_hash(k);
    const uint64_t want = KW == 1 ? k.lo : ((uint64_t)h << 32) | at;
    unsigned slot = __umulhi(h, (unsigned)kDedupSlots<KW>);
    for (int it = 0; it < kProbeMax; ++it) {
        unsigned long long *p = (unsigned long long *)S.slot + slot;
        unsigned long long v = *(volatile unsigned long long *)p;
        if (v == kFree) {
            v = atomicCAS(p, (unsigned long long)kFree, (unsigned long long)want);
            if (v == kFree) {
                S.list[atomicAdd(&S.nd, 1u)] = (uint16_t)slot;
                v = want;
            }
        }
        if (KW == 1 ? v == want
                    : (unsigned)(v >> 32) == h && (v == want || load_key<KW>(in, (unsigned)v) == k)) {
            atomicAdd(&S.cnt[slot], 1u);
            return;
        }
        if (++slot == (unsigned)kDedupSlots<KW>) slot = 0;
        if (it >= 16 && *(volatile unsigned *)&S.over) return;   // the round is lost anyway
    }
    S.over = 1;
}

template <int KW>
__global__ void __launch_bounds__(kDedupThreads, 3) dedup_big_kernel(DedupArgs x, int K) {
    constexpr int SLOTS = kDedupSlots<KW>, NT = kDedupThreads;
    extern __shared__ __align__(16) unsigned char dyn[];
    DedupSmem<KW> &S = *reinterpret_cast<DedupSmem<KW> *>(dyn);
    uint16_t *ord = (uint16_t *)S.stage;
    const unsigned tid = threadIdx.x;
    for (unsigned i = tid; i < (unsigned)SLOTS; i += NT) {
        S.slot[i] = kFree;
        S.cnt[i] = 0;
    }
    const uint64_t last = K >= 32 ? ~0ull : (1ull << (2 * K)) - 1;
    const unsigned n_big = x.meta->n_big;
    for (unsigned q = blockIdx.x; q < n_big; q += gridDim.x) {
        const unsigned g = x.big[q];
        RangeRuns cur;
        if (tid == 0) S.cut_by = range_cut<KW>(x, g, K, last);
        cur.load(x, g);
        unsigned n_all;   // windows of the range
        const unsigned pre0 = block_exclusive_scan<unsigned, NT>(cur.n, n_all);
        const unsigned m0 = n_all;
        if (cur.n_runs > NT) {
            unsigned n = 0;
            for (unsigned r = NT + tid; r < cur.n_runs; r += NT)
                n += (unsigned)cur.row0[(uint64_t)cur.n_runs + r] - cur.row0[r];
            block_exclusive_scan<unsigned, NT>(n, n);
            n_all += n;
        }
        if (S.cut_by.pure) {   // one key, however many windows
            __syncthreads();   // every thread has seen it
            if (tid == 0) {
                const RangeCut &cut = S.cut_by;
                const unsigned at = atomicAdd(&x.meta->out_cursor, 1u);
                Key<KW> k;
                k.lo = KW == 1 ? cut.lo : cut.lo2;
                k.hi = KW == 1 ? 0 : cut.lo >> (128 - 2 * K);
                store_key<KW>(x.out, at, k);
                x.mult[at] = n_all;
                if (x.ordered) {
                    x.places[g] = at;
                    x.counts[g] = 1;
                }
            }
            continue;
        }
        unsigned done = 0;    // distinct keys written
        unsigned depth = 0;   // bounds held
        Key<KW> lo, hi;
        lo.lo = lo.hi = 0;
        hi = lo;
        bool from = false, until = false;   // whether lo and hi bound this round
        bool first = true;
        for (bool again = true; again;) {
            __syncthreads();   // the last round's table is cleared
            if (tid == 0) S.nd = S.over = S.crowded = S.ones = 0;
            for (unsigned i = tid; i < (unsigned)kSubBins2; i += NT) S.sub[i] = 0;
            bool over = false;   // the same in every thread
            for (unsigned r0 = 0; r0 < cur.n_runs && !over; r0 += NT) {
                RangeRuns seg = cur;
                unsigned m = m0, pre = pre0;
                if (r0) {
                    seg.load_run(x, r0 + tid);
                    pre = block_exclusive_scan<unsigned, NT>(seg.n, m);
                }
                S.src[tid] = seg.src;
                S.pos[tid] = pre;
                if (tid == 0) S.pos[NT] = m;
                __syncthreads();
                const unsigned nr = min((unsigned)NT, cur.n_runs - r0);
                for (unsigned p0 = 0; p0 < m && !over; p0 += kDedupStage<KW>) {
                    const unsigned p1 = min(m, p0 + (unsigned)kDedupStage<KW>);
                    gather_runs<KW, NT>(x.in, S.src, S.pos, nr, p0, p1, S.stage,
                                        KW == 2 ? S.ref : nullptr);
                    if (first) {   // beside the first copies
                        first = false;
                        // the range's place in the output: room for all its windows
                        if (tid == 0 && x.ordered)
                            x.places[g] = S.out0 = atomicAdd(&x.meta->out_cursor, n_all);
                    }
                    copies_done();
                    __syncthreads();
                    for (unsigned i = tid; i < p1 - p0; i += NT) {
                        const Key<KW> k = load_key<KW>(S.stage, i);
                        if ((from && k < lo) || (until && !(k < hi))) continue;
                        table_add(S, k, x.in, KW == 2 ? S.ref[i] : 0u);
                    }
                    __syncthreads();
                    over = S.over != 0;   // written between the barriers around the additions
                }
            }
            const unsigned nd = S.nd;
            if (!over && !x.ordered) {
                const bool ones = KW == 1 && S.ones && !until;
                if (tid == 0) S.out0 = atomicAdd(&x.meta->out_cursor, nd + (ones ? 1u : 0u));
                __syncthreads();
                for (unsigned i = tid; i < nd; i += NT) {
                    const unsigned slot = S.list[i];
                    store_key<KW>(x.out, S.out0 + i, table_key(S, x.in, slot));
                    x.mult[S.out0 + i] = S.cnt[slot];
                }
                if (ones && tid == 0) {
                    x.out[S.out0 + nd] = ~0ull;
                    x.mult[S.out0 + nd] = S.ones;
                }
                again = until;
            } else if (!over) {
                const RangeCut cut = S.cut_by;
                for (unsigned i = tid; i < nd; i += NT) {
                    const Key<KW> k = table_key(S, x.in, S.list[i]);
                    atomicAdd(&S.sub[cut_of(cut, k, K)], 1u);
                }
                __syncthreads();
                unsigned most;
                scan_cuts<NT>(S.sub, most);
                if (most > kRankLimit) S.crowded = 1;
                __syncthreads();
                for (unsigned i = tid; i < nd; i += NT) {
                    const unsigned slot = S.list[i];
                    const Key<KW> k = table_key(S, x.in, slot);
                    ord[atomicAdd(&S.sub[cut_of(cut, k, K)], 1u)] = (uint16_t)slot;
                }
                __syncthreads();
                const uint64_t at = (uint64_t)S.out0 + done;
                if (!S.crowded) {
                    // a cut's keys end at its cursor and begin at the one before
                    for (unsigned i = tid; i < nd; i += NT) {
                        const unsigned slot = ord[i];
                        const Key<KW> k = table_key(S, x.in, slot);
                        const unsigned c = cut_of(cut, k, K);
                        const unsigned a0 = c ? S.sub[c - 1] : 0u, a1 = S.sub[c];
                        unsigned rk = a0;
                        if (a1 - a0 > 1)
                            for (unsigned j = a0; j < a1; ++j)
                                rk += table_key(S, x.in, ord[j]) < k ? 1u : 0u;
                        store_key<KW>(x.out, at + rk, k);
                        x.mult[at + rk] = S.cnt[slot];
                    }
                } else {
                    bitonic_places<NT>(ord, nd, [&](unsigned v) { return table_key(S, x.in, v); });
                    for (unsigned i = tid; i < nd; i += NT) {
                        const unsigned slot = ord[i];
                        store_key<KW>(x.out, at + i, table_key(S, x.in, slot));
                        x.mult[at + i] = S.cnt[slot];
                    }
                }
                done += nd;
                if (KW == 1 && S.ones && !until) {   // the largest key there is
                    if (tid == 0) {
                        x.out[at + nd] = ~0ull;
                        x.mult[at + nd] = S.ones;
                    }
                    ++done;
                }
                again = until;
            } else {
                // too many distinct keys: the round ends below the median of the
                // first keys found in 32 stretches of the table
                if (tid == 0) S.cut = 0;
                __syncthreads();
                if (tid < 32) {
                    const unsigned s0 = tid * (SLOTS / 32);
                    unsigned at = s0;
                    while (at < s0 + SLOTS / 32 && S.cnt[at] == 0) ++at;
                    const bool have = at < s0 + SLOTS / 32;
                    const unsigned held = __ballot_sync(0xffffffffu, have);
                    Key<KW> k;
                    k.lo = k.hi = 0;
                    if (have) k = table_key(S, x.in, at);
                    unsigned below = 0;
                    for (int j = 0; j < 32; ++j) {
                        Key<KW> o;
                        o.lo = __shfl_sync(0xffffffffu, k.lo, j);
                        o.hi = KW == 2 ? __shfl_sync(0xffffffffu, k.hi, j) : 0;
                        below += ((held >> j) & 1u) && o < k ? 1u : 0u;
                    }
                    if (have && below && below == (unsigned)__popc(held) / 2) {
                        S.pivot = k;
                        S.cut = 1;
                    }
                }
                __syncthreads();
                if (until && depth < kBoundsMax) {   // (else the rounds go on to the one before it)
                    if (tid == 0) S.bounds[depth] = hi;
                    ++depth;
                }
                hi = S.pivot;
                until = true;
                again = S.cut != 0;   // a full stretch of the table holds two keys at least
                if (!again && tid == 0) atomicOr(&x.ctr->error, kErrProbeLimit);
            }
            __syncthreads();
            if (!over && again) {   // on to the next bound
                lo = hi;
                from = true;
                until = depth != 0;
                if (until) hi = S.bounds[--depth];
            }
            for (unsigned i = tid; i < nd; i += NT) {
                const unsigned slot = S.list[i];
                S.slot[slot] = kFree;
                S.cnt[slot] = 0;
            }
        }
        if (tid == 0 && x.ordered) x.counts[g] = done;
    }
}

// offsets[g] = distinct keys in ranges before g, offsets[n] = all; one block.
__global__ void __launch_bounds__(1024) scan_counts_kernel(const uint32_t *counts, unsigned n,
                                                           uint32_t *offsets, DedupMeta *meta,
                                                           DevCounters *ctr, uint64_t list_cap) {
    constexpr unsigned E = 16;
    unsigned carry = 0;
    for (unsigned i0 = 0; i0 < n; i0 += 1024 * E) {
        unsigned v[E], sum = 0;
#pragma unroll
        for (unsigned j = 0; j < E; ++j) {
            const unsigned i = i0 + threadIdx.x * E + j;
            v[j] = i < n ? counts[i] : 0u;
            sum += v[j];
        }
        unsigned tot;
        unsigned pre = block_exclusive_scan<unsigned, 1024>(sum, tot) + carry;
#pragma unroll
        for (unsigned j = 0; j < E; ++j) {
            const unsigned i = i0 + threadIdx.x * E + j;
            if (i < n) offsets[i] = pre;
            pre += v[j];
        }
        carry += tot;
    }
    if (threadIdx.x == 0) {
        offsets[n] = carry;
        meta->distinct = carry;
        if (ctr) {
            ctr->distinct = carry;   // the list holds exactly these
            if (carry > list_cap) atomicOr(&ctr->error, kErrListFull);
        }
    }
}

// -------------------------------------------------------- 5. increments
// Walks distinct keys [begin, end) of the call in ascending order, EMIT_KEYS
// at a time: ranges hold their keys at places[g], numbered from offsets[g].
// win: a window of the offsets in shared memory.
constexpr unsigned kWin = 256;

// The range holding distinct key i (the last g with offsets[g] <= i).
__device__ __forceinline__ unsigned range_of(const uint32_t *offsets, unsigned n, unsigned i) {
    unsigned a = 0, b = n - 1;
    while (a < b) {
        const unsigned m = a + (b - a + 1) / 2;
        if (offsets[m] <= i)
            a = m;
        else
            b = m - 1;
    }
    return a;
}

// Loads offsets [g0, g0 + kWin] and places of those ranges into shared memory.
template <int NT>
__device__ __forceinline__ void load_window(const EmitArgs &e, unsigned g0, unsigned *off,
                                            unsigned *plc) {
    for (unsigned i = threadIdx.x; i <= kWin; i += NT) {
        const unsigned g = g0 + i;
        off[i] = g <= e.n_total ? e.offsets[g] : ~0u;
        if (i < kWin) plc[i] = g < e.n_total ? e.places[g] : 0u;
    }
}

// Where key i of the call is in e.keys / e.mult, for i inside the window.
__device__ __forceinline__ uint64_t place_in(const unsigned *off, const unsigned *plc, unsigned i) {
    unsigned a = 0, b = kWin - 1;
    while (a < b) {
        const unsigned m = (a + b + 1) / 2;
        if (off[m] <= i)
            a = m;
        else
            b = m - 1;
    }
    return (uint64_t)plc[a] + (i - off[a]);
}

// Partitioned update: one 32-bit code per (distinct key, hash), the cell
// within its coarse region, the counter within the cell and the increment
// less one; the codes of a chunk of keys are grouped by region in shared
// memory and appended to the regions' buffers, one cursor atomic per region.
// Codes that do not fit, and increments above a code's largest, are added to
// the countBF directly.
constexpr int kEmitThreads = 256;

// H hashes of PER keys a thread are in registers at a time: two of four, or, where
// three divide the hashes of a key, three of three, so that no pass over the
// regions is half empty (two-dimensional countBF, three hashes, 1.2e8 windows: a whole
// pass 4.60 -> 4.55 ms; of two-word keys 4.69 -> 4.65 ms).  MODE: the
// addressing of the usual countBFs (flat with 2^n counters, flat, two-dimensional;
// a power of two counters in a cell each), short enough to be unrolled over the
// keys and hashes; kAnyAddress: the general one, which is not (unrolled, the body
// would not fit the instruction cache).
enum AddressMode { kAnyAddress, kFlatPow2, kFlat, kTwoDim };

// Coarse region of hash h, and cell in it and counter in the cell as a code has
// them (at most 2^30 cells, so a cell's number has 32 bits).
template <int MODE>
__device__ __forceinline__ void code_of(const Geometry &G, int coarse_shift, int sb, uint64_t h,
                                        unsigned &bin, uint32_t &code) {
    if (MODE == kFlatPow2 || MODE == kFlat) {   // the counter's number is cell and counter
        const uint64_t g = MODE == kFlatPow2 ? h & G.m_mask : mod_by(h, G.m, G.mag_m);
        bin = (unsigned)(g >> (coarse_shift + sb));
        code = (uint32_t)g & ((1u << (coarse_shift + sb)) - 1);
        return;
    }
    uint64_t cell64;
    unsigned slot;
    if (MODE == kTwoDim) {
        cell64 = mod_by(h, G.dim_x, G.mag_x) * G.dim_y + mod_by(h, G.dim_y, G.mag_y);
        slot = (unsigned)h & (unsigned)(G.eta - 1);
    } else {
        address(G, h, cell64, slot);
    }
    const unsigned cell = (unsigned)cell64;
    bin = cell >> coarse_shift;
    code = ((cell & ((1u << coarse_shift) - 1)) << sb) | slot;
}

template <int KW, int MODE, unsigned H>
__global__ void __launch_bounds__(kEmitThreads, 4) emit_kernel(EmitArgs e) {
    constexpr int NT = kEmitThreads, PER = H == 3 ? 3 : 4;
    __shared__ uint32_t sorted[PER * NT * H];
    __shared__ uint8_t region[PER * NT * H];   // of sorted[i]
    __shared__ unsigned hist[kCoarseBins], start[kCoarseBins];
    __shared__ unsigned long long base[kCoarseBins];      // a code's place in e.coarse less its i
    __shared__ unsigned staged;
    __shared__ unsigned off[kWin + 1], plc[kWin];
    const unsigned tid = threadIdx.x, lane = tid & 31;
    const Geometry &G = e.G;
    const unsigned D = e.ordered ? e.meta->distinct : e.meta->out_cursor;
    const unsigned r0 = min(e.begin, D), r1 = min(e.end, D);
    const unsigned i_begin = r0 + (unsigned)((uint64_t)(r1 - r0) * blockIdx.x / gridDim.x);
    const unsigned i_end = r0 + (unsigned)((uint64_t)(r1 - r0) * (blockIdx.x + 1) / gridDim.x);
    if (i_begin >= i_end) return;
    unsigned g0 = e.ordered ? range_of(e.offsets, e.n_total, i_begin) : 0;
    const unsigned nh = (unsigned)G.nhash;
    const int wb = e.w_bits, sb = e.slot_bits;
    const uint32_t w_most = 1u << wb;   // wb is 16 at most
    if (e.ordered) load_window<NT>(e, g0, off, plc);
    else if (tid == 0) off[kWin] = ~0u;   // the keys stand one after the other
    __syncthreads();
    for (unsigned i0 = i_begin; i0 < i_end;) {
        if (off[kWin] <= i0) {   // i0 lies past the window of ranges: the next one
            __syncthreads();
            load_window<NT>(e, g0 += kWin, off, plc);
            __syncthreads();
            continue;
        }
        const unsigned i1 = min(min(i_end, i0 + PER * NT), off[kWin]);
        Key<KW> key[PER];
        uint32_t w[PER];
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            const unsigned i = i0 + q * NT + tid;
            w[q] = 0;
            if (i < i1) {
                const uint64_t at = e.ordered ? place_in(off, plc, i) : i;
                key[q] = load_key<KW>(e.keys, at);
                w[q] = e.mult ? (uint32_t)min((uint64_t)e.mult[at], G.maxc) : 1u;
                if (e.dlist && i < e.dlist_cap) store_key<KW>(e.dlist, i, key[q]);
                if (e.sure) e.sure[i] = w[q] > e.tau;
            }
        }
        for (unsigned a0 = 0; a0 < nh; a0 += H) {
            if (tid < kCoarseBins) hist[tid] = 0;
            __syncthreads();
            uint32_t code[PER][H];
            unsigned br[PER][H];
#pragma unroll(MODE != kAnyAddress ? PER : 1)
            for (int q = 0; q < PER; ++q) {
                const uint64_t k1m = KW == 1 ? premix8(key[q].lo) : 0;
#pragma unroll
                for (unsigned j = 0; j < H; ++j) {
                    br[q][j] = kNoKey;
                    if (w[q] && a0 + j < nh) {
                        uint64_t h1, h2;
                        if (KW == 1)
                            murmur8(k1m, a0 + j, h1, h2);
                        else
                            murmur16(key[q].lo, key[q].hi, a0 + j, h1, h2);
                        unsigned bin;
                        uint32_t in;
                        code_of<MODE>(G, e.coarse_shift, sb, h1, bin, in);
                        const uint32_t wc = min(w[q], w_most);
                        code[q][j] = (in << wb) | (wc - 1);
                        br[q][j] = (bin << 16) | atomicAdd(&hist[bin], 1u);
                        if (wc < w[q]) {
                            const uint64_t cell = ((uint64_t)bin << e.coarse_shift) | (in >> sb);
                            sat_add(G.cells, cell, (in & ((1u << sb) - 1)) * (unsigned)G.alpha, G.maxc,
                                    w[q] - wc, __ldcg(G.cells + cell), G.cas_limit, &e.ctr->error);
                        }
                    }
                }
            }
            __syncthreads();
            if (tid < kCoarseBins) {   // warps 0 and 1: prefix over the regions
                const unsigned n = hist[tid];
                unsigned incl = n, below = 0;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned t = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= (unsigned)o) incl += t;
                }
                if (tid >= 32) {   // warp 1 starts after all of warp 0's regions
                    below = hist[tid - 32];
#pragma unroll
                    for (int o = 16; o; o >>= 1) below += __shfl_xor_sync(0xffffffffu, below, o);
                }
                start[tid] = below + incl - n;
                if (tid == kCoarseBins - 1) staged = below + incl;
                unsigned long long b0 = ~0ull;
                if (n) {
                    b0 = atomicAdd(e.coarse_cursor + tid, (unsigned long long)n);
                    if (b0 + n > e.coarse_cap) {
                        b0 = ~0ull;   // region full: these go to the countBF directly
                    } else {
                        atomicAdd(e.coarse_written + tid, (unsigned long long)n);
                        b0 += (uint64_t)tid * e.coarse_cap - (below + incl - n);
                    }
                }
                base[tid] = b0;
            }
            __syncthreads();
#pragma unroll
            for (int q = 0; q < PER; ++q)
#pragma unroll
                for (unsigned j = 0; j < H; ++j)
                    if (br[q][j] != kNoKey) {
                        const unsigned at = start[br[q][j] >> 16] + (br[q][j] & 0xffffu);
                        sorted[at] = code[q][j];
                        region[at] = (uint8_t)(br[q][j] >> 16);
                    }
            __syncthreads();
            // runs of a region's codes leave together
            for (unsigned i = tid, n = staged; i < n; i += NT) {
                const uint32_t c = sorted[i];
                const unsigned bin = region[i];
                const unsigned long long b0 = base[bin];
                if (b0 != ~0ull) {
                    __stcs(e.coarse + (b0 + i), c);
                } else {
                    const uint64_t cell = ((uint64_t)bin << e.coarse_shift) | (c >> (sb + wb));
                    const unsigned slot = (c >> wb) & ((1u << sb) - 1);
                    sat_add(G.cells, cell, slot * (unsigned)G.alpha, G.maxc, (c & (w_most - 1)) + 1ull,
                            __ldcg(G.cells + cell), G.cas_limit, &e.ctr->error);
                }
            }
            __syncthreads();
        }
        i0 = i1;
    }
}

// Atomic update: the distinct keys' increments straight into the countBF (an
// L2-resident one), four first attempts of a key in flight together.
template <int KW>
__global__ void __launch_bounds__(kEmitThreads, 4) emit_atomic_kernel(EmitArgs e) {
    constexpr int NT = kEmitThreads;
    __shared__ unsigned off[kWin + 1], plc[kWin];
    const unsigned tid = threadIdx.x;
    const Geometry &G = e.G;
    const unsigned D = e.ordered ? e.meta->distinct : e.meta->out_cursor;
    const unsigned i_begin = (unsigned)((uint64_t)D * blockIdx.x / gridDim.x);
    const unsigned i_end = (unsigned)((uint64_t)D * (blockIdx.x + 1) / gridDim.x);
    if (i_begin >= i_end) return;
    unsigned g0 = e.ordered ? range_of(e.offsets, e.n_total, i_begin) : 0;
    if (e.ordered) load_window<NT>(e, g0, off, plc);
    else if (tid == 0) off[kWin] = ~0u;   // the keys stand one after the other
    __syncthreads();
    for (unsigned i0 = i_begin; i0 < i_end;) {
        if (off[kWin] <= i0) {
            __syncthreads();
            load_window<NT>(e, g0 += kWin, off, plc);
            __syncthreads();
            continue;
        }
        const unsigned i1 = min(min(i_end, i0 + NT), off[kWin]);
        const unsigned i = i0 + tid;
        i0 = i1;
        if (i >= i1) continue;
        const uint64_t at = e.ordered ? place_in(off, plc, i) : i;
        const Key<KW> key = load_key<KW>(e.keys, at);
        const uint64_t w = min((uint64_t)e.mult[at], G.maxc);
        if (e.dlist && i < e.dlist_cap) store_key<KW>(e.dlist, i, key);
        if (e.sure) e.sure[i] = w > e.tau;
        const uint64_t k1m = KW == 1 ? premix8(key.lo) : 0;
        for (int a0 = 0; a0 < G.nhash; a0 += 4) {
            uint64_t cell[4], cur[4], prev[4];
            unsigned sh[4];
            bool need[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                cell[j] = 0;
                sh[j] = 0;
                cur[j] = 0;
                if (a0 + j < G.nhash) {
                    uint64_t h1, h2;
                    unsigned slot;
                    if (KW == 1)
                        murmur8(k1m, (uint32_t)(a0 + j), h1, h2);
                    else
                        murmur16(key.lo, key.hi, (uint32_t)(a0 + j), h1, h2);
                    address(G, h1, cell[j], slot);
                    sh[j] = slot * (unsigned)G.alpha;
                }
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (a0 + j < G.nhash) cur[j] = __ldcg(G.cells + cell[j]);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint64_t room = G.maxc - ((cur[j] >> sh[j]) & G.maxc);
                need[j] = a0 + j < G.nhash && room != 0;
                prev[j] = cur[j];
                if (need[j])
                    prev[j] = atomicCAS((unsigned long long *)(G.cells + cell[j]),
                                        (unsigned long long)cur[j],
                                        (unsigned long long)(cur[j] + (min(w, room) << sh[j])));
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (need[j] && prev[j] != cur[j])
                    sat_add(G.cells, cell[j], sh[j], G.maxc, w, prev[j], G.cas_limit,
                            &e.ctr->error);
        }
    }
}

unsigned round_up(unsigned n, unsigned to) { return (n + to - 1) / to * to; }

// Sub-arrays of DedupBufs::meta.
struct MetaLayout {
    uint64_t size = 0;
    uint64_t take(uint64_t bytes) {
        const uint64_t at = size;
        size += (bytes + 255) & ~255ull;
        return at;
    }
    uint64_t meta, codes, valid, samples, samples_lo, spl, spl_lo, lut, piece, starts, places;
    uint64_t counts, offsets, big;
    uint64_t prefix, totals, tile_base, map, fine_spl, fine_lo, fine_lut, fine_starts;
    explicit MetaLayout(const DedupPlan &p) {
        meta = take(sizeof(DedupMeta));
        codes = take(p.chunks * p.chunk / 4 + 64);   // and 128 bases after the last chunk
        valid = take(p.chunks * p.chunk / 8);
        samples = take(round_up(p.samples, kSampleTile) * 8ull);
        samples_lo = take(p.kw == 2 ? round_up(p.samples, kSampleTile) * 8ull : 0);
        spl = take(kMaxRanges * 8ull);
        spl_lo = take(p.kw == 2 ? kMaxRanges * 8ull : 0);
        lut = take(kLutStride * 2ull);
        piece = take(p.chunks * 4);
        starts = take((p.n_ranges + 1ull) * p.chunks * 2);
        places = take(p.total() * 4);
        counts = take(p.total() * 4);
        offsets = take((p.total() + 1) * 4);
        big = take(p.total() * 4);
        prefix = totals = tile_base = map = fine_spl = fine_lo = fine_lut = fine_starts = size;
        if (p.n_fine) {
            prefix = take((uint64_t)p.n_ranges * p.chunks * 4);
            totals = take(p.n_ranges * 4ull);
            tile_base = take((p.n_ranges + 1) * 4ull);
            map = take(p.tiles() * sizeof(TileMap));
            fine_spl = take((uint64_t)p.n_ranges * kMaxRanges * 8);
            fine_lo = take(p.kw == 2 ? (uint64_t)p.n_ranges * kMaxRanges * 8 : 0);
            fine_lut = take((uint64_t)p.n_ranges * kLutStride * 2);
            fine_starts = take(p.tiles() * (p.n_fine + 1) * 2);
        }
    }
};

// Values a thread of block_sort holds for n of them (n <= kMaxSamples).
int sort_items(unsigned n) {
    int e = 1;
    while (1024u * e < n) e *= 2;
    return e;
}

uint64_t last_prefix(int K) { return K >= 32 ? ~0ull : (1ull << (2 * K)) - 1; }

template <typename F>
cudaError_t set_smem(F f, size_t bytes) {
    return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

#define DD_TRY(call)                              \
    do {                                          \
        const cudaError_t e_ = (call);            \
        if (e_ != cudaSuccess) return e_;         \
    } while (0)

template <int KW, int CHUNK>
cudaError_t extract_variant(int K, int canonical, const ExtractArgs &x, unsigned per_sm, int sms,
                            cudaStream_t s) {
    constexpr size_t smem = sizeof(GroupSmem<KW, CHUNK>);
    auto *k = canonical == 0   ? extract_kernel<KW, CHUNK, 0>
              : canonical == 1 ? extract_kernel<KW, CHUNK, 1> : extract_kernel<KW, CHUNK, 2>;
    DD_TRY(set_smem(k, smem));
    const unsigned grid = std::min(x.n_chunks, (unsigned)sms * per_sm);
    k<<<grid, CHUNK / 8, smem, s>>>(K, x);
    return cudaGetLastError();
}

RefineArgs refine_args(const DedupPlan &p, const DedupBufs &d, const MetaLayout &m,
                       uint64_t n_chunks) {
    RefineArgs r;
    r.in = d.a;
    r.out = d.b;
    r.n_chunks = (unsigned)n_chunks;
    r.n_ranges = p.n_ranges;
    r.n_fine = p.n_fine;
    r.target = p.target;
    r.spl = (const uint64_t *)(d.meta + m.spl);
    r.spl_lo = (const uint64_t *)(d.meta + m.spl_lo);
    r.piece = (const uint32_t *)(d.meta + m.piece);
    r.prefix = (const uint32_t *)(d.meta + m.prefix);
    r.totals = (const uint32_t *)(d.meta + m.totals);
    r.tile_base = (const uint32_t *)(d.meta + m.tile_base);
    r.starts = (const uint16_t *)(d.meta + m.starts);
    r.map = (const TileMap *)(d.meta + m.map);
    r.fine_spl = (uint64_t *)(d.meta + m.fine_spl);
    r.fine_lo = (uint64_t *)(d.meta + m.fine_lo);
    r.fine_lut = (uint16_t *)(d.meta + m.fine_lut);
    r.fine_starts = (uint16_t *)(d.meta + m.fine_starts);
    r.meta = (DedupMeta *)(d.meta + m.meta);
    return r;
}

template <int KW>
cudaError_t finish_variant(const DedupPlan &p, const DedupBufs &d, DevCounters *ctr,
                           uint64_t n_chunks, bool ordered, bool fresh, uint64_t list_cap, int sms,
                           cudaStream_t s, uint64_t &launches) {
    const MetaLayout m(p);
    DedupMeta *meta = (DedupMeta *)(d.meta + m.meta);
    const unsigned nc = (unsigned)n_chunks;
    if (p.n_fine) {
        const RefineArgs r = refine_args(p, d, m, n_chunks);
        row_prefix_kernel<<<p.n_ranges, 1024, 0, s>>>(r.starts, nc, (uint32_t *)r.prefix,
                                                     (uint32_t *)r.totals);
        const int E = sort_items(p.fine_samples);
        auto *fk = E == 1 ? fine_splitters_kernel<KW, 1> : E == 2 ? fine_splitters_kernel<KW, 2>
                 : E == 4 ? fine_splitters_kernel<KW, 4> : E == 8 ? fine_splitters_kernel<KW, 8>
                 : fine_splitters_kernel<KW, 16>;
        DD_TRY(set_smem(fk, std::max(E, 4) * 8192));
        fk<<<p.n_ranges, 1024, std::max(E, 4) * 8192, s>>>(r, p.K, p.fine_samples, last_prefix(p.K));
        tile_map_kernel<<<(unsigned)((p.tiles() + 1023) / 1024), 1024, 0, s>>>(
            r.totals, p.n_ranges, r.prefix, nc, (uint32_t *)r.tile_base, (TileMap *)r.map, meta);
        constexpr size_t smem = sizeof(RefineSmem<KW>);
        DD_TRY(set_smem(refine_kernel<KW>, smem));
        const uint64_t grid = std::min<uint64_t>(p.tiles(), (uint64_t)sms * 2);
        refine_kernel<KW><<<(unsigned)grid, kRefineThreads, smem, s>>>(r, p.K, last_prefix(p.K));
        launches += 4;
    }
    DedupArgs x;
    x.in = p.n_fine ? d.b : d.a;
    x.out = p.n_fine ? d.a : d.b;
    x.mult = d.mult;
    x.n_chunks = nc;
    x.n_fine = p.n_fine;
    x.piece = (const uint32_t *)(d.meta + m.piece);
    x.tile_base = (const uint32_t *)(d.meta + m.tile_base);
    x.starts = (const uint16_t *)(d.meta + (p.n_fine ? m.fine_starts : m.starts));
    x.n_ranges = p.n_ranges;
    x.n_total = (unsigned)p.total();
    x.spl = (const uint64_t *)(d.meta + m.spl);
    x.spl_lo = (const uint64_t *)(d.meta + m.spl_lo);
    x.fine_spl = (const uint64_t *)(d.meta + m.fine_spl);
    x.fine_lo = (const uint64_t *)(d.meta + m.fine_lo);
    x.places = (uint32_t *)(d.meta + m.places);
    x.counts = (uint32_t *)(d.meta + m.counts);
    x.meta = meta;
    x.ctr = ctr;
    x.big = (uint32_t *)(d.meta + m.big);
    x.ordered = ordered ? 1 : 0;
    constexpr size_t smem = sizeof(SmallSmem<KW>), big_smem = sizeof(DedupSmem<KW>);
    DD_TRY(set_smem(dedup_kernel<KW>, smem));
    DD_TRY(set_smem(dedup_big_kernel<KW>, big_smem));
    const unsigned total = (unsigned)p.total();
    dedup_kernel<KW><<<std::min(total, (unsigned)sms * 4), kSmallThreads, smem, s>>>(x, p.K);
    dedup_big_kernel<KW><<<std::min(total, (unsigned)sms * 3), kDedupThreads, big_smem, s>>>(x, p.K);
    launches += 2;
    if (!ordered) return cudaGetLastError();
    scan_counts_kernel<<<1, 1024, 0, s>>>(x.counts, (unsigned)p.total(),
                                          (uint32_t *)(d.meta + m.offsets), meta, fresh ? ctr : nullptr,
                                          list_cap);
    launches += 1;
    return cudaGetLastError();
}

}  // namespace

uint64_t DedupPlan::meta_bytes() const { return MetaLayout(*this).size; }

int dedup_chunk(uint64_t nbytes) {
    return nbytes / kExtractChunk < 4 * kPlanSms ? kExtractSmall : kExtractChunk;
}

// Ranges of about `target` windows each, so that few hold more than a dedup
// block's stage (the splitters' sampling spreads the sizes by a quarter); small calls
// are cut into at least two ranges per SM while those keep 512 windows.  Up
// to kMaxRanges ranges in one level; more in two levels of about equally many
// ranges, so that the runs a block gathers are about equally long at both.
DedupPlan plan_dedup(int K, uint64_t bound, uint64_t chunks, int chunk) {
    DedupPlan p;
    p.K = K;
    p.kw = K <= 32 ? 1 : 2;
    p.bound = bound;
    if (bound == 0 || bound > kMaxRangeWindows) return p;
    // a call of few ranges waits for its largest ones: smaller ones then
    p.target = bound < (1ull << 25) ? (p.kw == 1 ? 1280 : 896) : (p.kw == 1 ? 1664 : 1152);
    uint64_t ranges = (bound + p.target - 1) / p.target;
    ranges = std::max(ranges, std::min<uint64_t>(2 * kPlanSms, bound / 512));
    if (ranges < 1) ranges = 1;
    p.chunk = chunk;
    p.chunks = chunks;
    if (ranges <= kMaxRanges) {
        p.n_ranges = (unsigned)ranges;
    } else {
        unsigned c = 32;
        while ((uint64_t)c * c < ranges && c < kMaxRanges) ++c;
        // with the quarter, no more fine ranges than there may be
        c = std::max(c, (unsigned)std::min<uint64_t>((ranges * 5 / 4 + kMaxRanges - 1) / kMaxRanges,
                                                     kMaxRanges));
        p.n_ranges = c;
        const uint64_t mean = (ranges + c - 1) / c;   // and a quarter for the larger ones
        p.n_fine = (unsigned)std::min<uint64_t>(mean + mean / 4, kMaxRanges);
        p.fine_samples = std::min(16 * p.n_fine, kMaxSamples);
    }
    // sixteen spread the sizes by a quarter around their mean; ranges far below a
    // dedup block's room do with eight (with eight for 900 two-word windows a range,
    // many ranges went to dedup_big_kernel: 112 us of a 370 us call, now 21 of 260)
    const unsigned per_range = p.n_fine ? 32 : bound / ranges * 2 <= p.target ? 8 : 16;
    p.samples = std::min(per_range * p.n_ranges, kMaxSamples);
    p.on = true;
    return p;
}

DedupPlan plan_pack(int K, uint64_t nbytes) {
    DedupPlan p;
    p.K = K;
    p.kw = K <= 32 ? 1 : 2;
    p.chunk = dedup_chunk(nbytes);
    p.chunks = (nbytes + p.chunk - 1) / p.chunk;
    return p;
}

Packed packed_input(const DedupPlan &p, const DedupBufs &d) {
    const MetaLayout m(p);
    return Packed{(const uint32_t *)(d.meta + m.codes), (const uint16_t *)(d.meta + m.valid),
                  (DedupMeta *)(d.meta + m.meta)};
}

cudaError_t dedup_pack(const DedupPlan &p, const DedupBufs &d, const InsertArgs &a, uint64_t chunk0,
                       uint64_t n_chunks, uint64_t begin, uint64_t end, int sms, cudaStream_t s,
                       uint64_t &launches) {
    if (begin >= end) return cudaSuccess;
    const MetaLayout m(p);
    PackArgs x;
    x.chunk0 = chunk0;
    x.chunk_begin = begin;
    x.chunk_end = end;
    x.chunk_last = chunk0 + n_chunks;
    x.codes = (uint32_t *)(d.meta + m.codes);
    x.valid = (uint16_t *)(d.meta + m.valid);
    const bool small = p.chunk == kExtractSmall;   // resident blocks of 64 or 256 threads
    const unsigned grid = (unsigned)std::min<uint64_t>(end - begin, (uint64_t)sms * (small ? 24 : 8));
    if (small)
        pack_kernel<kExtractSmall><<<grid, kExtractSmall / 16, 0, s>>>(a, x);
    else
        pack_kernel<kExtractChunk><<<grid, kExtractChunk / 16, 0, s>>>(a, x);
    launches += 1;
    return cudaGetLastError();
}

cudaError_t dedup_extract(const DedupPlan &p, const DedupBufs &d, int canonical, uint64_t n_chunks,
                          uint64_t span, int sms, cudaStream_t s, uint64_t &launches) {
    const MetaLayout m(p);
    DedupMeta *meta = (DedupMeta *)(d.meta + m.meta);
    PackArgs pa;
    memset(&pa, 0, sizeof(pa));
    pa.codes = (uint32_t *)(d.meta + m.codes);
    pa.valid = (uint16_t *)(d.meta + m.valid);
    DD_TRY(cudaMemsetAsync(meta, 0, sizeof(DedupMeta), s));
    uint64_t *samples = (uint64_t *)(d.meta + m.samples);
    uint64_t *samples_lo = (uint64_t *)(d.meta + m.samples_lo);
    const unsigned n = round_up(p.samples, kSampleTile), tiles = n / kSampleTile;
    const size_t smem = std::max(n * sizeof(uint64_t), sizeof(unsigned) << kLutBits);
    auto *sk = p.kw == 1 ? sample_kernel<1> : sample_kernel<2>;
    sk<<<tiles, 1024, 0, s>>>(pa, p.K, canonical, span, p.samples, samples, samples_lo, meta);
    auto *rk = p.kw == 1 ? rank_kernel<1> : rank_kernel<2>;
    DD_TRY(set_smem(rk, smem));
    rk<<<tiles, 1024, smem, s>>>(samples, samples_lo, n, p.n_ranges, p.K, last_prefix(p.K), meta,
                                 (uint64_t *)(d.meta + m.spl), (uint64_t *)(d.meta + m.spl_lo),
                                 (uint16_t *)(d.meta + m.lut));
    ExtractArgs x;
    x.codes = pa.codes;
    x.valid = pa.valid;
    x.n_chunks = (unsigned)n_chunks;
    x.n_ranges = p.n_ranges;
    x.spl = (const uint64_t *)(d.meta + m.spl);
    x.spl_lo = (const uint64_t *)(d.meta + m.spl_lo);
    x.lut = (const uint16_t *)(d.meta + m.lut);
    x.out = d.a;
    x.piece = (uint32_t *)(d.meta + m.piece);
    x.starts = (uint16_t *)(d.meta + m.starts);
    x.meta = meta;
    launches += 3;
    if (p.kw == 1)
        return p.chunk == kExtractSmall
                   ? extract_variant<1, kExtractSmall>(p.K, canonical, x, 6, sms, s)
                   : extract_variant<1, kExtractChunk>(p.K, canonical, x, 2, sms, s);
    return p.chunk == kExtractSmall
               ? extract_variant<2, kExtractSmall>(p.K, canonical, x, 6, sms, s)
               : extract_variant<2, kExtractChunk>(p.K, canonical, x, 2, sms, s);
}

cudaError_t dedup_finish(const DedupPlan &p, const DedupBufs &d, DevCounters *ctr,
                         uint64_t n_chunks, bool ordered, bool fresh, uint64_t list_cap, int sms,
                         cudaStream_t s, uint64_t &launches) {
    return p.kw == 1
               ? finish_variant<1>(p, d, ctr, n_chunks, ordered, fresh, list_cap, sms, s, launches)
               : finish_variant<2>(p, d, ctr, n_chunks, ordered, fresh, list_cap, sms, s, launches);
}

EmitArgs dedup_result(const DedupPlan &p, const DedupBufs &d, const Geometry &G, DevCounters *ctr,
                      bool ordered) {
    const MetaLayout m(p);
    EmitArgs e;
    memset(&e, 0, sizeof(e));
    e.G = G;
    e.keys = p.n_fine ? d.a : d.b;
    e.mult = d.mult;
    e.places = (const uint32_t *)(d.meta + m.places);
    e.offsets = (const uint32_t *)(d.meta + m.offsets);
    e.n_total = (unsigned)p.total();
    e.ordered = ordered ? 1 : 0;
    e.begin = 0;
    e.end = ~0u;
    e.ctr = ctr;
    e.meta = (const DedupMeta *)(d.meta + m.meta);
    return e;
}

EmitArgs windows_result(const uint64_t *keys, const DedupMeta *meta, const Geometry &G,
                        DevCounters *ctr) {
    EmitArgs e;
    memset(&e, 0, sizeof(e));
    e.G = G;
    e.keys = keys;
    e.end = ~0u;
    e.ctr = ctr;
    e.meta = meta;
    return e;
}

template <int KW>
auto emit_variant(int mode, int nhash) -> void (*)(EmitArgs) {
    if (nhash % 3 == 0 && mode != kAnyAddress)
        return mode == kTwoDim     ? emit_kernel<KW, kTwoDim, 3>
               : mode == kFlatPow2 ? emit_kernel<KW, kFlatPow2, 3> : emit_kernel<KW, kFlat, 3>;
    return mode == kTwoDim     ? emit_kernel<KW, kTwoDim, 2>
           : mode == kFlatPow2 ? emit_kernel<KW, kFlatPow2, 2>
           : mode == kFlat     ? emit_kernel<KW, kFlat, 2> : emit_kernel<KW, kAnyAddress, 2>;
}

cudaError_t launch_emit(const EmitArgs &e, int kw, int sms, cudaStream_t s) {
    const int mode = e.G.eta_log2 < 0 ? kAnyAddress : e.G.dim_x ? kTwoDim : e.G.m_mask ? kFlatPow2 : kFlat;
    auto *k = kw == 1 ? emit_variant<1>(mode, e.G.nhash) : emit_variant<2>(mode, e.G.nhash);
    k<<<(unsigned)sms * 4, kEmitThreads, 0, s>>>(e);
    return cudaGetLastError();
}

cudaError_t launch_emit_atomic(const EmitArgs &e, int kw, int sms, cudaStream_t s) {
    if (kw == 1)
        emit_atomic_kernel<1><<<(unsigned)sms * 4, kEmitThreads, 0, s>>>(e);
    else
        emit_atomic_kernel<2><<<(unsigned)sms * 4, kEmitThreads, 0, s>>>(e);
    return cudaGetLastError();
}

}  // namespace countbf
