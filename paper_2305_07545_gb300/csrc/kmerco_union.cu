// Union of two ascending lists of distinct keys, ascending and without
// repetition: how a handle's list takes in the keys of a further insert by key
// ranges, or of another handle.  It streams both lists twice and writes the
// union once (10 to 13 ps a key; a probe of the distinct set takes 36 to 75 ps a
// key, and the list has to be sorted again afterwards).
//
// The merged sequence (a key of `a` before an equal one of `b`) is cut into
// tiles of kUnionTile keys: union_split_kernel finds where each tile begins in
// the two lists, union_count_kernel how many keys of b in it repeat one of a,
// union_scan_kernel the tiles' places, union_write_kernel writes them.
#include <algorithm>

#include "kmerco_internal.cuh"

namespace countbf {
namespace {

constexpr int kUnionThreads = 512;
constexpr int kUnionTile = 4096;

struct UnionMeta {
    unsigned long long na, nb;   // lengths of the lists
};

template <int KW>
struct UKey {
    uint64_t lo, hi;
    __device__ __forceinline__ bool operator==(const UKey &o) const {
        return lo == o.lo && (KW == 1 || hi == o.hi);
    }
    __device__ __forceinline__ bool operator<=(const UKey &o) const {
        if (KW == 1) return lo <= o.lo;
        return hi < o.hi || (hi == o.hi && lo <= o.lo);
    }
};

template <int KW>
__device__ __forceinline__ UKey<KW> ukey(const uint64_t *p, uint64_t i) {
    UKey<KW> k;
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
__device__ __forceinline__ void ustore(uint64_t *p, uint64_t i, const UKey<KW> &k) {
    if (KW == 1)
        p[i] = k.lo;
    else
        ((ulonglong2 *)p)[i] = make_ulonglong2(k.lo, k.hi);
}

// split[t]: keys of a among the first t * kUnionTile merged ones (one more entry
// than tiles: the last one is all of a).
template <int KW>
__global__ void __launch_bounds__(256) union_split_kernel(const uint64_t *a, const uint64_t *b,
                                                          const unsigned long long *na_dev,
                                                          const unsigned *nb32,
                                                          const unsigned long long *nb64,
                                                          unsigned *split, UnionMeta *meta) {
    const uint64_t na = *na_dev, nb = nb32 ? *nb32 : *nb64;
    const uint64_t t = blockIdx.x * 256ull + threadIdx.x;
    if (t == 0) {
        meta->na = na;
        meta->nb = nb;
    }
    const uint64_t d = min(t * (uint64_t)kUnionTile, na + nb);
    if (t > (na + nb + kUnionTile - 1) / kUnionTile) return;
    uint64_t lo = d > nb ? d - nb : 0, hi = min(d, na);   // keys of a: the fewest and most
    while (lo < hi) {
        const uint64_t m = lo + (hi - lo) / 2;   // a[m] belongs to the first d when a[m] <= b[d - 1 - m]
        if (ukey<KW>(a, m) <= ukey<KW>(b, d - 1 - m))
            lo = m + 1;
        else
            hi = m;
    }
    split[t] = (unsigned)lo;
}

// A tile of both lists in shared memory: na keys of a from a0 on with the key
// before them, nb keys of b.
template <int KW>
struct __align__(16) UnionSmem {
    uint64_t key[kUnionTile * KW];   // a's keys, then b's
    unsigned delta[kUnionTile + 1];  // new keys of b in front of a's key i
    UKey<KW> before;
    unsigned repeats;
};

struct UnionTileRange {
    unsigned a0, na, b0, nb;
};

template <int KW>
__device__ __forceinline__ UnionTileRange load_tile(UnionSmem<KW> &S, const uint64_t *a,
                                                    const uint64_t *b, const unsigned *split,
                                                    uint64_t t, uint64_t total) {
    UnionTileRange r;
    const uint64_t d0 = t * (uint64_t)kUnionTile, d1 = min(d0 + kUnionTile, total);
    r.a0 = split[t];
    r.na = split[t + 1] - r.a0;
    r.b0 = (unsigned)(d0 - r.a0);
    r.nb = (unsigned)(d1 - d0) - r.na;
    for (unsigned i = threadIdx.x; i < r.na; i += kUnionThreads)
        ustore<KW>(S.key, i, ukey<KW>(a, (uint64_t)r.a0 + i));
    for (unsigned i = threadIdx.x; i < r.nb; i += kUnionThreads)
        ustore<KW>(S.key, r.na + i, ukey<KW>(b, (uint64_t)r.b0 + i));
    if (threadIdx.x == 0 && r.a0) S.before = ukey<KW>(a, (uint64_t)r.a0 - 1);
    return r;
}

// Keys of a in the tile at or below b's key j, and whether that key repeats one.
template <int KW>
__device__ __forceinline__ unsigned place_of(const UnionSmem<KW> &S, const UnionTileRange &r,
                                             unsigned j, bool &repeats) {
    const UKey<KW> k = ukey<KW>(S.key, r.na + j);
    unsigned lo = 0, hi = r.na;
    while (lo < hi) {
        const unsigned m = (lo + hi) / 2;
        if (ukey<KW>(S.key, m) <= k)
            lo = m + 1;
        else
            hi = m;
    }
    repeats = lo ? ukey<KW>(S.key, lo - 1) == k : r.a0 && S.before == k;
    return lo;
}

template <int KW>
__global__ void __launch_bounds__(kUnionThreads) union_count_kernel(const uint64_t *a,
                                                                    const uint64_t *b,
                                                                    const unsigned *split,
                                                                    unsigned *counts,
                                                                    const UnionMeta *meta) {
    extern __shared__ __align__(16) unsigned char dyn[];
    UnionSmem<KW> &S = *reinterpret_cast<UnionSmem<KW> *>(dyn);
    const uint64_t total = meta->na + meta->nb;
    const uint64_t tiles = (total + kUnionTile - 1) / kUnionTile;
    for (uint64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        if (threadIdx.x == 0) S.repeats = 0;
        const UnionTileRange r = load_tile(S, a, b, split, t, total);
        __syncthreads();
        unsigned mine = 0;
        for (unsigned j = threadIdx.x; j < r.nb; j += kUnionThreads) {
            bool rep;
            place_of(S, r, j, rep);
            mine += rep;
        }
        mine = __reduce_add_sync(0xffffffffu, mine);
        if ((threadIdx.x & 31) == 0 && mine) atomicAdd(&S.repeats, mine);
        __syncthreads();
        if (threadIdx.x == 0) counts[t] = r.na + r.nb - S.repeats;
        __syncthreads();
    }
}

// counts[t] becomes the place of tile t's first key; the sum goes to *distinct.
__global__ void __launch_bounds__(1024) union_scan_kernel(unsigned *counts, const UnionMeta *meta,
                                                          unsigned long long *distinct) {
    const uint64_t n = (meta->na + meta->nb + kUnionTile - 1) / kUnionTile;
    constexpr unsigned E = 8;
    unsigned carry = 0;
    for (uint64_t i0 = 0; i0 < n; i0 += 1024 * E) {
        unsigned v[E], sum = 0;
#pragma unroll
        for (unsigned j = 0; j < E; ++j) {
            const uint64_t i = i0 + threadIdx.x * E + j;
            v[j] = i < n ? counts[i] : 0u;
            sum += v[j];
        }
        unsigned tot;
        unsigned pre = block_exclusive_scan<unsigned, 1024>(sum, tot) + carry;
#pragma unroll
        for (unsigned j = 0; j < E; ++j) {
            const uint64_t i = i0 + threadIdx.x * E + j;
            if (i < n) counts[i] = pre;
            pre += v[j];
        }
        carry += tot;
    }
    if (threadIdx.x == 0) *distinct = carry;
}

template <int KW>
__global__ void __launch_bounds__(kUnionThreads) union_write_kernel(const uint64_t *a,
                                                                    const uint64_t *b,
                                                                    const unsigned *split,
                                                                    const unsigned *places,
                                                                    const UnionMeta *meta,
                                                                    uint64_t *out) {
    constexpr unsigned E = kUnionTile / kUnionThreads;
    extern __shared__ __align__(16) unsigned char dyn[];
    UnionSmem<KW> &S = *reinterpret_cast<UnionSmem<KW> *>(dyn);
    const uint64_t total = meta->na + meta->nb;
    const uint64_t tiles = (total + kUnionTile - 1) / kUnionTile;
    for (uint64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        for (unsigned i = threadIdx.x; i <= (unsigned)kUnionTile; i += kUnionThreads) S.delta[i] = 0;
        const UnionTileRange r = load_tile(S, a, b, split, t, total);
        __syncthreads();
        const uint64_t base = places[t];
        // b: consecutive keys a thread, so that a scan numbers the new ones
        const unsigned per = (r.nb + kUnionThreads - 1) / kUnionThreads;
        const unsigned j0 = min(threadIdx.x * per, r.nb), j1 = min(j0 + per, r.nb);
        unsigned fresh = 0, at[E];
#pragma unroll
        for (unsigned e = 0; e < E; ++e) {
            at[e] = ~0u;
            if (j0 + e < j1) {
                bool rep;
                const unsigned p = place_of(S, r, j0 + e, rep);
                if (!rep) {
                    at[e] = p;
                    ++fresh;
                    atomicAdd(&S.delta[p], 1u);
                }
            }
        }
        unsigned tot;
        unsigned n = block_exclusive_scan<unsigned, kUnionThreads>(fresh, tot);
#pragma unroll
        for (unsigned e = 0; e < E; ++e)
            if (at[e] != ~0u) ustore<KW>(out, base + at[e] + n++, ukey<KW>(S.key, r.na + j0 + e));
        // a: moved up by the new keys of b in front
        unsigned d[E], sum = 0;
#pragma unroll
        for (unsigned e = 0; e < E; ++e) {
            const unsigned i = threadIdx.x * E + e;
            d[e] = i < r.na ? S.delta[i] : 0u;
            sum += d[e];
        }
        unsigned before = block_exclusive_scan<unsigned, kUnionThreads>(sum, tot);
#pragma unroll
        for (unsigned e = 0; e < E; ++e) {
            before += d[e];
            S.delta[threadIdx.x * E + e] = before;   // this thread's entries
        }
        __syncthreads();
        for (unsigned i = threadIdx.x; i < r.na; i += kUnionThreads)
            ustore<KW>(out, base + i + S.delta[i], ukey<KW>(S.key, i));
        __syncthreads();
    }
}

template <int KW>
cudaError_t union_variant(const uint64_t *a, uint64_t na_most, const uint64_t *b, uint64_t nb_most,
                          const unsigned *nb32, const unsigned long long *nb64, uint64_t *out,
                          unsigned *scratch, unsigned long long *distinct, cudaStream_t s) {
    const uint64_t tiles = (na_most + nb_most + kUnionTile - 1) / kUnionTile;
    UnionMeta *meta = (UnionMeta *)scratch;
    unsigned *split = scratch + 4, *counts = split + tiles + 2;
    constexpr size_t smem = sizeof(UnionSmem<KW>);
    cudaError_t e = cudaFuncSetAttribute(union_count_kernel<KW>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(union_write_kernel<KW>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const unsigned g = (unsigned)std::min<uint64_t>(tiles, 152 * (KW == 1 ? 4 : 2));
    union_split_kernel<KW><<<(unsigned)((tiles + 1 + 255) / 256), 256, 0, s>>>(a, b, distinct, nb32,
                                                                             nb64, split, meta);
    union_count_kernel<KW><<<g, kUnionThreads, smem, s>>>(a, b, split, counts, meta);
    union_scan_kernel<<<1, 1024, 0, s>>>(counts, meta, distinct);
    union_write_kernel<KW><<<g, kUnionThreads, smem, s>>>(a, b, split, counts, meta, out);
    return cudaGetLastError();
}

}  // namespace

uint64_t union_scratch_words(uint64_t na, uint64_t nb) {
    return 2 * ((na + nb + kUnionTile - 1) / kUnionTile) + 8;
}

cudaError_t launch_union(const uint64_t *a, uint64_t na_most, const uint64_t *b, uint64_t nb_most,
                         const unsigned *nb32, const unsigned long long *nb64, int kw, uint64_t *out,
                         unsigned *scratch, unsigned long long *distinct, cudaStream_t s) {
    if (na_most + nb_most == 0) return cudaSuccess;
    return kw == 1 ? union_variant<1>(a, na_most, b, nb_most, nb32, nb64, out, scratch, distinct, s)
                   : union_variant<2>(a, na_most, b, nb_most, nb32, nb64, out, scratch, distinct, s);
}

}  // namespace countbf
