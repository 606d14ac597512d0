// Insertion phase of KmerCo (Algorithm 1 with the countBF insert of
// Algorithm 3) on sm_103a.
//
// Two ways lead a call's windows into the countBF and the distinct set:
//  - by key ranges (kmerco_dedup.cu): the call's distinct keys with their
//    multiplicities first, then one weighted increment per key and hash; the
//    kernels that apply those in the partitioned update are here
//    (repartition_kernel, apply_count_kernel, apply_kernel);
//  - window by window (insert_kernel, insert_batch_kernel here): for small
//    calls, handles with a small retry limit, and when the buffers of the
//    first way cannot be had.
//
// insert_kernel: a work unit is a chunk of consecutive window starts of the
// flat bases array, regardless of read boundaries, so long and short reads
// balance the same way.  Per chunk a block
//   1. stages the chunk's bases (plus K-1 halo) in shared memory, 2-bit
//      packed (A=0 C=1 G=2 T=3, first base most significant), with an
//      invalid-base bitmap and the read starts inside it in a break bitmap,
//   2. keeps the window starts whose K bases are valid and lie in one read,
//   3. per window: the canonical key (the smaller of forward and reverse
//      complement by value, or by H_0; Sections 2.2-2.3), k_h MurmurHash3
//      hashes, one saturating counter increment per hash (Algorithm 3), each
//      a compare-and-swap on its 64-bit cell in global memory, and an insert
//      into the distinct-key set (open addressing, linear probing); keys new
//      to the set are staged in shared memory and appended to the distinct
//      list with one global atomic per chunk.
// Larger calls have their input packed first (pack_kernel): steps 1 and 2 read codes
// and window bits, and the caller's buffers are read within microseconds.  For the
// partitioned update the counters are left out and the windows' keys written to
// memory instead: pieces of 2.5e6 windows into 2^18 cells then take 238 us each
// with their increments, 282 with a compare-and-swap per window and hash.
//
// Partitioned update (at most 2^30 cells): emit_kernel (kmerco_dedup.cu) has
// appended the increments as 32-bit codes to 64 coarse countBF regions;
// repartition_kernel splits every region into slices, and one block per
// slice applies its increments in shared memory: apply_count_kernel
// (alpha <= 15) sums them in 32-bit lanes and adds the sums with saturation
// (the repartition then writes each increment as its lane index),
// apply_kernel uses shared-memory compare-and-swap on the cells.  Either
// writes the slice back once.  Increments that do not fit a buffer are added
// to the countBF directly.  Saturating increments commute, so every way gives
// the same countBF.
#include "kmerco_stage.cuh"

namespace countbf {
namespace {

template <int KW, int CHUNK>
struct __align__(16) InsertSmem {
    StageSmem<CHUNK> st;
    uint16_t vpos[CHUNK];                       // valid window starts
    uint64_t fresh[CHUNK * KW];                 // keys new to the distinct set
    unsigned nvalid;
    unsigned nfresh;
    unsigned staged_base;
    unsigned long long fresh_base;
};

__device__ __forceinline__ uint64_t load_cg(const uint64_t *p) { return __ldcg(p); }

// L2 eviction-priority policies.  The countBF is kept (evict_last) while
// the distinct set, touched once per window at random over a region much
// larger than L2, is let go first.
__device__ __forceinline__ uint64_t policy_keep() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t policy_stream() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
// 64-bit load that bypasses L1 (the value may be changed by other SMs'
// atomics) with an L2 eviction policy.
__device__ __forceinline__ uint64_t load_hint(const uint64_t *a, uint64_t pol) {
    uint64_t v;
    asm volatile("ld.global.cg.L2::cache_hint.b64 %0, [%1], %2;" : "=l"(v) : "l"(a), "l"(pol) : "memory");
    return v;
}

// 128-bit compare-and-swap (sm_90+), returns the previous slot contents.
__device__ __forceinline__ void cas128(uint64_t *addr, uint64_t cmp_lo, uint64_t cmp_hi,
                                       uint64_t new_lo, uint64_t new_hi, uint64_t &old_lo,
                                       uint64_t &old_hi) {
    asm volatile(
        "{\n\t.reg .b128 d, b, c;\n\t"
        "mov.b128 b, {%3, %4};\n\t"
        "mov.b128 c, {%5, %6};\n\t"
        "atom.global.cas.b128 d, [%2], b, c;\n\t"
        "mov.b128 {%0, %1}, d;\n\t}"
        : "=l"(old_lo), "=l"(old_hi)
        : "l"(addr), "l"(cmp_lo), "l"(cmp_hi), "l"(new_lo), "l"(new_hi)
        : "memory");
}

// Saturating increment of the counter at `shift` in cell `c`
// (Algorithm 3: extract, add one unless at 2^alpha - 1, write back).  `old`
// is a recent read of the cell; a failed CAS refreshes it.
__device__ __forceinline__ void sat_increment(uint64_t *cells, uint64_t c, unsigned shift,
                                              uint64_t maxc, uint64_t old, uint32_t limit,
                                              unsigned *err) {
    const uint64_t inc = 1ull << shift;
    for (uint32_t it = 0;; ++it) {
        if (((old >> shift) & maxc) == maxc) return;   // saturated: stays at the maximum
        uint64_t prev = atomicCAS((unsigned long long *)(cells + c), (unsigned long long)old,
                                  (unsigned long long)(old + inc));
        if (prev == old) return;
        old = prev;
        if (it >= limit) {
            atomicOr(err, kErrCasLimit);
            return;
        }
    }
}

// Insert a key into the distinct set; true when the key was not there yet.
// A slot stores the key with the set's generation tag in the unused top bits
// of its top word (SetTag): a slot whose tag differs from the current one is
// free, so a reset only moves to the next tag instead of clearing the table.
// Without spare bits (mask 0) a free slot is all ones, cleared at reset; the key
// that is all ones itself has the place after the last slot.
// For one-word keys `first` is an already loaded value of the home slot
// (kEmptyKey - 1 when none was loaded, a value no slot holds); for two-word
// keys *first2 is, when not null.
__device__ __forceinline__ bool slot_free(uint64_t top, const SetTag &t) {
    return t.mask ? (top & t.mask) != t.tag : top == kEmptyKey;
}

template <int KW>
__device__ __forceinline__ bool set_insert(uint64_t *table, uint64_t cap, uint64_t th,
                                           uint64_t klo, uint64_t khi, const SetTag &t,
                                           uint32_t limit, unsigned *err, uint64_t pol,
                                           uint64_t first = kEmptyKey - 1,
                                           const ulonglong2 *first2 = nullptr) {
    if (!t.mask && klo == kEmptyKey && (KW == 1 || khi == kEmptyKey))
        return atomicExch((unsigned long long *)(table + cap * KW), 0ull) != 0ull;
    uint64_t slot = __umul64hi(th, cap);
    for (uint32_t it = 0;; ++it) {
        if (KW == 1) {
            const uint64_t want = klo | t.tag;
            uint64_t v = (it == 0 && first != kEmptyKey - 1) ? first : load_hint(table + slot, pol);
            for (;;) {   // settle this slot
                if (v == want) return false;
                if (!slot_free(v, t)) break;   // another key
                const uint64_t prev = atomicCAS((unsigned long long *)(table + slot),
                                                (unsigned long long)v, (unsigned long long)want);
                if (prev == v) return true;
                v = prev;                      // written meanwhile: look again
            }
        } else {
            // A plain 16-byte load settles most probes without an atomic: the
            // key itself, or another key (a different top word: each slot is
            // written once per generation).  A free slot, or one showing our
            // top word with another low word (a different key, or ours half
            // written), is decided by the 128-bit compare-and-swap, whose
            // result is the slot's real contents.
            const uint64_t whi = khi | t.tag;
            ulonglong2 v = it == 0 && first2 ? *first2 : __ldcg((const ulonglong2 *)(table + 2 * slot));
            for (;;) {
                if (v.x == klo && v.y == whi) return false;
                const bool free = t.mask ? slot_free(v.y, t) : (v.x == kEmptyKey && v.y == kEmptyKey);
                // without a tag: one word of all ones is a key's, or not written yet
                const bool unsure = !t.mask && !free && (v.x == kEmptyKey || v.y == kEmptyKey);
                if (!free && !unsure && v.y != whi) break;
                const uint64_t elo = free ? v.x : kEmptyKey, ehi = free ? v.y : kEmptyKey;
                uint64_t olo, ohi;
                cas128(table + 2 * slot, elo, ehi, klo, whi, olo, ohi);
                if (olo == elo && ohi == ehi) return true;
                if (!free && olo == v.x && ohi == v.y) break;   // a different key, settled
                v.x = olo;
                v.y = ohi;
            }
        }
        if (++slot == cap) slot = 0;
        if (it >= limit) {
            atomicOr(err, kErrProbeLimit);
            return false;
        }
    }
}

// One chunk of CHUNK window starts (the steps above) for the sample
// described by `a`; counts its windows into my_windows / my_skipped.
template <int KW, int CHUNK, bool PACKED = false, bool STAGED = false>
__device__ __forceinline__ void process_chunk(const InsertArgs &a, uint64_t chunk,
                                              InsertSmem<KW, CHUNK> &S, uint64_t pol_keep,
                                              uint64_t pol_stream,
                                              unsigned long long &my_windows,
                                              unsigned long long &my_skipped) {
    constexpr int kPack32 = ChunkDims<CHUNK>::kPack32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int K = a.K;
    const Geometry &G = a.G;
    unsigned nb = 0;
    if (PACKED) {
        const uint32_t *codes = a.codes + chunk * (CHUNK / 16);
        for (int i = tid; i < kPack32; i += kInsertThreads) S.st.pk[i] = codes[i];
    } else {
        nb = stage_chunk<CHUNK, kInsertThreads>(a, chunk, S.st);
    }
    if (tid == 0) {
        S.nvalid = 0;
        S.nfresh = 0;
    }
    __syncthreads();

    // window starts: inside one read, K valid bases
    const uint64_t *inv64 = (const uint64_t *)S.st.inv;
    const uint64_t *brk64 = (const uint64_t *)S.st.brk;
    const uint64_t maskK = K == 64 ? ~0ull : ((1ull << K) - 1);
    const uint64_t maskK1 = (1ull << (K - 1)) - 1;
    for (int p0 = 0; p0 < CHUNK; p0 += kInsertThreads) {
        unsigned p = (unsigned)(p0 + tid);
        bool valid;
        if (PACKED) {   // the windows were counted when they were packed
            valid = (a.valid[chunk * (CHUNK / 16) + (p >> 4)] >> (p & 15)) & 1u;
        } else {
            const bool window = p + (unsigned)K <= nb && (bits_at(brk64, p + 1) & maskK1) == 0;
            valid = window && (bits_at(inv64, p) & maskK) == 0;
            my_windows += window;
            my_skipped += window && !valid;
        }
        unsigned bal = __ballot_sync(0xffffffffu, valid);
        unsigned base = 0;
        if (lane == 0 && bal) base = atomicAdd(&S.nvalid, (unsigned)__popc(bal));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (valid) S.vpos[base + __popc(bal & ((1u << lane) - 1))] = (uint16_t)p;
    }
    __syncthreads();

    // per valid window: canonical key, hashes, counter updates, set insert
    for (int i = tid; !PACKED && i < kPack32 / 2; i += kInsertThreads)
        S.st.brk[i] = 0;   // for the next chunk
    const unsigned nvalid = S.nvalid;
    if (STAGED) {
        if (tid == 0 && nvalid) S.staged_base = atomicAdd(a.n_staged, nvalid);
        __syncthreads();
    }
    const uint64_t *pk64 = (const uint64_t *)S.st.pk;
    for (unsigned i0 = (unsigned)warp * 32; i0 < nvalid; i0 += kInsertThreads) {
        const unsigned i = i0 + lane;
        const bool active = i < nvalid;
        uint64_t klo = 0, khi = 0;
        if (active) {
            const unsigned p = S.vpos[i];
            const unsigned w = p >> 5, s = (p & 31) * 2;
            const uint64_t x0 = pk64[w], x1 = pk64[w + 1];
            const uint64_t t0 = s ? (x0 << s) | (x1 >> (64 - s)) : x0;
            if (KW == 1) {
                const uint64_t fwd = t0 >> (64 - 2 * K);
                klo = fwd;
                if (a.canonical == 1) {
                    const uint64_t rc = revcomp64(fwd, K);
                    klo = rc < fwd ? rc : fwd;
                } else if (a.canonical == 2) {   // the strand with the smaller H_0
                    const uint64_t rc = revcomp64(fwd, K);
                    uint64_t hf, hr, t;
                    murmur8(premix8(fwd), 0u, hf, t);
                    murmur8(premix8(rc), 0u, hr, t);
                    klo = hf < hr ? fwd : rc;
                }
            } else {
                const uint64_t x2 = pk64[w + 2];
                const uint64_t t1 = s ? (x1 << s) | (x2 >> (64 - s)) : x1;
                const int r = 128 - 2 * K;   // 0..62
                uint64_t fhi, flo;
                if (r == 0) {
                    fhi = t0;
                    flo = t1;
                } else {
                    flo = (t1 >> r) | (t0 << (64 - r));
                    fhi = t0 >> r;
                }
                klo = flo;
                khi = fhi;
                if (a.canonical) {
                    uint64_t rhi, rlo;
                    revcomp128(fhi, flo, K, rhi, rlo);
                    bool take_rc;
                    if (a.canonical == 2) {   // the strand with the smaller H_0
                        uint64_t hf, hr, t;
                        murmur16(flo, fhi, 0u, hf, t);
                        murmur16(rlo, rhi, 0u, hr, t);
                        take_rc = !(hf < hr);
                    } else {
                        take_rc = rhi < fhi || (rhi == fhi && rlo < flo);
                    }
                    if (take_rc) {
                        klo = rlo;
                        khi = rhi;
                    }
                }
            }
        }

        uint64_t table_hash = 0, table_first = kEmptyKey - 1;
        const uint64_t k1m = KW == 1 ? premix8(klo) : 0;
        if (STAGED && active) {
            const uint64_t at = (uint64_t)S.staged_base + i;
            uint64_t h1;
            if (KW == 1) {
                __stcs((unsigned long long *)a.staged + at, (unsigned long long)klo);
                murmur8(k1m, 0u, h1, table_hash);
                table_first = load_hint(a.table + __umul64hi(table_hash, a.cap), pol_stream);
            } else {
                __stcs((ulonglong2 *)a.staged + at, make_ulonglong2(klo, khi));
                murmur16(klo, khi, 0u, h1, table_hash);
            }
        }
        // All loads of a group of four hashes (and, in the first group, the
        // distinct-set home slot) are issued together, then all first
        // compare-and-swap attempts; only failed attempts retry.
        for (int a0 = 0; !STAGED && a0 < G.nhash; a0 += 4) {
            uint64_t cell[4], cur[4], prev[4];
            unsigned sh[4], slot[4];
            bool use[4], need[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                use[j] = active && (a0 + j < G.nhash);
                cell[j] = 0;
                sh[j] = 0;
                slot[j] = 0;
                if (use[j]) {
                    uint64_t h1, h2;
                    if (KW == 1)
                        murmur8(k1m, (uint32_t)(a0 + j), h1, h2);
                    else
                        murmur16(klo, khi, (uint32_t)(a0 + j), h1, h2);
                    if (a0 + j == 0) table_hash = h2;
                    address(G, h1, cell[j], slot[j]);
                    sh[j] = slot[j] * (unsigned)G.alpha;
                }
            }
            if (KW == 1 && a0 == 0 && active)
                table_first = load_hint(a.table + __umul64hi(table_hash, a.cap), pol_stream);
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (use[j]) cur[j] = load_hint(G.cells + cell[j], pol_keep);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                need[j] = use[j] && ((cur[j] >> sh[j]) & G.maxc) != G.maxc;
                prev[j] = cur[j];
                if (need[j])
                    prev[j] = atomicCAS((unsigned long long *)(G.cells + cell[j]),
                                        (unsigned long long)cur[j],
                                        (unsigned long long)(cur[j] + (1ull << sh[j])));
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (need[j] && prev[j] != cur[j])
                    sat_increment(G.cells, cell[j], sh[j], G.maxc, prev[j], G.cas_limit,
                                  &a.ctr->error);
        }

        bool isnew = false;
        if (active)
            isnew = set_insert<KW>(a.table, a.cap, table_hash, klo, khi, a.set_tag,
                                   G.probe_limit, &a.ctr->error, pol_stream, table_first);
        const unsigned bal = __ballot_sync(0xffffffffu, isnew);
        unsigned base = 0;
        if (lane == 0 && bal) base = atomicAdd(&S.nfresh, (unsigned)__popc(bal));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (isnew) {
            const unsigned slot = base + __popc(bal & ((1u << lane) - 1));
            S.fresh[slot * KW] = klo;
            if (KW == 2) S.fresh[slot * KW + 1] = khi;
        }
    }
    __syncthreads();

    // the distinct-list run of this chunk's new keys
    const unsigned nfresh = S.nfresh;
    if (tid == 0 && nfresh) {
        unsigned long long b = atomicAdd(&a.ctr->distinct, (unsigned long long)nfresh);
        if (b + nfresh > a.dlist_cap) {
            atomicOr(&a.ctr->error, kErrListFull);
            b = ~0ull;
        }
        S.fresh_base = b;
    }
    __syncthreads();

    if (nfresh) {
        const unsigned long long b = S.fresh_base;
        if (b != ~0ull)
            for (unsigned i = tid; i < nfresh * KW; i += kInsertThreads)
                a.dlist[b * KW + i] = S.fresh[i];
    }
    __syncthreads();
}

// Warp totals of windows and skipped windows into a sample's counters.
__device__ __forceinline__ void flush_totals(DevCounters *ctr, unsigned long long &w,
                                             unsigned long long &k) {
    for (int o = 16; o; o >>= 1) {
        w += __shfl_down_sync(0xffffffffu, w, o);
        k += __shfl_down_sync(0xffffffffu, k, o);
    }
    if ((threadIdx.x & 31) == 0 && w) {
        atomicAdd(&ctr->windows, w);
        atomicAdd(&ctr->skipped, k);
        atomicAdd(&ctr->inserted, w - k);
    }
    w = 0;
    k = 0;
}

template <int KW, int CHUNK, bool PACKED, bool STAGED>
__global__ void __launch_bounds__(kInsertThreads, 4) insert_kernel(InsertArgs a) {
    __shared__ InsertSmem<KW, CHUNK> S;
    for (int i = threadIdx.x; i < ChunkDims<CHUNK>::kPack32 / 2; i += kInsertThreads) S.st.brk[i] = 0;
    __syncthreads();
    const uint64_t pol_keep = policy_keep(), pol_stream = policy_stream();
    unsigned long long my_windows = 0, my_skipped = 0;
    for (uint64_t chunk = a.chunk_begin + blockIdx.x; chunk < a.nchunks; chunk += gridDim.x)
        process_chunk<KW, CHUNK, PACKED, STAGED>(a, chunk, S, pol_keep, pol_stream, my_windows,
                                                 my_skipped);
    if (!PACKED) flush_totals(a.ctr, my_windows, my_skipped);
}

// Many samples in one persistent launch (atomic update design): the chunks
// of all samples form one index space, sample s owning chunks
// [chunk_end[s-1], chunk_end[s]).  A block walks its chunks in increasing
// order, so the sample only moves forward; its arguments are kept in
// shared memory and its totals are flushed when it changes.
template <int KW, int CHUNK>
__global__ void __launch_bounds__(kInsertThreads, 4) insert_batch_kernel(
    const InsertArgs *args, const unsigned long long *chunk_end, int nsamples,
    unsigned long long total_chunks) {
    __shared__ InsertSmem<KW, CHUNK> S;
    __shared__ InsertArgs A;
    const uint64_t pol_keep = policy_keep(), pol_stream = policy_stream();
    unsigned long long my_windows = 0, my_skipped = 0;
    for (int i = threadIdx.x; i < ChunkDims<CHUNK>::kPack32 / 2; i += kInsertThreads) S.st.brk[i] = 0;
    int s = -1;
    unsigned long long s_begin = 0;
    for (unsigned long long chunk = blockIdx.x; chunk < total_chunks; chunk += gridDim.x) {
        int t = s < 0 ? 0 : s;
        while (t < nsamples && chunk >= chunk_end[t]) ++t;   // uniform across the block
        if (t != s) {
            if (s >= 0) flush_totals(A.ctr, my_windows, my_skipped);
            __syncthreads();
            if (threadIdx.x == 0) A = args[t];
            s = t;
            s_begin = t ? chunk_end[t - 1] : 0;
            __syncthreads();
        }
        process_chunk<KW, CHUNK>(A, chunk - s_begin, S, pol_keep, pol_stream, my_windows,
                                 my_skipped);
    }
    if (s >= 0) flush_totals(A.ctr, my_windows, my_skipped);
}

// Sum over reads of max(0, len - K + 1); flags decreasing offsets.
__global__ void window_bound_kernel(const uint64_t *offsets, uint64_t nreads, int K,
                                    DevCounters *ctr) {
    unsigned long long sum = 0;
    bool bad = false;
    for (uint64_t r = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; r < nreads;
         r += (uint64_t)gridDim.x * blockDim.x) {
        uint64_t s = offsets[r], e = offsets[r + 1];
        if (e < s) {
            bad = true;
            continue;
        }
        if (e - s >= (uint64_t)K) sum += e - s - K + 1;
    }
    for (int o = 16; o; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o);
    if ((threadIdx.x & 31) == 0 && sum) atomicAdd(&ctr->bound, sum);
    if (bad) atomicOr(&ctr->bad_offsets, 1u);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ctr->first = offsets[0];
        ctr->last = offsets[nreads];
    }
}

// first_read[c] = smallest r in [0, nreads] with offsets[r] - first >= c * chunk.
// Eight lanes probe eight places of what is left at a time: a chain of 5 loads
// for 30,000 reads, where halving took 15.
__global__ void __launch_bounds__(256) first_read_kernel(const uint64_t *offsets, uint64_t nreads,
                                                         uint64_t first, uint64_t nchunks,
                                                         uint64_t chunk, uint32_t *first_read) {
    const uint64_t c = (blockIdx.x * 256ull + threadIdx.x) >> 3;
    const unsigned sub = threadIdx.x & 7, group = threadIdx.x & 24;
    const uint64_t target = first + c * chunk;
    uint64_t lo = 0, hi = c < nchunks ? nreads : 0;   // answer in [lo, hi]
    while (__any_sync(0xffffffffu, lo < hi)) {
        const uint64_t n = hi - lo, step = n > 8 ? n / 9 : 1;
        const uint64_t m = lo + step * (n > 8 ? sub + 1 : sub);
        const bool above = m >= hi || offsets[m] >= target;
        const unsigned any = (__ballot_sync(0xffffffffu, above) >> group) & 0xffu;
        const unsigned k = any ? __ffs(any) - 1 : 8;   // the first probe at or above the target
        const uint64_t at = lo + step * (n > 8 ? k + 1 : k);
        const uint64_t below = lo + step * (n > 8 ? k : k - 1);
        if (k) lo = below + 1;
        if (k < 8) hi = min(hi, at);
    }
    if (c < nchunks && sub == 0) first_read[c] = (uint32_t)lo;
}

// Window bound of many samples in one launch: block (x, s) scans reads of
// sample s.  out[s] = {sum of max(0, len - K + 1), first offset, last offset,
// decreasing-offsets flag}.
struct BoundOut {
    unsigned long long bound, first, last, bad;
};
__global__ void window_bound_batch_kernel(const uint64_t *const *offsets, const uint64_t *nreads,
                                          int K, BoundOut *out) {
    const int smp = blockIdx.y;
    const uint64_t *off = offsets[smp];
    const uint64_t n = nreads[smp];
    unsigned long long sum = 0;
    bool bad = false;
    for (uint64_t r = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; r < n;
         r += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t a = off[r], b = off[r + 1];
        if (b < a) {
            bad = true;
            continue;
        }
        if (b - a >= (uint64_t)K) sum += b - a - K + 1;
    }
    for (int o = 16; o; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o);
    if ((threadIdx.x & 31) == 0 && sum) atomicAdd(&out[smp].bound, sum);
    if (bad) atomicOr(&out[smp].bad, 1ull);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        out[smp].first = off[0];
        out[smp].last = off[n];
    }
}

// first_read of every sample's chunks in one launch (chunk index space as in
// insert_batch_kernel).
__global__ void first_read_batch_kernel(const InsertArgs *args, const unsigned long long *chunk_end,
                                        int nsamples, unsigned long long total_chunks,
                                        uint64_t chunk) {
    const unsigned long long c = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
    if (c >= total_chunks) return;
    int lo = 0, hi = nsamples - 1;   // sample owning chunk c
    while (lo < hi) {
        const int mid = (lo + hi) / 2;
        if (c < chunk_end[mid])
            hi = mid;
        else
            lo = mid + 1;
    }
    const InsertArgs &a = args[lo];
    const unsigned long long local = c - (lo ? chunk_end[lo - 1] : 0);
    const uint64_t target = a.first + local * chunk;
    uint64_t rlo = 0, rhi = a.nreads;
    while (rlo < rhi) {
        const uint64_t mid = rlo + (rhi - rlo) / 2;
        if (a.offsets[mid] >= target)
            rhi = mid;
        else
            rlo = mid + 1;
    }
    const_cast<uint32_t *>(a.first_read)[local] = (uint32_t)rlo;
}

// Insert keys into a distinct set (filling or growing a set, a call's or
// another handle's distinct keys).  With dlist != nullptr keys new to the set
// are appended.  n32 / n64: when not null, the number of keys, at most n, is
// read there.
// A block takes PER keys a thread at a time and reserves the list places of
// its new keys with one atomic (an atomic per warp, all on one address, took
// most of the kernel's time).
template <int KW, int PER>
__global__ void __launch_bounds__(256) reinsert_kernel(const uint64_t *keys, uint64_t n,
                                                       const unsigned *n32,
                                                       const unsigned long long *n64,
                                                       uint64_t *table, uint64_t cap, SetTag tag,
                                                       uint64_t *dlist, uint64_t dlist_cap,
                                                       DevCounters *ctr, uint32_t probe_limit) {
    constexpr int kTile = PER * 256;
    __shared__ unsigned long long at0;
    if (n32) n = min(n, (uint64_t)*n32);
    if (n64) n = min(n, (uint64_t)*n64);
    for (uint64_t i0 = (uint64_t)blockIdx.x * kTile; i0 < n;
         i0 += (uint64_t)gridDim.x * kTile) {
        uint64_t klo[PER], khi[PER];
        unsigned fresh = 0;   // bit q: key q is new
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            const uint64_t i = i0 + q * 256 + threadIdx.x;
            klo[q] = khi[q] = 0;
            if (i < n) {
                klo[q] = keys[i * KW];
                if (KW == 2) khi[q] = keys[i * KW + 1];
            }
        }
        uint64_t th[PER], first[PER];
        ulonglong2 first2[KW == 2 ? PER : 1];
#pragma unroll
        for (int q = 0; q < PER; ++q) {   // the home slots' loads in flight together
            uint64_t h1;
            if (KW == 1)
                murmur8(premix8(klo[q]), 0, h1, th[q]);
            else
                murmur16(klo[q], khi[q], 0, h1, th[q]);
            first[q] = kEmptyKey - 1;
            if (i0 + q * 256 + threadIdx.x < n) {
                const uint64_t home = __umul64hi(th[q], cap);
                if (KW == 1)
                    first[q] = load_hint(table + home, policy_stream());
                else
                    first2[q] = __ldcg((const ulonglong2 *)(table + 2 * home));
            }
        }
#pragma unroll
        for (int q = 0; q < PER; ++q)
            if (i0 + q * 256 + threadIdx.x < n &&
                set_insert<KW>(table, cap, th[q], klo[q], khi[q], tag, probe_limit, &ctr->error,
                               policy_stream(), first[q], KW == 2 ? &first2[q] : nullptr))
                fresh |= 1u << q;
        if (!dlist) continue;
        unsigned tot;
        unsigned at = block_exclusive_scan<unsigned, 256>(__popc(fresh), tot);
        if (threadIdx.x == 0) at0 = tot ? atomicAdd(&ctr->distinct, (unsigned long long)tot) : 0;
        __syncthreads();
        const unsigned long long base = at0;
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            if (!((fresh >> q) & 1u)) continue;
            const uint64_t slot = base + at++;
            if (slot < dlist_cap) {
                dlist[slot * KW] = klo[q];
                if (KW == 2) dlist[slot * KW + 1] = khi[q];
            } else {
                atomicOr(&ctr->error, kErrListFull);
            }
        }
    }
}

// Exclusive prefix sum of v[0..n) into out[0..n), n <= E * kRepartThreads,
// by the whole block (E entries per thread).
template <int E>
__device__ __forceinline__ void repart_scan(const unsigned *v, unsigned *out, unsigned n) {
    const unsigned tid = threadIdx.x;
    unsigned x[E], sum = 0;
#pragma unroll
    for (int q = 0; q < E; ++q) {
        x[q] = E * tid + q < n ? v[E * tid + q] : 0u;
        sum += x[q];
    }
    unsigned tot;
    unsigned off = block_exclusive_scan<unsigned, kRepartThreads>(sum, tot);
#pragma unroll
    for (int q = 0; q < E; ++q) {
        if (E * tid + q < n) out[E * tid + q] = off;
        off += x[q];
    }
}

// Split each coarse region's increment codes into slices of 2^slice_shift
// cells.  The blocks walk the tiles of all regions (the regions' code counts
// are on the device, so an idle pass costs one short launch).  MAXF bounds
// the slices per region (2^(coarse_shift - slice_shift)).  With LANES a slice
// code is the counting lane (counter << slice_shift) | cell in its low
// kLaneBits bits with the increment less one above, else the region's code
// less the slice's bits.
template <int MAXF, bool LANES>
__global__ void __launch_bounds__(kRepartThreads, 3) repartition_kernel(PartArgs p) {
    extern __shared__ uint32_t sorted[];   // the tile's codes grouped by slice
    __shared__ unsigned hist[MAXF], start[MAXF], fill[MAXF];
    __shared__ unsigned long long base[MAXF];
    __shared__ unsigned tiles[kCoarseBins + 1];   // tiles of the regions before each one
    const unsigned tid = threadIdx.x;
    if (tid == 0) tiles[0] = 0;
    if (tid < kCoarseBins)
        tiles[tid + 1] = (unsigned)((p.coarse_written[tid] + kRepartTile - 1) / kRepartTile);
    __syncthreads();
    if (tid == 0)
        for (int i = 0; i < kCoarseBins; ++i) tiles[i + 1] += tiles[i];
    __syncthreads();
    const unsigned total = tiles[kCoarseBins];
    const int lb = p.slot_bits + p.w_bits;                        // bits under the cell
    const int fsh = lb + p.slice_shift;                           // code >> fsh = slice
    const unsigned fpc = 1u << (p.coarse_shift - p.slice_shift);  // slices per coarse region
    const uint32_t smask = (1u << p.slice_shift) - 1, fmask = (1u << fsh) - 1;
    const uint32_t slot_mask = (1u << p.slot_bits) - 1, w_mask = (1u << p.w_bits) - 1;
    for (unsigned t = blockIdx.x; t < total; t += gridDim.x) {
        unsigned b = 0;   // the region of tile t
        for (unsigned step = kCoarseBins / 2; step; step >>= 1)
            if (tiles[b + step] <= t) b += step;
        const uint64_t n = p.coarse_written[b];
        const uint64_t t0 = (uint64_t)(t - tiles[b]) * kRepartTile;
        const unsigned cnt = (unsigned)min((uint64_t)kRepartTile, n - t0);
        for (unsigned f = tid; f < fpc; f += kRepartThreads) {
            hist[f] = 0;
            fill[f] = 0;
        }
        __syncthreads();
        // 16 codes per thread, all loads issued before use (the region is 16-byte
        // aligned: coarse_cap is a multiple of 4 and t0 of kRepartTile)
        const uint32_t *src = p.coarse + (uint64_t)b * p.coarse_cap + t0;
        uint32_t c16[16];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const unsigned i = 4 * (tid + j * kRepartThreads);
            if (i + 4 <= cnt) {
                const uint4 v = __ldcs((const uint4 *)(src + i));
                c16[4 * j] = v.x;
                c16[4 * j + 1] = v.y;
                c16[4 * j + 2] = v.z;
                c16[4 * j + 3] = v.w;
            } else {
#pragma unroll
                for (int q = 0; q < 4; ++q) c16[4 * j + q] = i + q < cnt ? src[i + q] : 0u;
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const unsigned i = 4 * (tid + j * kRepartThreads);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (i + q < cnt) atomicAdd(&hist[c16[4 * j + q] >> fsh], 1u);
        }
        __syncthreads();
        if (MAXF <= 64) {
            if (tid < fpc) {
                unsigned pre = 0;
                for (unsigned f = 0; f < tid; ++f) pre += hist[f];
                start[tid] = pre;
            }
        } else {
            repart_scan<(MAXF + kRepartThreads - 1) / kRepartThreads>(hist, start, fpc);
        }
        for (unsigned f = tid; f < fpc; f += kRepartThreads) {
            const unsigned m = hist[f];
            unsigned long long b0 = ~0ull;
            if (m) {
                const uint64_t F = (uint64_t)b * fpc + f;
                b0 = atomicAdd(p.fine_cursor + F, (unsigned long long)m);
                if (b0 + m > p.fine_cap)
                    b0 = ~0ull;
                else
                    atomicAdd(p.fine_written + F, (unsigned long long)m);
            }
            base[f] = b0;
        }
        __syncthreads();
        // group the codes by slice, straight from registers
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const unsigned i = 4 * (tid + j * kRepartThreads);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (i + q < cnt) {
                    const unsigned f = c16[4 * j + q] >> fsh;
                    sorted[start[f] + atomicAdd(&fill[f], 1u)] = c16[4 * j + q];
                }
            }
        }
        __syncthreads();
        for (unsigned i = tid; i < cnt; i += kRepartThreads) {
            const uint32_t code = sorted[i];
            const unsigned f = code >> fsh;
            const unsigned long long b0 = base[f];
            const uint32_t slot = (code >> p.w_bits) & slot_mask;
            if (b0 != ~0ull) {
                const uint64_t F = (uint64_t)b * fpc + f;
                const uint64_t at = F * p.fine_cap + b0 + (i - start[f]);
                const uint32_t out =
                    LANES ? ((code & w_mask) << kLaneBits) | (slot << p.slice_shift) |
                                ((code >> lb) & smask)
                          : code & fmask;
                __stcs(p.fine + at, out);
            } else {
                const uint64_t cell = ((uint64_t)b << p.coarse_shift) | (code >> lb);
                sat_add(p.G.cells, cell, slot * (unsigned)p.G.alpha, p.G.maxc,
                        (code & w_mask) + 1ull, load_cg(p.G.cells + cell), p.G.cas_limit,
                        &p.ctr->error);
            }
        }
        __syncthreads();   // sorted, start and base are free again
    }
}

// One slice of 2^slice_shift cells per block: load it into shared memory,
// apply its increment codes with shared-memory compare-and-swap (saturating
// at 2^alpha - 1), write it back.  With HALF (alpha divides 32, so no counter
// straddles the middle of a cell) each update is a 32-bit compare-and-swap on
// the half-cell that holds the counter.  Slices are 64 KiB, three blocks per
// SM, so one block's slice load and store overlap the other blocks' updates.
template <bool HALF>
__global__ void __launch_bounds__(kCasApplyThreads, 3) apply_kernel(ApplyArgs p) {
    extern __shared__ unsigned long long cells_s[];
    const uint64_t s = blockIdx.x;
    const uint64_t w0 = s << p.slice_shift;
    const uint64_t slice = 1ull << p.slice_shift;
    const unsigned nw = (unsigned)min(slice, p.G.words - w0);
    const uint64_t n = p.written[s];
    if (n == 0) return;   // no increments for this slice
    for (unsigned i = threadIdx.x; i < nw; i += kCasApplyThreads) cells_s[i] = p.G.cells[w0 + i];
    __syncthreads();
    const uint32_t *src = p.codes + s * p.cap;   // 16-byte aligned: cap is a multiple of 4
    const uint32_t wmask = (uint32_t)(slice - 1);
    const uint32_t slot_mask = (1u << p.slot_bits) - 1, inc_mask = (1u << p.w_bits) - 1;
    const int lb = p.slot_bits + p.w_bits;
    const uint64_t maxc = p.G.maxc;
    const unsigned alpha = (unsigned)p.G.alpha;
    // eight codes per thread in flight (two 16-byte loads), then their updates
    constexpr unsigned kStep = kCasApplyThreads * 8;
    for (uint64_t i0 = 0; i0 < n; i0 += kStep) {
        uint32_t code[8];
        unsigned valid = 0;
        const uint64_t i = i0 + threadIdx.x * 4ull;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint64_t j = i + (uint64_t)h * kCasApplyThreads * 4;
            if (j + 4 <= n) {
                const uint4 v = __ldcs((const uint4 *)(src + j));
                code[4 * h] = v.x;
                code[4 * h + 1] = v.y;
                code[4 * h + 2] = v.z;
                code[4 * h + 3] = v.w;
                valid |= 0xFu << (4 * h);
            } else {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    code[4 * h + q] = j + q < n ? src[j + q] : 0u;
                    valid |= (j + q < n ? 1u : 0u) << (4 * h + q);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            if (!((valid >> q) & 1u)) continue;   // past the end
            const unsigned w = (code[q] >> lb) & wmask;
            const unsigned shift = ((code[q] >> p.w_bits) & slot_mask) * alpha;
            const unsigned inc = (code[q] & inc_mask) + 1;
            if (HALF) {   // the little-endian half-cell holding the counter
                unsigned *h32 = (unsigned *)cells_s + 2 * w + (shift >> 5);
                const unsigned sh = shift & 31u, mc = (unsigned)maxc;
                unsigned old = *h32;
                for (uint32_t it = 0;; ++it) {
                    const unsigned room = mc - ((old >> sh) & mc);
                    if (room == 0) break;
                    const unsigned prev = atomicCAS(h32, old, old + (min(inc, room) << sh));
                    if (prev == old) break;
                    old = prev;
                    if (it >= kCasLimit) {
                        atomicOr(&p.ctr->error, kErrCasLimit);
                        break;
                    }
                }
                continue;
            }
            unsigned long long old = cells_s[w];
            for (uint32_t it = 0;; ++it) {
                const unsigned long long room = maxc - ((old >> shift) & maxc);
                if (room == 0) break;
                const unsigned long long add = inc < room ? inc : room;
                const unsigned long long prev = atomicCAS(cells_s + w, old, old + (add << shift));
                if (prev == old) break;
                old = prev;
                if (it >= kCasLimit) {
                    atomicOr(&p.ctr->error, kErrCasLimit);
                    break;
                }
            }
        }
    }
    __syncthreads();
    for (unsigned i = threadIdx.x; i < nw; i += kCasApplyThreads) p.G.cells[w0 + i] = cells_s[i];
}

// Counting apply (alpha <= 15): one slice of 2^slice_shift cells per block.
// The slice's increments are summed in 32-bit shared-memory lanes, counter
// (cell, l) at lane l * 2^slice_shift + cell.  Then every counter becomes
// min(old + sum, 2^alpha - 1) and the slice is written back once.  With
// LANES the codes hold the lanes themselves, else cell and counter.
// A lane's sum is at most k_h times the call's windows; where that could
// pass 2^32 (p.guard), lanes that already saturate their counter are left
// alone, which keeps a sum below 2^15 plus the block's increments in flight.
//
// The last step costs more than the additions on a countBF with few increments
// a cell (570 instructions a cell counter by counter), so 4- and 8-bit counters
// have one that clamps the sums into a packed word and adds the counters of a
// cell side by side.
template <int ALPHA, bool LANES>
__global__ void __launch_bounds__(kApplyThreads, 2) apply_count_kernel(ApplyArgs p) {
    extern __shared__ __align__(16) uint32_t lanes[];   // one 32-bit sum per counter of the slice
    const uint64_t s = blockIdx.x;
    const uint64_t n = p.written[s];
    if (n == 0) return;   // no increments for this slice
    const int ssh = p.slice_shift;
    const uint64_t w0 = s << ssh;
    const uint64_t slice = 1ull << ssh;
    const unsigned nw = (unsigned)min(slice, p.G.words - w0);
    const unsigned eta = (unsigned)p.G.eta;
    const unsigned nwords = eta << ssh;
    if (nwords % 4 == 0) {
        for (unsigned i = threadIdx.x; i < nwords / 4; i += kApplyThreads)
            ((uint4 *)lanes)[i] = make_uint4(0, 0, 0, 0);
    } else {
        for (unsigned i = threadIdx.x; i < nwords; i += kApplyThreads) lanes[i] = 0;
    }
    __syncthreads();
    constexpr unsigned kStep = kApplyThreads * 8;   // two 16-byte loads per thread in flight
    const uint32_t wmask = (uint32_t)(slice - 1);
    const uint32_t slot_mask = (1u << p.slot_bits) - 1, inc_mask = (1u << p.w_bits) - 1;
    const int lb = p.slot_bits + p.w_bits;
    const uint32_t *src = p.codes + s * p.cap;   // 16-byte aligned: cap is a multiple of 4
    const bool guard = p.guard != 0;
    const uint32_t sat = (uint32_t)p.G.maxc;
    for (uint64_t i0 = 0; i0 < n; i0 += kStep) {
        uint32_t code[8];
        unsigned valid = 0;
        const uint64_t i = i0 + threadIdx.x * 4ull;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint64_t j = i + (uint64_t)h * kApplyThreads * 4;
            if (j + 4 <= n) {
                const uint4 v = __ldcs((const uint4 *)(src + j));
                code[4 * h] = v.x;
                code[4 * h + 1] = v.y;
                code[4 * h + 2] = v.z;
                code[4 * h + 3] = v.w;
                valid |= 0xFu << (4 * h);
            } else {
#pragma unroll
                for (unsigned q = 0; q < 4; ++q) {
                    code[4 * h + q] = j + q < n ? src[j + q] : 0u;
                    valid |= (j + q < n ? 1u : 0u) << (4 * h + q);
                }
            }
        }
#pragma unroll
        for (unsigned q = 0; q < 8; ++q) {
            if (!((valid >> q) & 1u)) continue;   // past the end
            const uint32_t c = code[q];
            const unsigned lane = LANES ? c & ((1u << kLaneBits) - 1)
                                        : (((c >> p.w_bits) & slot_mask) << ssh) | ((c >> lb) & wmask);
            const unsigned inc = (LANES ? c >> kLaneBits : c & inc_mask) + 1;
            if (guard && *(volatile uint32_t *)(lanes + lane) >= sat) continue;
            atomicAdd(lanes + lane, inc);
        }
    }
    __syncthreads();
    if (ALPHA) {
        // counters two apart lie in fields of 2 * ALPHA bits, which hold the sum of
        // a counter and a clamped addend; a carry out of the counter fills it
        constexpr int A = ALPHA ? ALPHA : 4, F = 2 * A, ETA = 64 / A;
        constexpr uint64_t kOnes = A == 4 ? 0x0101010101010101ull : 0x0001000100010001ull;
        constexpr uint64_t kMax = kOnes * ((1ull << A) - 1);
        for (unsigned i = threadIdx.x; i < nw; i += kApplyThreads) {
            const uint64_t old = p.G.cells[w0 + i];
            uint32_t add[2][2] = {{0, 0}, {0, 0}};   // [counter parity][half]
#pragma unroll
            for (int l = 0; l < ETA; ++l) {
                const uint32_t c = min(lanes[((unsigned)l << ssh) | i], (1u << A) - 1);
                add[l & 1][(l / 2) * F / 32] += c << ((l / 2) * F % 32);
            }
            uint64_t out = 0;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint64_t v = ((old >> (h * A)) & kMax) + (((uint64_t)add[h][1] << 32) | add[h][0]);
                const uint64_t carry = (v >> A) & kOnes;
                v = (v | ((carry << A) - carry)) & kMax;
                out |= v << (h * A);
            }
            p.G.cells[w0 + i] = out;
        }
        return;
    }
    const unsigned alpha = (unsigned)p.G.alpha;
    const uint64_t maxc = p.G.maxc;
    for (unsigned i = threadIdx.x; i < nw; i += kApplyThreads) {
        const uint64_t old = p.G.cells[w0 + i];
        uint64_t out = 0;
        for (unsigned l = 0; l < eta; ++l) {
            const uint64_t v = ((old >> (l * alpha)) & maxc) + lanes[((uint64_t)l << ssh) | i];
            out |= (v < maxc ? v : maxc) << (l * alpha);
        }
        p.G.cells[w0 + i] = out;
    }
}

}  // namespace

int insert_blocks_per_sm(int kw) {
    int n = 0;
    const cudaError_t e =
        kw == 1 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, insert_kernel<1, kChunk, false, false>,
                                                                kInsertThreads, 0)
                : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, insert_kernel<2, kChunk, false, false>,
                                                                kInsertThreads, 0);
    return e == cudaSuccess && n > 0 ? n : 1;
}

cudaError_t launch_window_bound(const uint64_t *offsets, uint64_t nreads, int K, DevCounters *ctr,
                                cudaStream_t s) {
    uint64_t blocks = (nreads + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    if (blocks == 0) blocks = 1;
    window_bound_kernel<<<(unsigned)blocks, 256, 0, s>>>(offsets, nreads, K, ctr);
    return cudaGetLastError();
}

cudaError_t launch_first_read(const uint64_t *offsets, uint64_t nreads, uint64_t first,
                              uint64_t nchunks, uint64_t chunk, uint32_t *first_read,
                              cudaStream_t s) {
    if (nchunks == 0) return cudaSuccess;
    first_read_kernel<<<(unsigned)((nchunks + 31) / 32), 256, 0, s>>>(offsets, nreads, first,
                                                                       nchunks, chunk, first_read);
    return cudaGetLastError();
}

int insert_batch_blocks_per_sm(int kw, int chunk) {
    int n = 0;
    if (kw == 1 && chunk == 1024)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, insert_batch_kernel<1, 1024>, kInsertThreads, 0);
    else if (kw == 1)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, insert_batch_kernel<1, 2048>, kInsertThreads, 0);
    else if (chunk == 1024)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, insert_batch_kernel<2, 1024>, kInsertThreads, 0);
    else
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, insert_batch_kernel<2, 2048>, kInsertThreads, 0);
    return n > 0 ? n : 1;
}

cudaError_t launch_window_bound_batch(const uint64_t *const *offsets, const uint64_t *nreads,
                                      int n, int K, void *out, uint64_t max_reads, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(out, 0, (size_t)n * sizeof(BoundOut), s);
    if (e != cudaSuccess || n == 0) return e;
    uint64_t bx = (max_reads + 255) / 256;
    if (bx > 256) bx = 256;
    if (bx == 0) bx = 1;
    window_bound_batch_kernel<<<dim3((unsigned)bx, (unsigned)n), 256, 0, s>>>(offsets, nreads, K,
                                                                              (BoundOut *)out);
    return cudaGetLastError();
}

cudaError_t launch_insert_batch(const InsertArgs *args, const unsigned long long *chunk_end,
                                int nsamples, unsigned long long total_chunks, int kw, int chunk,
                                int grid, cudaStream_t s) {
    if (total_chunks == 0) return cudaSuccess;
    first_read_batch_kernel<<<(unsigned)((total_chunks + 255) / 256), 256, 0, s>>>(
        args, chunk_end, nsamples, total_chunks, (uint64_t)chunk);
    const unsigned g = (unsigned)(total_chunks < (unsigned long long)grid ? total_chunks : grid);
    if (kw == 1 && chunk == 1024)
        insert_batch_kernel<1, 1024><<<g, kInsertThreads, 0, s>>>(args, chunk_end, nsamples, total_chunks);
    else if (kw == 1)
        insert_batch_kernel<1, 2048><<<g, kInsertThreads, 0, s>>>(args, chunk_end, nsamples, total_chunks);
    else if (chunk == 1024)
        insert_batch_kernel<2, 1024><<<g, kInsertThreads, 0, s>>>(args, chunk_end, nsamples, total_chunks);
    else
        insert_batch_kernel<2, 2048><<<g, kInsertThreads, 0, s>>>(args, chunk_end, nsamples, total_chunks);
    return cudaGetLastError();
}

cudaError_t launch_repartition(const PartArgs &p, int sms, cudaStream_t s) {
    if (p.coarse_shift - p.slice_shift > kMaxCoarseShift - kSliceShift ||
        p.coarse_shift <= p.slice_shift)
        return cudaErrorInvalidValue;
    const int smem = kRepartTile * (int)sizeof(uint32_t);
    if (p.lane_codes && (((uint64_t)p.G.eta << p.slice_shift) > (uint64_t)kCountLanes ||
                         p.w_bits > 32 - kLaneBits))
        return cudaErrorInvalidValue;   // a lane must fit its bits
    // slices per coarse region: up to 64, 1,024 or kMaxFine (2,048)
    const int fbits = p.coarse_shift - p.slice_shift;
    void (*k)(PartArgs) =
        fbits <= 6    ? (p.lane_codes ? repartition_kernel<64, true> : repartition_kernel<64, false>)
        : fbits <= 10 ? (p.lane_codes ? repartition_kernel<1024, true>
                                      : repartition_kernel<1024, false>)
                      : (p.lane_codes ? repartition_kernel<kMaxFine, true>
                                      : repartition_kernel<kMaxFine, false>);
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    const uint64_t tiles = (p.coarse_cap + kRepartTile - 1) / kRepartTile * kCoarseBins;
    k<<<(unsigned)(tiles < (uint64_t)sms * 3 ? tiles : (uint64_t)sms * 3), kRepartThreads, smem, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_apply(const ApplyArgs &p, uint64_t nslices, cudaStream_t s) {
    if (nslices == 0) return cudaSuccess;
    if (p.lane_codes || p.cap % 4) return cudaErrorInvalidValue;   // 16-byte aligned slices
    const size_t smem = (size_t)8 << p.slice_shift;
    void (*k)(ApplyArgs) = 32 % p.G.alpha == 0 ? apply_kernel<true> : apply_kernel<false>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(8 << kSliceShift));
    if (e != cudaSuccess) return e;
    k<<<(unsigned)nslices, kCasApplyThreads, smem, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_apply_count(const ApplyArgs &p, uint64_t nslices, cudaStream_t s) {
    if (nslices == 0) return cudaSuccess;
    const size_t smem = ((size_t)p.G.eta << p.slice_shift) * 4;
    if (smem > (size_t)kCountLanes * 4 || p.G.alpha > 15) return cudaErrorInvalidValue;
    if (p.cap % 4) return cudaErrorInvalidValue;   // 16-byte aligned slices
    void (*k)(ApplyArgs) =
        p.G.alpha == 4   ? (p.lane_codes ? apply_count_kernel<4, true> : apply_count_kernel<4, false>)
        : p.G.alpha == 8 ? (p.lane_codes ? apply_count_kernel<8, true> : apply_count_kernel<8, false>)
                         : (p.lane_codes ? apply_count_kernel<0, true> : apply_count_kernel<0, false>);
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kCountLanes * 4);
    if (e != cudaSuccess) return e;
    k<<<(unsigned)nslices, kApplyThreads, smem, s>>>(p);
    return cudaGetLastError();
}

template <bool PACKED, bool STAGED>
auto insert_variant(int K, int chunk) -> void (*)(InsertArgs) {
    if (K <= 32)
        return chunk == kChunk ? insert_kernel<1, kChunk, PACKED, STAGED>
                               : insert_kernel<1, kSmallChunk, PACKED, STAGED>;
    return chunk == kChunk ? insert_kernel<2, kChunk, PACKED, STAGED>
                           : insert_kernel<2, kSmallChunk, PACKED, STAGED>;
}

cudaError_t launch_insert(const InsertArgs &a, int grid, int chunk, cudaStream_t s) {
    if (a.nchunks <= a.chunk_begin) return cudaSuccess;
    const uint64_t n = a.nchunks - a.chunk_begin;
    const unsigned g = (unsigned)(n < (uint64_t)grid ? n : (uint64_t)grid);
    if (chunk != kChunk && chunk != kSmallChunk) return cudaErrorInvalidValue;
    auto *k = !a.codes   ? insert_variant<false, false>(a.K, chunk)
              : a.staged ? insert_variant<true, true>(a.K, chunk) : insert_variant<true, false>(a.K, chunk);
    k<<<g, kInsertThreads, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_reinsert(const uint64_t *keys, uint64_t n, const unsigned *n32,
                            const unsigned long long *n64, int kw, uint64_t *table, uint64_t cap,
                            SetTag tag, uint64_t *dlist, uint64_t dlist_cap, DevCounters *ctr,
                            uint32_t probe_limit, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    // four keys a thread once that still gives every resident block a tile
    const bool many = n > 152ull * 8 * 1024;
    const uint64_t tile = many ? 1024 : 256;
    uint64_t blocks = (n + tile - 1) / tile;
    if (blocks > 152 * 8) blocks = 152 * 8;   // resident ones: the rest by stride
    auto *k = kw == 1 ? (many ? reinsert_kernel<1, 4> : reinsert_kernel<1, 1>)
                      : (many ? reinsert_kernel<2, 4> : reinsert_kernel<2, 1>);
    k<<<(unsigned)blocks, 256, 0, s>>>(keys, n, n32, n64, table, cap, tag, dlist, dlist_cap, ctr,
                                       probe_limit);
    return cudaGetLastError();
}

}  // namespace countbf
