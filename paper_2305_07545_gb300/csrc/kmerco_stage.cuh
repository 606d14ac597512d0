// Staging of one chunk of reads in shared memory, used by every kernel that
// walks the windows of an input: 2-bit codes, invalid-base bitmap and
// read-start bitmap of CHUNK window starts and the K - 1 bases after them.
#pragma once

#include "kmerco_internal.cuh"

namespace countbf {

// Sizes for a chunk of CHUNK window starts: 16 bases per 32-bit word, the
// chunk and 128 more bases.
template <int CHUNK>
struct ChunkDims {
    static constexpr int kPack32 = CHUNK / 16 + 8;
};

template <int CHUNK>
struct __align__(16) StageSmem {
    uint32_t pk[ChunkDims<CHUNK>::kPack32];     // codes; word t at t ^ 1 so pairs read as u64
    uint16_t inv[ChunkDims<CHUNK>::kPack32];    // bit j of inv[t]: base 16t + j is not ACGTacgt
    uint32_t brk[ChunkDims<CHUNK>::kPack32 / 2];  // bit q: a read starts at base q of the chunk
};

// 64 bits of a bitmap starting at bit p.
__device__ __forceinline__ uint64_t bits_at(const uint64_t *bm, unsigned p) {
    unsigned w = p >> 6, s = p & 63;
    uint64_t v = bm[w] >> s;
    if (s) v |= bm[w + 1] << (64 - s);
    return v;
}

// Four bases (one byte each, first base in the low byte): their 2-bit codes
// A,a->0 C,c->1 G,g->2 T,t->3, first base most significant, and a bit per
// base that is not one of those letters (bit 0: the first base).  The code
// of a byte is ((c >> 1) ^ (c >> 2)) & 3; a byte is a letter when it equals,
// case aside, the letter its code stands for (one byte permute looks all four
// up), so four bases take about as many instructions as one did bytewise.
__device__ __forceinline__ void pack4(uint32_t x, uint32_t &code, uint32_t &bad) {
    const uint32_t y = ((x >> 1) ^ (x >> 2)) & 0x03030303u;
    const uint32_t z = (y | (y >> 4)) & 0x00ff00ffu;
    const uint32_t sel = z | (z >> 8);   // the four codes as nibbles (low 16 bits)
    const uint32_t letters = __byte_perm(0x54474341u, 0u, sel & 0x3333u);
    const uint32_t d = letters ^ (x & 0xDFDFDFDFu);
    const uint32_t t = ((((d & 0x7f7f7f7fu) + 0x7f7f7f7fu) | d) >> 7) & 0x01010101u;
    bad = (t * 0x10204080u) >> 28;
    code = (y * 0x40100401u) >> 24;
}

// Stages chunk `chunk` of the reads of `a` with NT threads; S.brk must be
// zero on entry.  Returns the bases of the chunk's span (its window starts
// and the K - 1 after them).  The caller synchronises before reading S.
template <int CHUNK, int NT>
__device__ __forceinline__ unsigned stage_chunk(const InsertArgs &a, uint64_t chunk,
                                                StageSmem<CHUNK> &S) {
    constexpr int kPack32 = ChunkDims<CHUNK>::kPack32;
    const int tid = threadIdx.x;
    const uint64_t total = a.last - a.first;
    const uint64_t c0 = chunk * (uint64_t)CHUNK;
    const uint64_t e = min(c0 + (uint64_t)(CHUNK + a.K - 1), total);
    const unsigned nb = (unsigned)(e - c0);
    const uintptr_t src = (uintptr_t)(a.bases + c0);
    const unsigned head = (unsigned)(src & 15);
    const uintptr_t abase = src - head;

    // read starts inside the chunk's span (none when the reads are one sequence)
    for (uint64_t r = (uint64_t)a.first_read[chunk] + tid; !a.whole_file && r < a.nreads; r += NT) {
        uint64_t s = a.offsets[r] - a.first;
        if (s >= c0 + nb) break;
        if (s < c0) continue;   // only with decreasing offsets, which the host rejects
        unsigned q = (unsigned)(s - c0);
        if (q > 0) atomicOr(&S.brk[q >> 5], 1u << (q & 31));
    }
    // bases [16t, 16t + 16) of the span straight from global memory (the two
    // 16-byte vectors holding them: whole ones with streaming loads, the
    // partial ones at the span's ends bytewise, 'N' outside it)
    for (int t = tid; t < kPack32; t += NT) {
        uint32_t w[8];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const unsigned lo = (unsigned)(t + h) << 4;
            if (lo >= head && lo + 16 <= head + nb) {
                const uint4 v = __ldcs((const uint4 *)(abase + lo));
                w[4 * h] = v.x;
                w[4 * h + 1] = v.y;
                w[4 * h + 2] = v.z;
                w[4 * h + 3] = v.w;
            } else {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    uint32_t word = 0;
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const unsigned b = lo + 4 * q + k;
                        const unsigned c = b >= head && b < head + nb
                                               ? *(const uint8_t *)(abase + b) : (unsigned)'N';
                        word |= c << (8 * k);
                    }
                    w[4 * h + q] = word;
                }
            }
        }
        // the 16 bytes start `head` bytes into the 32 loaded ones
        const unsigned hb = (head & 3) * 8;
        uint32_t x[4];
        switch (head >> 2) {
        case 0:
#pragma unroll
            for (int i = 0; i < 4; ++i) x[i] = __funnelshift_r(w[i], w[i + 1], hb);
            break;
        case 1:
#pragma unroll
            for (int i = 0; i < 4; ++i) x[i] = __funnelshift_r(w[i + 1], w[i + 2], hb);
            break;
        case 2:
#pragma unroll
            for (int i = 0; i < 4; ++i) x[i] = __funnelshift_r(w[i + 2], w[i + 3], hb);
            break;
        default:
#pragma unroll
            for (int i = 0; i < 4; ++i) x[i] = __funnelshift_r(w[i + 3], w[i + 4], hb);
            break;
        }
        uint32_t code = 0, bad = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            uint32_t c4, b4;
            pack4(x[i], c4, b4);
            code = (code << 8) | c4;
            bad |= b4 << (4 * i);
        }
        S.pk[t ^ 1] = code;
        S.inv[t] = (uint16_t)bad;
    }
    return nb;
}

}  // namespace countbf
