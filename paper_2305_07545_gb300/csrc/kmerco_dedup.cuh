// Declarations of the insertion by key ranges (kmerco_dedup.cu): plan,
// buffers and launcher.  Internal; nothing here is part of the public ABI.
#pragma once

#include "kmerco_internal.cuh"

namespace countbf {

constexpr unsigned kMaxRanges = 1024;    // ranges one level cuts at most
constexpr int kLutBits = 13;             // entries of a splitter lookup table
constexpr unsigned kLutStride = 1u << kLutBits;
constexpr int kExtractChunk = 4096;      // window starts per extract block
constexpr int kExtractSmall = 1024;      // the same for inputs too small to fill the GPU
constexpr int kRefineTile = 4096;        // keys per refine tile
constexpr int kRefineThreads = 512;
// dedup_kernel: windows of a range it takes, its table's slots; the cuts of the
// sort.  Four blocks an SM.
constexpr int kSmallThreads = 256;
template <int KW> constexpr int kStage = KW == 1 ? 2560 : 1792;
constexpr unsigned kTableSlots = 4096;
constexpr unsigned kMaxLeft = 1024;       // windows that do not settle in the first round
// dedup_big_kernel: its table's slots, three blocks an SM.
constexpr int kDedupThreads = 384;
template <int KW> constexpr int kDedupSlots = KW == 1 ? 3072 : 2048;
template <int KW> constexpr int kDedupStage = KW == 1 ? 2560 : 1536;   // windows of a batch
constexpr int kSubBits2 = 9;
constexpr int kSubBins2 = (1 << kSubBits2) + 1;   // the range's last prefix may open one more
constexpr uint64_t kMaxRangeWindows = 1ull << 31;   // of one pass (32-bit key indexes)
constexpr uint64_t kPlanSms = 152;       // SMs of a GB300: plans follow from the input alone
constexpr unsigned kMaxSamples = 16384;  // samples that cut a level's ranges, at most

struct DedupMeta {
    unsigned cursor;       // keys reserved by extract_kernel
    unsigned out_cursor;   // keys reserved by dedup_kernel
    unsigned distinct;     // distinct keys of the call
    unsigned n_tiles;      // refine tiles
    unsigned sampled;      // samples that are keys
    unsigned ranked;       // blocks of rank_kernel that are done
    unsigned n_big;        // ranges left to dedup_big_kernel
    unsigned crowd;        // sample tiles that have the low words of two-word keys
};

struct TileMap {
    uint32_t range, piece;
};

struct PackArgs {
    uint64_t chunk0, chunk_last;        // the pass's first chunk; the one past its last
    uint64_t chunk_begin, chunk_end;    // chunks of this launch
    uint32_t *codes;       // 16 bases a word, words swapped in pairs
    uint16_t *valid;       // a bit per window start
};

struct ExtractArgs {
    const uint32_t *codes;
    const uint16_t *valid;
    unsigned n_chunks;     // chunks of the pass
    unsigned n_ranges;
    const uint64_t *spl, *spl_lo;   // prefixes of the splitters, low words of two-word keys
    const uint16_t *lut;
    uint64_t *out;
    uint32_t *piece;       // first key of every chunk's piece
    uint16_t *starts;      // n_ranges + 1 rows of n_chunks
    DedupMeta *meta;
};

struct RefineArgs {
    const uint64_t *in;
    uint64_t *out;
    unsigned n_chunks, n_ranges, n_fine;
    unsigned target;         // windows of a fine range
    const uint64_t *spl, *spl_lo;
    const uint32_t *piece, *prefix, *totals, *tile_base;
    const uint16_t *starts;
    const TileMap *map;
    uint64_t *fine_spl, *fine_lo;   // kMaxRanges per range
    uint16_t *fine_lut;      // kLutStride per range
    uint16_t *fine_starts;   // per range: n_fine + 1 rows of its tiles
    DedupMeta *meta;
};

struct DedupArgs {
    const uint64_t *in;
    uint64_t *out;
    uint32_t *mult;          // multiplicity of out[i]
    unsigned n_chunks;       // one level: runs of every range
    unsigned n_fine;         // two levels: fine ranges per coarse range; 0: one level
    unsigned n_ranges, n_total;
    int ordered;             // write every range's keys in order, and where they are
    const uint64_t *spl, *spl_lo, *fine_spl, *fine_lo;
    const uint32_t *piece, *tile_base;
    const uint16_t *starts;  // of the last level
    uint32_t *places, *counts;   // per range: first key in out, distinct keys
    uint32_t *big;           // ranges left to dedup_big_kernel
    DedupMeta *meta;
    DevCounters *ctr;
};

struct EmitArgs {
    Geometry G;
    const uint64_t *keys;
    const uint32_t *mult, *places, *offsets;   // mult null: each key once
    unsigned n_total;        // ranges
    int ordered;             // keys in the order of the ranges (places, offsets), else as they stand
    unsigned begin, end;     // distinct keys of this pass
    uint64_t *dlist;         // distinct list to write, or null
    uint64_t dlist_cap;      // keys it holds: those after them are left out
    uint8_t *sure;           // key i has more than tau windows (or null)
    uint32_t tau;
    int coarse_shift, slot_bits, w_bits;
    uint32_t *coarse;
    uint64_t coarse_cap;
    unsigned long long *coarse_cursor, *coarse_written;
    DevCounters *ctr;
    const DedupMeta *meta;
};

// How one pass of an insert call is cut into ranges; sizes of its buffers.
// Every size follows from the pass's window bound and chunk count.
struct DedupPlan {
    bool on = false;
    int kw = 1, K = 0;
    int chunk = 0;              // window starts per chunk
    uint64_t bound = 0;         // windows of a pass at most
    uint64_t chunks = 0;        // chunks of a pass at most
    unsigned target = 0;        // windows of a final range
    unsigned n_ranges = 1;      // coarse ranges (one level: the final ones)
    unsigned n_fine = 0;        // fine ranges per coarse one; 0: one level
    unsigned samples = 0, fine_samples = 0;
    uint64_t total() const { return (uint64_t)n_ranges * (n_fine ? n_fine : 1); }
    uint64_t tiles() const { return n_fine ? bound / kRefineTile + n_ranges + 1 : 0; }
    uint64_t keys_a() const { return (bound + chunks + 2) * kw; }   // words
    uint64_t keys_b() const { return (n_fine ? tiles() * kRefineTile : bound + 2) * kw; }
    uint64_t mult_words() const { return bound + 2; }               // uint32
    uint64_t meta_bytes() const;
};

struct DedupBufs {
    uint64_t *a, *b;       // keys
    uint32_t *mult;
    unsigned char *meta;   // everything else, meta_bytes()
};

// Window starts per chunk for an input of nbytes bases: a small one gives every
// resident block a chunk.
int dedup_chunk(uint64_t nbytes);
// A pass over `chunks` chunks that hold at most `bound` windows; not on when
// that is more than one pass takes.
DedupPlan plan_dedup(int K, uint64_t bound, uint64_t chunks, int chunk);

// A call that is only packed (kmerco_insert.cu then takes its windows one by one).
DedupPlan plan_pack(int K, uint64_t nbytes);
// Where the packed input and the pass's counts are.
struct Packed {
    const uint32_t *codes;
    const uint16_t *valid;
    DedupMeta *meta;
};
Packed packed_input(const DedupPlan &p, const DedupBufs &d);

// The pass over n_chunks chunks from chunk0 on: first its bases are packed,
// chunk range [begin, end) by chunk range (nothing reads the caller's buffers
// after these); then the windows' keys are cut into ranges (span: bases of the
// pass); then everything up to the distinct keys with their multiplicities.
// ordered: in ascending order; fresh: the handle's list is empty (ctr->distinct
// becomes the call's count, and more than list_cap of them the list-full error).
cudaError_t dedup_pack(const DedupPlan &p, const DedupBufs &d, const InsertArgs &a, uint64_t chunk0,
                       uint64_t n_chunks, uint64_t begin, uint64_t end, int sms, cudaStream_t s,
                       uint64_t &launches);
cudaError_t dedup_extract(const DedupPlan &p, const DedupBufs &d, int canonical, uint64_t n_chunks,
                          uint64_t span, int sms, cudaStream_t s, uint64_t &launches);
cudaError_t dedup_finish(const DedupPlan &p, const DedupBufs &d, DevCounters *ctr,
                         uint64_t n_chunks, bool ordered, bool fresh, uint64_t list_cap, int sms,
                         cudaStream_t s, uint64_t &launches);
// The arguments every consumer of the distinct keys takes.  Of a pass that is not
// ordered, e.keys holds them one after the other in no order, e.meta->out_cursor of them.
EmitArgs dedup_result(const DedupPlan &p, const DedupBufs &d, const Geometry &G, DevCounters *ctr,
                      bool ordered);
// n keys of one window each, in no order, their number in meta->out_cursor.
EmitArgs windows_result(const uint64_t *keys, const DedupMeta *meta, const Geometry &G,
                        DevCounters *ctr);
cudaError_t launch_emit(const EmitArgs &e, int kw, int sms, cudaStream_t s);
cudaError_t launch_emit_atomic(const EmitArgs &e, int kw, int sms, cudaStream_t s);

}  // namespace countbf
