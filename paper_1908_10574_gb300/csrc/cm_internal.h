// Internal declarations shared by the libcm CUDA sources (not part of the C ABI).
#pragma once

#include <cstdint>
#include <cstddef>
#include <string>
#include <vector>
#include <cuda_runtime.h>

#include "../../include/cm.h"

namespace cm {

// ---- residue streams -------------------------------------------------------------------
// A block's subjects are concatenated into one byte stream, one byte per DP row:
// bits 0-4 residue code (0..23, 24 = pad row whose scores are all non-positive),
// bit 7 = first row of a subject, bit 6 = last row of a subject.  Every subject occupies a
// multiple of kRowGroup rows (pad rows follow it), so subjects start on group boundaries and a
// kernel step can cover up to kRowGroup rows; an empty subject is one group of pad rows, the
// first carrying both flags, so its score comes out 0.
constexpr uint8_t kFirst = 0x80;
constexpr uint8_t kLast = 0x40;
// Residue codes: ARNDCQEGHILKMFPSTWYV = 0..19, then B, Z, X, * = 20..23 (24-letter matrices,
// CM_MATRIX24); a 20 x 20 matrix sits in the top-left corner of the 24 x 24 one every kernel
// reads, and calls with it accept codes 0..19 only.
constexpr int kAlpha = 24;             // letters of the largest alphabet (matrix stride)
constexpr uint8_t kPadCode = 24;
constexpr int kProfRows = 25;          // 24 residues + pad row

// rows a subject of `len` residues occupies in a stream: a multiple of kRowGroup (at least
// one group), so subjects start on group boundaries and a kernel step can cover a group
constexpr int kRowGroup = 4;
inline int64_t stream_rows(int64_t len)
{
    return len <= 0 ? kRowGroup : (len + kRowGroup - 1) / kRowGroup * kRowGroup;
}

// longest sequence accepted: keeps every warp stream of the kernels below 2^31 rows
constexpr int64_t kMaxSeqLen = int64_t(1) << 28;

// ---- pair blocks -----------------------------------------------------------------------
// A block is a set of pairs between queries A (held in registers, one column per residue)
// and subjects B (streamed row by row).  CROSS: query k pairs with every subject s < nb.
// TRI: A == B sorted by length; query k pairs with subjects s < k.
enum BlockKind : int32_t { kCross = 0, kTri = 1 };

struct SwBlock {
    int32_t kind;       // BlockKind
    int32_t swap;       // 0: cell score M[q][x] (query = pair's first); 1: M[x][q]
    int32_t na, nb;     // |A|, |B|
    int64_t a_ids;      // offset of A's sequence ids in the id pool
    int64_t b_ids;      // offset of B's sequence ids in the id pool
    int64_t stream;     // byte offset of B's row stream in the stream pool
    int64_t srow;       // offset of B's row table (nb+1 entries) in the row pool
    int64_t out_base;   // output slot of the block's first pair
    int32_t k0;         // first query index covered (TRI: slot = tri(k) - tri(k0) + s)
    int32_t has_map;    // 1: slot -> user index through out_map[]
};

// Launch modes of the int16x2 kernel (see sw16_kernel): query pair over 32 lanes; single
// query with two subject streams in the word halves; query pair with two subject streams,
// one per 16-lane half-warp segment; single query with four subject streams (two 16-lane
// segments x two halves).  The 16-lane modes serve queries of at most kSeg16MaxCols.
enum SwMode : int32_t { kModePair = 0, kModeTwo = 1, kModeSeg16 = 2, kModeTwo16 = 3 };
constexpr int kSeg16MaxCols = 16 * 32;   // longest query tile of the 16-lane pair mode
constexpr int kTwo16MaxCols = 16 * 16;   // ... of the 16-lane single-query mode (registers)
constexpr int kTwoPassCols = 32 * 16;    // column pass of the 32-lane single-query mode

// One CTA task: query k (single-query modes) or the query pair (k, k+1) (pair modes, the two
// queries in the two 16-bit halves) of a block against subjects [s0, s1), whose rows are split
// over the CTA's subject streams.  `mode` is the SwMode of the launch the task belongs to.
struct SwTask {
    int32_t block;
    int32_t k;          // lo query index; hi = k+1 (if hi_valid)
    int32_t s0, s1;     // subjects covered (rows split over the CTA's streams)
    int32_t npass;      // column passes of SEG*R columns
    int32_t hi_valid;   // 0 when the lo query has no partner
    int32_t mode;
    int32_t R;          // columns per lane
};

// One work unit of the single-query launch: a task's passes [pass, pass_end).  A unit with all
// passes runs them one after another over its warp's boundary slot, in pieces of its subjects
// that fit the slot (piece_end).  A unit of one pass of several (a pipelined task: its passes are
// consecutive units) reads and then overwrites, row by row, the boundary column that the unit
// before it writes at piped + bnd_row.
struct SwUnit {
    int32_t block, k, s0, s1;
    int32_t npass, pass, pass_end;
    int32_t mode, R;
    int32_t rows;       // pipelined: rows of the boundary column
    int64_t bnd_row;    // pipelined: its first row in SwArgs::piped, else -1
};

// End of the piece of subjects [s0, s1) that a unit of several passes runs at once over a boundary
// slot of `slot` rows: as many whole subjects as have that many rows together (so no split of them
// over streams is longer), one at least.  A task's rows are only about its target where its list
// was cut by count (device-built lists), so a run of long subjects may be several pieces.
inline __host__ __device__ int32_t piece_end(const int64_t* srow, int32_t s0, int32_t s1, int64_t slot)
{
    int32_t lo = s0 + 1, hi = s1;                  // the last end in [lo, hi] that fits
    while (lo < hi) {
        const int32_t mid = lo + (hi - lo + 1) / 2;
        if (srow[mid] - srow[s0] <= slot) lo = mid; else hi = mid - 1;
    }
    return lo;
}

struct CellUnit;

struct SwArgs {
    const uint8_t* db;          // residue codes of all sequences
    const int64_t* off;         // n_seqs+1 offsets
    const SwBlock* blocks;
    const SwTask* tasks;
    int32_t ntasks;
    int32_t* task_counter;      // zeroed before launch
    const struct SwUnit* units; // single-query launch: its work units (instead of tasks)
    const int32_t* ranges;      // ... first unit of each range (nranges + 1)
    const int32_t* homes;       // ... the range each CTA starts with
    int32_t nranges;
    int32_t* progress;          // ... boundary row groups written by each unit (zeroed)
    uint2* piped;               // ... boundary columns of the pipelined units
    const CellUnit* cell_units; // int32 launch: its units (null: the huge-score kernel)
    int32_t ncells;
    int32_t num_sms;
    int4* cell_best;            // ... best so far up to each unit's strip
    const int32_t* ids;         // id pool
    const uint8_t* streams;     // stream pool
    const int64_t* srows;       // row pool
    int32_t* out;               // output slots (int32 scores, kSat = needs int32 rerun)
    const int64_t* out_map;     // slot -> user index (blocks with has_map)
    uint2* bnd;                 // multi-pass boundary columns, bnd_stride rows per warp
    int64_t bnd_stride;
    int32_t* err;               // set non-zero by a kernel's own bounds checks
    int16_t mat[kAlpha * kAlpha];   // substitution matrix, [first residue][second residue]
    int32_t gap_open;           // first-gap cost (already includes extend for BLAST mode)
    int32_t gap_extend;
    // the same constants in both halves of a word, as kernel parameters: the query-pair kernels'
    // inner loop takes them as operands without a register (or its read port)
    uint32_t beta2, bmo2, open2, ext2, nege2;   // beta, beta - o, o, e, -e
    int32_t beta;               // int16 bias: stored = true + beta
    int32_t sat_thr;            // stored best >= sat_thr -> rerun in int32
    int32_t wait_limit;         // polls of a bounded device wait before it gives up (long pairs)
};

constexpr int32_t kSat = INT32_MIN;   // output slot marker: saturated in int16, rerun pending

// One pair for the int32 rerun / cells kernels.
struct PairRef {
    int32_t q, x;       // query (columns) and subject (rows) sequence ids
    int32_t swap;       // as SwBlock::swap
    int32_t pad;
    int64_t slot;       // output slot (final index)
};

// One job of the alignment-cells kernel: rows a[0..m), columns b[0..n) (both reversed when
// `reverse`), result = (best, first row, first column) in row-major order, 0-based.
struct CellJob {
    int32_t a, b;
    int32_t m, n;
    int32_t reverse;
    int32_t pad;
};

// Strips of the int32 wavefront (wave32.cuh): at most 32 lanes x kWaveMaxR columns, of equal
// width; a unit of its launches (strips.cu) is one strip of one job.
constexpr int kWaveMaxR = 8;           // columns per lane: two profile words
constexpr int64_t kWaveScoreLimit = (int64_t)1 << 28;
constexpr int32_t kPollLimit = 1 << 24;   // polls of ~100 ns before a device wait gives up
inline __host__ __device__ int32_t wave_strips(int64_t n)
{
    return n <= 0 ? 1 : (int32_t)((n + 32 * kWaveMaxR - 1) / (32 * kWaveMaxR));
}
inline __host__ __device__ int32_t wave_R(int64_t n)
{
    const int64_t per = (n + wave_strips(n) - 1) / wave_strips(n);
    return per <= 0 ? 1 : (int32_t)((per + 31) / 32);
}
inline __host__ __device__ int32_t cell_strips(int64_t m, int64_t n) { return m <= 0 ? 1 : wave_strips(n); }
// Row groups of a boundary column that a pass of one warp publishes after step t of its wavefront
// (lane 31 is 31 groups behind): 1, 33, 65, ..., and 0 for none.  Never the last group: the pass
// publishes that one itself, behind a fence, once everything else it hands on is written.
inline __host__ __device__ int32_t groups_after_step(int32_t t, int32_t groups)
{
    return (t & 31) == 31 && t - 30 < groups ? t - 30 : 0;
}
struct CellUnit {
    int32_t job, strip;
    int32_t limit;                     // polls of its wait for the strip before
    int32_t pad;
    int64_t bnd_row;                   // first row of the job's boundary column in SwArgs::bnd
};

// One subject list of a ranked block, selected by bitmap rows of the ranker's pair selection:
// op 0 = row a, 1 = row a AND row b, 2 = row a AND NOT row b, 3 = row b AND NOT row a.  Bit i
// of a row selects subject reps[b0 + i].  The list's subjects become global subjects g0 ..,
// its stream rows start at rowbase.
enum KeptOp : int32_t { kKeepA = 0, kKeepAnd = 1, kKeepAOnly = 2, kKeepBOnly = 3 };
struct KeptList {
    int64_t row_a, row_b;   // word offsets of the two bitmap rows (row_b unused for kKeepA)
    int32_t words;          // words per row
    int32_t op;             // KeptOp
    int64_t b0;             // offset of the subject reps in `reps`
    int64_t g0;             // first global subject index of the list
    int64_t rowbase;        // first stream row of the list
};

// ---- launchers (sw16.cu, sw16_pair.cu, sw16_single.cu) ---------------------------------
// Words per lane in a profile row of the query-pair kernel: R rounded up to a multiple of 4
// (16-byte loads), plus 4 more when that is an even number of 16-byte units, so that the eight
// lanes of a quarter warp always read eight distinct 16-byte bank groups whatever residues they
// look up.
inline __host__ __device__ constexpr int lane_stride(int R)
{
    return (((R + 3) / 4) & 1) ? (R + 3) / 4 * 4 : (R + 3) / 4 * 4 + 4;
}
// shared memory of a query-pair CTA: the profile of one tile
inline constexpr int sw16_pair_smem(int R, int mode)
{
    return kProfRows * (mode == kModeSeg16 ? 16 : 32) * lane_stride(R) * 4;
}
int sw16_ctas_per_sm(int R, int W, int mode);
// query pairs: the tasks of one tile and mode, or (weak, see launch_sw16_single) of all of them
cudaError_t launch_sw16(int R, int W, int mode, int grid, const SwArgs& a, cudaStream_t st);
cudaError_t launch_sw16_pairs(int W, int grid, int smem, const SwArgs& a, cudaStream_t st)
    __attribute__((weak));
// Every single-query task (kModeTwo, kModeTwo16; any tile width) in one launch of `grid` CTAs of
// `warps` warps, a unit per warp at a time; range r holds the units [ranges[r], ranges[r + 1]),
// task_counter[r] is its ticket.  Slots of bnd_stride rows for the units of all passes are
// at bnd, one per warp.  Weak: a build with its own launch_sw16 and without this gets a launch
// per bin.
constexpr int kSingleWarps = 12;       // one CTA per SM: shared memory of the profiles
cudaError_t launch_sw16_single(int grid, int warps, const SwArgs& a, cudaStream_t st)
    __attribute__((weak));
cudaError_t launch_sw32(int R, int grid, const SwArgs& a, const PairRef* pr, int32_t npairs,
                        int32_t* counter, cudaStream_t st);
// int32 passes over lists of pairs (strips.cu): a.cell_units, a.ncells, a.progress, a.cell_best
// hold the list's units.  Long pairs (kLongMinCols, kLongMinRows) have launches of their own,
// whose waits cm_set_wait_limit bounds.
constexpr int64_t kLongMinCols = 2048, kLongMinRows = 512;
cudaError_t launch_long_sw32(int grid, const SwArgs& a, const PairRef* pr, int32_t npairs,
                             int32_t* counter, cudaStream_t st);
cudaError_t launch_long_cells(int grid, const SwArgs& a, const CellJob* jobs, int32_t njobs,
                              int32_t* counter, int32_t* res, cudaStream_t st);
cudaError_t launch_cells_wf(int grid, const SwArgs& a, const CellJob* jobs, int32_t njobs,
                            int32_t* counter, int32_t* res, cudaStream_t st);
// alignment cells where scores may reach 2^28 (longpair.cu; launch_long_cells without
// a.cell_units): kLongSlots boundary slots of bnd_stride rows per CTA
constexpr int kLongSlots = 8;
cudaError_t launch_huge_cells(int grid, const SwArgs& a, const CellJob* jobs, int32_t njobs,
                              int32_t* counter, int32_t* res, cudaStream_t st);

// ---- pack.cu ---------------------------------------------------------------------------
// letters of the 20-letter alphabet (alpha 20) or also B, Z, X, * (alpha 24) -> codes
cudaError_t launch_ascii_to_codes(const uint8_t* in, uint8_t* out, int64_t n, int32_t alpha,
                                  int32_t* bad, cudaStream_t st);
cudaError_t launch_check_codes(const uint8_t* in, int64_t n, int32_t alpha, int32_t* bad,
                               cudaStream_t st);
cudaError_t launch_gather_stream(const uint8_t* db, const int64_t* off, const int32_t* ids,
                                 int32_t nb, const int64_t* srow, uint8_t* stream,
                                 cudaStream_t st);
cudaError_t launch_collect_saturated(const int32_t* out, int64_t nslots, const SwBlock* blocks,
                                     int32_t nblocks, const int64_t* block_first_slot,
                                     const int32_t* ids, const int64_t* out_map,
                                     PairRef* list, int32_t* count, int32_t cap,
                                     cudaStream_t st);
cudaError_t launch_compact_tri(const int32_t* out, int64_t nslots, int32_t k0,
                               const int32_t* order, int32_t T, int32_t* pairs_out,
                               int32_t* scores_out, int64_t* chunk_counts, int64_t nchunks,
                               int phase, cudaStream_t st);
cudaError_t launch_scan_chunks(int64_t* counts, int64_t nchunks, int64_t* total,
                               cudaStream_t st);
cudaError_t launch_compact_slots(const int32_t* out, int64_t nslots, int32_t T,
                                 int64_t* slots_out, int32_t* scores_out, int64_t* chunk_counts,
                                 int64_t nchunks, int phase, cudaStream_t st);
int64_t compact_chunks(int64_t nslots);
// per list: stream rows and residues of its subjects (totals[2*l], totals[2*l + 1])
cudaError_t launch_kept_totals(const KeptList* lists, int32_t nlists, const uint32_t* bits,
                               const int32_t* reps, const int64_t* off, int64_t* totals,
                               cudaStream_t st);
// per list: subject ids (ids[g0 + s]) and row table (srow[g0 + s + 1]) in bitmap order
cudaError_t launch_kept_expand(const KeptList* lists, int32_t nlists, const uint32_t* bits,
                               const int32_t* reps, const int64_t* off, int32_t* ids,
                               int64_t* srow, cudaStream_t st);

}  // namespace cm
