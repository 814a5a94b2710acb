// Fused schedule of the FDMT: several merge levels per launch.
//
// A launch covers the levels (lb, lt] of the addition rule (section 4 of
// arXiv:1411.5373).  Its work items are "cones": one band B of level lt, a
// range of its delay rows, and one time tile [T0, T0 + W).  Following the
// addition rule down from those rows gives, for every sub-band of B at every
// level l in [lb, lt), a contiguous row range and a time window
// [T0 - o, T0 - o + W + s): the lower half keeps the parent's window, the
// upper half's window starts dl(last row) samples earlier and is
// dl(last) - dl(first) samples wider.  The level-lb rows of the cone are
// staged in shared memory by TMA (zero-filled outside [0, Nt), which is the
// paper's copy rule), the levels in between are computed in shared memory,
// and level lt is written to global memory.  A launch that starts at level 0
// stages input channels and computes the Option-1 partial sums itself.
#pragma once

#include <cstdint>
#include <string>
#include <vector>

#include "fdmt_tables.h"

namespace fdmt {

// Warps per block of the fused kernel (the planner balances work over them).
constexpr int32_t kFusedBlockWarps = 8;
// Row blocks are copied 2^p rows at a time, p <= kMaxBlockP.
constexpr int32_t kMaxBlockP = 5;

// TMA copy into shared memory of rows of the launch's base level (or of
// the input).  Row boxes: global row `row`, columns T0 + xoff + [0, nbox *
// box) in nbox copies of the launch's box width.  Row blocks: rows row ..
// row + 2^nbox - 1, columns T0 + xoff + [0, kchunks * chunk) in one copy,
// landing with row pitch kchunks * chunk.
struct FusedLoad {
  int32_t row;
  int32_t smem;  // byte offset in the block's shared memory
  int32_t xoff;  // first column relative to T0 (<= 0; 16-byte aligned, a chunk multiple for row blocks)
  int32_t nbox;  // row boxes: number of boxes; row blocks: log2 of the rows copied
};

// Compute stages of a work item.  The levels (lb, lt] of a cone are not all
// stored: a stage computes one level from the stored level below it
// (kStageSingle), two levels at once with the level between them never
// stored (kStagePair), or, in a launch that starts at the input, level 1
// straight from the staged input samples (kStageWalk: the Option-1 partial
// sums of level 0 are running sums in registers and are never stored).  The
// last stage writes the group's top level to global memory.
enum : int32_t { kStageWalk = 0, kStageSingle = 1, kStagePair = 2, kStageSearch = 3 };
// Stage word flag: the stage writes the group's top level into shared memory
// in the search layout (pidx) for the search stage that follows it.
constexpr int32_t kStagePadded = 16;
constexpr int32_t kStageKindMask = 15;
// Stage word flag: some op of the stage has a passed-up or one-term half
// (kOpLoOne, kOpHiOne, kOpNoHi; walks: kWalkNoUpper), which only Nf not a
// power of two produces; stages without it run code without those tests.
constexpr int32_t kStageGeneral = 32;
// Stage word flag: some walk of the stage is kWalkMoves.
constexpr int32_t kStageMoves = 128;

// Boxcar search in the last launch (section 4.2, pulse profile): widths
// 2^k, k < K <= kSearchMaxWidths; the top level's time window carries
// search_hist(K) columns of history before the tile.
#if defined(__CUDACC__)
#define FDMT_HOST_DEVICE __host__ __device__
#else
#define FDMT_HOST_DEVICE
#endif
constexpr int32_t kSearchMaxWidths = 9;
inline int32_t search_hist(int32_t k) { return k <= 1 ? 0 : (((1 << (k - 1)) - 1) + 15) / 16 * 16; }
// Search-layout index of column c of a row of 4-byte values: 4 words of
// padding after every 16 columns (no bank conflicts between the 16-column
// runs of neighbouring lanes).
FDMT_HOST_DEVICE inline int32_t search_pidx(int32_t c) { return c + 4 * (c >> 4); }

// Columns of one op: 32 lanes x kLaneCols columns each (lane l holds columns
// l, l + 32, ...).
#ifndef FDMT_LANE_COLS
#define FDMT_LANE_COLS 8
#endif
constexpr int32_t kLaneCols = FDMT_LANE_COLS;
constexpr int32_t kPieceCols = 32 * kLaneCols;
// Ops read whole pieces whatever their width: the block's shared memory
// ends with this much slack so those reads stay inside it.
constexpr int32_t kOverRead = kPieceCols * 4;
// At least this much of a block's shared memory lies between the last
// region and the slack (the programme slots; unused where a launch's
// programmes stay in global memory).
constexpr int32_t kProgMinBytes = 3712;

// Reuse flags of an op against the op before it in the same warp's list (same
// column piece).  No kernel reads them: they say what the runs (FusedRun) keep
// in registers, for the tables that tests execute and the ops' share of work:
//   kOpLoSame  the lower operand (single) or lower half sum (pair) is the
//              previous op's (same lower row: the addition rule's dl did not
//              change);
//   kOpHiShift the upper half sum (pair) is the previous op's one column
//              later (same upper row, dl one larger).
constexpr int32_t kOpLoSame = 1;
constexpr int32_t kOpHiShift = 2;
// Terms of an op where a band has no channel above its border (Nf not a
// power of two, section 4.2: its lower half's rows pass up unchanged):
//   kOpLoOne  the lower half sum is the single term s[p0]
//   kOpHiOne  the upper half sum is the single term s[p2]
//   kOpNoHi   no upper part: the output is the lower part (single: s[p0])
constexpr int32_t kOpLoOne = 4;
constexpr int32_t kOpHiOne = 8;
constexpr int32_t kOpNoHi = 16;
// Walk flags: the band has a single channel (no upper channel); where the
// delay grows, the walk moves its upper sums between lanes instead of reading
// them again.
constexpr int32_t kWalkNoUpper = 1;
constexpr int32_t kWalkMoves = 2;

// One output row piece of a single or pair stage.  Columns tau in
// [0, width) of the piece:
//   single: out[tau] = s[p0 + tau] + s[p1 + tau]
//   pair:   out[tau] = (s[p0 + tau] + s[p1 + tau]) + (s[p2 + tau] + s[p3 + tau])
// (s = shared memory; p0..p3 are byte offsets that already include the
// sources' column offsets; the bracketing is the level-by-level order).  dst
// is the output's byte offset, or for the top stage its global row, written
// at columns T0 + col + tau.
struct FusedOp {
  int32_t dst;
  int32_t p0, p1, p2, p3;
  int32_t width;
  int32_t flags;
  int32_t col;
};

// Level 1 of one band of two input channels, rows a..e (e - a < 32), over
// one column piece, from the staged samples of the two channels (section 4:
// Option-1 sums, then the addition rule).  Row Dt = dl + j sums
//   x_lo[tau] + ... + x_lo[tau - dl]  and  x_hi[tau - dl] + ... + x_hi[tau - dl - j]
// (each in that order) and adds the two; dl starts at dl0 for row a and
// grows by one at row a + 1 + i when bit i of `bits` is set (else j grows).
struct FusedWalk {
  int32_t dst;      // byte offset of row a at the piece's first column; top stage: global row of row a
  int32_t dst_row;  // bytes from one output row to the next in shared memory
  int32_t x_lo, x_hi;  // byte offsets of the two channels' staged samples at the piece's first column
  int32_t width, col;  // columns of the piece, first column within the tile
  int32_t a, e, dl0;
  int32_t bits;
  int32_t chan;     // lower channel (channel weights; the upper one is chan + 1)
  int32_t flags;    // kWalkNoUpper (a single channel, whose Option-1 rows pass up), kWalkMoves
};
// The ops of one node's rows, lowered for the kernel.  A run computes rows
// 0 .. n - 1 of a strip of kPieceCols columns that moves with the delay: row
// r writes columns c(r) + i, c(0) = col and c one larger after every row
// whose lower row grows, so that the upper half's samples keep their place
// in the strip (the upper half is read dl columns earlier, and dl grows with
// c) and stay in registers.  Row r is (s[p0] + s[p1]) + (s[p2] + s[p3]) for a
// pair, s[p0] + s[p2] for a single level, at byte offsets that step from row
// to row by two bits:
//   inc = 1 (the lower row grows): p0, p1 one column later, and
//     sub = 1: p0 a row later (g0), p1 a column earlier (its half's dl grew),
//     sub = 0: p1 a row later (g1);
//   inc = 0 (the upper row grows):
//     sub = 1: p2 a row later (g2), p3 a column earlier,
//     sub = 0: p3 a row later (g3).
// (single levels: p0 or p2 a row later).  The columns outside [0, width) hold
// sums of whatever lies beside the rows; they are written only under
// kRunWhole, where the row pitch leaves room for whole strips beside the
// node's columns.
struct FusedRun {
  int32_t dst;      // byte offset of row 0 at column col; top stage: global row of row 0
  int32_t dst_row;  // bytes from one output row to the next in shared memory
  int32_t col;      // first column of row 0 (may be negative)
  int32_t width;    // the node's columns
  int32_t p0, p1, p2, p3;
  int32_t g0, g1, g2, g3;
  int32_t n;        // rows, at most kRunRows
  uint32_t inc, sub;  // bit r: the step from row r to row r + 1
  int32_t flags;    // kOpLoOne, kOpHiOne, kOpNoHi (every row of the run), kRunWhole
};
constexpr int32_t kRunRows = 32;
constexpr int32_t kRunWhole = 256;
// Columns a run's strip may move over its rows: a stored row's pitch leaves
// at least this many columns free.
constexpr int32_t kRunGrow = 16;
// Bytes kept free below the staged rows: a run reads its lower rows from up
// to kRunRows - 1 columns before their first, a walk that moves its upper sums
// up to 32 samples before them.
constexpr int32_t kUnderRead = 128;
// Stages over the runs: as the stages, with single and pair stages' offsets
// into the runs, and this bit set in their kind.
constexpr int32_t kStageRuns = 64;

// What the kernel needs of a work item besides its rows, as one block that
// is copied to shared memory with them: per stage kProgStageBytes (the kind,
// then the byte offsets within the block of each warp's first walk or run
// and of the stage's end; a search stage has its first and last op instead),
// then the walks and runs.  A launch whose items leave no room for it in
// shared memory reads it in global memory (far).
struct FusedProg {
  int32_t load_begin, load_count;  // the item's row copies
  int32_t tx_bytes;                // bytes the copies and the block deliver
  int32_t n_stages;
  int32_t prog;        // first 16-byte word of the block in FusedPlan::prog
  int32_t prog_bytes;  // a multiple of 16
  int32_t far;         // 1: the block is not copied
  int32_t pad;
};
constexpr int32_t kProgStageBytes = 48;

// Per stage of a template: kind, then the first op (or walk) of each warp
// and the end of the stage's ops.
constexpr int32_t kStageWords = 2 + kFusedBlockWarps;

struct FusedTemplate {
  int32_t load_begin, load_count;
  int32_t walk_begin, walk_count;
  int32_t stage_begin;  // index into FusedPlan::stages (kStageWords per stage)
  int32_t n_stages;     // the last writes global memory
  int32_t tx_bytes;     // bytes the TMA loads deliver
  int32_t smem_bytes;   // dynamic shared memory this template needs
};

// Arguments of a launch that ends with the boxcar search.
struct SearchArgs {
  void *part_v;    // per (row, width, tile): the largest value (A's accumulator type)
  int *part_r;     //   and the region where it first occurs
  int32_t nk;      // widths searched
  int32_t nseg;    // tiles of the launch (partial slots per row and width)
  uint32_t q_off;  // byte offset of the item's per (row, width) bests in shared memory
  uint32_t q_row;  //   and their bytes
};

struct FusedGroup {
  int32_t lb = 0, lt = 0;
  int32_t W = 0;              // time tile of this launch
  int32_t in_size = 4;        // bytes per staged sample (input, or the level-lb state)
  int32_t out_size = 4;       // bytes per sample of the level-lt state written
  int32_t box = 0;            // row boxes: TMA box width, elements (a multiple of 128 bytes)
  int32_t chunk = 0;          // row blocks (chunk > 0): chunk elements, chunks per copy,
  int32_t kchunks = 0;        //   and the largest copy (2^max_p rows)
  int32_t max_p = 0;
  bool from_input = false;
  bool moves = false;         // some walk is kWalkMoves
  int32_t tpl_begin = 0, tpl_count = 0;
  int32_t smem_bytes = 0;     // group-wide layout: barrier + S + Pa + Pb (+ Pt + Q with a search)
                              //   + two programme slots + slack
  int32_t prog_off = 0, prog_slot = 0;  // byte offset of the first programme slot, bytes of one (0: far)
  int32_t s_end = 0, pa_end = 0;  // byte offsets where S and Pa end
  int32_t search_k = 0;       // boxcar widths searched in this launch (0 = none; last group only)
  int32_t hist = 0;           // history columns of the top level's window (search)
  int32_t q_off = 0;          // search: byte offset of an item's per (row, width) bests
  int32_t q_row = 0;          //   and their bytes
  int64_t ntiles = 0;
  int32_t min_x = 0;          // earliest column a copy reads, relative to its tile's first (<= 0)
  double hbm_bytes = 0;       // model: loaded + written bytes per launch
  double smem_traffic = 0;    // model: shared-memory bytes moved per launch
  double ops = 0;             // model: ops and walks per launch
  double block_slots = 0;     // model: resident blocks on the GPU
  double seconds = 0;         // model: launch time
};

struct FusedParams {
  int32_t W = 0;              // time tile of every group (multiple of 64); 0 = per group by the model
  int32_t smem_budget = 112 * 1024;
  std::vector<int32_t> bounds;  // level boundaries 0 = b0 < b1 < ... = L; empty = choose
  std::vector<int32_t> group_W;       // with bounds: tile per group (0 = W / choose)
  std::vector<int32_t> group_budget;  // with bounds: budget per group (0 = smem_budget)
  int32_t staging = 0;                // 0 = row blocks where nt allows, 1 = row boxes, 2 = row blocks
  bool narrow = false;                // store launch-boundary levels whose uint8 sums fit as uint16
  int32_t search_k = 0;               // boxcar widths searched by the last launch (0 = none)
  // Input mapping (d_min, channel order): the first launch's copies read
  // channel k at row nf - 1 - k (descending) and in_shift[k] samples earlier.
  const std::vector<int32_t> *in_shift = nullptr;
  bool descending = false;
};

struct FusedPlan {
  int32_t W = 0;  // tile of the first group (each group has its own)
  int64_t state_nt = 0;  // samples from one row to the next of the levels between launches (>= nt)
  int32_t state_size = 4, input_size = 4, acc_size = 4;
  std::vector<int32_t> level_size;  // [l]: bytes per stored sample of level l (level L: the output)
  std::vector<FusedGroup> groups;
  std::vector<FusedTemplate> tpls;
  std::vector<FusedLoad> loads;
  std::vector<FusedWalk> walks;
  std::vector<FusedOp> ops;
  std::vector<int32_t> stages;
  std::vector<FusedRun> runs;       // the ops as the kernel runs them
  std::vector<int32_t> run_stages;  //   and the stages over them (kStageRuns)
  std::vector<FusedProg> progs;     // per template: its programme
  std::vector<int32_t> prog;        //   in here
  // Workspace: intermediate level states between launches (ping-pong).
  size_t ws_split = 0, ws_bytes = 0;
  double model_seconds = 0;
  bool moves = false;    // walks move their upper sums where that is less work
  bool general = false;  // some stage holds passed-up or one-term halves (kStageGeneral)
};

// Output columns a caller wants of a transform: those from `first` on,
// column t of a row at out[row * pitch + t - first].
struct OutView {
  int64_t first = 0, pitch = 0;
};

// First tile of every group when only output columns from `first` on are
// wanted: a group computes the tiles its successor's copies reach.
struct FirstTiles {
  int64_t tile[64];  // (a plan has at most one group per level)
};
void first_tiles(const FusedPlan &fp, int64_t first, FirstTiles &out);

// Levels a group (lb, lt] keeps in shared memory (see fdmt_fused_plan.cpp).
std::vector<int32_t> stored_levels(int32_t lb, int32_t lt);

// Builds the cone templates for the given parameters.  Returns "" on
// success, else why the schedule does not fit.
std::string plan_fused(const Tables &t, int64_t nt, int32_t state_size, int32_t input_size,
                       const FusedParams &p, FusedPlan &out);

}  // namespace fdmt
