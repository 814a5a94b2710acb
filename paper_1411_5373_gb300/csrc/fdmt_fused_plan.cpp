// Host planner of the fused schedule (see fdmt_fused.h).
//
// For one group of levels (lb, lt] and one tile width W, every band of level
// lt is split into the fewest row ranges whose cones fit the shared-memory
// budget.  A cone is unrolled top-down with the addition rule of section 4:
// parent rows [a, e] with window offset o and spread s have
//   lower half rows [dl(a), dl(e)], offset o,          spread s
//   upper half rows [a - dl(a), e - dl(e)], offset o + dl(e), spread s + dl(e) - dl(a)
// and parent row Dt reads the upper half at column tau + dl(e) - dl(Dt).
//
// Staged rows reach shared memory by TMA in one of two formats per launch:
// row boxes (a 2-D [rows][nt] map; each row window is copied by whole boxes
// of up to 256 elements) or row blocks (a 3-D [rows][nt / C][C] map, C
// elements = 128 bytes or 64; one copy brings 2^p consecutive rows of K
// chunks, landing with row pitch K * C, so a node of R rows takes popcount(R)
// copies).  Row blocks need nt to be a multiple of C and windows that start
// on a chunk boundary; the input channels of a from-input cone share one
// window (the union of theirs) so they form one block.
//
// The level grouping, W and, where few items would leave SMs idle, the
// shared memory per item are chosen by a cost model (dynamic programming
// over group boundaries).  A launch's time is the 3.3-norm of its HBM time
// (the rows it reads and writes, each once) and its on-chip time (work items
// per block slot of the GPU times the time of one item, a sum over its
// stages, row strips, runs, walks and copies), plus a constant.  The
// constants are a least-squares fit to 7710 launches measured on a GB300 (11
// shapes from 64 x 1024 to 4096 x 65536, 3 data types, random level
// groupings, 9 tiles, 3 budgets; mean absolute error 7 %).
#include "fdmt_fused.h"

#include <algorithm>
#include <cmath>
#include <limits>

namespace fdmt {
namespace {

constexpr int32_t kBarrierBytes = 128 + kUnderRead;  // mbarrier slot and slack, keeps regions 128-byte aligned
constexpr double kHbmRate = 6.74e12;         // bytes/s of unique rows in and out
constexpr double kL2Rate = 14.0e12;          // bytes/s of staged rows (halos and overlaps come from L2)
constexpr double kNorm = 3.3;
constexpr double kLaunchSeconds = 6.6e-6;
constexpr double kStageSeconds = 0.325e-6;   // one item, two blocks on its SM: per stage,
constexpr double kPairSeconds = 16.9e-9;     //   row strip of a pair stage,
constexpr double kSingleSeconds = 6.3e-9;    //   of a single stage,
constexpr double kTopSeconds = 16.6e-9;      //   of the top stage (its stores) on top of that,
constexpr double kRunSeconds = 6.9e-9;       //   run,
constexpr double kWalkSeconds = 8.3e-9;      //   sample read or row written of a walk,
constexpr double kCopySeconds = 27.3e-9;     //   copy instruction
constexpr double kByteSeconds = 0.67e-12;    //   and byte copied
constexpr double kAloneShare = 0.6;          // time of an item whose block has an SM to itself
constexpr double kWaveTail = 0.7;            // a started wave counts as at most this much more than its items
constexpr double kSms = 152;
constexpr int64_t kPadRows = 4096;           // rows from this length on are padded between launches
constexpr double kMaxBlocksPerSm = 2;        // the fused kernel's register budget

int64_t round_up(int64_t v, int64_t a) { return (v + a - 1) / a * a; }
int64_t ceil_to(int64_t v, int64_t a) { return round_up(v, a); }

struct Node {
  int32_t band, a, e;  // band index at its level, first and last row
  int32_t o, s;        // window [T0 - o, T0 - o + W + s)
  int32_t smem = 0;    // byte offset of row a
  int32_t stride = 0;  // elements per row in shared memory
  int32_t delta = 0;   // column of time T0 - o within the stored row
  int32_t xsmem = 0, xstride = 0, xdelta = 0;  // staged input (level 0 of an input cone)
  int32_t klo = -1, khi = -1;  // the halves in the level below (khi < 0: none, rows pass up)
};

// The rows of one node of a single or pair stage: its first column piece's
// ops, ops[op .. op + n), and what a run needs beside them.
struct NodeRows {
  int32_t op, n;
  int32_t width;         // the node's columns
  int32_t pitch;         // columns from one output row to the next (shared memory)
  int32_t es;            // bytes per source sample
  int32_t g[4];          // row strides of the sources
  int32_t flags;         // kOpLoOne, kOpHiOne, kOpNoHi
  int32_t step;          // first of n - 1 row steps (bit 0 inc, bit 1 sub; see FusedRun)
};
struct StageRows {
  std::vector<NodeRows> nodes;
  std::vector<uint8_t> steps;
};

struct ConeOut {
  FusedTemplate tpl{};
  std::vector<FusedLoad> loads;
  std::vector<FusedWalk> walks;                 // the first stage of a launch from the input
  std::vector<double> walk_cost;                //   and what each costs (shared-memory pipe slots)
  std::vector<std::vector<FusedOp>> stage_ops;  // single / pair stages, in row order (before the warp split)
  std::vector<StageRows> stage_rows;            // the same by node (empty for the search)
  std::vector<int32_t> kinds;                   // stage kinds
  double hbm = 0;
  double slots = 0;  // shared-memory pipe slots of one tile (warp instructions), for inspection
  double nops = 0;   // ops and walks of one tile, for inspection
  double work = 0;   // cost model: seconds of the stages of one tile
};

// Region sizes of one cone: S = staged source rows (input channels or the
// base level), Pa / Pb = computed levels, alternating.  A group lays all its
// cones out at the same region bases (the maxima over its cones) so that a
// block can stage the next cone into S while it still computes in Pa / Pb.
struct ConeShape {
  std::vector<std::vector<Node>> nodes;  // [level - lb]
  int64_t s_bytes = 0, pa_bytes = 0, pb_bytes = 0;
  int64_t pt_bytes = 0;  // search: the top level in the search layout
  int32_t top_rows = 0;  // rows of the top node
  int64_t prog_bytes = 0;  // at most this much of the item's programme (walks and runs)
  std::vector<std::pair<int32_t, int32_t>> needs;  // (window elements from the aligned start, rows) per staged node
  int32_t x_o = 0;  // row blocks, from input: the channels' common window starts at T0 - x_o
  // Empty, for levels lb .. lb + m, in the memory it has (a plan shapes cones by
  // the hundred thousand).
  void reset(int32_t m) {
    nodes.resize(m + 1);
    for (std::vector<Node> &v : nodes) v.clear();
    needs.clear();
    s_bytes = pa_bytes = pb_bytes = pt_bytes = prog_bytes = 0;
    top_rows = x_o = 0;
  }
};

// Staging format of a launch.  chunk == 0: row boxes of `box` elements.
// chunk > 0: row blocks of kchunks chunks (kchunks == 0 while the windows
// are being measured: each cone then uses its own widest window).
struct StageFmt {
  int32_t box = 0;
  int32_t chunk = 0, kchunks = 0;
  int32_t max_p = 0;  // copies bring at most 2^max_p rows
  int32_t search_k = 0;  // > 0: the launch ends with the boxcar search of this many widths
  bool compact = false;  // least shared memory: tight row pitches, programmes in global memory
  const std::vector<int32_t> *in_shift = nullptr;  // mapped input (row boxes): each channel's delay
  bool descending = false;
  int32_t shift(int32_t channel) const { return in_shift != nullptr ? (*in_shift)[channel] : 0; }
};

}  // namespace

// The levels a group (lb, lt] stores: lb (staged, or the input when lb = 0),
// then every level a stage ends on.  From the input the first stage ends on
// level 1; an odd number of levels left takes one single-level stage first;
// the rest are pairs.
std::vector<int32_t> stored_levels(int32_t lb, int32_t lt) {
  std::vector<int32_t> v{lb};
  int32_t cur = lb;
  if (lb == 0) {
    v.push_back(1);
    cur = 1;
  }
  if (((lt - cur) & 1) != 0) v.push_back(++cur);
  while (cur < lt) {
    cur += 2;
    v.push_back(cur);
  }
  return v;
}

namespace {

// Row pitch of a stored level's node of `cols` columns.  Rows that nearly
// fill whole strips get the room of whole strips, so that runs store them
// without testing columns (kRunWhole): a strip may start up to kRunGrow
// columns before its row (in the free columns of the row before it) and
// reaches at most the end of its row's pitch.
int32_t stored_pitch(int32_t cols, bool tight) {
  const int32_t whole = (int32_t)round_up(cols + kRunGrow, kPieceCols);
  if (tight) return (int32_t)round_up(cols, 4);
  return whole - cols <= cols / 6 + kRunGrow ? whole : (int32_t)round_up(cols + kRunGrow, 4);
}

void shape_cone(const Tables &t, int32_t lb, int32_t lt, int32_t band, int32_t r0, int32_t r1,
                int32_t W, const FusedPlan &fp, const StageFmt &f, ConeShape &cs) {
  const bool from_input = (lb == 0);
  const int32_t sA = fp.acc_size, sB = fp.level_size[lb], sI = fp.input_size;
  const int32_t alignB = f.chunk > 0 ? f.chunk : 16 / sB, alignI = f.chunk > 0 ? f.chunk : 16 / sI;
  const int32_t m = lt - lb;
  cs.reset(m);
  std::vector<std::vector<Node>> &nodes = cs.nodes;
  const int32_t hist = f.search_k > 0 ? search_hist(f.search_k) : 0;
  nodes[m].push_back(Node{band, r0, r1, hist, hist});
  for (int32_t l = lt; l > lb; --l) {
    std::vector<Node> &kids = nodes[l - 1 - lb];
    for (Node &p : nodes[l - lb]) {
      p.klo = (int32_t)kids.size();
      if (!has_upper(t, l, p.band)) {
        // Nf not a power of two: a band with no channel above its border
        // passes its lower half's rows up unchanged (same rows, same window).
        kids.push_back(Node{2 * p.band, p.a, p.e, p.o, p.s});
        continue;
      }
      const std::vector<int32_t> &dl = t.dl[l][p.band];
      const int32_t da = dl[p.a], de = dl[p.e];
      kids.push_back(Node{2 * p.band, da, de, p.o, p.s});
      p.khi = (int32_t)kids.size();
      kids.push_back(Node{2 * p.band + 1, p.a - da, p.e - de, p.o + de, p.s + de - da});
    }
  }
  // Row pitch of a staged row whose window needs `need` elements.
  auto pitch = [&](int32_t need, int32_t own_max) -> int32_t {
    if (f.chunk == 0) return (int32_t)round_up(need, f.box);
    return f.kchunks > 0 ? f.kchunks * f.chunk : (int32_t)round_up(own_max, f.chunk);
  };
  int32_t own_max = 0;  // widest staged window of this cone (row blocks, measuring)
  if (from_input && f.chunk > 0) {
    for (const Node &n : nodes[0]) cs.x_o = std::max(cs.x_o, n.o + n.e);
    cs.x_o = (int32_t)ceil_to(cs.x_o, alignI);
    for (const Node &n : nodes[0]) own_max = std::max(own_max, W + n.s + cs.x_o - n.o);
  } else if (!from_input) {
    for (const Node &n : nodes[0]) own_max = std::max(own_max, W + n.s + (int32_t)ceil_to(n.o, alignB) - n.o);
  }
  // Level index i = l - lb for l in [lb, lt).  Only the stored levels of
  // the group's stage sequence take shared memory: the staged base level
  // (S), then the stored computed levels alternately in Pa and Pb.  In a
  // launch from the input, level 0 is never stored (the first stage walks
  // the staged input samples).
  const std::vector<int32_t> st = stored_levels(lb, lt);
  int64_t pa = 0, pb = 0;
  int32_t k = 0;  // index among stored computed levels
  for (int32_t i = 0; i < m; ++i) {
    const bool staged = (i == 0 && !from_input);
    int64_t off = staged ? 0 : kUnderRead;
    const bool stored = !(i == 0 && from_input) &&
                        std::find(st.begin(), st.end(), lb + i) != st.end();
    for (Node &n : nodes[i]) {
      const int32_t rows = n.e - n.a + 1;
      n.delta = 0;
      n.smem = -1;
      if (staged) {
        const int32_t ceil_o = (int32_t)ceil_to(n.o, alignB);
        n.delta = ceil_o - n.o;
        cs.needs.emplace_back(W + n.s + n.delta, n.e - n.a + 1);
        n.stride = pitch(W + n.s + n.delta, own_max);
        n.smem = (int32_t)off;
        off += round_up((int64_t)rows * n.stride * sB, 128);
      } else if (stored) {
        n.stride = stored_pitch(W + n.s, f.compact);
        n.smem = (int32_t)off;
        off += round_up((int64_t)rows * n.stride * sA, 128);
      }
      if (i == 0 && from_input) {
        if (f.chunk > 0) {
          // One block of consecutive channels, one common window.
          n.xdelta = cs.x_o - n.o;
          n.xstride = pitch(W + n.s + n.xdelta, own_max);
          n.xsmem = (int32_t)cs.s_bytes;
          cs.s_bytes += (int64_t)n.xstride * sI;
        } else {
          // (a mapped channel is read its delay earlier: zeros before the raw row)
          const int32_t at = n.o + f.shift(n.band);
          n.xdelta = (int32_t)ceil_to((int64_t)at + n.e, alignI) - at;
          n.xstride = pitch(W + n.s + n.xdelta, 0);
          n.xsmem = (int32_t)cs.s_bytes;
          cs.s_bytes += round_up((int64_t)n.xstride * sI, 128);
        }
        cs.needs.emplace_back(W + n.s + n.xdelta, 1);
      }
    }
    if (i == 0 && from_input) cs.s_bytes = round_up(cs.s_bytes, 128);
    if (staged) {
      cs.s_bytes = off;
    } else if (stored) {  // (the region starts with the slack before its first row)
      if ((k & 1) == 0) pa = std::max(pa, off);
      else pb = std::max(pb, off);
      ++k;
    }
  }
  cs.pa_bytes = pa;
  cs.pb_bytes = pb;
  // Walks and runs of the stages' nodes: their rows are cut after 32 rows or
  // (lower_stage) where the delay has grown by 9 .. 17 columns.
  for (size_t si = 1; si < st.size(); ++si) {
    const int32_t i = st[si] - lb;
    for (const Node &n : nodes[i]) {
      const int64_t cols = (i == m && f.search_k == 0) ? W : W + n.s, rows = n.e - n.a + 1;
      if (from_input && si == 1) {
        cs.prog_bytes += (rows + 31) / 32 * ((cols + kPieceCols - 1) / kPieceCols) * (int64_t)sizeof(FusedWalk);
        continue;
      }
      const std::vector<int32_t> &dl = t.dl[lb + i][n.band];
      const int64_t grow = n.khi >= 0 ? dl[n.e] - dl[n.a] : 0;
      const int64_t strips = (cols + kRunGrow + kPieceCols - 1) / kPieceCols;
      cs.prog_bytes += (1 + rows / kRunRows + grow / 9) * strips * (int64_t)sizeof(FusedRun);
    }
  }
  if (f.search_k > 0) {
    // The top rows, W + hist columns each in the search layout (region Pt).
    Node &n = nodes[m].front();
    n.delta = 0;
    n.smem = 0;
    // rows 4 words apart modulo the 32 banks: 16-byte loads of eight rows
    // at the same column hit distinct banks
    n.stride = (int32_t)round_up(search_pidx(W + n.s), 4);
    n.stride += (4 - n.stride % 32 + 32) % 32;
    cs.pt_bytes = round_up((int64_t)(n.e - n.a + 1) * n.stride * sA, 128);
    cs.top_rows = n.e - n.a + 1;
  }
}

// The search's per (row, width) bests of a work item with `rows` top rows
// (one 64-bit word each).
int64_t search_q_bytes(const StageFmt &f, int64_t rows) {
  if (f.search_k <= 0) return 0;
  return round_up(rows * f.search_k * 8, 128);
}

// Bytes of one programme slot (0: far) for items of `stages` stages and at most
// `descs` bytes of walks and runs (a stage's split over the warps can cut a
// run in two at each of its seven borders).
int64_t prog_slot_bytes(const StageFmt &f, int64_t stages, int64_t descs) {
  if (f.compact) return 0;
  const int64_t n = stages * (kProgStageBytes + (kFusedBlockWarps - 1) * (int64_t)sizeof(FusedRun)) + descs;
  return std::max<int64_t>(kProgMinBytes / 2, round_up(n, 128));
}

int64_t prog_area(int64_t slot) { return std::max<int64_t>(kProgMinBytes, 2 * slot); }

int64_t cone_bytes(const StageFmt &f, const ConeShape &cs, int64_t stages) {
  return kBarrierBytes + cs.s_bytes + cs.pa_bytes + cs.pb_bytes + cs.pt_bytes +
         prog_area(prog_slot_bytes(f, stages, cs.prog_bytes)) + kOverRead;
}

// Emits the loads, inits and ops of a shaped cone at the given region bases.
// Row blocks: copies of 2^p rows (p <= max_p) covering rows [0, rows) of a
// block, largest first; calls emit(first row, p).
template <class F>
void row_pieces(int32_t rows, int32_t max_p, F emit) {
  for (int32_t r = 0; r < rows;) {
    int32_t p = max_p;
    while ((1 << p) > rows - r) --p;
    emit(r, p);
    r += 1 << p;
  }
}

// Shared-memory pipe slots (warp instructions, 32 columns each) of one op
// per 32 columns: its loads, the shuffle of a shifted upper half, the store.
double op_slots(int32_t kind, int32_t flags) {
  const double hi = (flags & kOpNoHi) ? 0 : 1;
  if (kind == kStageSingle) return ((flags & kOpLoSame) ? 0 : 1) + hi + 1;
  const double lo = (flags & kOpLoSame) ? 0 : ((flags & kOpLoOne) ? 1 : 2);
  const double up = (flags & kOpNoHi) ? 0 : ((flags & kOpHiShift) ? 1 : ((flags & kOpHiOne) ? 1 : 2));
  return lo + up + 1;
}

// Rows ra .. re of level-1 band `band` as a walk: its row steps, and with
// `moves` whether its upper sums move.  *cost: the same slots of the walk: the
// first row's samples of both channels, then one sample more per row, or,
// where the lower row grows, one and the upper channel's j + 1 again or 9
// shuffles and 8 selections of 8 columns each (kWalkMoves); and the rows'
// stores.
FusedWalk walk_rows(const Tables &t, int32_t band, bool upper, int32_t ra, int32_t re, bool moves, double *cost) {
  const std::vector<int32_t> &dl = t.dl[1][band];
  FusedWalk wk{};
  wk.a = ra;
  wk.e = re;
  wk.dl0 = dl[ra];
  int32_t j = ra - wk.dl0;
  double again = wk.dl0 + 1 + (upper ? j + 1 : 0) + 1, moved = again;
  for (int32_t r = ra + 1; r <= re; ++r) {
    const bool grows = dl[r] > dl[r - 1];
    if (grows) wk.bits |= 1 << (r - ra - 1);
    again += upper && grows ? 2 + j + 1 : 2;
    moved += upper && grows ? 2 + 17.0 / 8 : 2;
    j += grows ? 0 : 1;
  }
  wk.flags = !upper ? kWalkNoUpper : (moves && moved < again ? kWalkMoves : 0);
  *cost = wk.flags & kWalkMoves ? moved : again;
  return wk;
}

// Whether a plan's walks move their upper sums where that is less work: if it
// saves enough of all walks (whole bands counted), since the launch's other
// walks pay for the code.  Measured on a GB300, walks' cost without over with
// moves and the first launch without / with them, us: 1024 x 65536 x 2048
// float32 1.01, 185 / 193; 139 x 48444 x 541 float32 1.12, 46.0 / 47.1; 1024 x
// 65536 x 4096 float32 1.13, 340 / 335; 366 x 8424 x 2258 fp16 state 1.31,
// 43.3 / 41.3; 64 x 47828 x 847 float32 1.85, 72.5 / 57.7; 32 x 150000 x 4000
// float32 5.4, 2516 / 505.
constexpr double kMovesPay = 1.3;
bool moves_pay(const Tables &t) {
  if (t.levels < 1) return false;
  double again = 0, least = 0;
  for (int32_t b = 0; b < (int32_t)t.band_rows[1].size(); ++b) {
    if (!has_upper(t, 1, b)) continue;
    for (int32_t r = 0; r < t.band_rows[1][b]; r += 32) {
      const int32_t e = std::min(t.band_rows[1][b], r + 32) - 1;
      double cost = 0;
      walk_rows(t, b, true, r, e, false, &cost);
      again += cost;
      walk_rows(t, b, true, r, e, true, &cost);
      least += cost;
    }
  }
  return again > kMovesPay * least;
}

// Cost model: the rows of one node of a single or pair stage.
double stage_work(const Tables &t, int32_t level, const Node &p, int32_t cols, bool pair, bool to_global) {
  const std::vector<int32_t> &dl = t.dl[level][p.band];
  const int32_t grow = p.khi >= 0 ? std::min(kRunGrow, dl[p.e] - dl[p.a]) : 0;
  const double strips = (cols + grow + kPieceCols - 1) / kPieceCols;
  return strips * ((p.e - p.a + 1) * ((pair ? kPairSeconds : kSingleSeconds) + (to_global ? kTopSeconds : 0)) + kRunSeconds);
}

// Emits the loads, walks and stage ops of a shaped cone at the given region
// bases.
void emit_cone(const Tables &t, int32_t lb, int32_t lt, int32_t W, const FusedPlan &fp, const StageFmt &f,
               ConeShape &cs, int64_t base_s, int64_t base_a, int64_t base_b, int64_t base_t, ConeOut &c) {
  const bool search = f.search_k > 0;
  const bool from_input = (lb == 0);
  const int32_t sA = fp.acc_size, sB = fp.level_size[lb], sI = fp.input_size;
  const int32_t m = lt - lb;
  std::vector<std::vector<Node>> &nodes = cs.nodes;
  const std::vector<int32_t> st = stored_levels(lb, lt);
  {
    int32_t k = 0;
    for (int32_t i = 0; i < m; ++i) {
      const bool staged = (i == 0 && !from_input);
      bool any = false;
      for (Node &n : nodes[i]) {
        if (n.smem >= 0) {
          any = true;
          n.smem += (int32_t)(staged ? base_s : ((k & 1) == 0 ? base_a : base_b));
        }
        n.xsmem += (int32_t)base_s;
      }
      if (any && !staged) ++k;
    }
    if (search) nodes[m].front().smem += (int32_t)base_t;
  }
  c = ConeOut();
  int64_t tx = 0;
  if (from_input && f.chunk > 0) {
    const Node &n0 = nodes[0].front();
    row_pieces((int32_t)nodes[0].size(), f.max_p, [&](int32_t r, int32_t p) {
      c.loads.push_back(FusedLoad{n0.band + r, n0.xsmem + r * n0.xstride * sI, -cs.x_o, p});
      tx += ((int64_t)n0.xstride * sI) << p;
    });
  }
  if (from_input) {
    if (f.chunk == 0)
      for (const Node &n : nodes[0]) {
        c.loads.push_back(FusedLoad{f.descending ? t.nf - 1 - n.band : n.band, n.xsmem,
                                    -(int32_t)ceil_to((int64_t)n.o + n.e + f.shift(n.band), 16 / sI),
                                    n.xstride / f.box});
        tx += (int64_t)n.xstride * sI;
      }
  } else {
    for (const Node &n : nodes[0]) {
      const int32_t row0 = t.band_row0[lb][n.band];
      const int32_t xoff = -(int32_t)ceil_to(n.o, f.chunk > 0 ? f.chunk : 16 / sB);
      if (f.chunk > 0) {
        row_pieces(n.e - n.a + 1, f.max_p, [&](int32_t r, int32_t p) {
          c.loads.push_back(FusedLoad{row0 + n.a + r, n.smem + r * n.stride * sB, xoff, p});
          tx += ((int64_t)n.stride * sB) << p;
        });
        continue;
      }
      for (int32_t j = n.a; j <= n.e; ++j) {
        c.loads.push_back(FusedLoad{row0 + j, n.smem + (j - n.a) * n.stride * sB, xoff, n.stride / f.box});
        tx += (int64_t)n.stride * sB;
      }
    }
  }
  c.tpl.tx_bytes = (int32_t)tx;
  c.hbm += (double)tx;
  c.slots += (double)tx / 128.0;  // the copies' writes into shared memory

  // Byte offset of row r, column col (relative to the window start) of a
  // stored node at level index i.
  auto leaf = [&](int32_t i, const Node &n, int32_t r, int32_t col) -> int32_t {
    const int32_t es = (i == 0 && !from_input) ? sB : sA;
    return n.smem + ((r - n.a) * n.stride + n.delta + col) * es;
  };
  auto dlv = [&](int32_t l, int32_t band, int32_t r) { return t.dl[l][band][r]; };

  for (size_t si = 0; si + 1 < st.size(); ++si) {
    const int32_t l1 = st[si + 1];          // level the stage ends on
    const int32_t io = l1 - lb;             // its level index
    const bool top = (l1 == lt);
    const std::vector<Node> &par = nodes[io];
    if (from_input && si == 0) {
      // Level 1 from the staged input: one walk per node, row run and piece.
      c.kinds.push_back(kStageWalk);
      const std::vector<Node> &ch = nodes[0];
      for (size_t pi = 0; pi < par.size(); ++pi) {
        const Node &p = par[pi];
        const bool upper = p.khi >= 0;
        const Node &clo = ch[p.klo], &chi = upper ? ch[p.khi] : ch[p.klo];
        const int32_t de = upper ? dlv(1, p.band, p.e) : 0;
        const int32_t wp = top ? W : W + p.s;
        for (int32_t c0 = 0; c0 < wp; c0 += kPieceCols) {
          for (int32_t ra = p.a; ra <= p.e; ra += 32) {
            const int32_t re = std::min(p.e, ra + 31);
            double cost = 0;
            FusedWalk wk = walk_rows(t, p.band, upper, ra, re, fp.moves, &cost);
            wk.dst = top ? (t.band_row0[lt][p.band] + ra) : leaf(io, p, ra, c0);
            wk.dst_row = top ? 0 : p.stride * sA;
            wk.x_lo = clo.xsmem + (clo.xdelta + c0) * sI;
            wk.x_hi = chi.xsmem + (chi.xdelta + c0 + de) * sI;
            wk.width = std::min(kPieceCols, wp - c0);
            wk.col = c0;
            wk.chan = clo.band;
            c.walks.push_back(wk);
            c.walk_cost.push_back(cost);
            c.slots += cost * kLaneCols;
            c.work += cost * kWalkSeconds + (top ? (re - ra + 1) * kTopSeconds : 0);
            c.nops += 1;
            if (top) c.hbm += (double)std::min(kPieceCols, W - c0) * (re - ra + 1) * fp.level_size[lt];
          }
        }
      }
      continue;
    }
    const bool pair = (l1 - st[si] == 2);
    const int32_t kind = pair ? kStagePair : kStageSingle;
    // With a search the top level goes to Pt (search layout), all W + hist
    // columns; otherwise to global memory, W columns.
    const bool to_global = top && !search;
    c.kinds.push_back(kind | (top && search ? kStagePadded : 0));
    std::vector<FusedOp> ops;
    StageRows sr;
    const int32_t wmax = to_global ? W : [&] {
      int32_t v = 0;
      for (const Node &p : par) v = std::max(v, W + p.s);
      return v;
    }();
    for (int32_t c0 = 0; c0 < wmax; c0 += kPieceCols) {
      for (size_t pi = 0; pi < par.size(); ++pi) {
        const Node &p = par[pi];
        const int32_t wp = to_global ? W : W + p.s;
        if (c0 >= wp) continue;
        const int32_t width = std::min(kPieceCols, wp - c0);
        const bool upper = p.khi >= 0;
        const int32_t de = dlv(l1, p.band, p.e);
        const std::vector<Node> &kid = nodes[io - 1];
        const Node &klo = kid[p.klo], &khi = upper ? kid[p.khi] : kid[p.klo];
        if (c0 == 0) {
          NodeRows nr{};
          nr.op = (int32_t)ops.size();
          nr.n = p.e - p.a + 1;
          nr.width = wp;
          nr.pitch = to_global ? 0 : p.stride;
          const int32_t is = pair ? io - 2 : io - 1;  // level index of the sources
          nr.es = (is == 0 && !from_input) ? sB : sA;
          nr.flags = upper ? 0 : kOpNoHi;
          if (!pair) {
            nr.g[0] = klo.stride * nr.es;
            nr.g[2] = khi.stride * nr.es;
          } else {
            const std::vector<Node> &g = nodes[io - 2];
            nr.g[0] = g[klo.klo].stride * nr.es;
            nr.g[2] = g[khi.klo].stride * nr.es;
            if (klo.khi >= 0) nr.g[1] = g[klo.khi].stride * nr.es;
            else nr.flags |= kOpLoOne;
            if (upper) {
              if (khi.khi >= 0) nr.g[3] = g[khi.khi].stride * nr.es;
              else nr.flags |= kOpHiOne;
            }
          }
          nr.step = (int32_t)sr.steps.size();
          for (int32_t dt = p.a; dt < p.e; ++dt) {
            const int32_t j = dlv(l1, p.band, dt), inc = dlv(l1, p.band, dt + 1) - j;
            const Node &k = inc ? klo : khi;
            const int32_t r = inc ? j : dt - j;  // the row of k that grows
            const int32_t sub = (pair && k.khi >= 0) ? dlv(l1 - 1, k.band, r + 1) - dlv(l1 - 1, k.band, r) : 1;
            sr.steps.push_back((uint8_t)(inc | sub << 1));
          }
          c.work += stage_work(t, l1, p, wp, pair, to_global);
          sr.nodes.push_back(nr);
        }
        int32_t pj = -1, pm = -1;
        for (int32_t dt = p.a; dt <= p.e; ++dt) {
          // (a band without an upper half has dl = dt: row dt is its lower row dt)
          const int32_t j = dlv(l1, p.band, dt), mrow = dt - j, q = de - j;
          FusedOp op{};
          if (to_global)
            op.dst = t.band_row0[lt][p.band] + dt;
          else if (top)  // Pt: the row's base plus the piece's first column in the search layout
            op.dst = p.smem + ((dt - p.a) * p.stride + search_pidx(c0)) * sA;
          else
            op.dst = leaf(io, p, dt, c0);
          op.width = width;
          op.col = c0;
          op.flags = 0;
          if (!pair) {
            op.p0 = leaf(io - 1, klo, j, c0);
            if (upper) op.p1 = leaf(io - 1, khi, mrow, c0 + q);
            else op.flags |= kOpNoHi;
          } else {
            // klo / khi are not stored: expand them into their halves (one
            // term where a half passes its lower rows up).
            const std::vector<Node> &g = nodes[io - 2];
            const int32_t l0 = l1 - 1;
            if (klo.khi >= 0) {
              const int32_t j1 = dlv(l0, klo.band, j), q1 = dlv(l0, klo.band, klo.e) - j1;
              op.p0 = leaf(io - 2, g[klo.klo], j1, c0);
              op.p1 = leaf(io - 2, g[klo.khi], j - j1, c0 + q1);
            } else {
              op.p0 = leaf(io - 2, g[klo.klo], j, c0);
              op.flags |= kOpLoOne;
            }
            if (!upper) {
              op.flags |= kOpNoHi;
            } else if (khi.khi >= 0) {
              const int32_t j2 = dlv(l0, khi.band, mrow), q2 = dlv(l0, khi.band, khi.e) - j2;
              op.p2 = leaf(io - 2, g[khi.klo], j2, c0 + q);
              op.p3 = leaf(io - 2, g[khi.khi], mrow - j2, c0 + q + q2);
            } else {
              op.p2 = leaf(io - 2, g[khi.klo], mrow, c0 + q);
              op.flags |= kOpHiOne;
            }
          }
          if (dt > p.a && j == pj) op.flags |= kOpLoSame;
          if (pair && upper && dt > p.a && mrow == pm && j == pj + 1) op.flags |= kOpHiShift;
          pj = j;
          pm = mrow;
          ops.push_back(op);
          c.slots += op_slots(kind, op.flags) * kLaneCols;
          c.nops += 1;
          if (to_global) c.hbm += (double)width * fp.level_size[lt];
        }
      }
    }
    c.stage_ops.push_back(std::move(ops));
    c.stage_rows.push_back(std::move(sr));
  }
  if (search) {
    // One search op per top row: the row in Pt, its global row, the W
    // owned columns after hist columns of history.
    c.kinds.push_back(kStageSearch);
    std::vector<FusedOp> ops;
    const Node &p = nodes[m].front();
    for (int32_t dt = p.a; dt <= p.e; ++dt) {
      FusedOp op{};
      op.dst = t.band_row0[lt][p.band] + dt;
      op.p0 = p.smem + (dt - p.a) * p.stride * sA;
      op.width = W;
      op.col = p.s;
      ops.push_back(op);
      c.slots += 6.0 * (W + p.s) / 32;
      c.nops += 1;
      c.hbm += (double)W * fp.level_size[lt];
    }
    c.stage_ops.push_back(std::move(ops));
  }
  c.tpl.n_stages = (int32_t)c.kinds.size();
}

// What emit_cone adds to the cost model, without the loads, walks and ops:
// `work`, `hbm`, the bytes copied and the number of copies.  The search over
// groupings and tiles compares launches by this alone.
void count_cone(const Tables &t, int32_t lb, int32_t lt, int32_t W, const FusedPlan &fp, const StageFmt &f,
                const ConeShape &cs, ConeOut &c, int32_t &copies) {
  const bool from_input = (lb == 0);
  const int32_t sB = fp.level_size[lb], sI = fp.input_size;
  const std::vector<int32_t> st = stored_levels(lb, lt);
  int64_t tx = 0;
  const std::vector<Node> &base = cs.nodes[0];
  if (from_input && f.chunk > 0) {
    row_pieces((int32_t)base.size(), f.max_p, [&](int32_t, int32_t) { ++copies; });
    for (const Node &n : base) tx += (int64_t)n.xstride * sI;
  } else {
    for (const Node &n : base) {
      const int32_t rows = from_input ? 1 : n.e - n.a + 1;
      tx += (int64_t)rows * (from_input ? n.xstride * sI : n.stride * sB);
      if (f.chunk > 0) row_pieces(rows, f.max_p, [&](int32_t, int32_t) { ++copies; });
      else copies += rows;
    }
  }
  c.tpl.tx_bytes = (int32_t)tx;
  c.hbm = (double)tx;
  for (size_t si = 0; si + 1 < st.size(); ++si) {
    const int32_t l1 = st[si + 1], io = l1 - lb;
    const bool top = (l1 == lt), to_global = top && f.search_k == 0;
    for (const Node &p : cs.nodes[io]) {
      const bool upper = p.khi >= 0;
      const int32_t n = p.e - p.a + 1, wp = to_global ? W : W + p.s;
      if (from_input && si == 0) {
        const double pieces = (wp + kPieceCols - 1) / kPieceCols;
        for (int32_t ra = p.a; ra <= p.e; ra += 32) {
          double cost = 0;
          const FusedWalk wk = walk_rows(t, p.band, upper, ra, std::min(p.e, ra + 31), fp.moves, &cost);
          c.work += pieces * (cost * kWalkSeconds + (top ? (wk.e - ra + 1) * kTopSeconds : 0));
        }
      } else {
        c.work += stage_work(t, l1, p, wp, l1 - st[si] == 2, to_global);
      }
      if (to_global) c.hbm += (double)W * n * fp.level_size[lt];
    }
  }
  if (f.search_k > 0) c.hbm += (double)W * (cs.nodes[lt - lb].front().e - cs.nodes[lt - lb].front().a + 1) * fp.level_size[lt];
}

// Splits a stage's ops (or walks) into kFusedBlockWarps contiguous runs of
// about equal cost; returns the first index of each run and the end.
std::vector<int32_t> split_warps(const std::vector<double> &cost) {
  double total = 0;
  for (double v : cost) total += v;
  std::vector<int32_t> b(kFusedBlockWarps + 1, (int32_t)cost.size());
  b[0] = 0;
  double acc = 0;
  int32_t w = 1;
  for (int32_t i = 0; i < (int32_t)cost.size() && w < kFusedBlockWarps; ++i) {
    acc += cost[i];
    while (w < kFusedBlockWarps && acc >= total * w / kFusedBlockWarps) b[w++] = i + 1;
  }
  for (; w < kFusedBlockWarps; ++w) b[w] = (int32_t)cost.size();
  return b;
}

// One work item (template): the cones of a bundle, their stage ops merged
// and split over the warps.  Stage offsets are relative to the item's walks
// and ops until the group is appended to the plan.
struct ItemOut {
  FusedTemplate tpl{};
  std::vector<FusedLoad> loads;
  std::vector<FusedWalk> walks;
  std::vector<FusedOp> ops;
  std::vector<int32_t> stages;  // kStageWords per stage
  std::vector<StageRows> rows;  // per stage: its nodes' rows, op indices into `ops` (empty: walk, search)
  double hbm = 0, slots = 0, nops = 0, work = 0;
};

// Cost model: one item beside its rows.
double item_work(int64_t stages, int32_t copies, int32_t tx_bytes) {
  return (double)stages * (kStageSeconds + (kFusedBlockWarps - 1) * kRunSeconds) + copies * kCopySeconds +
         tx_bytes * kByteSeconds;
}

struct GroupBuild {
  bool ok = false;
  FusedGroup g;
  int64_t items = 0;           // templates
  std::vector<ItemOut> cones;  // filled when emitted
  int32_t budget = 0;
  double seconds = 0;
};

// All cones of group (lb, lt] for tile W: each band of level lt is split
// into the fewest equal row ranges whose cones fit `budget`; the cones are
// then laid out at the group's region bases.  The group total can exceed the
// per-cone budget slightly (maxima of different cones); the budget is
// lowered until the total fits.
// TMA box width for staged rows with the given (window, rows) needs, of
// `es`-byte elements: a multiple of 128 bytes (every copy lands 128-byte
// aligned in shared memory) and at most 256 elements, chosen to minimise
// the copied bytes plus a fixed cost per copy (a copy's issue and
// completion cost about as much as moving kCopyBytes more).
constexpr int64_t kCopyBytes = 1024;
int32_t choose_box(const std::vector<std::pair<int32_t, int32_t>> &needs, int32_t es) {
  const int32_t q = 128 / es;
  int32_t best = 0;
  int64_t best_cost = std::numeric_limits<int64_t>::max();
  for (int32_t box = q; box <= 256; box += q) {
    int64_t cost = 0;
    for (const auto &nr : needs) {
      const int64_t nbox = (nr.first + box - 1) / box;
      cost += nr.second * nbox * ((int64_t)box * es + kCopyBytes);
    }
    if (cost < best_cost) {
      best_cost = cost;
      best = box;
    }
  }
  return best;
}

// What a build of a group is for: the windows of its cones (`needs`), its
// cost as well, or its descriptors as well.
enum class Build { kMeasure, kCount, kEmit };

GroupBuild build_group_fmt(const Tables &t, int64_t nt, int32_t lb, int32_t lt, int32_t W,
                           const FusedPlan &fp, int32_t budget, const StageFmt &f,
                           std::vector<std::pair<int32_t, int32_t>> *needs, Build what) {
  GroupBuild gb;
  const int32_t nb = bands_at(t.nf, lt);
  const int64_t nst = (int64_t)stored_levels(lb, lt).size() - 1 + (f.search_k > 0 ? 1 : 0);
  ConeShape trial;
  for (int32_t cone_budget = budget; cone_budget >= 4096; cone_budget = cone_budget * 7 / 8) {
    std::vector<ConeShape> shapes;
    bool ok = true;
    for (int32_t b = 0; b < nb && ok; ++b) {
      const int32_t rows = t.band_rows[lt][b];
      auto fits = [&](int32_t per, std::vector<ConeShape> *keep) {
        for (int32_t r0 = 0; r0 < rows; r0 += per) {
          shape_cone(t, lb, lt, b, r0, std::min(rows, r0 + per) - 1, W, fp, f, trial);
          if (cone_bytes(f, trial, nst) + search_q_bytes(f, trial.top_rows) > cone_budget) return false;
          if (keep) keep->push_back(trial);
        }
        return true;
      };
      int32_t lo = 0, hi = rows;
      if (fits(rows, nullptr)) {
        lo = rows;
      } else {
        while (hi - lo > 1) {
          const int32_t mid = lo + (hi - lo) / 2;
          if (fits(std::max(mid, 1), nullptr)) lo = mid; else hi = mid;
        }
      }
      if (lo < 1) {
        ok = false;
        break;
      }
      const int32_t parts = (rows + lo - 1) / lo;
      const int32_t per = (rows + parts - 1) / parts;
      ok = fits(per, &shapes);
    }
    if (!ok) return gb;  // even single rows do not fit
    // Work items: runs of consecutive cones that fit the budget together
    // (their regions stacked), so that small cones share the per-item cost;
    // at most as many per item as leaves two items per block slot.
    const int64_t ntiles = (nt + W - 1) / W;
    const int64_t cap = std::max<int64_t>(
        1, (int64_t)shapes.size() * ntiles / (int64_t)(2 * kSms * kMaxBlocksPerSm));
    std::vector<std::vector<int32_t>> bundles;
    int64_t bs = 0, ba = 0, bb = 0, bt = 0, br = 0, bp = 0;
    for (int32_t i = 0; i < (int32_t)shapes.size(); ++i) {
      const ConeShape &cs = shapes[i];
      if (!bundles.empty() && (int64_t)bundles.back().size() < cap &&
          kBarrierBytes + bs + cs.s_bytes + ba + cs.pa_bytes + bb + cs.pb_bytes + bt + cs.pt_bytes +
                  search_q_bytes(f, br + cs.top_rows) + prog_area(prog_slot_bytes(f, nst, bp + cs.prog_bytes)) + kOverRead <=
              cone_budget) {
        bundles.back().push_back(i);
        bs += cs.s_bytes;
        ba += cs.pa_bytes;
        bb += cs.pb_bytes;
        bt += cs.pt_bytes;
        br += cs.top_rows;
        bp += cs.prog_bytes;
      } else {
        bundles.push_back({i});
        bs = cs.s_bytes;
        ba = cs.pa_bytes;
        bb = cs.pb_bytes;
        bt = cs.pt_bytes;
        br = cs.top_rows;
        bp = cs.prog_bytes;
      }
    }
    int64_t ms = 0, ma = 0, mb = 0, mt = 0, mr = 0, mp = 0;
    for (const std::vector<int32_t> &bu : bundles) {
      int64_t s1 = 0, a1 = 0, b1 = 0, t1 = 0, r1 = 0, p1 = 0;
      for (int32_t i : bu) {
        s1 += shapes[i].s_bytes;
        a1 += shapes[i].pa_bytes;
        b1 += shapes[i].pb_bytes;
        t1 += shapes[i].pt_bytes;
        r1 += shapes[i].top_rows;
        p1 += shapes[i].prog_bytes;
      }
      ms = std::max(ms, s1);
      ma = std::max(ma, a1);
      mb = std::max(mb, b1);
      mt = std::max(mt, t1);
      mr = std::max(mr, r1);
      mp = std::max(mp, p1);
    }
    const int64_t qb = search_q_bytes(f, mr);
    const int64_t slot = prog_slot_bytes(f, nst, mp);
    const int64_t total = kBarrierBytes + ms + ma + mb + mt + qb + prog_area(slot) + kOverRead;
    if (total > budget && total > 227 * 1024 - 1024) continue;
    if (total > budget && cone_budget > 4096) continue;
    gb = GroupBuild();
    gb.items = (int64_t)bundles.size();
    gb.budget = budget;
    gb.g.lb = lb;
    gb.g.lt = lt;
    gb.g.W = W;
    gb.g.in_size = (lb == 0) ? fp.input_size : fp.level_size[lb];
    gb.g.out_size = fp.level_size[lt];
    gb.g.box = f.box;
    gb.g.chunk = f.chunk;
    gb.g.kchunks = f.kchunks;
    gb.g.max_p = f.max_p;
    gb.g.from_input = (lb == 0);
    gb.g.search_k = f.search_k;
    gb.g.hist = f.search_k > 0 ? search_hist(f.search_k) : 0;
    gb.g.q_off = (int32_t)(kBarrierBytes + ms + ma + mb + mt);
    gb.g.q_row = (int32_t)qb;
    gb.g.ntiles = (nt + W - 1) / W;
    gb.g.smem_bytes = (int32_t)total;
    gb.g.prog_slot = (int32_t)slot;
    gb.g.prog_off = (int32_t)(total - kOverRead - prog_area(slot));
    gb.g.s_end = (int32_t)(kBarrierBytes + ms);
    gb.g.pa_end = (int32_t)(kBarrierBytes + ms + ma);
    double hbm = 0, sl = 0, nops = 0, work = 0;
    for (const std::vector<int32_t> &bu : bundles) {
      // Each cone of the item gets its own slice of S, Pa and Pb; the item's
      // stage ops are merged stage by stage, then split over the warps.
      ItemOut item;
      if (what != Build::kEmit) {
        int32_t copies = 0;
        for (int32_t i : bu) {
          if (needs) needs->insert(needs->end(), shapes[i].needs.begin(), shapes[i].needs.end());
          if (what == Build::kMeasure) continue;
          ConeOut c;
          count_cone(t, lb, lt, W, fp, f, shapes[i], c, copies);
          item.tpl.tx_bytes += c.tpl.tx_bytes;
          hbm += c.hbm;
          work += c.work;
        }
        work += item_work(nst, copies, item.tpl.tx_bytes);
        continue;
      }
      int64_t so = 0, ao = 0, bo = 0, to = 0;
      std::vector<ConeOut> cos;
      for (int32_t i : bu) {
        ConeShape &cs = shapes[i];
        if (needs) needs->insert(needs->end(), cs.needs.begin(), cs.needs.end());
        ConeOut c;
        emit_cone(t, lb, lt, W, fp, f, cs, kBarrierBytes + so, kBarrierBytes + ms + ao,
                  kBarrierBytes + ms + ma + bo, kBarrierBytes + ms + ma + mb + to, c);
        so += cs.s_bytes;
        ao += cs.pa_bytes;
        bo += cs.pb_bytes;
        to += cs.pt_bytes;
        item.loads.insert(item.loads.end(), c.loads.begin(), c.loads.end());
        item.tpl.tx_bytes += c.tpl.tx_bytes;
        item.hbm += c.hbm;
        item.slots += c.slots;
        item.nops += c.nops;
        item.work += c.work;
        cos.push_back(std::move(c));
      }
      const std::vector<int32_t> &kinds = cos.front().kinds;
      for (size_t si = 0; si < kinds.size(); ++si) {
        std::vector<double> cost;
        int32_t base;
        if ((kinds[si] & kStageKindMask) == kStageWalk) {
          base = (int32_t)item.walks.size();
          for (const ConeOut &c : cos) {
            item.walks.insert(item.walks.end(), c.walks.begin(), c.walks.end());
            cost.insert(cost.end(), c.walk_cost.begin(), c.walk_cost.end());
          }
        } else {
          base = (int32_t)item.ops.size();
          const size_t k = (lb == 0) ? si - 1 : si;
          const int32_t kind = kinds[si] & kStageKindMask;
          for (const ConeOut &c : cos)
            for (const FusedOp &op : c.stage_ops[k]) {
              item.ops.push_back(op);
              // an op loads and stores whole pieces whatever its width
              cost.push_back(kind == kStageSearch ? 1.0 : op_slots(kind, op.flags) * kLaneCols + 2.0);
            }
        }
        StageRows rows;
        const size_t rk = (lb == 0) ? si - 1 : si;
        if ((kinds[si] & kStageKindMask) == kStageSingle || (kinds[si] & kStageKindMask) == kStagePair) {
          int32_t at = base;
          for (const ConeOut &c : cos) {
            const int32_t s0 = (int32_t)rows.steps.size();
            for (NodeRows nr : c.stage_rows[rk].nodes) {
              nr.op += at;
              nr.step += s0;
              rows.nodes.push_back(nr);
            }
            rows.steps.insert(rows.steps.end(), c.stage_rows[rk].steps.begin(), c.stage_rows[rk].steps.end());
            at += (int32_t)c.stage_ops[rk].size();
          }
        }
        item.rows.push_back(std::move(rows));
        const std::vector<int32_t> b = split_warps(cost);
        bool general = false, moves = false;
        if ((kinds[si] & kStageKindMask) == kStageWalk) {
          for (size_t i = (size_t)base; i < item.walks.size(); ++i) {
            general |= (item.walks[i].flags & kWalkNoUpper) != 0;
            moves |= (item.walks[i].flags & kWalkMoves) != 0;
          }
        } else {
          for (size_t i = (size_t)base; i < item.ops.size(); ++i)
            general |= (item.ops[i].flags & (kOpLoOne | kOpHiOne | kOpNoHi)) != 0;
        }
        item.stages.push_back(kinds[si] | (general ? kStageGeneral : 0) | (moves ? kStageMoves : 0));
        for (int32_t w = 0; w <= kFusedBlockWarps; ++w) {
          item.stages.push_back(base + b[w]);
          // A warp's first op has nothing earlier to reuse.
          if ((kinds[si] & kStageKindMask) != kStageWalk && w < kFusedBlockWarps && b[w] < b[w + 1])
            item.ops[base + b[w]].flags &= ~(kOpLoSame | kOpHiShift);
        }
      }
      item.tpl.n_stages = (int32_t)kinds.size();
      item.tpl.smem_bytes = (int32_t)total;
      hbm += item.hbm;
      sl += item.slots;
      nops += item.nops;
      work += item.work + item_work(nst, (int32_t)item.loads.size(), item.tpl.tx_bytes);
      gb.cones.push_back(std::move(item));
    }
    gb.g.hbm_bytes = hbm * (double)gb.g.ntiles;
    gb.g.smem_traffic = sl * 128.0 * (double)gb.g.ntiles;
    const double tiles = (double)gb.g.ntiles;
    const double items = (double)gb.items * tiles;
    const double slots =
        kSms * std::min(kMaxBlocksPerSm, std::max(1.0, std::floor((228.0 * 1024) / (total + 1024.0))));
    const double waves = items / slots;
    const double on_chip = work / (double)gb.items * (items <= kSms ? kAloneShare : 1.0) *
                           std::max(waves, std::min(std::ceil(waves), waves + kWaveTail));
    // DRAM sees each base row and each output row once (neighbouring cones'
    // halos and overlaps are L2 hits); the staged bytes go through L2.
    const double unique = (double)nt * ((lb == 0 ? (double)t.nf * fp.input_size
                                                  : (double)t.level_rows[lb] * fp.level_size[lb]) +
                                        (double)t.level_rows[lt] * fp.level_size[lt]);
    const double mem = std::max(unique / kHbmRate, gb.g.hbm_bytes / kL2Rate);
    gb.seconds = kLaunchSeconds + std::pow(std::pow(on_chip, kNorm) + std::pow(mem, kNorm), 1.0 / kNorm);
    gb.g.ops = nops * tiles;
    gb.g.block_slots = slots;
    gb.g.seconds = gb.seconds;
    gb.ok = true;
    return gb;
  }
  return gb;
}

// Group (lb, lt] for tile W.  The staging format follows the windows of
// the group's own cones: a first build with provisional boxes measures
// them, the second uses the chosen box or block width.
GroupBuild build_group_mode(const Tables &t, int64_t nt, int32_t lb, int32_t lt, int32_t W,
                       const FusedPlan &fp, int32_t budget, const FusedParams &prm, int32_t search_k, bool emit,
                            bool compact, int32_t staging) {
  const int32_t es = (lb == 0) ? fp.input_size : fp.level_size[lb];
  const int64_t rows = (lb == 0) ? t.nf : t.level_rows[lb];
  // Row blocks: chunks of 128 bytes (64 for 1-byte samples, so that a tile
  // start, a multiple of 64 samples, is a chunk boundary).
  const int32_t chunk = std::min(128 / es, 64);
  // (mapped channels start at their own columns: row boxes)
  const bool mapped = lb == 0 && prm.in_shift != nullptr;
  const bool blocks = staging != 1 && (lb == 0 ? nt : fp.state_nt) % chunk == 0 && !mapped;
  if (staging == 2 && nt % chunk != 0) return GroupBuild();
  StageFmt boxes;
  boxes.search_k = search_k;
  boxes.compact = compact;
  if (mapped) {
    boxes.in_shift = prm.in_shift;
    boxes.descending = prm.descending;
  }
  StageFmt f = boxes;
  if (blocks) {
    f.chunk = chunk;
    f.max_p = 0;
    while (f.max_p < 5 && (int64_t(2) << f.max_p) <= rows) ++f.max_p;
  } else {
    f.box = 128 / es;
  }
  std::vector<std::pair<int32_t, int32_t>> needs;
  GroupBuild gb = build_group_fmt(t, nt, lb, lt, W, fp, budget, f, &needs, Build::kMeasure);
  if (!gb.ok) return gb;
  int32_t widest = 0;
  for (const auto &nr : needs) widest = std::max(widest, nr.first);
  if (blocks) {
    // Every staged row of the launch gets the widest window; a copy's row
    // pitch stays a multiple of 128 bytes.  The cones of the rebuilt group
    // can differ (other row splits, other window alignments), so the width
    // is checked again and widened until it covers all of them.
    for (int iter = 0; iter < 4; ++iter) {
      int32_t k = (widest + chunk - 1) / chunk;
      while ((k * chunk * es) % 128 != 0) ++k;
      if (k > 256 || (int64_t)k * chunk > nt) break;
      f.kchunks = std::max(f.kchunks, k);
      std::vector<std::pair<int32_t, int32_t>> got;
      GroupBuild g2 = build_group_fmt(t, nt, lb, lt, W, fp, budget, f, &got, Build::kCount);
      if (!g2.ok) break;
      widest = 0;
      for (const auto &nr : got) widest = std::max(widest, nr.first);
      if (widest <= f.kchunks * chunk)
        return emit ? build_group_fmt(t, nt, lb, lt, W, fp, budget, f, nullptr, Build::kEmit) : g2;
    }
    if (staging == 2) return GroupBuild();
    f = boxes;  // fall back to row boxes
    f.box = 128 / es;
    needs.clear();
    gb = build_group_fmt(t, nt, lb, lt, W, fp, budget, f, &needs, Build::kMeasure);
    if (!gb.ok) return gb;
  }
  f.box = choose_box(needs, es);
  return build_group_fmt(t, nt, lb, lt, W, fp, budget, f, nullptr, emit ? Build::kEmit : Build::kCount);
}

// The same in a layout: roomy; compact, where a budget fits no roomy one; and
// compact with row boxes (whose windows are not rounded to chunks), where it
// fits neither.
enum : int32_t { kRoomy = 0, kCompact = 1, kCompactBoxes = 2 };
GroupBuild build_group(const Tables &t, int64_t nt, int32_t lb, int32_t lt, int32_t W, const FusedPlan &fp,
                       int32_t budget, const FusedParams &prm, int32_t search_k, bool emit, int32_t layout) {
  if (layout == kCompactBoxes && prm.staging != 0) return GroupBuild();
  return build_group_mode(t, nt, lb, lt, W, fp, budget, prm, search_k, emit, layout != kRoomy,
                          layout == kCompactBoxes ? 1 : prm.staging);
}

// Shared-memory pipe slots per 32 columns of the first row of a run (all its
// sources, the store) and of a later row (one half's sources, on average 1.5
// of a pair's two, the store).
double run_first_cost(bool pair) { return pair ? 5.5 : 3.5; }
double run_step_cost(bool pair) { return pair ? 2.75 : 2.25; }

// Lowers a stage's rows to runs split over the warps at about equal cost.
// A node's rows are first cut into chunks whose delay growth is at most
// kRunGrow and still fits the columns left free in the node's last strip (a
// strip moves a column with every step of the lower row, so more growth
// would take one more strip); the strips of all chunks, in order, are then dealt to the warps, each warp
// taking rows up to the smallest cost at which the block's warps suffice.
// dst_moves: the rows go to plain rows of shared memory (dst at column col).
void lower_stage(const StageRows &sr, const std::vector<FusedOp> &ops, bool pair, bool dst_moves,
                 std::vector<FusedRun> &runs, int32_t begin[kFusedBlockWarps + 1]) {
  struct Strip {
    int32_t node, first, n, col;  // rows first .. first + n - 1 of the node; column of the first row
  };
  std::vector<Strip> strips;
  for (size_t i = 0; i < sr.nodes.size(); ++i) {
    const NodeRows &nr = sr.nodes[i];
    const int32_t free_cols = (nr.width + kPieceCols - 1) / kPieceCols * kPieceCols - nr.width;
    const bool moves = !(nr.flags & kOpNoHi);  // rows without an upper half keep their columns
    for (int32_t r = 0; r < nr.n;) {
      int32_t grow = 0, k = 1;
      while (r + k < nr.n && k < kRunRows) {
        const int32_t inc = moves ? sr.steps[nr.step + r + k - 1] & 1 : 0;
        if (grow + inc > kRunGrow || (grow + inc > free_cols && free_cols >= 8)) break;
        grow += inc;
        ++k;
      }
      for (int32_t c = -grow; c < nr.width; c += kPieceCols) strips.push_back(Strip{(int32_t)i, r, k, c});
      r += k;
    }
  }
  auto deal = [&](double cap, std::vector<FusedRun> *out) {
    int32_t w = 0;
    double load = 0;
    if (out) begin[0] = (int32_t)out->size();
    for (const Strip &s : strips) {
      const NodeRows &nr = sr.nodes[s.node];
      int32_t col = s.col;
      for (int32_t r = 0; r < s.n;) {
        // rows this warp still takes (at least one if it has none)
        const double room = cap - load - run_first_cost(pair);
        int32_t k = room < 0 ? 0 : std::min<int32_t>(s.n - r, 1 + (int32_t)(room / run_step_cost(pair)));
        if (k < 1) {
          if (load > 0) {
            if (++w >= kFusedBlockWarps) return false;
            if (out) begin[w] = (int32_t)out->size();
            load = 0;
            continue;
          }
          k = 1;
        }
        FusedRun run{};
        int32_t moved = 0;
        const uint8_t *st = sr.steps.data() + nr.step + s.first + r;
        for (int32_t i = 0; i < k; ++i) {
          if (s.first + r + i + 1 >= nr.n) break;
          const int32_t inc = st[i] & 1;
          if (i + 1 < k) {
            run.inc |= (uint32_t)inc << i;
            run.sub |= (uint32_t)(st[i] >> 1) << i;
          }
          moved += nr.flags & kOpNoHi ? 0 : inc;  // columns moved by the row after this part
        }
        if (out) {
          const FusedOp &op = ops[nr.op + s.first + r];
          run.dst = dst_moves ? op.dst + col * 4 : op.dst;
          run.dst_row = nr.pitch * 4;
          run.col = col;
          run.width = nr.width;
          run.p0 = op.p0 + col * nr.es;
          run.p1 = op.p1 + col * nr.es;
          run.p2 = (pair ? op.p2 : op.p1) + col * nr.es;
          run.p3 = op.p3 + col * nr.es;
          if (!pair) run.p1 = run.p3 = 0;
          if (nr.flags & kOpLoOne) run.p1 = 0;
          if (nr.flags & kOpHiOne) run.p3 = 0;
          if (nr.flags & kOpNoHi) run.p2 = run.p3 = 0;
          run.g0 = nr.g[0];
          run.g1 = nr.g[1];
          run.g2 = nr.g[2];
          run.g3 = nr.g[3];
          run.n = k;
          run.flags = nr.flags;
          if (dst_moves && nr.pitch % kPieceCols == 0 && nr.pitch - nr.width >= kRunGrow) run.flags |= kRunWhole;
          out->push_back(run);
        }
        load += run_first_cost(pair) + (k - 1) * run_step_cost(pair);
        col += moved;
        r += k;
      }
    }
    if (out)
      while (w < kFusedBlockWarps) begin[++w] = (int32_t)out->size();
    return true;
  };
  double total = 0;
  for (const Strip &s : strips) total += run_first_cost(pair) + (s.n - 1) * run_step_cost(pair);
  double lo = total / kFusedBlockWarps, hi = std::max(lo, run_first_cost(pair));
  while (!deal(hi, nullptr)) hi *= 1.25;
  while (hi - lo > 0.5) {
    const double mid = 0.5 * (lo + hi);
    if (deal(mid, nullptr)) hi = mid; else lo = mid;
  }
  deal(hi, &runs);
}

// False if a programme outgrows the room its group has for it.
bool append_group(FusedPlan &fp, GroupBuild &gb) {
  FusedGroup g = gb.g;
  g.tpl_begin = (int32_t)fp.tpls.size();
  g.tpl_count = (int32_t)gb.cones.size();
  for (ItemOut &c : gb.cones) {
    FusedTemplate tp = c.tpl;
    tp.load_begin = (int32_t)fp.loads.size();
    tp.load_count = (int32_t)c.loads.size();
    tp.walk_begin = (int32_t)fp.walks.size();
    tp.walk_count = (int32_t)c.walks.size();
    tp.stage_begin = (int32_t)fp.stages.size();
    const int32_t w0 = (int32_t)fp.walks.size(), o0 = (int32_t)fp.ops.size();
    for (size_t i = 0; i < c.stages.size(); i += kStageWords) {
      const int32_t off = (c.stages[i] & kStageKindMask) == kStageWalk ? w0 : o0;
      fp.general |= (c.stages[i] & kStageGeneral) != 0;
      g.moves |= (c.stages[i] & kStageMoves) != 0;
      fp.stages.push_back(c.stages[i]);
      for (int32_t w = 1; w < kStageWords; ++w) fp.stages.push_back(c.stages[i + w] + off);
      const int32_t kind = c.stages[i] & kStageKindMask;
      if (kind == kStageSingle || kind == kStagePair) {
        const bool dst_moves = i + kStageWords < c.stages.size() && !(c.stages[i] & kStagePadded);
        int32_t begin[kFusedBlockWarps + 1];
        lower_stage(c.rows[i / kStageWords], c.ops, kind == kStagePair, dst_moves, fp.runs, begin);
        fp.run_stages.push_back(c.stages[i] | kStageRuns);
        fp.run_stages.insert(fp.run_stages.end(), begin, begin + kFusedBlockWarps + 1);
      } else {
        fp.run_stages.insert(fp.run_stages.end(), fp.stages.end() - kStageWords, fp.stages.end());
      }
    }
    for (const FusedLoad &ld : c.loads) g.min_x = std::min(g.min_x, ld.xoff);
    FusedProg pr{};
    pr.load_begin = tp.load_begin;
    pr.load_count = tp.load_count;
    pr.n_stages = tp.n_stages;
    pr.prog = (int32_t)(fp.prog.size() / 4);
    std::vector<int32_t> words((size_t)tp.n_stages * (kProgStageBytes / 4), 0);
    for (int32_t st = 0; st < tp.n_stages; ++st) {
      const int32_t *src = fp.run_stages.data() + tp.stage_begin + st * kStageWords;
      const size_t at = (size_t)st * (kProgStageBytes / 4);
      const int32_t kind = src[0] & kStageKindMask;
      words[at] = src[0];
      if (kind == kStageSearch) {
        for (int32_t w = 1; w < kStageWords; ++w) words[at + w] = src[w];
        continue;
      }
      const int32_t size = kind == kStageWalk ? (int32_t)sizeof(FusedWalk) : (int32_t)sizeof(FusedRun);
      for (int32_t w = 1; w < kStageWords; ++w) words[at + w] = (int32_t)words.size() * 4 + (src[w] - src[1]) * size;
      const int32_t *d = kind == kStageWalk ? reinterpret_cast<const int32_t *>(c.walks.data() + (src[1] - w0))
                                            : reinterpret_cast<const int32_t *>(fp.runs.data() + src[1]);
      words.insert(words.end(), d, d + (size_t)(src[kStageWords - 1] - src[1]) * size / 4);
    }
    pr.prog_bytes = (int32_t)words.size() * 4;
    pr.far = g.prog_slot == 0 ? 1 : 0;
    pr.tx_bytes = tp.tx_bytes + (pr.far ? 0 : pr.prog_bytes);
    if (!pr.far && pr.prog_bytes > g.prog_slot) return false;
    fp.prog.insert(fp.prog.end(), words.begin(), words.end());
    fp.progs.push_back(pr);
    fp.loads.insert(fp.loads.end(), c.loads.begin(), c.loads.end());
    fp.walks.insert(fp.walks.end(), c.walks.begin(), c.walks.end());
    fp.ops.insert(fp.ops.end(), c.ops.begin(), c.ops.end());
    fp.tpls.push_back(tp);
  }
  fp.groups.push_back(g);
  return true;
}

}  // namespace

void first_tiles(const FusedPlan &fp, int64_t first, FirstTiles &out) {
  for (size_t g = fp.groups.size(); g-- > 0;) {
    out.tile[g] = first / fp.groups[g].W;
    first = std::max<int64_t>(0, out.tile[g] * fp.groups[g].W + fp.groups[g].min_x);
  }
}

std::string plan_fused(const Tables &t, int64_t nt, int32_t state_size, int32_t input_size,
                       const FusedParams &p, FusedPlan &out) {
  const int32_t L = t.levels;
  std::vector<int32_t> widths;
  if (p.W > 0) {
    if (p.W % 64 != 0) return "tile width must be a multiple of 64";
    widths.push_back(p.W);
  } else {
    // (whole strips of 256 columns less the windows' growth, and small ones)
    widths = {64, 128, 192, 256, 384, 448, 704, 960};
  }
  if (p.search_k < 0 || p.search_k > kSearchMaxWidths || (p.search_k > 0 && L < 2))
    return "the search in the last launch takes 1 .. 9 widths and at least two merge levels";
  if (p.search_k > 0 && p.W > 0 && p.W + search_hist(p.search_k) > 16 * kFusedBlockWarps * 32)
    return "the searched window must fit one wave of the block";
  FusedPlan fp;
  fp.state_size = state_size;
  fp.input_size = input_size;
  // Rows between launches are padded to whole chunks so that they can be
  // staged as row blocks whatever nt (a row box takes two to four copies per
  // row: 1000 x 50004 x 777 float32, launches [3,6] [6,10]: 87 and 88 us with
  // boxes, 64 and 65 us with padded rows).  Columns past nt are never needed.
  // Short rows keep their length: their launches are not bound by copies.
  fp.state_nt = p.staging == 0 && nt >= kPadRows ? round_up(nt, 64) : nt;
  fp.acc_size = 4;
  fp.moves = moves_pay(t);
  // Stored element size of each level at a launch boundary; the output
  // (level L) is 4 bytes.  With p.narrow (integer sums of uint8 samples), a
  // level whose sums stay below 2^16 is stored as uint16: row Dt of a band
  // of 2^l channels sums 2^l + Dt samples (the path's sample counts
  // telescope, section 4), each at most 255.
  fp.level_size.assign(L + 1, state_size);
  fp.level_size[L] = 4;
  if (p.narrow) {
    for (int32_t l = 1; l < L; ++l) {
      int32_t rmax = 0;
      for (int32_t r : t.band_rows[l]) rmax = std::max(rmax, r);
      if (255LL * ((1LL << l) + rmax - 1) <= 65535 && (nt * 2) % 16 == 0) fp.level_size[l] = 2;
    }
  }
  // Best tile for one group (lb, lt] (optionally a given tile and budget),
  // counted only.  `known`: the tile that was best before.
  struct Segment {
    GroupBuild gb;
    int32_t layout = kRoomy;
  };
  auto best_segment = [&](int32_t lb, int32_t lt, int32_t forced_W = 0, int32_t budget = 0, bool refine = false,
                          int32_t known = 0) {
    Segment best;
    const std::vector<int32_t> ws = forced_W > 0 ? std::vector<int32_t>{forced_W} : widths;
    auto tries = [&](int32_t W, int32_t layout, int32_t bytes) {
      GroupBuild gb = build_group(t, nt, lb, lt, W, fp, bytes, p, lt == L ? p.search_k : 0, false, layout);
      const bool ok = gb.ok;
      if (ok && (!best.gb.ok || gb.seconds < best.gb.seconds)) best = Segment{std::move(gb), layout};
      return ok;
    };
    // Long rows take the other layouts only where no tile fits the roomy one
    // (planning 1000 x 50004 x 777: 218 ms, 364 ms with all of them tried
    // tile by tile); short calls are bound by launches and latency, where a
    // lesser layout that saves a launch can win.
    const bool all = nt < kPadRows;
    for (int32_t layout = kRoomy; layout <= kCompactBoxes && !best.gb.ok; ++layout)
      for (int32_t W : ws) {
        if (known > 0 && W != known) continue;
        if (best.gb.ok && W / 2 >= nt) break;  // (no wider than one tile needs)
        for (int32_t l = layout; !tries(W, l, budget > 0 ? budget : p.smem_budget) && all && l < kCompactBoxes;) ++l;
      }
    // Few items leave SMs idle: smaller ones (more row ranges) may be faster
    // (tried once the boundaries stand).
    for (int32_t kib = 56; refine && budget == 0 && p.smem_budget == FusedParams().smem_budget && kib >= 14; kib /= 2) {
      if (!best.gb.ok || best.gb.items * best.gb.g.ntiles >= best.gb.g.block_slots) break;
      for (int32_t W : ws)
        for (int32_t l = kRoomy; !tries(W, l, kib * 1024) && all && l < kCompactBoxes;) ++l;
    }
    return best;
  };
  std::vector<int32_t> bounds = p.bounds, tile(L + 1, 0);  // tile[j]: of the group that ends at level j, if searched
  if (bounds.empty()) {
    // Dynamic programming over boundaries: cost[j] = best time to reach level j.
    std::vector<double> cost(L + 1, std::numeric_limits<double>::infinity());
    std::vector<int32_t> from(L + 1, -1);
    cost[0] = 0;
    for (int32_t j = 1; j <= L; ++j)
      for (int32_t i = std::max(0, j - 6); i < j; ++i) {
        if (!std::isfinite(cost[i])) continue;
        const GroupBuild gb = best_segment(i, j).gb;
        if (!gb.ok) continue;
        if (cost[i] + gb.seconds < cost[j]) {
          cost[j] = cost[i] + gb.seconds;
          from[j] = i;
          tile[j] = gb.g.W;
        }
      }
    if (!std::isfinite(cost[L])) return "no fused schedule fits the shared-memory budget";
    std::vector<int32_t> rev;
    for (int32_t j = L; j > 0; j = from[j]) rev.push_back(j);
    bounds = {0};
    for (auto it = rev.rbegin(); it != rev.rend(); ++it) bounds.push_back(*it);
  }
  if (bounds.size() < 2 || bounds.front() != 0 || bounds.back() != L)
    return "level boundaries must run from 0 to L";
  double secs = 0;
  for (size_t i = 0; i + 1 < bounds.size(); ++i) {
    if (bounds[i + 1] <= bounds[i]) return "level boundaries must increase";
    const int32_t gw = i < p.group_W.size() ? p.group_W[i] : 0;
    const int32_t gbud = i < p.group_budget.size() ? p.group_budget[i] : 0;
    if (gw < 0 || gw % 64 != 0 || gbud < 0 || gbud > 227 * 1024) return "bad per-group parameters";
    const Segment seg = best_segment(bounds[i], bounds[i + 1], gw, gbud, true,
                                     gw == 0 && gbud == 0 ? tile[bounds[i + 1]] : 0);
    GroupBuild gb;
    if (seg.gb.ok)
      gb = build_group(t, nt, bounds[i], bounds[i + 1], seg.gb.g.W, fp, seg.gb.budget, p,
                       bounds[i + 1] == L ? p.search_k : 0, true, seg.layout);
    if (!gb.ok) return "a level group does not fit the shared-memory budget";
    secs += gb.seconds;
    if (!append_group(fp, gb)) return "a programme outgrew its slot";
  }
  fp.W = fp.groups.front().W;
  fp.model_seconds = secs;
  // Intermediate states between groups: group g writes buffer g % 2.
  size_t even = 0, odd = 0;
  for (size_t g = 0; g + 1 < fp.groups.size(); ++g) {
    const size_t bytes = (size_t)t.level_rows[fp.groups[g].lt] * (size_t)fp.state_nt * (size_t)fp.level_size[fp.groups[g].lt];
    if (g & 1) odd = std::max(odd, bytes); else even = std::max(even, bytes);
  }
  fp.ws_split = (size_t)round_up((int64_t)even, 256);
  fp.ws_bytes = fp.ws_split + (size_t)round_up((int64_t)odd, 256);
  out = std::move(fp);
  return "";
}

}  // namespace fdmt
