// Device-side building blocks of the fused-schedule kernels (single beam
// in fdmt_fused.cu, batches in fdmt_batch_fused.cu): mbarrier and TMA
// wrappers, the staging of one work item, and its compute stages (level 1
// walked from the staged input, single levels and pairs of levels).
#pragma once

#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <climits>
#include <cstdint>
#include <type_traits>

#include "fdmt_common.cuh"
#include "fdmt_fused.h"

namespace fdmt {

constexpr int kFusedWarps = kFusedBlockWarps;
constexpr int kFusedThreads = 32 * kFusedWarps;
constexpr int kFusedMinBlocks = 2;  // resident blocks per SM the register budget allows
constexpr int kWaitTries = 4000;            // x the suspend hint below: a ~2 s bound
constexpr uint32_t kSuspendHintNs = 500000;

// ---------------------------------------------------------------------------
// PTX helpers (mbarrier + TMA)

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// try_wait with a suspend-time hint: a waiting thread sleeps in hardware
// until the phase completes or the hint elapses, instead of spinning.
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(kSuspendHintNs)
      : "memory");
  return ok != 0;
}

// Bounded wait for phase `parity`; false if it did not complete in time.
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t parity) {
  for (int i = 0; i < kWaitTries; ++i)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}

__device__ __forceinline__ void tma_load_row(uint32_t dst, const CUtensorMap *map, int32_t x,
                                             int32_t y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}

// Row block: chunks [x, x + kchunks) of rows [y, y + 2^p) through a map of
// the [rows][nt / chunk][chunk] view whose box is (chunk, kchunks, 2^p).
__device__ __forceinline__ void tma_load_block(uint32_t dst, const CUtensorMap *map, int32_t x, int32_t y,
                                               uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(x), "r"(y), "r"(bar)
      : "memory");
}

// The tensor maps of a launch: row boxes use m[0]; row blocks use m[p] for
// copies of 2^p rows.
struct TmaMaps {
  CUtensorMap m[kMaxBlockP + 1];
};

template <bool R16>
__device__ __forceinline__ float round_state(float v) {
  if constexpr (R16) return __half2float(__float2half_rn(v));
  return v;
}
template <bool R16>
__device__ __forceinline__ int32_t round_state(int32_t v) { return v; }

template <class T> __device__ __forceinline__ T to_store(float v);
template <> __device__ __forceinline__ float to_store<float>(float v) { return v; }
template <> __device__ __forceinline__ __half to_store<__half>(float v) { return __float2half_rn(v); }
template <class T> __device__ __forceinline__ T to_store(int32_t v) { return v; }

__device__ __forceinline__ float lds_f32(uint32_t a) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ int32_t lds_s32(uint32_t a) {
  int32_t v;
  asm volatile("ld.shared.s32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ float lds_h2f(uint32_t a) {
  unsigned short v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a) : "memory");
  return __half2float(__ushort_as_half(v));
}
__device__ __forceinline__ void sts_f32(uint32_t a, float v) {
  asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void sts_s32(uint32_t a, int32_t v) {
  asm volatile("st.shared.s32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

template <class TI, class A> __device__ __forceinline__ A load_input(uint32_t a);
template <> __device__ __forceinline__ float load_input<float, float>(uint32_t a) { return lds_f32(a); }
template <> __device__ __forceinline__ int32_t load_input<uint8_t, int32_t>(uint32_t a) {
  unsigned short v;
  asm volatile("ld.shared.u8 %0, [%1];" : "=h"(v) : "r"(a) : "memory");
  return (int32_t)v;
}

template <class T> struct Lds;
template <> struct Lds<float> {
  static __device__ __forceinline__ float get(uint32_t a) { return lds_f32(a); }
};
template <> struct Lds<int32_t> {
  static __device__ __forceinline__ int32_t get(uint32_t a) { return lds_s32(a); }
};
template <> struct Lds<__half> {
  static __device__ __forceinline__ float get(uint32_t a) { return lds_h2f(a); }
};
template <> struct Lds<uint16_t> {  // uint16-stored integer state
  static __device__ __forceinline__ int32_t get(uint32_t a) {
    unsigned short v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a) : "memory");
    return (int32_t)v;
  }
};
__device__ __forceinline__ void sts(uint32_t a, float v) { sts_f32(a, v); }
__device__ __forceinline__ void sts(uint32_t a, int32_t v) { sts_s32(a, v); }

// ---------------------------------------------------------------------------
// Stages of a work item.  Each warp runs its own list of ops (the planner
// splits every stage into kFusedBlockWarps contiguous lists); lane l handles
// columns l, l + 32, ..., l + 32 (kLaneCols - 1) of an op's piece, so every
// shared-memory access of a warp touches 32 consecutive words (no bank
// conflicts).  Values that an op's reuse flags carry over stay in registers.

// Descriptors: every lane reads the same address (one broadcast request).
__device__ __forceinline__ FusedOp ld_op(const FusedOp *__restrict__ p) {
  const int4 a = __ldg(reinterpret_cast<const int4 *>(p));
  const int4 b = __ldg(reinterpret_cast<const int4 *>(p) + 1);
  return FusedOp{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
}
__device__ __forceinline__ void sts_v4(uint32_t a, int4 v) {
  asm volatile("st.shared.v4.s32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
               : "memory");
}
__device__ __forceinline__ int4 lds_v4(uint32_t a) {
  int4 v;
  asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a)
               : "memory");
  return v;
}

// A descriptor read from shared memory as broadcasts.
template <class D> __device__ __forceinline__ D lds_desc(uint32_t a);
template <> __device__ __forceinline__ FusedOp lds_desc<FusedOp>(uint32_t at) {
  const int4 a = lds_v4(at), b = lds_v4(at + 16u);
  return FusedOp{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
}
template <> __device__ __forceinline__ FusedRun lds_desc<FusedRun>(uint32_t at) {
  const int4 a = lds_v4(at), b = lds_v4(at + 16u), c = lds_v4(at + 32u), d = lds_v4(at + 48u);
  return FusedRun{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y, c.z, c.w, d.x, (uint32_t)d.y, (uint32_t)d.z, d.w};
}
template <> __device__ __forceinline__ FusedWalk lds_desc<FusedWalk>(uint32_t at) {
  const int4 x = lds_v4(at), y = lds_v4(at + 16u), z = lds_v4(at + 32u);
  return FusedWalk{x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w, z.x, z.y, z.z, z.w};
}

// A value every lane of the warp holds, as one the compiler knows to be
// uniform (branches on it then need no reconvergence).
__device__ __forceinline__ int32_t warp_all(int32_t v) { return __shfl_sync(0xffffffffu, v, 0); }
__device__ __forceinline__ uint32_t warp_all(uint32_t v) { return __shfl_sync(0xffffffffu, v, 0); }

// An item's programme: a slot of shared memory, or (far) global memory.
struct Prog {
  uint32_t near;
  const int4 *far;  // null: near
};
__device__ __forceinline__ int32_t prog_word(const Prog &p, uint32_t off) {
  return p.far != nullptr ? __ldg(reinterpret_cast<const int32_t *>(p.far) + (off >> 2)) : lds_s32(p.near + off);
}
template <class D>
__device__ __forceinline__ D prog_desc(const Prog &p, uint32_t off) {
  if (p.far == nullptr) return lds_desc<D>(p.near + off);
  alignas(16) D d;
  int4 *o = reinterpret_cast<int4 *>(&d);
#pragma unroll
  for (int i = 0; i < (int)(sizeof(D) / 16); ++i) o[i] = __ldg(p.far + (off >> 4) + i);
  return d;
}

// Stage s of a programme for one warp: its kind and the offsets of the
// warp's first descriptor and of their end.
struct StageRange {
  int kind;
  uint32_t first, end;
  Prog prog;
};
__device__ __forceinline__ StageRange prog_stage(const Prog &p, int s, int warp) {
  const uint32_t at = (uint32_t)(s * kProgStageBytes);
  return StageRange{warp_all(prog_word(p, at)), (uint32_t)warp_all(prog_word(p, at + 4u + 4u * (uint32_t)warp)),
                    (uint32_t)warp_all(prog_word(p, at + 8u + 4u * (uint32_t)warp)), p};
}

// The warps that compute (kFusedThreads threads) wait for each other.  The
// copying warp of the single-beam kernel takes no part.
__device__ __forceinline__ void compute_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kFusedThreads) : "memory"); }
// The same, and whether `ok` held in every thread.
__device__ __forceinline__ bool compute_sync_and(bool ok) {
  uint32_t r;
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\t"
               "barrier.cta.red.and.pred q, 1, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
               : "=r"(r) : "r"((uint32_t)ok), "n"(kFusedThreads) : "memory");
  return r != 0;
}

// kLaneCols columns of a row piece from shared memory.  The loads are
// unconditional (no branch or predicate between them): columns at or beyond
// the op's width read whatever lies there, which the planner keeps inside
// the block's shared memory (kOverRead bytes of slack after the last
// region), and those values never reach a stored column.
template <class TSrc, class A>
__device__ __forceinline__ void ld_piece(A (&v)[kLaneCols], uint32_t addr, int lane) {
  constexpr uint32_t es = sizeof(TSrc);
  addr += (uint32_t)lane * es;
#pragma unroll
  for (int k = 0; k < kLaneCols; ++k) v[k] = (A)Lds<TSrc>::get(addr + (uint32_t)(32 * k) * es);
}

// The same of staged input samples.
template <class TI, class A>
__device__ __forceinline__ void ld_samples(A (&v)[kLaneCols], uint32_t addr, int lane) {
  addr += (uint32_t)lane * (uint32_t)sizeof(TI);
#pragma unroll
  for (int k = 0; k < kLaneCols; ++k) v[k] = load_input<TI, A>(addr + (uint32_t)(32 * k) * (uint32_t)sizeof(TI));
}

// Where a merge stage writes: shared memory (a stored level), global memory
// (the group's top level), or shared memory in the search layout (the top
// level of a launch that ends with the boxcar search).
enum : int { kOutSmem = 0, kOutGlobal = 1, kOutPadded = 2 };

// Stores that write only where column c (as unsigned, so that a negative one
// never qualifies) lies below n.
__device__ __forceinline__ void sts_below(uint32_t a, float v, int c, int n) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.lt.u32 q, %2, %3;\n\t@q st.shared.f32 [%0], %1;\n\t}"
               ::"r"(a), "f"(v), "r"((uint32_t)c), "r"((uint32_t)n) : "memory");
}
__device__ __forceinline__ void sts_below(uint32_t a, int32_t v, int c, int n) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.lt.u32 q, %2, %3;\n\t@q st.shared.s32 [%0], %1;\n\t}"
               ::"r"(a), "r"(v), "r"((uint32_t)c), "r"((uint32_t)n) : "memory");
}
__device__ __forceinline__ void stg_below(float *g, float v, int c, int n) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.lt.u32 q, %2, %3;\n\t@q st.global.f32 [%0], %1;\n\t}"
               ::"l"(g), "f"(v), "r"((uint32_t)c), "r"((uint32_t)n) : "memory");
}
__device__ __forceinline__ void stg_below(int32_t *g, int32_t v, int c, int n) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.lt.u32 q, %2, %3;\n\t@q st.global.s32 [%0], %1;\n\t}"
               ::"l"(g), "r"(v), "r"((uint32_t)c), "r"((uint32_t)n) : "memory");
}
__device__ __forceinline__ void stg_below(__half *g, float v, int c, int n) {
  const unsigned short h = __half_as_ushort(__float2half_rn(v));
  asm volatile("{\n\t.reg .pred q;\n\tsetp.lt.u32 q, %2, %3;\n\t@q st.global.u16 [%0], %1;\n\t}"
               ::"l"(g), "h"(h), "r"((uint32_t)c), "r"((uint32_t)n) : "memory");
}
__device__ __forceinline__ void stg_below(uint16_t *g, int32_t v, int c, int n) {
  const unsigned short h = (unsigned short)v;
  asm volatile("{\n\t.reg .pred q;\n\tsetp.lt.u32 q, %2, %3;\n\t@q st.global.u16 [%0], %1;\n\t}"
               ::"l"(g), "h"(h), "r"((uint32_t)c), "r"((uint32_t)n) : "memory");
}

// o = a + b over a lane's columns, each sum rounded by itself; float sums
// two at a time (add.rn.f32x2: one issue slot for two columns).
__device__ __forceinline__ void add_piece(float (&o)[kLaneCols], const float (&a)[kLaneCols],
                                          const float (&b)[kLaneCols]) {
  static_assert(kLaneCols % 2 == 0, "columns are added in pairs");
#pragma unroll
  for (int k = 0; k < kLaneCols; k += 2)
    asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\t"
        "add.rn.f32x2 x, x, y;\n\tmov.b64 {%0, %1}, x;\n\t}"
        : "=f"(o[k]), "=f"(o[k + 1])
        : "f"(a[k]), "f"(a[k + 1]), "f"(b[k]), "f"(b[k + 1]));
}
__device__ __forceinline__ void add_piece(int32_t (&o)[kLaneCols], const int32_t (&a)[kLaneCols],
                                          const int32_t (&b)[kLaneCols]) {
#pragma unroll
  for (int k = 0; k < kLaneCols; ++k) o[k] = a[k] + b[k];
}
__device__ __forceinline__ float no_term(float) { return -0.0f; }
__device__ __forceinline__ int32_t no_term(int32_t) { return 0; }
template <bool R16, class A>
__device__ __forceinline__ void round_piece(A (&v)[kLaneCols]) {
#pragma unroll
  for (int k = 0; k < kLaneCols; ++k) v[k] = round_state<R16>(v[k]);
}

// The runs of a single (PAIR false) or pair stage.  A row's four (two)
// sources and half sums stay in registers: from one row to the next the
// strip moves with the delay (FusedRun), so one half is unchanged and of the
// other half's two sources one (sub = 1 below, sub = 0 above) or both are
// read again -- on average 1.5 reads and one write per output of a pair,
// against the four reads its sum has.  The next row's reads are issued
// before the row is stored, so their latency overlaps the stores.  The half
// sums belong to a level below the top: fp16-state mode rounds them.  The
// words that steer the rows are broadcast by a shuffle, which makes the
// branches on them uniform.
// Bound: instruction issue, then the shared-memory pipe (one 128-byte access
// per clock and SM).
template <class TSrc, class A, class TO, bool R16, int OUT, bool PAIR, bool GEN>
__device__ __forceinline__ void stage_runs(uint32_t sbase, const StageRange &range, int lane, TO *__restrict__ out,
                                           int64_t nt, int64_t T0, int lo, int lim) {
  constexpr uint32_t es = sizeof(TSrc);
  for (uint32_t at = range.first; at != range.end; at += (uint32_t)sizeof(FusedRun)) {
    const FusedRun run = prog_desc<FusedRun>(range.prog, at);
    const uint32_t flags = warp_all((uint32_t)run.flags);
    const bool lo_one = GEN && (flags & kOpLoOne) != 0, hi_one = GEN && (flags & kOpHiOne) != 0;
    const bool no_hi = GEN && (flags & kOpNoHi) != 0;
    const uint32_t move = no_hi ? 0u : 1u;  // columns the strip moves when the lower row grows
    uint32_t inc = warp_all(run.inc), sub = warp_all(run.sub);
    uint32_t p0 = sbase + (uint32_t)run.p0, p1 = sbase + (uint32_t)run.p1;
    uint32_t p2 = sbase + (uint32_t)run.p2, p3 = sbase + (uint32_t)run.p3;
    const uint32_t e = move * es, g0 = (uint32_t)run.g0 + e, g1 = (uint32_t)run.g1 + e;
    int c = warp_all(run.col);
    int limit = warp_all(run.width);
    if constexpr (OUT == kOutGlobal) limit = max(min(limit, lim) - lo, 0);
    uint32_t dst = sbase + (uint32_t)run.dst;
    TO *g = nullptr;
    if constexpr (OUT == kOutGlobal) {
      g = out + (int64_t)run.dst * nt + T0 + c + lane;
      c -= lo;  // columns count from the first one wanted
    }
    if constexpr (OUT == kOutSmem) dst += (uint32_t)lane * sizeof(A);
    A a0[kLaneCols], b1[kLaneCols], a2[kLaneCols], b3[kLaneCols], lp[kLaneCols], hp[kLaneCols], v[kLaneCols];
    auto lower = [&]() {
      if constexpr (PAIR) {
        add_piece(lp, a0, b1);
        round_piece<R16>(lp);
      } else {
#pragma unroll
        for (int k = 0; k < kLaneCols; ++k) lp[k] = a0[k];
      }
    };
    auto upper = [&]() {
      if constexpr (PAIR) {
        add_piece(hp, a2, b3);
        round_piece<R16>(hp);
      } else {
#pragma unroll
        for (int k = 0; k < kLaneCols; ++k) hp[k] = a2[k];
      }
    };
    auto sum = [&]() { add_piece(v, lp, hp); };
    if constexpr (GEN) {
      // a term that a band does not have is -0 (0 for integers): adding it
      // changes no value, the sign of a zero included
#pragma unroll
      for (int k = 0; k < kLaneCols; ++k) b1[k] = a2[k] = b3[k] = no_term(A());
    }
    auto store = [&]() {
      if constexpr (OUT == kOutGlobal) {
        if (c >= 0 && c + kPieceCols <= limit) {
#pragma unroll
          for (int k = 0; k < kLaneCols; ++k) g[32 * k] = to_store<TO>(v[k]);
        } else {
#pragma unroll
          for (int k = 0; k < kLaneCols; ++k) stg_below(g + 32 * k, v[k], c + lane + 32 * k, limit);
        }
      } else if constexpr (OUT == kOutSmem) {
        round_piece<R16>(v);
        if (flags & kRunWhole) {
#pragma unroll
          for (int k = 0; k < kLaneCols; ++k) sts(dst + (uint32_t)(32 * k) * sizeof(A), v[k]);
        } else {
#pragma unroll
          for (int k = 0; k < kLaneCols; ++k)
            sts_below(dst + (uint32_t)(32 * k) * sizeof(A), v[k], c + lane + 32 * k, limit);
        }
      } else {
        // the top level of a searched launch (column c of a row at word c +
        // 4 (c / 16)); it is the output level, never rounded
        const int cl = c + lane;
        const uint32_t at = dst + (uint32_t)(cl + 4 * (cl >> 4)) * (uint32_t)sizeof(A);
#pragma unroll
        for (int k = 0; k < kLaneCols; ++k) sts_below(at + (uint32_t)(40 * k) * sizeof(A), v[k], cl + 32 * k, limit);
      }
    };
    ld_piece<TSrc, A>(a0, p0, lane);
    if (PAIR && !lo_one) ld_piece<TSrc, A>(b1, p1, lane);
    if (!no_hi) {
      ld_piece<TSrc, A>(a2, p2, lane);
      if (PAIR && !hi_one) ld_piece<TSrc, A>(b3, p3, lane);
    }
    lower();
    upper();
    for (int left = warp_all(run.n) - 1; left > 0; --left) {
      sum();
      if (inc & 1u) {
        if (!PAIR || (sub & 1u)) {
          p0 += g0;
          ld_piece<TSrc, A>(a0, p0, lane);
          if constexpr (PAIR && GEN) {
            p1 += e - es;
            if (no_hi && !lo_one) ld_piece<TSrc, A>(b1, p1, lane);
          }
        } else {
          p0 += e;
          p1 += g1;
          ld_piece<TSrc, A>(a0, p0, lane);
          ld_piece<TSrc, A>(b1, p1, lane);
        }
        store();
        c += (int)move;
        if constexpr (OUT == kOutGlobal) g += nt + move;
        dst += (uint32_t)run.dst_row + (OUT == kOutSmem ? move * (uint32_t)sizeof(A) : 0u);
        lower();
      } else {
        if (!PAIR || (sub & 1u)) {
          p2 += (uint32_t)run.g2;
          ld_piece<TSrc, A>(a2, p2, lane);
          if constexpr (PAIR) {
            p3 -= es;
            if (!hi_one) ld_piece<TSrc, A>(b3, p3, lane);
          }
        } else {
          p3 += (uint32_t)run.g3;
          ld_piece<TSrc, A>(b3, p3, lane);
        }
        store();
        if constexpr (OUT == kOutGlobal) g += nt;
        dst += (uint32_t)run.dst_row;
        upper();
      }
      inc >>= 1;
      sub >>= 1;
    }
    sum();
    store();
  }
}

// Level 1 straight from the staged input (section 4: the Option-1 partial
// sums of level 0 and one merge).  The running sums plo = x_lo[tau] + ... +
// x_lo[tau - dl] and phi = x_hi[tau - dl] + ... + x_hi[tau - dl - j] are
// kept in registers in the oracle's order (each adds one earlier sample);
// when dl grows the upper sums move a column.  A walk reads them again a
// column earlier (j + 1 reads; j is 0 or 1 on most rows) or, with many delays
// per channel (kWalkMoves), moves them between lanes, the first column coming
// from 32 more columns of sums that are kept before the piece (`before`; each
// move uses up one, and a walk makes at most 31).  A row's reads are issued before the row before it
// is stored.  SCALE multiplies every sample by its channel's weight first.
// MOVES: the stage has walks that move their sums.
// Bound: instruction issue.  Launch [0,1] of 32 x 159808 x 2738 with fp16
// state, 86 level-0 rows per channel: 1648 us with every upper sum read again,
// 386 us with the moves.
template <class TI, class A, class TO, bool R16, bool SCALE, bool TOP, bool GEN, bool MOVES>
__device__ __forceinline__ void stage_walk(uint32_t sbase, const StageRange &range, int lane,
                                           const float *__restrict__ w, TO *__restrict__ out, int64_t nt, int64_t T0,
                                           int lo, int lim) {
  constexpr uint32_t es = (uint32_t)sizeof(TI);
  for (uint32_t at = range.first; at != range.end; at += (uint32_t)sizeof(FusedWalk)) {
    const FusedWalk wk = prog_desc<FusedWalk>(range.prog, at);
    float wl = 1.0f, wh = 1.0f;
    if constexpr (SCALE) {
      wl = __ldg(w + wk.chan);
      if (!GEN || !(wk.flags & kWalkNoUpper)) wh = __ldg(w + wk.chan + 1);
    }
    const uint32_t xl = sbase + (uint32_t)wk.x_lo, xh = sbase + (uint32_t)wk.x_hi;
    // A channel's samples s columns earlier (scaled).
    auto samples = [&](A (&x)[kLaneCols], uint32_t base, int s, float wt) {
      ld_samples<TI, A>(x, base - (uint32_t)s * es, lane);
      if constexpr (SCALE) {
#pragma unroll
        for (int k = 0; k < kLaneCols; ++k) x[k] = __fmul_rn(x[k], wt);
      }
    };
    const bool upper = !GEN || !(warp_all(wk.flags) & kWalkNoUpper);
    int dl = warp_all(wk.dl0), j = warp_all(wk.a) - dl;
    uint32_t bits = (uint32_t)warp_all(wk.bits);
    const bool moves = MOVES && (warp_all(wk.flags) & kWalkMoves) != 0;
    const int skip = TOP ? max(lo - wk.col, 0) : 0;  // columns before the first one wanted
    const bool whole = TOP ? warp_all(wk.width) >= kPieceCols && warp_all(wk.col) + kPieceCols <= lim && warp_all(skip) == 0
                           : warp_all(wk.width) >= kPieceCols || (warp_all(wk.dst_row) & (kPieceCols * 4 - 1)) == 0;
    const int limit = TOP ? max(min(wk.width, lim - wk.col) - skip, 0) : wk.width;
    uint32_t dst = sbase + (uint32_t)wk.dst + (uint32_t)lane * (uint32_t)sizeof(A);
    TO *g = nullptr;
    if constexpr (TOP) g = out + (int64_t)wk.dst * nt + T0 + wk.col + lane;
    A plo[kLaneCols], phi[kLaneCols], v[kLaneCols], t[kLaneCols], before = A(0);
    // The upper channel's sample s columns before column lane - 32 (scaled);
    // those that no move brings into the piece may lie up to 32 samples before
    // the staged rows, in the slack below them (kUnderRead).
    auto sample_before = [&](int s) -> A {
      A x = load_input<TI, A>(xh + (uint32_t)(lane - 32 - s) * es);
      if constexpr (SCALE) x = __fmul_rn(x, wh);
      return x;
    };
    auto move_upper = [&]() {
      const int from = (lane + 31) & 31;
      A in = __shfl_sync(0xffffffffu, before, from);
      before = in;
#pragma unroll
      for (int k = 0; k < kLaneCols; ++k) {
        const A x = __shfl_sync(0xffffffffu, phi[k], from);
        phi[k] = lane == 0 ? in : x;
        in = x;
      }
    };
    auto store = [&]() {
      if constexpr (TOP) {
        if (whole) {
#pragma unroll
          for (int k = 0; k < kLaneCols; ++k) g[32 * k] = to_store<TO>(v[k]);
        } else {
#pragma unroll
          for (int k = 0; k < kLaneCols; ++k) stg_below(g + 32 * k, v[k], lane + 32 * k - skip, limit);
        }
        g += nt;
      } else {
        round_piece<R16>(v);
        if (whole) {
#pragma unroll
          for (int k = 0; k < kLaneCols; ++k) sts(dst + (uint32_t)(32 * k) * sizeof(A), v[k]);
        } else {
#pragma unroll
          for (int k = 0; k < kLaneCols; ++k)
            sts_below(dst + (uint32_t)(32 * k) * sizeof(A), v[k], lane + 32 * k, limit);
        }
        dst += (uint32_t)wk.dst_row;
      }
    };
    auto sum = [&]() {
      if constexpr (R16) {
#pragma unroll
        for (int k = 0; k < kLaneCols; ++k) v[k] = acc_add(round_state<R16>(plo[k]), round_state<R16>(phi[k]));
      } else {
        add_piece(v, plo, phi);
      }
    };
    samples(plo, xl, 0, wl);
    if constexpr (GEN) {
#pragma unroll
      for (int k = 0; k < kLaneCols; ++k) phi[k] = no_term(A());
    }
    if (upper) samples(phi, xh, dl, wh);
    for (int i = 1; i <= dl; ++i) {
      samples(t, xl, i, wl);
      add_piece(plo, plo, t);
    }
    if (upper)
      for (int i = 1; i <= j; ++i) {
        samples(t, xh, dl + i, wh);
        add_piece(phi, phi, t);
      }
    if (moves) {
      before = sample_before(dl);
      for (int i = 1; i <= j; ++i) before = acc_add(before, sample_before(dl + i));
    }
    for (int left = warp_all(wk.e - wk.a); left > 0; --left) {
      sum();
      if (!upper || (bits & 1u)) {  // (a single channel: row r is its Option-1 row r, dl = r)
        ++dl;
        samples(t, xl, dl, wl);
        if (moves) move_upper();
        else if (upper) samples(phi, xh, dl, wh);
        store();
        add_piece(plo, plo, t);
        if (upper && !moves)
          for (int i = 1; i <= j; ++i) {
            samples(t, xh, dl + i, wh);
            add_piece(phi, phi, t);
          }
      } else {
        ++j;
        samples(t, xh, dl + j, wh);
        if (moves) before = acc_add(before, sample_before(dl + j));
        store();
        add_piece(phi, phi, t);
      }
      bits >>= 1;
    }
    sum();
    store();
  }
}

// The walk stage writing the top level (global memory) or a stored one.
template <class TI, class A, class TO, bool R16, bool SCALE, bool GEN, bool MOVES>
__device__ __forceinline__ void walk_out(bool top, uint32_t sbase, const StageRange &r, int lane,
                                         const float *__restrict__ w, TO *__restrict__ out, int64_t nt, int64_t T0,
                                         int lo, int lim) {
  if (top) stage_walk<TI, A, TO, R16, SCALE, true, GEN, MOVES>(sbase, r, lane, w, out, nt, T0, lo, lim);
  else stage_walk<TI, A, TO, R16, SCALE, false, GEN, MOVES>(sbase, r, lane, w, out, nt, T0, lo, lim);
}

// A single or pair stage of an item; TSrc is the type of the stage's source
// rows (the staged base level for the first stage, the accumulator type
// after it).  GEN: the plan may hold stages with passed-up or one-term
// halves (else only the code without those tests is compiled in).
template <class TSrc, class A, class TO, bool R16, int OUT, bool GEN = true>
__device__ __forceinline__ void run_merge_stage(const StageRange &r, uint32_t sbase, int lane, TO *__restrict__ out,
                                                int64_t nt, int64_t T0, int lo, int lim) {
  const bool gen = GEN && (r.kind & kStageGeneral) != 0;
  if ((r.kind & kStageKindMask) == kStagePair) {
    if (gen) stage_runs<TSrc, A, TO, R16, OUT, true, true>(sbase, r, lane, out, nt, T0, lo, lim);
    else stage_runs<TSrc, A, TO, R16, OUT, true, false>(sbase, r, lane, out, nt, T0, lo, lim);
  } else {
    if (gen) stage_runs<TSrc, A, TO, R16, OUT, false, true>(sbase, r, lane, out, nt, T0, lo, lim);
    else stage_runs<TSrc, A, TO, R16, OUT, false, false>(sbase, r, lane, out, nt, T0, lo, lim);
  }
}

// ---------------------------------------------------------------------------
// Boxcar search of the top level (section 4.2, pulse profile) in the last
// launch.  For width w = 2^k the boxcar sum B_w[t] = A[t - w + 1] + ... +
// A[t] is built as the binary tree B_1 = A, B_2w[t] = B_w[t] + B_w[t - w];
// per (row, width) the largest value over the tile's own columns and the
// region where it first occurs are kept, to be resolved to a time by the
// search's finalize kernel, which recomputes the region from A.  Regions
// are 16 samples for widths 1 .. 16 and 256 samples for widths 32 .. 256,
// named by the time of their first sample.

constexpr int kSearchNoRegion = INT32_MIN;

__device__ __forceinline__ float search_lowest(float) { return -__int_as_float(0x7f800000); }
__device__ __forceinline__ int32_t search_lowest(int32_t) { return INT32_MIN; }
__device__ __forceinline__ float search_max(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ int32_t search_max(int32_t a, int32_t b) { return max(a, b); }

// Per (row, width) best of an item, one 64-bit word in shared memory
// reduced with atomicMax: the value's order-preserving bits above the
// complement of its region, so the maximum is the largest value and, among
// equal values, the earliest region.  0 = nothing seen.
__device__ __forceinline__ uint32_t search_order(float v) {
  const uint32_t b = __float_as_uint(v);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ uint32_t search_order(int32_t v) { return (uint32_t)v ^ 0x80000000u; }
__device__ __forceinline__ float search_value(uint32_t o, float) {
  return __uint_as_float((o & 0x80000000u) ? (o & 0x7fffffffu) : ~o);
}
__device__ __forceinline__ int32_t search_value(uint32_t o, int32_t) { return (int32_t)(o ^ 0x80000000u); }
__device__ __forceinline__ bool search_nan(float v) { return v != v; }
__device__ __forceinline__ bool search_nan(int32_t) { return false; }

// The key of the largest of x[16 .. 31] over the columns c0 + S (i - 16) in
// [lo, hi), with `region` (the time of the region's first sample); 0 when
// `use` is false or nothing qualifies.  NaN never qualifies (the transform
// of finite input is finite).
template <class A, int S>
__device__ __forceinline__ unsigned long long search_key(const A (&x)[32], bool use, int c0, int lo, int hi,
                                                         int region) {
  if (!use) return 0ull;
  A m;
  if (c0 >= lo && c0 + 15 * S < hi) {
    A t[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) t[i] = search_max(x[16 + i], x[24 + i]);
#pragma unroll
    for (int i = 0; i < 4; ++i) t[i] = search_max(t[i], t[i + 4]);
    m = search_max(search_max(t[0], t[2]), search_max(t[1], t[3]));
  } else {
    m = search_lowest(A());
    bool any = false;
#pragma unroll
    for (int i = 16; i < 32; ++i) {
      const int c = c0 + S * (i - 16);
      if (c >= lo && c < hi) {
        m = search_max(m, x[i]);
        any = true;
      }
    }
    if (!any) return 0ull;
  }
  if (search_nan(m)) return 0ull;
  return ((unsigned long long)search_order(m) << 32) | (uint32_t)(0x7fffffff - region);
}

// Joins the keys of a warp into the best words they name: lanes naming the
// same word are reduced in registers first (largest value, then earliest
// region), then one atomicMax per word.  Every lane of the warp calls it.
__device__ __forceinline__ void search_join_warp(unsigned long long key, uint32_t addr, int lane) {
  const unsigned group = __match_any_sync(0xffffffffu, addr);
  const uint32_t hi = (uint32_t)(key >> 32);
  const uint32_t mhi = __reduce_max_sync(group, hi);
  const uint32_t mlo = __reduce_max_sync(group, hi == mhi ? (uint32_t)key : 0u);
  if (lane == __ffs(group) - 1 && (mhi | mlo) != 0u) {
    const unsigned long long k = ((unsigned long long)mhi << 32) | mlo;
    asm volatile("atom.shared.max.u64 _, [%0], %1;" ::"r"(addr), "l"(k) : "memory");
  }
}

__device__ __forceinline__ int4 lds128(uint32_t a) {
  int4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a)
               : "memory");
  return v;
}
__device__ __forceinline__ void sts128(uint32_t a, int4 v) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
               : "memory");
}

// The boxcar search of an item's top rows (Pt, search layout), all threads
// of the block together.  The stage's ops are the rows (dst = global row,
// p0 = the row in Pt, width = own columns W, col = history columns).
// Phase 1 takes (row, run of 16 columns) units, whole rows per wave, lane
// after lane along a row: a unit loads its run and the run before it, then
// (after a block barrier) writes the run's own columns to A, doubles four
// times in registers (widths 1 .. 16) and stores B_16 over its run in place
// (no later wave reads those rows).  Phase 2 takes (256-column group, row,
// residue) units over B_16 at stride 16 (widths 32 .. 256).  Each unit's
// best per width joins the row's best in shared memory (`best`, rows x
// widths words); the bests are written as the tile's partials.
template <class A, class TO>
__device__ __forceinline__ void stage_search_block(uint32_t sbase, const FusedOp *__restrict__ ops, int op0,
                                                   int op1, TO *__restrict__ out, int64_t nt, int64_t T0, int lim,
                                                   int64_t tile, const SearchArgs &sa) {
  const int tid = threadIdx.x, R = op1 - op0, nk = sa.nk;
  if (R <= 0) return;
  const uint32_t best = sbase + sa.q_off;
  for (int i = tid; i < R * nk; i += kFusedThreads)
    asm volatile("st.shared.u64 [%0], %1;" ::"r"(best + 8u * i), "l"(0ull) : "memory");
  const FusedOp op_first = ld_op(ops + op0);
  const int hist = op_first.col, n = op_first.width + hist, own_hi = hist + lim, runs = n >> 4;
  const int32_t t0 = (int32_t)(T0 - hist);  // time of window column 0
  const int per_wave = kFusedThreads / runs;  // whole rows per wave (runs <= kFusedThreads)
  compute_sync();
  const int lane = tid & 31;
  for (int row0 = 0; row0 < R; row0 += per_wave) {
    const int ri = row0 + tid / runs, r = tid % runs;
    const bool valid = tid < per_wave * runs && ri < R;
    FusedOp op{};
    A x[32];
    uint32_t cur = 0;
    if (valid) {
      op = ld_op(ops + op0 + ri);
      cur = sbase + op.p0 + (uint32_t)(20 * r) * sizeof(A);
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int4 hi = lds128(cur + 16u * v);
        const int4 lo = r > 0 ? lds128(cur - 80u + 16u * v) : make_int4(0, 0, 0, 0);
        const A *ph = reinterpret_cast<const A *>(&hi);
        const A *pl = reinterpret_cast<const A *>(&lo);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          x[16 + 4 * v + e] = ph[e];
          x[4 * v + e] = pl[e];
        }
      }
    } else {
#pragma unroll
      for (int j = 0; j < 32; ++j) x[j] = A(0);
    }
    compute_sync();  // the wave's rows are all loaded before any run is overwritten
    const int c0 = 16 * r;
    if (valid) {
      TO *arow = out + (int64_t)op.dst * nt + T0 - hist;
      if (c0 >= hist && c0 + 16 <= own_hi) {
        int4 *dv = reinterpret_cast<int4 *>(arow + c0);
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          TO o[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) o[e] = to_store<TO>(x[16 + 4 * v + e]);
          dv[v] = *reinterpret_cast<const int4 *>(o);
        }
      } else {
#pragma unroll
        for (int e = 0; e < 16; ++e)
          if (c0 + e >= hist && c0 + e < own_hi) arow[c0 + e] = to_store<TO>(x[16 + e]);
      }
    }
    const bool owned = valid && c0 + 15 >= hist && c0 < own_hi;
    const uint32_t brow = best + 8u * (uint32_t)((valid ? ri : 0) * nk);
    search_join_warp(search_key<A, 1>(x, owned, c0, hist, own_hi, t0 + c0), brow, lane);
#pragma unroll
    for (int m = 1; m <= 4; ++m) {
      const int h = 1 << (m - 1);
#pragma unroll
      for (int j = 31; j >= (1 << m); --j) x[j] = acc_add(x[j], x[j - h]);
      if (m < nk) search_join_warp(search_key<A, 1>(x, owned, c0, hist, own_hi, t0 + c0), brow + 8u * m, lane);
    }
    if (nk > 5 && valid) {
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        int4 o;
        A *po = reinterpret_cast<A *>(&o);
#pragma unroll
        for (int e = 0; e < 4; ++e) po[e] = x[16 + 4 * v + e];
        sts128(cur + 16u * v, o);
      }
    }
    compute_sync();  // before the next wave (and phase 2) reads its rows
  }
  if (nk > 5) {
    const int groups = (n + 255) >> 8;
    const int U2 = R * groups * 16;
    for (int u0 = 0; u0 < U2; u0 += kFusedThreads) {
      const int u = u0 + tid;
      const int rho = u & 15, ri = (u >> 4) % R, g = (u >> 4) / R;
      const int base = 256 * g;
      // groups without an own column take no part (but every lane joins)
      const bool use = u < U2 && base + 256 > hist && base < own_hi;
      A x[32];
      uint32_t brow = best;
      if (use) {
        const FusedOp op = ld_op(ops + op0 + ri);
        const uint32_t row = sbase + op.p0;
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          const int c = base + rho + 16 * (j - 16);
          x[j] = (c >= 0 && c < n) ? Lds<A>::get(row + (uint32_t)search_pidx(c) * sizeof(A)) : A(0);
        }
        brow = best + 8u * (uint32_t)(ri * nk);
      } else {
#pragma unroll
        for (int j = 0; j < 32; ++j) x[j] = A(0);
      }
#pragma unroll
      for (int m = 1; m <= 4; ++m) {
        const int h = 1 << (m - 1);
#pragma unroll
        for (int j = 31; j >= (1 << m); --j) x[j] = acc_add(x[j], x[j - h]);
        if (4 + m < nk)
          search_join_warp(search_key<A, 16>(x, use, base + rho, hist, own_hi, t0 + base), brow + 8u * (4 + m),
                           lane);
      }
    }
    compute_sync();
  }
  // The row bests become the tile's partials.
  for (int i = tid; i < R * nk; i += kFusedThreads) {
    const int ri = i / nk, k = i - ri * nk;
    unsigned long long key;
    asm volatile("ld.shared.u64 %0, [%1];" : "=l"(key) : "r"(best + 8u * i) : "memory");
    const FusedOp op = ld_op(ops + op0 + ri);
    const int64_t slot = ((int64_t)op.dst * nk + k) * sa.nseg + tile;
    if (key == 0) {
      sa.part_r[slot] = kSearchNoRegion;
    } else {
      static_cast<A *>(sa.part_v)[slot] = search_value((uint32_t)(key >> 32), A());
      sa.part_r[slot] = 0x7fffffff - (int32_t)(uint32_t)key;
    }
  }
}

// The first stage of an item: level 1 walked from the staged input
// (FROM_INPUT) or the first single / pair stage over the staged base rows.
// TB is the staged base level's type and TO the type written to global memory when this stage is
// the top.  With SEARCH the stage before the search writes the top level
// into Pt instead.  Rows of the top level are nt apart in `out`; its columns
// T0 + [lo, lim) are written.  GEN as for run_merge_stage; SCALE: the input
// is multiplied by channel weights (float input only); MOVES: some stage is
// kStageMoves.
template <class TI, class TB, class A, class TO, bool R16, bool FROM_INPUT, bool SEARCH, bool GEN, bool SCALE, bool MOVES>
__device__ __forceinline__ void item_first_stage(uint32_t sbase, const Prog &prog, int n_stages,
                                                 const float *__restrict__ w, int warp, int lane,
                                                 TO *__restrict__ out, int64_t nt, int64_t T0, int lo, int lim) {
  const StageRange r = prog_stage(prog, 0, warp);
  const bool top = !SEARCH && n_stages == 1;
  if constexpr (FROM_INPUT) {
    constexpr bool kScale = SCALE && std::is_floating_point<A>::value;
    const bool gen = GEN && (r.kind & kStageGeneral) != 0;
    if (MOVES && (r.kind & kStageMoves) != 0)
      walk_out<TI, A, TO, R16, kScale, GEN, MOVES>(top, sbase, r, lane, w, out, nt, T0, lo, lim);
    else if (gen) walk_out<TI, A, TO, R16, kScale, GEN, false>(top, sbase, r, lane, w, out, nt, T0, lo, lim);
    else walk_out<TI, A, TO, R16, kScale, false, false>(top, sbase, r, lane, w, out, nt, T0, lo, lim);
  } else if constexpr (SEARCH) {
    if (n_stages == 2) run_merge_stage<TB, A, TO, R16, kOutPadded, GEN>(r, sbase, lane, out, nt, T0, lo, lim);
    else run_merge_stage<TB, A, TO, R16, kOutSmem, GEN>(r, sbase, lane, out, nt, T0, lo, lim);
  } else {
    if (top) run_merge_stage<TB, A, TO, R16, kOutGlobal, GEN>(r, sbase, lane, out, nt, T0, lo, lim);
    else run_merge_stage<TB, A, TO, R16, kOutSmem, GEN>(r, sbase, lane, out, nt, T0, lo, lim);
  }
}

// Stages 1 .. n - 1 of an item (sources in Pa / Pb), a barrier of the
// computing warps before each; the last writes global memory (with SEARCH:
// the one before it writes Pt and the last is the search).
template <class A, class TO, bool R16, bool SEARCH, bool GEN = true>
__device__ __forceinline__ void item_later_stages(uint32_t sbase, const Prog &prog, int n_stages,
                                                  const FusedOp *__restrict__ ops, int warp, int lane,
                                                  TO *__restrict__ out, int64_t nt, int64_t T0, int lo, int lim,
                                                  int64_t tile, const SearchArgs &sa) {
  for (int s = 1; s < n_stages; ++s) {
    compute_sync();
    if constexpr (SEARCH) {
      if (s == n_stages - 1) {
        // every thread: the whole stage's rows (warp 0's first to the end)
        const uint32_t at = (uint32_t)(s * kProgStageBytes);
        stage_search_block<A, TO>(sbase, ops, prog_word(prog, at + 4u), prog_word(prog, at + 4u * (kStageWords - 1)), out,
                                  nt, T0, lim, tile, sa);
        return;
      }
    }
    const StageRange r = prog_stage(prog, s, warp);
    if (SEARCH && s == n_stages - 2) run_merge_stage<A, A, TO, R16, kOutPadded, GEN>(r, sbase, lane, out, nt, T0, lo, lim);
    else if (!SEARCH && s == n_stages - 1) run_merge_stage<A, A, TO, R16, kOutGlobal, GEN>(r, sbase, lane, out, nt, T0, lo, lim);
    else run_merge_stage<A, A, TO, R16, kOutSmem, GEN>(r, sbase, lane, out, nt, T0, lo, lim);
  }
}

// Row copies of an item.
__device__ __forceinline__ FusedLoad fetch_load(const FusedProg &tp, const FusedLoad *__restrict__ loads, int i) {
  if (i < tp.load_count) return loads[tp.load_begin + i];
  return FusedLoad{0, 0, 0, 0};
}

// Stage the rows of a work item into region S: one warp; lane 0 announces
// the bytes on the mbarrier, then the lanes issue the copies.  `first` is
// load `lane` of the item, fetched ahead of time, so the copies go out
// without waiting on a descriptor read.  cshift > 0: row blocks of
// 2^cshift-element chunks; else row boxes of `box` elements.
template <class TS>
__device__ __forceinline__ void stage_item(unsigned char *smem, uint32_t bar, const CUtensorMap *maps, const FusedProg &tp,
                                           const FusedLoad *__restrict__ loads, const FusedLoad &first, int64_t T0,
                                           int32_t box, int32_t cshift, int lane) {
  // Order this block's earlier generic-proxy accesses of S before the
  // async-proxy copies that overwrite it.
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (lane == 0) mbar_arrive_expect_tx(bar, (uint32_t)tp.tx_bytes);
  __syncwarp();
  const uint32_t box_bytes = (uint32_t)box * (uint32_t)sizeof(TS);
  for (int i = lane; i < tp.load_count; i += 32) {
    const FusedLoad ld = (i == lane) ? first : loads[tp.load_begin + i];
    const int32_t x = (int32_t)(T0 + ld.xoff);
    const uint32_t dst = smem_u32(smem + ld.smem);
    if (cshift > 0) {
      tma_load_block(dst, maps + ld.nbox, x >> cshift, ld.row, bar);
    } else {
      for (int b = 0; b < ld.nbox; ++b) tma_load_row(dst + b * box_bytes, maps, x + b * box, ld.row, bar);
    }
  }
}

// Ask for the rows of a work item to be brought into L2 (the same copies as
// stage_item, without their shared memory).
template <class TS>
__device__ __forceinline__ void prefetch_item(const CUtensorMap *maps, const FusedProg &tp,
                                              const FusedLoad *__restrict__ loads, const FusedLoad &first, int64_t T0,
                                              int32_t box, int32_t cshift, int lane) {
  for (int i = lane; i < tp.load_count; i += 32) {
    const FusedLoad ld = (i == lane) ? first : loads[tp.load_begin + i];
    const int32_t x = (int32_t)(T0 + ld.xoff);
    if (cshift > 0) {
      asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(
                       reinterpret_cast<uint64_t>(maps + ld.nbox)),
                   "r"(0), "r"(x >> cshift), "r"(ld.row)
                   : "memory");
    } else {
      for (int b = 0; b < ld.nbox; ++b)
        asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(
                         reinterpret_cast<uint64_t>(maps)),
                     "r"(x + b * box), "r"(ld.row)
                     : "memory");
    }
  }
}

// Copy an item's programme to its slot at shared address dst, on the same
// barrier phase (its bytes are part of tx_bytes); one lane.
__device__ __forceinline__ void stage_prog(uint32_t dst, const FusedProg &pr, const int4 *__restrict__ prog,
                                           uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(prog + pr.prog), "r"((uint32_t)pr.prog_bytes), "r"(bar)
               : "memory");
}

// ---------------------------------------------------------------------------
// Blocks of eight computing warps and a copying one.  The barrier slot holds
// the `full` mbarrier (an item's rows and programme have landed), the `free`
// mbarrier (every computing warp is done with the staged rows) and two item
// headers (tile, columns of the tile inside [0, nt), stages, programme).

constexpr int kFusedLaunchThreads = kFusedThreads + 32;
constexpr uint32_t kFreeBar = 8, kItemHeader = 32;
constexpr int32_t kTileChunk = 304;  // time tiles of one chunk of items

__device__ __forceinline__ void init_item_barriers(uint32_t full) {
  if (threadIdx.x == 0) {
    mbar_init(full, 1);
    mbar_init(full + kFreeBar, kFusedWarps);
    fence_mbar_init();
  }
  __syncthreads();
}

// The copying warp: stages item i + 1 (its rows into S, its programme into
// one of two slots, its place into one of two headers) as soon as the
// computing warps have arrived at `free`, behind their first stage of item
// i, the only one that reads S; its own bookkeeping is off their path.
// Items go tile chunk by tile chunk, template by template within a chunk,
// tile by tile within a template: neighbouring templates share staged rows,
// and a chunk keeps their second reading within reach of L2 whatever the row
// length.  Row blocks are also asked for one item ahead: L2 hides the HBM
// latency that a block's single staging region cannot.  1024 x 65536 x 1024
// float32 306 us without, 289 us with; 4096 x 2^18 x 4096, HBM-bound in its
// cones, 5.67 ms without, 5.70 with, 6.36 with the requests but template by
// template.  (Row boxes are bound by the rate of copies: asking twice made
// them 5 % slower.)  also_ahead(programme, T0) asks for whatever else the next
// item reads.
template <class TS, class Ahead>
__device__ __forceinline__ void copy_items(unsigned char *smem, const TmaMaps &maps, int64_t nt, int32_t W,
                                           int32_t tile0, int32_t ntiles, int64_t items,
                                           const FusedProg *__restrict__ progs, const int4 *__restrict__ prog,
                                           const FusedLoad *__restrict__ loads, int32_t box, int32_t cshift,
                                           int32_t prog_off, int32_t prog_slot, int *__restrict__ status, int lane,
                                           Ahead also_ahead) {
  const uint32_t full = smem_u32(smem), free_bar = full + kFreeBar, header = full + kItemHeader;
  int64_t item = blockIdx.x;
  if (item >= items) return;
  const int32_t ntpl = (int32_t)(items / ntiles);
  const int64_t per_chunk = (int64_t)kTileChunk * ntpl;
  int32_t tile = 0, tpl = 0;
  auto place = [&](int64_t i) {
    const int64_t chunk = i / per_chunk;
    const int32_t first_tile = (int32_t)(chunk * kTileChunk), n = min(kTileChunk, ntiles - first_tile);
    const int32_t r = (int32_t)(i - chunk * per_chunk);
    tpl = r / n;
    tile = first_tile + r % n;
  };
  place(item);
  FusedProg pr = progs[tpl];
  FusedLoad ld = fetch_load(pr, loads, lane);
  uint32_t slot = 0, phase = 0;
  for (bool first = true; item < items; item += gridDim.x, first = false) {
    if (!first) {
      if (!mbar_wait_bounded(free_bar, phase)) {
        // The computing warps gave up (or never arrived): let the copies in
        // flight land before the block ends.
        atomicExch(status, 1);
        mbar_wait_bounded(full, phase);
        return;
      }
      phase ^= 1u;
    }
    const int64_t T0 = (int64_t)(tile0 + tile) * W;
    if (lane == 0) {
      const int lim = (int)((nt - T0) < (int64_t)W ? (nt - T0) : (int64_t)W);
      sts_v4(header + 16u * slot, make_int4(tile0 + tile, lim, pr.n_stages, pr.prog));
    }
    stage_item<TS>(smem, full, maps.m, pr, loads, ld, T0, box, cshift, lane);
    if (lane == 0 && prog_slot > 0) stage_prog(full + (uint32_t)(prog_off + (int)slot * prog_slot), pr, prog, full);
    slot ^= 1u;
    if (item + gridDim.x < items) {
      place(item + gridDim.x);
      pr = progs[tpl];
      ld = fetch_load(pr, loads, lane);
      const int64_t T1 = (int64_t)(tile0 + tile) * W;
      if (cshift > 0) prefetch_item<TS>(maps.m, pr, loads, ld, T1, box, cshift, lane);
      also_ahead(pr, T1);
    }
  }
  // The last copies land before the block ends: the computing warps wait
  // for them (or give up, which the bounded wait covers).
  mbar_wait_bounded(full, phase);
}

}  // namespace fdmt
