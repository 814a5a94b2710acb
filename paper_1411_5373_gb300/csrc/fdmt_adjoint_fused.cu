// Fused-schedule kernel of the FDMT adjoint (pull cones of several
// transposed levels per launch; planner in fdmt_adjoint_plan.cpp, layout in
// fdmt_adjoint_fused.h).
//
// One block computes one cone for one time tile, persistent over items as
// the forward cone kernel: a copying warp stages the cone's level-lt gradient
// rows by TMA (zeros past Nt) with the item's programme, the computing warps
// wait on the mbarrier (bounded: on timeout the block sets the plan's status
// word and returns), then the stages run level by level, each child row summing its run of parent rows
// in increasing row order; the last stage writes the owned level-lb rows,
// or the input gradient (the Option-1 transpose) in the launch that ends at
// level 0.  The next item's copies go out as soon as the first stage has
// read the staged rows.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "fdmt_adjoint_fused.h"
#include "fdmt_fused_dev.cuh"
#include "fdmt_internal.h"
#include "fdmt_residency.h"
#include "fdmt_tma.h"

namespace fdmt {

namespace {

// Predicated stores (no branch): only columns below the limit are written.
__device__ __forceinline__ void sts_if(uint32_t a, float v, bool p) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q st.shared.f32 [%0], %1;\n\t}"
               ::"r"(a), "f"(v), "r"((uint32_t)p) : "memory");
}
__device__ __forceinline__ void stg_if(float *g, float v, bool p) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q st.global.f32 [%0], %1;\n\t}"
               ::"l"(g), "f"(v), "r"((uint32_t)p) : "memory");
}

// A gather op's result to shared memory; a whole piece without predicates.
__device__ __forceinline__ void st_piece_smem(uint32_t addr, const float (&v)[kLaneCols], int width, int lane) {
  addr += (uint32_t)lane * 4u;
  if (width >= kPieceCols) {
#pragma unroll
    for (int k = 0; k < kLaneCols; ++k) sts_f32(addr + 128u * (uint32_t)k, v[k]);
  } else {
#pragma unroll
    for (int k = 0; k < kLaneCols; ++k) sts_if(addr + 128u * (uint32_t)k, v[k], lane + 32 * k < width);
  }
}

// out_row[t] for t = t0 + lane + 32 k: written where the piece column is
// below `width` and 0 <= t < nt (bands tile time with their own offset, so
// t0 may be negative).
__device__ __forceinline__ void adj_store_global(float *__restrict__ out_row, int64_t t0,
                                                 const float (&v)[kLaneCols], int width, int64_t nt, int lane) {
  if (width == kPieceCols && t0 >= 0 && t0 + kPieceCols <= nt) {  // a whole piece inside [0, nt)
    float *p = out_row + t0 + lane;
#pragma unroll
    for (int k = 0; k < kLaneCols; ++k) p[32 * k] = v[k];
    return;
  }
#pragma unroll
  for (int k = 0; k < kLaneCols; ++k) {
    const int tau = lane + 32 * k;
    const int64_t t = t0 + tau;
    const bool ok = tau < width && t >= 0 && t < nt;
    stg_if(out_row + (ok ? t : 0), v[k], ok);
  }
}

// The columns [first, end) of an init op's piece that lie below its width and
// inside [0, nt).
struct Inside {
  int first, end;
  __device__ __forceinline__ Inside(int64_t t0, int width, int64_t nt)
      : first(t0 < 0 ? (int)max(t0, (int64_t)-kPieceCols) * -1 : 0),
        end(nt - t0 < width ? (int)max(nt - t0, (int64_t)0) : width) {}
  __device__ __forceinline__ bool whole() const { return first == 0 && end == kPieceCols; }
  __device__ __forceinline__ bool holds(int col) const { return col >= first && col < end; }
};

// One transposed level: each op sums its run of p2 parent rows (stride p1
// bytes; the upper half's stride includes the one-column shift per row).
template <int OUT>
__device__ __forceinline__ void adj_gather_stage(uint32_t sbase, const StageRange &range, int lane,
                                                 float *__restrict__ out, int64_t nt, int64_t T0) {
  for (uint32_t at = range.first; at != range.end; at += (uint32_t)sizeof(FusedOp)) {
    const FusedOp op = prog_desc<FusedOp>(range.prog, at);
    const int terms = warp_all(op.p2);
    // the sum starts from the first row of the run and adds the others in
    // row order; runs of one to three rows (nearly all) are straight-line
    float v[kLaneCols];
    const uint32_t a0 = sbase + (uint32_t)op.p0;
    const uint32_t step = (uint32_t)op.p1;
    ld_piece<float, float>(v, a0, lane);
    if (terms == 2) {
      float x[kLaneCols];
      ld_piece<float, float>(x, a0 + step, lane);
      add_piece(v, v, x);
    } else if (terms == 3) {
      float x[kLaneCols], y[kLaneCols];
      ld_piece<float, float>(x, a0 + step, lane);
      ld_piece<float, float>(y, a0 + 2 * step, lane);
      add_piece(v, v, x);
      add_piece(v, v, y);
    } else if (terms > 3) {
      uint32_t a = a0 + step;
      for (int j = 1; j < terms; ++j, a += step) {
        float x[kLaneCols];
        ld_piece<float, float>(x, a, lane);
        add_piece(v, v, x);
      }
    }
    if constexpr (OUT == kOutSmem)
      st_piece_smem(sbase + (uint32_t)op.dst, v, op.width, lane);
    else
      adj_store_global(out + (int64_t)op.dst * nt, T0 + op.col, v, op.width, nt, lane);
  }
}

// Transpose of the Option-1 initialisation for one channel:
//   g_in[tau] = sum_{j < rows} sum_{i <= j} g0[j][tau + i]
// (j outer, i inner), scaled by the channel weight when w is given.  With
// `part`, each op also writes its piece's share of the weight gradient,
// sum_tau x[k][t] g_in[tau] (unscaled), summed in a fixed order: per lane
// over its columns, then a butterfly over the lanes; slot (channel, tile,
// piece).
__device__ __forceinline__ void adj_init_load_x(float (&xv)[kLaneCols], const FusedOp &op,
                                                const float *__restrict__ x, int64_t nt, int64_t T0, int lane) {
  const int64_t t0 = T0 + op.col;
  const Inside in(t0, op.width, nt);
  const float *p = x + (int64_t)op.dst * nt + t0 + lane;
  if (in.whole()) {
#pragma unroll
    for (int k = 0; k < kLaneCols; ++k) xv[k] = __ldg(p + 32 * k);
  } else {
#pragma unroll
    for (int k = 0; k < kLaneCols; ++k) xv[k] = in.holds(lane + 32 * k) ? __ldg(p + 32 * k) : 0.f;
  }
}

// Asks L2 for the input samples that an item's init ops will read (whole 16
// bytes inside [0, nt); the ragged ends come with their first reader).
__device__ __forceinline__ void adj_init_ahead(const FusedProg &pr, const int4 *__restrict__ prog,
                                               const float *__restrict__ x, int64_t nt, int64_t T0, int lane) {
  const char *words = reinterpret_cast<const char *>(prog + pr.prog);
  const int32_t *stage = reinterpret_cast<const int32_t *>(words + (pr.n_stages - 1) * kProgStageBytes);
  const int32_t first = stage[1], n = (stage[kStageWords - 1] - first) / (int32_t)sizeof(FusedOp);
  const FusedOp *ops = reinterpret_cast<const FusedOp *>(words + first);
  for (int32_t i = lane; i < n; i += 32) {
    const int64_t t = T0 + ops[i].col, a = t < 0 ? 0 : t, b = t + ops[i].width < nt ? t + ops[i].width : nt;
    const float *row = x + (int64_t)ops[i].dst * nt;
    const uint64_t from = (reinterpret_cast<uint64_t>(row + a) + 15) & ~15ull;
    const uint64_t to = reinterpret_cast<uint64_t>(row + b) & ~15ull;
    if (a < b && from < to)
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(from), "r"((uint32_t)(to - from)) : "memory");
  }
}

// FOLD: the op is kAdjInitF (level-0 values re-formed from level-1 runs).
template <bool FOLD>
__device__ __forceinline__ void adj_init_op(uint32_t sbase, const FusedOp &op, const float (&xv)[kLaneCols],
                                            int lane, float *__restrict__ out, int64_t nt, int64_t T0,
                                            const float *__restrict__ w, float *__restrict__ part,
                                            int64_t part_row) {
  // (j, i) = (0, 0) first, then the other terms in order
  float v[kLaneCols];
  if constexpr (FOLD) {
    // term (j, i) is level-0 row j at column tau + i: its run of level-1
    // rows summed in row order, as the gather would have stored it (runs of
    // one or two rows, nearly all, without a loop)
    uint32_t pj = sbase + (uint32_t)op.p0;
    const uint32_t step = (uint32_t)op.p1, back = 4u * (uint32_t)(op.flags & 1);
    uint32_t runs = (uint32_t)warp_all(op.flags) >> 1;
    const int rows = warp_all(op.p2);
    auto term = [&](float (&r)[kLaneCols], uint32_t a, int cnt) {
      ld_piece<float, float>(r, a, lane);
      if (cnt > 1) {
        float y[kLaneCols];
        ld_piece<float, float>(y, a + step, lane);
        add_piece(r, r, y);
        for (int q = 2; q < cnt; ++q) {
          ld_piece<float, float>(y, a + (uint32_t)q * step, lane);
          add_piece(r, r, y);
        }
      }
    };
    int cnt = (int)(runs & 15u);
    term(v, pj, cnt);
    for (int j = 1; j < rows; ++j) {
      pj += (uint32_t)cnt * step - back;
      runs >>= 4;
      cnt = (int)(runs & 15u);
      for (int ii = 0; ii <= j; ++ii) {
        float r[kLaneCols];
        term(r, pj + 4u * (uint32_t)ii, cnt);
        add_piece(v, v, r);
      }
    }
  } else {
    ld_piece<float, float>(v, sbase + (uint32_t)op.p0, lane);
    for (int j = 1; j < op.p2; ++j) {
      const uint32_t row = sbase + (uint32_t)op.p0 + (uint32_t)(j * op.p1);
      for (int ii = 0; ii <= j; ++ii) {
        float y[kLaneCols];
        ld_piece<float, float>(y, row + (uint32_t)(4 * ii), lane);
        add_piece(v, v, y);
      }
    }
  }
  const Inside in(T0 + op.col, op.width, nt);
  if (part != nullptr) {
    float d = 0.f;
    if (in.whole()) {
#pragma unroll
      for (int k = 0; k < kLaneCols; ++k) d = __fadd_rn(d, __fmul_rn(xv[k], v[k]));
    } else {
#pragma unroll
      for (int k = 0; k < kLaneCols; ++k)
        d = __fadd_rn(d, in.holds(lane + 32 * k) ? __fmul_rn(xv[k], v[k]) : 0.f);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) d = __fadd_rn(d, __shfl_xor_sync(0xffffffffu, d, off));
    if (lane == 0) part[(int64_t)op.dst * part_row + op.p3] = d;
  }
  if (w != nullptr) {
    const float wk = __ldg(w + op.dst);
#pragma unroll
    for (int k = 0; k < kLaneCols; ++k) v[k] = __fmul_rn(v[k], wk);
  }
  float *p = out + (int64_t)op.dst * nt + T0 + op.col + lane;
  if (in.whole()) {
#pragma unroll
    for (int k = 0; k < kLaneCols; ++k) p[32 * k] = v[k];
  } else {
#pragma unroll
    for (int k = 0; k < kLaneCols; ++k)
      if (in.holds(lane + 32 * k)) p[32 * k] = v[k];
  }
}

// The init stage takes its ops two at a time: the input samples of both
// (for the weight gradient) are requested before either op's sums, so the
// two loads' latencies overlap.
template <bool FOLD>
__device__ __forceinline__ void adj_init_stage(uint32_t sbase, const StageRange &range, int lane,
                                               float *__restrict__ out, int64_t nt, int64_t T0,
                                               const float *__restrict__ w, const float *__restrict__ x,
                                               float *__restrict__ part, int64_t part_row) {
  constexpr uint32_t kOp = (uint32_t)sizeof(FusedOp);
  for (uint32_t at = range.first; at != range.end;) {
    const bool two = at + kOp != range.end;
    const FusedOp a = prog_desc<FusedOp>(range.prog, at), b = prog_desc<FusedOp>(range.prog, two ? at + kOp : at);
    at += two ? 2 * kOp : kOp;
    float xa[kLaneCols], xb[kLaneCols];
    if (part != nullptr) {
      adj_init_load_x(xa, a, x, nt, T0, lane);
      if (two) adj_init_load_x(xb, b, x, nt, T0, lane);
    }
    adj_init_op<FOLD>(sbase, a, xa, lane, out, nt, T0, w, part, part_row);
    if (two) adj_init_op<FOLD>(sbase, b, xb, lane, out, nt, T0, w, part, part_row);
  }
}

// Persistent blocks as the forward cone kernel: eight computing warps, one
// that copies (copy_items).  INIT: the last stage is the initialisation
// transpose.
// Bound: latency and HBM alike.  1024 x 65536 x 1024 on a GB300, launches 10
// -> 8 -> 6 -> 4 -> 2 -> 0 with the weight gradient: 112, 110, 116, 126 and
// 264 us with ops read through L2 and warp 0 copying; 98, 97, 101, 104 and
// 248 us with programmes and a copying warp.  The last launch reads a second
// input: 237 us with it asked for ahead, 195 with the init stage's columns
// tested once per piece and its runs straight-line (instruction issue).
template <bool INIT>
__global__ void __launch_bounds__(kFusedLaunchThreads, kFusedMinBlocks)
adjoint_cone_kernel(const __grid_constant__ TmaMaps maps, float *__restrict__ out, int64_t nt, int32_t W,
                    int32_t ntiles, int64_t items, const FusedProg *__restrict__ progs, const int4 *__restrict__ prog,
                    const FusedLoad *__restrict__ loads, const float *__restrict__ w, int32_t box, int32_t cshift,
                    int32_t prog_off, int32_t prog_slot, int *__restrict__ status, const float *__restrict__ x,
                    float *__restrict__ part, int32_t pieces) {
  extern __shared__ __align__(128) unsigned char smem[];
  const int warp = warp_all((int)(threadIdx.x >> 5)), lane = threadIdx.x & 31;
  const uint32_t full = smem_u32(smem);
  init_item_barriers(full);
  if (warp == kFusedWarps) {
    copy_items<float>(smem, maps, nt, W, 0, ntiles, items, progs, prog, loads, box, cshift, prog_off, prog_slot, status,
                      lane, [&](const FusedProg &pr, int64_t T0) {
                        if (INIT && part != nullptr) adj_init_ahead(pr, prog, x, nt, T0, lane);
                      });
    return;
  }
  uint32_t slot = 0, phase = 0;
  for (int64_t item = blockIdx.x; item < items; item += gridDim.x) {
    const bool ok = mbar_wait_bounded(full, phase);
    phase ^= 1u;
    // every computing warp has left the item before, whose regions the
    // first stage overwrites
    if (!compute_sync_and(ok)) {
      atomicExch(status, 1);
      return;
    }
    const int4 h = lds_v4(full + kItemHeader + 16u * slot);
    const int n_stages = warp_all(h.z);
    const int64_t T0 = (int64_t)h.x * W;
    const Prog prg{full + (uint32_t)(prog_off + (int)slot * prog_slot), prog_slot > 0 ? nullptr : prog + h.w};
    float *const pt = INIT && part != nullptr ? part + (int64_t)h.x * pieces : nullptr;
    for (int s = 0; s < n_stages; ++s) {
      if (s > 0) compute_sync();
      const StageRange r = prog_stage(prg, s, warp);
      if (s < n_stages - 1) {
        adj_gather_stage<kOutSmem>(full, r, lane, out, nt, T0);
      } else if (!INIT) {
        adj_gather_stage<kOutGlobal>(full, r, lane, out, nt, T0);
      } else if (r.kind == kAdjInitF) {
        adj_init_stage<true>(full, r, lane, out, nt, T0, w, x, pt, (int64_t)ntiles * pieces);
      } else {
        adj_init_stage<false>(full, r, lane, out, nt, T0, w, x, pt, (int64_t)ntiles * pieces);
      }
      if (s == 0) {
        __syncwarp();
        if (lane == 0) mbar_arrive(full + kFreeBar);  // this warp reads S no more
      }
    }
    slot ^= 1u;
  }
}

// The weight gradient from the init launch's partials: one warp per
// channel sums its (tile, piece) slots in a fixed order.
__global__ void __launch_bounds__(256)
adj_weights_finalize_kernel(const float *__restrict__ part, int32_t nf, int64_t per_channel,
                            float *__restrict__ gw) {
  const int lane = threadIdx.x & 31;
  const int64_t k = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (k >= nf) return;
  const float *p = part + k * per_channel;
  float d = 0.f;
  for (int64_t i = lane; i < per_channel; i += 32) d = __fadd_rn(d, p[i]);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) d = __fadd_rn(d, __shfl_xor_sync(0xffffffffu, d, off));
  if (lane == 0) gw[k] = d;
}

template <bool INIT>
cudaError_t launch_adj_group(const DeviceTables &dt, const AdjGroup &g, const float *base, int64_t base_rows,
                             int64_t base_nt, float *dst, const float *w, int64_t nt, cudaStream_t s,
                             const float *x = nullptr, float *part = nullptr) {
  auto kern = adjoint_cone_kernel<INIT>;
  FusedGroup mg;  // the staged rows: row boxes of g.box samples or row blocks
  mg.box = g.box;
  mg.chunk = g.chunk;
  mg.kchunks = g.kchunks;
  mg.max_p = g.max_p;
  TmaMaps maps;
  int32_t cshift = 0;
  if (!make_group_maps(maps.m, mg, base, map_type<float>(), sizeof(float), (uint64_t)base_rows, (uint64_t)base_nt,
                       &cshift))
    return cudaErrorInvalidValue;
  const int64_t items = (int64_t)g.tpl_count * g.ntiles;
  if (items == 0) return cudaSuccess;
  int resident = 0;
  const cudaError_t e = resident_blocks(reinterpret_cast<const void *>(kern), kFusedLaunchThreads, g.smem_bytes, &resident);
  if (e != cudaSuccess) return e;
  const int64_t blocks = std::min<int64_t>(items, resident);
  dt.prof->begin(s, K_ADJ_CONE, g.lb * 100 + g.lt);
  kern<<<(unsigned)blocks, kFusedLaunchThreads, g.smem_bytes, s>>>(
      maps, dst, nt, g.W, (int32_t)g.ntiles, items, dt.a_progs + g.tpl_begin,
      reinterpret_cast<const int4 *>(dt.a_prog), dt.a_loads, w, g.box, cshift, g.prog_off, g.prog_slot, dt.status, x,
      part, g.pieces);
  dt.prof->end(s);
  return cudaGetLastError();
}

}  // namespace

cudaError_t run_adjoint_fused(const DeviceTables &dt, const float *grad_out, const float *w, float *grad_in,
                              void *const bufs[2], int64_t nt, cudaStream_t s, const float *x, float *part,
                              float *grad_w) {
  if (dt.adj_fused == nullptr) return cudaErrorInvalidValue;
  const AdjFusedPlan &ap = *dt.adj_fused;
  const int G = (int)ap.groups.size();
  for (int g = 0; g < G; ++g) {
    const AdjGroup &gr = ap.groups[g];
    const float *base = g == 0 ? grad_out : static_cast<const float *>(bufs[(g - 1) & 1]);
    float *dst = (g == G - 1) ? grad_in : static_cast<float *>(bufs[g & 1]);
    const int64_t rows = dt.level_rows[gr.lt];
    const int64_t base_nt = g == 0 ? nt : ap.state_nt;
    const cudaError_t e = gr.init ? launch_adj_group<true>(dt, gr, base, rows, base_nt, dst, w, nt, s, x,
                                                           grad_w != nullptr ? part : nullptr)
                                  : launch_adj_group<false>(dt, gr, base, rows, base_nt, dst, nullptr, ap.state_nt, s);
    if (e != cudaSuccess) return e;
  }
  if (grad_w == nullptr) return cudaSuccess;
  const AdjGroup &gl = ap.groups.back();
  dt.prof->begin(s, K_ADJ_WFINAL, 0);
  adj_weights_finalize_kernel<<<(unsigned)((dt.nf + 7) / 8), 256, 0, s>>>(part, dt.nf, gl.ntiles * gl.pieces,
                                                                          grad_w);
  dt.prof->end(s);
  return cudaGetLastError();
}

}  // namespace fdmt
