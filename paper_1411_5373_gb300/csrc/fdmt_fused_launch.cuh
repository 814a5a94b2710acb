// Fused-schedule kernel and its launch (shared by the translation units that
// instantiate it: fdmt_fused_f32.cu for float32, fdmt_fused.cu for fp16
// state, fdmt_fused_u8.cu for uint8).  The schedule: fdmt_fused.h; the planner: fdmt_fused_plan.cpp.
//
// One block computes one cone for one time tile:
//   1. a copying warp issues TMA copies of the cone's base rows (or input
//      channels) and of its stage programme into shared memory; out-of-range
//      columns arrive as zeros, which is the paper's copy rule for t < 0;
//   2. the computing warps wait on the mbarrier (bounded: on timeout the
//      block sets the plan's status word and returns instead of hanging);
//   3. the stages run: a cone that starts at the input walks level 1
//      straight from the staged samples (the Option-1 partial sums of
//      section 4 are running sums in registers); the other levels are
//      computed one (single) or two (pair) at a time, the level between the
//      two of a pair never stored; each warp runs its own list of row
//      pieces, lanes over time (conflict-free: consecutive lanes touch
//      consecutive words);
//   4. the group's top level is written to global memory, coalesced.

#pragma once

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <type_traits>

#include "fdmt_fused.h"
#include "fdmt_fused_dev.cuh"
#include "fdmt_internal.h"
#include "fdmt_residency.h"
#include "fdmt_tma.h"

namespace fdmt {

// Persistent blocks: block b handles items b, b + gridDim.x, ...  Warps 0 ..
// 7 compute; warp 8 copies (copy_items).  The computing warps wait for an
// item's rows (`full`), then for each other (every one of them has left item
// i - 1, whose Pa / Pb the first stage overwrites), run
// the first stage (level 1 walked from the staged input, or the first single
// / pair stage over the staged base rows) and the remaining stages in Pa /
// Pb; the last writes global memory.
// GEN: the plan holds stages with passed-up or one-term halves (Nf not a
// power of two); SCALE: channel weights multiply the input.  Each launch
// takes the variant it needs, so a kernel carries only its own stage code.
// MOVES: walks that move their upper sums as well (the code alone, not run,
// cost the first launch of other plans up to a tenth: 2078 x 5536 x 2697
// uint8, [0,4] 45 -> 49 us).
// The register budget is set for two resident blocks per SM (a run keeps
// four sources and two half sums of eight columns in registers).
// Bound: the computing warps' instruction issue and latency (without copies
// the launches below take 0.8 .. 0.9 of their time), then HBM.  Measured on
// a GB300, 1024 x 65536 x 1024 float32, launches [0,3] [3,7] [7,10] with a
// 112 KiB block: 166, 137 and 121 us with ops read one by one through L2, a
// pair's upper half moved by shuffles and warp 0 copying; 168, 136 and 109
// us with the ops as runs; 139, 137 and 109 us with the walks' code
// straightened as well; 105, 113 and 92 us with the programmes in shared
// memory and a copying warp.
template <class TI, class TB, class TO, class A, bool FROM_INPUT, bool R16, bool SEARCH, bool GEN, bool SCALE, bool MOVES>
__global__ void __launch_bounds__(kFusedLaunchThreads, kFusedMinBlocks)
fused_kernel(const __grid_constant__ TmaMaps maps, TO *__restrict__ out, int64_t nt, int64_t pitch, int64_t first,
             int32_t W, int32_t tile0, int32_t ntiles, int64_t items, const FusedProg *__restrict__ progs,
             const int4 *__restrict__ prog, const FusedLoad *__restrict__ loads, const FusedOp *__restrict__ ops,
             const float *__restrict__ w, int32_t box, int32_t cshift, int32_t prog_off, int32_t prog_slot,
             int *__restrict__ status, const SearchArgs sa) {
  using TS = typename std::conditional<FROM_INPUT, TI, TB>::type;  // staged element type
  extern __shared__ __align__(128) unsigned char smem[];
  const int warp = warp_all((int)(threadIdx.x >> 5)), lane = threadIdx.x & 31;
  const uint32_t full = smem_u32(smem), free_bar = full + kFreeBar, header = full + kItemHeader;
  init_item_barriers(full);
  if (warp == kFusedWarps) {
    copy_items<TS>(smem, maps, nt, W, tile0, ntiles, items, progs, prog, loads, box, cshift, prog_off, prog_slot, status,
                   lane, [](const FusedProg &, int64_t) {});
    return;
  }
  uint32_t slot = 0, phase = 0;
  for (int64_t item = blockIdx.x; item < items; item += gridDim.x) {
    const bool ok = mbar_wait_bounded(full, phase);
    phase ^= 1u;
    if (!compute_sync_and(ok)) {
      // The copies did not complete in time: report it; the copying warp
      // gives them one more bounded wait.
      atomicExch(status, 1);
      return;
    }
    const int4 h = lds_v4(header + 16u * slot);
    const int lim = h.y, n_stages = warp_all(h.z);
    const int64_t tile = h.x, T0 = tile * W;
    const Prog prg{full + (uint32_t)(prog_off + (int)slot * prog_slot), prog_slot > 0 ? nullptr : prog + h.w};
    const int lo = first > T0 ? (int)(first - T0) : 0;
    item_first_stage<TI, TB, A, TO, R16, FROM_INPUT, SEARCH, GEN, SCALE, MOVES>(full, prg, n_stages, w, warp, lane, out,
                                                                         pitch, T0, lo, lim);
    __syncwarp();
    if (lane == 0) mbar_arrive(free_bar);  // this warp reads S no more
    item_later_stages<A, TO, R16, SEARCH, GEN>(full, prg, n_stages, ops, warp, lane, out, pitch, T0, lo, lim, tile, sa);
    slot ^= 1u;
  }
}

namespace {

template <class TI, class TB, class TO, class A, bool FI, bool R16, bool SEARCH, bool GEN, bool SCALE, bool MOVES = false>
cudaError_t launch_variant(const DeviceTables &dt, const FusedGroup &g, const void *base, int64_t base_rows,
                           void *dst, const float *w, int64_t nt, cudaStream_t s, const SearchArgs *sa,
                           int64_t tile0, const OutView *view) {
  auto kern = fused_kernel<TI, TB, TO, A, FI, R16, SEARCH, GEN, SCALE, MOVES>;
  using TS = typename std::conditional<FI, TI, TB>::type;
  TmaMaps maps;
  int32_t cshift = 0;
  // Rows of the levels between launches are state_nt apart.
  const int64_t state_nt = dt.fused->state_nt, base_nt = FI ? nt : state_nt;
  if (!make_group_maps(maps.m, g, base, map_type<TS>(), sizeof(TS), (uint64_t)base_rows, (uint64_t)base_nt, &cshift))
    return cudaErrorInvalidValue;
  const int32_t box = g.box;
  const int64_t ntiles = g.ntiles - tile0, items = (int64_t)g.tpl_count * ntiles;
  const OutView v = view != nullptr ? *view : OutView{0, g.lt == dt.levels ? nt : state_nt};
  int resident = 0;
  const cudaError_t e = resident_blocks(reinterpret_cast<const void *>(kern), kFusedLaunchThreads, g.smem_bytes, &resident);
  if (e != cudaSuccess) return e;
  const int64_t blocks = std::min<int64_t>(items, resident);
  dt.prof->begin(s, FI ? K_FUSED_LOCAL : K_FUSED_CONE, g.lb * 100 + g.lt);
  kern<<<(unsigned)blocks, kFusedLaunchThreads, g.smem_bytes, s>>>(
      maps, static_cast<TO *>(dst) - v.first, nt, v.pitch, v.first, g.W, (int32_t)tile0, (int32_t)ntiles, items,
      dt.f_progs + g.tpl_begin, reinterpret_cast<const int4 *>(dt.f_prog), dt.f_loads, dt.f_ops, w, box, cshift,
      g.prog_off, g.prog_slot, dt.status, sa ? *sa : SearchArgs{});
  dt.prof->end(s);
  return cudaGetLastError();
}

// The launch of one group, with the kernel variant the plan and the
// arguments need: with or without pass-through stage code (GEN), moving walks
// (from the input) and weights (only for float input from the input).
template <class TI, class TB, class TO, class A, bool FI, bool R16, bool SEARCH = false>
cudaError_t launch_group(const DeviceTables &dt, const FusedGroup &g, const void *base, int64_t base_rows,
                         void *dst, const float *w, int64_t nt, cudaStream_t s, const SearchArgs *sa, int64_t tile0,
                         const OutView *view) {
  const bool gen = dt.fused->general;
  if constexpr (FI) {
    if (g.moves) {  // (few channels, many delays: one variant for all of them)
      if constexpr (std::is_floating_point<A>::value) {
        if (w != nullptr)
          return launch_variant<TI, TB, TO, A, FI, R16, SEARCH, true, true, true>(dt, g, base, base_rows, dst, w, nt, s,
                                                                                  sa, tile0, view);
      }
      return launch_variant<TI, TB, TO, A, FI, R16, SEARCH, true, false, true>(dt, g, base, base_rows, dst, w, nt, s,
                                                                               sa, tile0, view);
    }
  }
  if constexpr (FI && std::is_floating_point<A>::value) {
    if (w != nullptr)
      return gen ? launch_variant<TI, TB, TO, A, FI, R16, SEARCH, true, true>(dt, g, base, base_rows, dst, w, nt, s, sa,
                                                                              tile0, view)
                 : launch_variant<TI, TB, TO, A, FI, R16, SEARCH, false, true>(dt, g, base, base_rows, dst, w, nt, s,
                                                                               sa, tile0, view);
  }
  return gen ? launch_variant<TI, TB, TO, A, FI, R16, SEARCH, true, false>(dt, g, base, base_rows, dst, w, nt, s, sa,
                                                                           tile0, view)
             : launch_variant<TI, TB, TO, A, FI, R16, SEARCH, false, false>(dt, g, base, base_rows, dst, w, nt, s, sa,
                                                                            tile0, view);
}

// The launches of a float plan (A the sums' type, R16: fp16-state rounding).
template <class TI, class TB, class TO, class A, bool R16>
cudaError_t run_fused_typed(const DeviceTables &dt, const void *in, const float *w, void *out,
                            void *const bufs[2], int64_t nt, cudaStream_t s, const SearchArgs *sa,
                            const OutView *view) {
  const FusedPlan &fp = *dt.fused;
  const int G = (int)fp.groups.size();
  FirstTiles ft;
  first_tiles(fp, view != nullptr ? view->first : 0, ft);
  for (int g = 0; g < G; ++g) {
    const FusedGroup &gr = fp.groups[g];
    const bool last = (g == G - 1);
    void *dst = last ? out : bufs[g & 1];
    cudaError_t e;
    if (last && gr.search_k > 0) {
      // The last launch ends with the boxcar search (a search needs at
      // least two merge levels, so a launch from the input walks level 1
      // into Pa before its top level goes to Pt).
      if (sa == nullptr) return cudaErrorInvalidValue;
      e = gr.from_input ? launch_group<TI, TB, TO, A, true, R16, true>(dt, gr, in, dt.nf, dst, w, nt, s, sa, ft.tile[g], view)
                        : launch_group<TI, TB, TO, A, false, R16, true>(dt, gr, bufs[(g - 1) & 1],
                                                                        dt.level_rows[gr.lb], dst, w, nt, s, sa, ft.tile[g], view);
    } else if (gr.from_input) {
      e = last ? launch_group<TI, TB, TO, A, true, R16>(dt, gr, in, dt.nf, dst, w, nt, s, nullptr, ft.tile[g], view)
               : launch_group<TI, TB, TB, A, true, R16>(dt, gr, in, dt.nf, dst, w, nt, s, nullptr, ft.tile[g], nullptr);
    } else {
      const void *base = bufs[(g - 1) & 1];
      const int64_t rows = dt.level_rows[gr.lb];
      e = last ? launch_group<TI, TB, TO, A, false, R16>(dt, gr, base, rows, dst, w, nt, s, nullptr, ft.tile[g], view)
               : launch_group<TI, TB, TB, A, false, R16>(dt, gr, base, rows, dst, w, nt, s, nullptr, ft.tile[g], nullptr);
    }
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace

// uint8 input (fdmt_fused_u8.cu).
cudaError_t run_fused_u8(const DeviceTables &dt, const void *in, void *out, void *const bufs[2], int64_t nt,
                         cudaStream_t s, const SearchArgs *sa, const OutView *view);
// float32 input and state (fdmt_fused_f32.cu).
cudaError_t run_fused_f32(const DeviceTables &dt, const void *in, const float *w, void *out, void *const bufs[2],
                          int64_t nt, cudaStream_t s, const SearchArgs *sa, const OutView *view);

}  // namespace fdmt
