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
#include <mutex>
#include <type_traits>

#include "fdmt_fused.h"
#include "fdmt_fused_dev.cuh"
#include "fdmt_internal.h"
#include "fdmt_tma.h"

namespace fdmt {

// Persistent blocks: block b handles items b, b + gridDim.x, ...  Warps 0 ..
// 7 compute; warp 8 copies.  The
// copying warp stages item i + 1 (its rows into S, its programme into one of
// two slots, its place into one of two headers) as soon as the computing
// warps have arrived at the `free` barrier, behind their first stage of item
// i, the only one that reads S; its own bookkeeping is off their path.  The
// computing warps wait for the rows (`full`), then for each other (every one
// of them has left item i - 1, whose Pa / Pb the first stage overwrites), run
// the first stage (level 1 walked from the staged input, or the first single
// / pair stage over the staged base rows) and the remaining stages in Pa /
// Pb; the last writes global memory.
// GEN: the plan holds stages with passed-up or one-term halves (Nf not a
// power of two); SCALE: channel weights multiply the input.  Each launch
// takes the variant it needs, so a kernel carries only its own stage code.
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
constexpr int kFusedLaunchThreads = kFusedThreads + 32;
constexpr int32_t kTileChunk = 304;  // time tiles of one chunk of items

template <class TI, class TB, class TO, class A, bool FROM_INPUT, bool R16, bool SEARCH, bool GEN, bool SCALE>
__global__ void __launch_bounds__(kFusedLaunchThreads, kFusedMinBlocks)
fused_kernel(const __grid_constant__ TmaMaps maps, TO *__restrict__ out, int64_t nt, int64_t pitch, int64_t first,
             int32_t W, int32_t tile0, int32_t ntiles, int64_t items, const FusedProg *__restrict__ progs,
             const int4 *__restrict__ prog, const FusedLoad *__restrict__ loads, const FusedOp *__restrict__ ops,
             const float *__restrict__ w, int32_t box, int32_t cshift, int32_t prog_off, int32_t prog_slot,
             int *__restrict__ status, const SearchArgs sa) {
  using TS = typename std::conditional<FROM_INPUT, TI, TB>::type;  // staged element type
  extern __shared__ __align__(128) unsigned char smem[];
  const int warp = warp_all((int)(threadIdx.x >> 5)), lane = threadIdx.x & 31;
  // The barrier slot: the `full` and `free` mbarriers, then two item headers
  // (first column, columns, stages, tile).
  const uint32_t full = smem_u32(smem), free_bar = full + 8u, header = full + 32u;
  if (threadIdx.x == 0) {
    mbar_init(full, 1);
    mbar_init(free_bar, kFusedWarps);
    fence_mbar_init();
  }
  __syncthreads();
  if (warp == kFusedWarps) {
    // Items go tile chunk by tile chunk, template by template within a
    // chunk, tile by tile within a template: neighbouring templates share
    // staged rows, and a chunk keeps their second reading within reach of L2
    // whatever the row length.  Row blocks are also asked for one item ahead:
    // L2 hides the HBM latency that a block's single staging region cannot.
    // 1024 x 65536 x 1024 float32 306 us without, 289 us with; 4096 x 2^18 x
    // 4096, HBM-bound in its cones, 5.67 ms without, 5.70 with, 6.36 with the
    // requests but template by template.  (Row boxes are bound by the rate
    // of copies: asking twice made them 5 % slower.)
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
    bool first = true;
    for (; item < items; item += gridDim.x) {
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
      first = false;
      const int64_t T0 = (int64_t)(tile0 + tile) * W;
      if (lane == 0) {
        const int lim = (int)((nt - T0) < (int64_t)W ? (nt - T0) : (int64_t)W);
        sts_v4(header + 16u * slot, make_int4(tile0 + tile, lim, pr.n_stages, 0));
      }
      stage_item<TS>(smem, full, maps.m, pr, loads, ld, T0, box, cshift, lane);
      if (lane == 0) stage_prog(full + (uint32_t)(prog_off + (int)slot * prog_slot), pr, prog, full);
      slot ^= 1u;
      if (item + gridDim.x < items) {
        place(item + gridDim.x);
        pr = progs[tpl];
        ld = fetch_load(pr, loads, lane);
        if (cshift > 0) prefetch_item<TS>(maps.m, pr, loads, ld, (int64_t)(tile0 + tile) * W, box, cshift, lane);
      }
    }
    // The last copies land before the block ends: the computing warps wait
    // for them (or give up, which the bounded wait covers).
    mbar_wait_bounded(full, phase);
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
    const uint32_t prg = full + (uint32_t)(prog_off + (int)slot * prog_slot);
    const int lo = first > T0 ? (int)(first - T0) : 0;
    item_first_stage<TI, TB, A, TO, R16, FROM_INPUT, SEARCH, GEN, SCALE>(full, prg, n_stages, w, warp, lane, out,
                                                                         pitch, T0, lo, lim);
    __syncwarp();
    if (lane == 0) mbar_arrive(free_bar);  // this warp reads S no more
    item_later_stages<A, TO, R16, SEARCH, GEN>(full, prg, n_stages, ops, warp, lane, out, pitch, T0, lo, lim, tile, sa);
    slot ^= 1u;
  }
}

namespace {

template <class TI, class TB, class TO, class A, bool FI, bool R16, bool SEARCH, bool GEN, bool SCALE>
cudaError_t launch_variant(const DeviceTables &dt, const FusedGroup &g, const void *base, int64_t base_rows,
                           void *dst, const float *w, int64_t nt, cudaStream_t s, const SearchArgs *sa,
                           int64_t tile0, const OutView *view) {
  auto kern = fused_kernel<TI, TB, TO, A, FI, R16, SEARCH, GEN, SCALE>;
  static std::once_flag attr_once;
  static cudaError_t attr_err = cudaSuccess;
  std::call_once(attr_once, [&] {
    attr_err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  });
  if (attr_err != cudaSuccess) return attr_err;
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
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kFusedLaunchThreads, g.smem_bytes);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  int dev = 0, sms = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  const int64_t blocks = std::min<int64_t>(items, (int64_t)per_sm * sms);
  dt.prof->begin(s, FI ? K_FUSED_LOCAL : K_FUSED_CONE, g.lb * 100 + g.lt);
  kern<<<(unsigned)blocks, kFusedLaunchThreads, g.smem_bytes, s>>>(
      maps, static_cast<TO *>(dst) - v.first, nt, v.pitch, v.first, g.W, (int32_t)tile0, (int32_t)ntiles, items,
      dt.f_progs + g.tpl_begin, reinterpret_cast<const int4 *>(dt.f_prog), dt.f_loads, dt.f_ops, w, box, cshift,
      g.prog_off, g.prog_slot, dt.status, sa ? *sa : SearchArgs{});
  dt.prof->end(s);
  return cudaGetLastError();
}

// The launch of one group, with the kernel variant the plan and the
// arguments need: with or without pass-through stage code (GEN) and weights
// (only for float input from the input).
template <class TI, class TB, class TO, class A, bool FI, bool R16, bool SEARCH = false>
cudaError_t launch_group(const DeviceTables &dt, const FusedGroup &g, const void *base, int64_t base_rows,
                         void *dst, const float *w, int64_t nt, cudaStream_t s, const SearchArgs *sa, int64_t tile0,
                         const OutView *view) {
  const bool gen = dt.fused->general;
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
