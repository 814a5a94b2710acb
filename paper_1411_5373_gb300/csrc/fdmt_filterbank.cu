// STFT filterbank in front of the transform (contracts in include/fdmt.h).
//
// Section 2 of Zackay & Ofek (arXiv:1411.5373): the voltage series is cut
// into blocks of Nf samples, each block is Fourier transformed (STFT) and
// the squared magnitude at each frequency is kept, optionally binned in
// time (the footnote): I[c][t] = sum_{b < nbin} |X_{t nbin + b}[k(c)]|^2,
// with channel c in ascending frequency holding DFT bin k = (c + Nf/2) mod Nf
// of the complex (baseband) voltages.
//
// A block of 256 threads (512 and 1024 for the largest Nf, where there are
// transforms enough) transforms 16 samples per thread at a time, in registers,
// with Stockham passes of radix 16: the first pass reads the voltages from
// global memory, a pass reads all its values before any is stored, so one
// shared buffer serves every exchange, and the last pass stores squared
// magnitudes.  Blocks are persistent: the twiddle table is made once per block.
// Bound: the shared-memory pipe, then HBM.  64 M voltages into 1024 x 65536 on a
// GB300: 334 us with two exchange buffers (two blocks per SM), twiddles made
// anew for every 4096 samples and the two parts of a complex sum added one
// by one; 217 us now.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "../../include/fdmt.h"
#include "fdmt_residency.h"
#include "fdmt_stockham.cuh"
#include "fdmt_tma.h"

namespace fdmt {
namespace {

constexpr int kFbValues = 16;  // complex samples per thread
constexpr int kFbThreads = 256;
// Threads of a block (TH below) for 2^LN channels: larger blocks transform
// more times at once, so that a tile's rows stay 16 bytes or wider.
__host__ __device__ constexpr int fb_threads(int ln) { return ln <= 9 ? kFbThreads : (ln == 10 ? 512 : 1024); }
__host__ __device__ constexpr int fb_samples(int th) { return kFbValues * th; }

// Shared-memory index of squared magnitude i: the times of a channel, a
// multiple of Nf apart, land 32 / T banks apart when they are read back.
__device__ __forceinline__ constexpr int pad_power(int i) { return i + (i >> 7); }

// The values of pass (NS, R) in registers: work item w = threadIdx.x + it
// threads holds elements base + r NF / R of its transform.
template <int LN, int TH, int R>
struct FbItem {
  static constexpr int NF = 1 << LN, LR = fft::ilog2(R), LPER = LN - LR, PER = 1 << LPER;
  int f, j;
  __device__ __forceinline__ explicit FbItem(int it) {
    const int w = (int)threadIdx.x + it * TH;
    f = w >> LPER;
    j = w & (PER - 1);
  }
};

// pad16(i + r STEP) and pad_power(i + r STEP) for i = i0 + r STEP with i0
// padded already: linear in r where the padding is (a step of whole runs, or
// single steps from the start of a run), so that a pass's addresses are
// constant offsets from one base.
template <int STEP, bool RUN>
__device__ __forceinline__ int step16(int i0, int p0, int r) {
  if constexpr (STEP % 16 == 0) return p0 + r * (STEP + STEP / 16);
  if constexpr (RUN) return p0 + r * STEP;
  return fft::pad16(i0 + r * STEP);
}
template <int STEP>
__device__ __forceinline__ int step_power(int i0, int p0, int r) {
  if constexpr (STEP % 128 == 0) return p0 + r * (STEP + STEP / 128);
  return pad_power(i0 + r * STEP);
}

// One pass over F transforms: `v` holds its values; the outputs go to `buf`
// (element order), or, in the last pass (NS R = NF), their squared
// magnitudes to `power`.
// TILE: `power` is the [channel][time] tile of samples / NF times that a tensor
// copy writes out, which may still be reading the last one when the first
// pass stores.
template <int LN, int TH, int NS, int R, bool TILE>
__device__ __forceinline__ void fb_finish(float2 (&v)[kFbValues / R][R], float2 *buf, float *power,
                                          const float2 *__restrict__ tw, int F) {
  constexpr int NF = 1 << LN, LR = fft::ilog2(R), LNS = fft::ilog2(NS);
#pragma unroll
  for (int it = 0; it < kFbValues / R; ++it) {
    const FbItem<LN, TH, R> w(it);
    const int k = w.j & (NS - 1);
    if constexpr (NS > 1) {
      // exp(-2 pi i r k / (NS R)) = tw[r k NF / (NS R)]
      constexpr int SH = LN - LNS - LR;
      const int step = k << SH;
#pragma unroll
      for (int r = 1; r < R; ++r)
        v[it][r] = fft::cmul(v[it][r], tw[SH >= 2 ? r * fft::pad4(step) : fft::pad4(r * step)]);
    }
    fft::dft_regs<R>(v[it]);
  }
  if constexpr (TILE && NS == 1) {
    if (threadIdx.x == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
    __syncthreads();
  }
  if constexpr (NS > 1) __syncthreads();  // every value of the pass has been read
#pragma unroll
  for (int it = 0; it < kFbValues / R; ++it) {
    const FbItem<LN, TH, R> w(it);
    if (w.f >= F) continue;
    const int out0 = w.f * NF + (w.j >> LNS) * NS * R + (w.j & (NS - 1));
    const int at = NS * R == NF ? pad_power(out0) : fft::pad16(out0);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float2 z = v[it][fft::bitrev_small(r, LR)];
      if constexpr (NS * R == NF && TILE) {
        constexpr int kT = fb_samples(TH) / NF;
        const int k = out0 - w.f * NF + r * NS;
        power[((k + NF / 2) & (NF - 1)) * kT + w.f] = __fadd_rn(__fmul_rn(z.x, z.x), __fmul_rn(z.y, z.y));
      } else if constexpr (NS * R == NF)
        power[step_power<NS>(out0, at, r)] = __fadd_rn(__fmul_rn(z.x, z.x), __fmul_rn(z.y, z.y));
      else  // (the first pass stores whole runs of 16)
        buf[step16<NS, NS == 1 && R == 16>(out0, at, r)] = z;
    }
  }
  if constexpr (TILE && NS * R == NF) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
}

// The passes after transforms of size NS.
template <int LN, int TH, int NS, bool TILE>
__device__ __forceinline__ void fb_rest(float2 *buf, float *power, const float2 *__restrict__ tw, int F) {
  constexpr int NF = 1 << LN;
  if constexpr (NS < NF) {
    constexpr int R = NF / NS >= 16 ? 16 : NF / NS, PER = NF / R;
    float2 v[kFbValues / R][R];
#pragma unroll
    for (int it = 0; it < kFbValues / R; ++it) {
      const FbItem<LN, TH, R> w(it);
      const int i0 = w.f * NF + w.j, at = fft::pad16(i0);
#pragma unroll
      for (int r = 0; r < R; ++r) v[it][r] = buf[step16<PER, false>(i0, at, r)];
    }
    fb_finish<LN, TH, NS, R, TILE>(v, buf, power, tw, F);
    fb_rest<LN, TH, NS * R, TILE>(buf, power, tw, F);
  }
}

// Squared magnitudes of F <= samples / NF transforms of the voltages at x, in
// `power` (element f NF + k at pad_power); a barrier at the end.
template <int LN, int TH, bool TILE>
__device__ __forceinline__ void fb_transform(const float2 *__restrict__ x, float2 *buf, float *power,
                                             const float2 *__restrict__ tw, int F) {
  constexpr int NF = 1 << LN, R = NF >= 16 ? 16 : NF;
  float2 v[kFbValues / R][R];
#pragma unroll
  for (int it = 0; it < kFbValues / R; ++it) {
    const FbItem<LN, TH, R> w(it);
    const float2 *from = x + (w.f < F ? w.f * NF + w.j : 0);  // (a work item past the last transform stores nothing)
#pragma unroll
    for (int r = 0; r < R; ++r) v[it][r] = __ldg(from + r * FbItem<LN, TH, R>::PER);
  }
  fb_finish<LN, TH, 1, R, TILE>(v, buf, power, tw, F);
  fb_rest<LN, TH, R, TILE>(buf, power, tw, F);
}

template <int LN, int TH>
__global__ void __launch_bounds__(TH, 1024 / TH)
filterbank_kernel(const float2 *__restrict__ v, int nbin, int64_t nt, int T, float *__restrict__ out) {
  constexpr int NF = 1 << LN;
  extern __shared__ __align__(16) float2 sm[];
  float2 *buf = sm;                                // samples, padded
  float *power = reinterpret_cast<float *>(sm);    // the same memory, after the last pass
  float2 *tw = sm + fft::pad16(fb_samples(TH));        // [nf], padded by pad4
  fft::twiddles<TH, LN>(tw);
  __syncthreads();
  const int lT = 31 - __clz(T);
  constexpr int kRound = fb_samples(TH) / NF, kThreads = TH;  // transforms at once
  for (int64_t t_first = (int64_t)blockIdx.x * T; t_first < nt; t_first += (int64_t)gridDim.x * T) {
    const float2 *x = v + t_first * nbin * (int64_t)NF;
    if (T * nbin <= kRound) {
      const int T_here = (int)((nt - t_first) < (int64_t)T ? (nt - t_first) : (int64_t)T);
      fb_transform<LN, TH, false>(x, buf, power, tw, T_here * nbin);
      // Consecutive threads take consecutive times of one channel row (T is
      // a power of two; the last tile may hold fewer times): thread i time i
      // mod T of channels i / T, i / T + threads / T, ...  (T can exceed the
      // block only for Nf < 16.)
      for (int tt = threadIdx.x & (T - 1); tt < T_here; tt += kThreads) {
        const int dc = T < kThreads ? kThreads >> lT : 1;
        float *o = out + (int64_t)((int)threadIdx.x >> lT) * nt + t_first + tt;
        for (int c = (int)threadIdx.x >> lT; c < NF; c += dc, o += (int64_t)dc * nt) {
          const int k = (c + NF / 2) & (NF - 1);
          float acc = 0.0f;
          for (int b = 0; b < nbin; ++b) acc = __fadd_rn(acc, power[pad_power((tt * nbin + b) * NF + k)]);
          *o = acc;
        }
      }
      __syncthreads();  // before the next tile's first pass stores
    } else {
      // One time (T = 1) whose bin takes more than one round: every thread
      // keeps the sums of its channels.
      constexpr int kOwn = (NF + kThreads - 1) / kThreads;
      float acc[kOwn];
#pragma unroll
      for (int q = 0; q < kOwn; ++q) acc[q] = 0.0f;
      for (int b0 = 0; b0 < nbin; b0 += kRound) {
        const int F = min(kRound, nbin - b0);
        fb_transform<LN, TH, false>(x + (int64_t)b0 * NF, buf, power, tw, F);
#pragma unroll
        for (int q = 0; q < kOwn; ++q) {
          const int c = (int)threadIdx.x + q * kThreads, k = (c + NF / 2) & (NF - 1);
          if (c < NF)
            for (int b = 0; b < F; ++b) acc[q] = __fadd_rn(acc[q], power[pad_power(b * NF + k)]);
        }
        __syncthreads();
      }
#pragma unroll
      for (int q = 0; q < kOwn; ++q) {
        const int c = (int)threadIdx.x + q * kThreads;
        if (c < NF) out[(int64_t)c * nt + t_first] = acc[q];
      }
    }
  }
}

// The same without binning where the output takes tensor copies (16-byte
// aligned, nt a multiple of 4): the last pass stores its powers as an
// [Nf][T] tile, which one thread writes out by copies of [256][T], off the
// other threads' path and behind the next tile's first pass.  Taken for T
// <= 16 times per tile, where the threads write only a part of a row's 128
// bytes at a time, and for Nf = 16; between them whole segments cost less
// than the tile's bank conflicts.  64 M voltages, tile against threads, us:
// Nf = 16 251 / 292, 32 272 / 229, 64 242 / 193, 256 169 / 176, 512 192 / 205,
// 1024 217 / 226, 2048 295 / 307, 4096 360 / 415 (before: 391, 315, 255, 385,
// 321, 335, 447, 690).
template <int LN, int TH>
__global__ void __launch_bounds__(TH, 1024 / TH)
filterbank_tile_kernel(const __grid_constant__ CUtensorMap map, const float2 *__restrict__ v, int64_t nt) {
  constexpr int NF = 1 << LN, T = fb_samples(TH) / NF, kRows = NF < 256 ? NF : 256;
  extern __shared__ __align__(128) float2 sm[];
  float2 *buf = sm;
  float *power = reinterpret_cast<float *>(sm);
  float2 *tw = sm + fft::pad16(fb_samples(TH));
  fft::twiddles<TH, LN>(tw);
  __syncthreads();
  for (int64_t t_first = (int64_t)blockIdx.x * T; t_first < nt; t_first += (int64_t)gridDim.x * T) {
    const int F = (int)((nt - t_first) < (int64_t)T ? (nt - t_first) : (int64_t)T);
    // (ends with a barrier; columns past nt of the last tile are clipped)
    fb_transform<LN, TH, true>(v + t_first * (int64_t)NF, buf, power, tw, F);
    if (threadIdx.x == 0) {
      const uint32_t src = static_cast<uint32_t>(__cvta_generic_to_shared(power));
      for (int c = 0; c < NF; c += kRows)
        asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];" ::"l"(
                         reinterpret_cast<uint64_t>(&map)),
                     "r"((int)t_first), "r"(c), "r"(src + (uint32_t)(c * T * 4))
                     : "memory");
      asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    }
  }
  if (threadIdx.x == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

constexpr size_t fb_smem(int ln, int th) {
  return ((size_t)fft::pad16(fb_samples(th)) + (size_t)fft::pad4(1 << ln)) * sizeof(float2);
}

template <int LN, int TH>
cudaError_t launch_filterbank(const float2 *v, int nbin, int64_t nt, int T, float *out, cudaStream_t s) {
  constexpr size_t smem = fb_smem(LN, TH);
  cudaError_t e;
  int resident = 0;
  constexpr int kTile = fb_samples(TH) >> LN;
  if constexpr (LN >= 4 && kTile >= 4 && (kTile <= 16 || kTile >= 256)) {
    constexpr int kT = kTile, kRows = LN < 8 ? 1 << LN : 256;
    if (nbin == 1 && T == kT && nt % 4 == 0 && nt < ((int64_t)1 << 31) - kT &&
        (reinterpret_cast<uintptr_t>(out) & 15u) == 0) {
      auto kern = filterbank_tile_kernel<LN, TH>;
      if ((e = resident_blocks(reinterpret_cast<const void *>(kern), TH, smem, &resident)) != cudaSuccess)
        return e;
      CUtensorMap map;
      if (!make_store_map(&map, out, 1u << LN, (uint64_t)nt, kT, kRows)) return cudaErrorInvalidValue;
      const int64_t tiles = std::min<int64_t>((nt + kT - 1) / kT, resident);
      kern<<<(unsigned)tiles, TH, smem, s>>>(map, v, nt);
      return cudaGetLastError();
    }
  }
  auto kern = filterbank_kernel<LN, TH>;
  if ((e = resident_blocks(reinterpret_cast<const void *>(kern), TH, smem, &resident)) != cudaSuccess)
    return e;
  const int64_t blocks = std::min<int64_t>((nt + T - 1) / T, resident);
  kern<<<(unsigned)blocks, TH, smem, s>>>(v, nbin, nt, T, out);
  return cudaGetLastError();
}

// Output times per block of `th` threads: a power of two, as many transforms as
// a block takes at once (at least one time's bin).
int times(int nf, int nbin, int th) {
  int n = std::max(1, fb_samples(th) / (nf * nbin));
  while (n & (n - 1)) n &= n - 1;
  return n;
}

// The larger blocks of Nf = 1024 and more leave SMs idle where a call has few
// blocks, and a bin that is no power of two leaves part of them idle.  On a
// GB300, blocks of 256 / 512 / 1024 threads, us (before the larger blocks):
//   2048 channels: 100 times 7.9 / 8.6 / 14.7 (8.5), 608 10.9 / 9.0 / 13.7
//   (12.6), 2432 29.5 / 21.0 / 23.1 (35.4), 32768 402 / 306 / 293 (450); in bins
//   of three, 400 18.9 / 17.0 / 21.0 (19.0); in bins of five, 400 25.0 / 26.2 /
//   29.1 (23.1), 2432 126 / 140 / 147 (144);
//   4096 channels: 100 10.4 / 12.6 / 16.7 (10.4), 304 14.9 / 12.6 / 16.7 (15.2),
//   400 20.7 / 19.0 / 16.7 (22.9), 2432 98.8 / 74.1 / 55.7 (109).
// So 256 threads up to one such block per SM (and for bins that a block of 512
// does not hold), 512 up to four for 2048 channels and one for 4096.
template <int LN>
cudaError_t run_filterbank(const float2 *v, int nbin, int64_t nt, float *out, cudaStream_t s) {
  constexpr int kTH = fb_threads(LN), NF = 1 << LN;
  if constexpr (kTH > kFbThreads) {
    int resident = 0;  // 1024 / kTH blocks per SM
    const cudaError_t e = resident_blocks(reinterpret_cast<const void *>(filterbank_kernel<LN, kTH>), kTH,
                                          fb_smem(LN, kTH), &resident);
    if (e != cudaSuccess) return e;
    const int64_t sms = resident * kTH / 1024;
    auto holds = [&](int th) { return nbin * NF <= fb_samples(th); };
    auto blocks = [&](int th) { return (nt + times(NF, nbin, th) - 1) / times(NF, nbin, th); };
    if ((holds(256) && blocks(256) <= sms) || (LN == 11 && !holds(512)))
      return launch_filterbank<LN, 256>(v, nbin, nt, times(NF, nbin, 256), out, s);
    if constexpr (kTH > 512)
      if (holds(512) && blocks(512) <= (LN == 11 ? 4 : 1) * sms)
        return launch_filterbank<LN, 512>(v, nbin, nt, times(NF, nbin, 512), out, s);
  }
  return launch_filterbank<LN, kTH>(v, nbin, nt, times(NF, nbin, kTH), out, s);
}

}  // namespace
}  // namespace fdmt

extern "C" int fdmt_filterbank(const void *volts, int64_t n, int32_t nf, int32_t nbin, float *out, int64_t nt,
                               void *stream) {
  if (volts == nullptr || out == nullptr || (reinterpret_cast<uintptr_t>(volts) & 15u) ||
      (reinterpret_cast<uintptr_t>(out) & 3u))
    return FDMT_ERR_INVALID_ARG;
  if (nf < 2 || nf > 4096 || (nf & (nf - 1)) != 0 || nbin < 1 || nbin > 1024) return FDMT_ERR_INVALID_ARG;
  if (nt < 1 || n < 0 || nt > n / ((int64_t)nf * nbin)) return FDMT_ERR_INVALID_ARG;
  int log2nf = 0;
  while ((1 << log2nf) < nf) ++log2nf;
  // (one time's bin: at most as many samples as two padded buffers and the
  // twiddles held in 200 KiB)
  const int ref = fdmt::times(nf, nbin, fdmt::kFbThreads);
  const size_t padded = (size_t)ref * nbin * nf + ((size_t)ref * nbin * nf >> 4);
  if ((2 * padded + (size_t)nf + (size_t)nf / 4) * sizeof(float2) > 200 * 1024) return FDMT_ERR_UNSUPPORTED;
  const int T = fdmt::times(nf, nbin, fdmt::fb_threads(log2nf));
  if ((nt + T - 1) / T > INT32_MAX) return FDMT_ERR_UNSUPPORTED;
  const float2 *vv = static_cast<const float2 *>(volts);
  cudaStream_t cs = static_cast<cudaStream_t>(stream);
  cudaError_t e;
  switch (log2nf) {
    case 1: e = fdmt::run_filterbank<1>(vv, nbin, nt, out, cs); break;
    case 2: e = fdmt::run_filterbank<2>(vv, nbin, nt, out, cs); break;
    case 3: e = fdmt::run_filterbank<3>(vv, nbin, nt, out, cs); break;
    case 4: e = fdmt::run_filterbank<4>(vv, nbin, nt, out, cs); break;
    case 5: e = fdmt::run_filterbank<5>(vv, nbin, nt, out, cs); break;
    case 6: e = fdmt::run_filterbank<6>(vv, nbin, nt, out, cs); break;
    case 7: e = fdmt::run_filterbank<7>(vv, nbin, nt, out, cs); break;
    case 8: e = fdmt::run_filterbank<8>(vv, nbin, nt, out, cs); break;
    case 9: e = fdmt::run_filterbank<9>(vv, nbin, nt, out, cs); break;
    case 10: e = fdmt::run_filterbank<10>(vv, nbin, nt, out, cs); break;
    case 11: e = fdmt::run_filterbank<11>(vv, nbin, nt, out, cs); break;
    default: e = fdmt::run_filterbank<12>(vv, nbin, nt, out, cs); break;
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    return FDMT_ERR_CUDA;
  }
  return FDMT_OK;
}
