// Overlap-save streaming of the transform (contracts in include/fdmt.h).
//
// Output column t depends only on input columns [t - Nd + 1, t] (the
// recursion only ever looks back in time, Algorithm 1, and treats samples
// before the first as zero, the copy rule of section 4).  A continuous
// stream is therefore transformed chunk by chunk: each chunk is appended to
// the last `carry` >= Nd - 1 input columns of the previous one, the window
// (carry + chunk columns) is transformed with an ordinary plan, and the
// window's last `chunk` output columns are exactly the stream's output for
// that chunk.  The first chunk sees a carry of zeros, which is the copy rule.
//
// One kernel lays a window out (carry and chunk rows, 16 bytes per thread).
// A fused plan writes the chunk's columns straight to the caller's output
// and computes only the tiles they need; a plain plan's window output is
// copied.  The stream owns its window buffers, allocated once at creation.
// Four pushes of 16384 samples, 1024 channels and delays, uint8, fused, on a
// GB300: 724 us with two 2-D copies in, the whole window
// transformed and a 2-D copy out, 370 us now.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <new>

#include "../../include/fdmt.h"
#include "fdmt_internal.h"

struct fdmt_stream_s {
  fdmt_plan_t plan = nullptr;
  int32_t nf = 0, nd = 0, dtype = 0;
  int64_t chunk = 0, carry = 0, window = 0;
  size_t in_es = 0;
  void *win[2] = {nullptr, nullptr};  // input windows [nf][window], ping-pong
  void *wout = nullptr;               // plain plans: window output [nd][window]
  bool fused = false;
  void *ws = nullptr;
  size_t ws_bytes = 0;
  int cur = 0;                        // window holding the latest chunk
};

namespace {

size_t in_size(int32_t dtype) { return dtype == FDMT_U8_I32 ? 1 : 4; }

constexpr int kWindowThreads = 256;

// Row blockIdx.y of a window: the last `carry` 16-byte words of `prev`, then
// `chunk` words of the new chunk.
__global__ void __launch_bounds__(kWindowThreads)
window_kernel(const int4 *__restrict__ prev, const int4 *__restrict__ in, int4 *__restrict__ win, int64_t carry,
              int64_t chunk) {
  const int64_t i = (int64_t)blockIdx.x * kWindowThreads + threadIdx.x, row = blockIdx.y, pitch = carry + chunk;
  if (i >= pitch) return;
  win[row * pitch + i] = i >= carry ? __ldg(in + row * chunk + (i - carry)) : __ldg(prev + row * pitch + chunk + i);
}

void release(fdmt_stream_s *s) {
  if (s == nullptr) return;
  if (s->plan != nullptr) fdmt_destroy(s->plan);
  cudaFree(s->win[0]);
  cudaFree(s->win[1]);
  cudaFree(s->wout);
  cudaFree(s->ws);
  delete s;
}

}  // namespace

extern "C" {

int fdmt_stream_create(double f_min, double f_max, int32_t nf, int64_t chunk, int32_t nd, int32_t dtype,
                       uint32_t flags, fdmt_stream_t *out) {
  if (out == nullptr) return FDMT_ERR_INVALID_ARG;
  *out = nullptr;
  if (chunk < 16 || chunk % 16 != 0 || nd < 1 || (flags & FDMT_PLAN_HOST_ONLY)) return FDMT_ERR_INVALID_ARG;
  if (dtype != FDMT_U8_I32 && dtype != FDMT_F32_F32 && dtype != FDMT_F32_F16STATE) return FDMT_ERR_INVALID_ARG;
  const int64_t carry = ((int64_t)nd - 1 + 15) / 16 * 16;
  const int64_t window = carry + chunk;
  // Validate the shape on the host before any device allocation.
  fdmt_plan_t probe = nullptr;
  int st = fdmt_plan(f_min, f_max, nf, window, nd, dtype, flags | FDMT_PLAN_HOST_ONLY, &probe);
  if (st != FDMT_OK) return st;
  fdmt_destroy(probe);

  fdmt_stream_s *s = new (std::nothrow) fdmt_stream_s;
  if (s == nullptr) return FDMT_ERR_NO_MEMORY;
  s->nf = nf;
  s->nd = nd;
  s->dtype = dtype;
  s->chunk = chunk;
  s->carry = carry;
  s->window = window;
  s->in_es = in_size(dtype);
  if ((st = fdmt_plan(f_min, f_max, nf, window, nd, dtype, flags, &s->plan)) != FDMT_OK) {
    release(s);
    return st;
  }
  if ((st = fdmt_workspace_bytes(s->plan, &s->ws_bytes)) != FDMT_OK) {
    release(s);
    return st;
  }
  const size_t in_bytes = (size_t)nf * window * s->in_es;
  const size_t out_bytes = (size_t)nd * window * 4;
  s->fused = (flags & FDMT_SCHED_FUSED) != 0;
  if (cudaMalloc(&s->win[0], in_bytes) != cudaSuccess || cudaMalloc(&s->win[1], in_bytes) != cudaSuccess ||
      (!s->fused && cudaMalloc(&s->wout, out_bytes) != cudaSuccess) ||
      cudaMalloc(&s->ws, s->ws_bytes > 0 ? s->ws_bytes : 256) != cudaSuccess) {
    cudaGetLastError();
    release(s);
    return FDMT_ERR_NO_MEMORY;
  }
  // The carry before the first chunk is zero (the copy rule).
  if (s->carry > 0 && cudaMemset2D(static_cast<char *>(s->win[0]) + (size_t)chunk * s->in_es, (size_t)window * s->in_es, 0,
                                   (size_t)carry * s->in_es, (size_t)nf) != cudaSuccess) {
    cudaGetLastError();
    release(s);
    return FDMT_ERR_CUDA;
  }
  *out = s;
  return FDMT_OK;
}

int fdmt_stream_info(fdmt_stream_t s, int64_t *carry, int64_t *window) {
  if (s == nullptr) return FDMT_ERR_INVALID_ARG;
  if (carry != nullptr) *carry = s->carry;
  if (window != nullptr) *window = s->window;
  return FDMT_OK;
}

int fdmt_stream_push(fdmt_stream_t s, const void *in, void *out, void *stream) {
  if (s == nullptr || in == nullptr || out == nullptr) return FDMT_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out)) & 15u) return FDMT_ERR_INVALID_ARG;
  // (before the window's kernel is launched: the plan's own check comes later)
  fdmt::PlanView view;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) return FDMT_ERR_CUDA;
  if (!fdmt::plan_view(s->plan, &view) || dev != view.device) return FDMT_ERR_INVALID_ARG;
  cudaStream_t cs = static_cast<cudaStream_t>(stream);
  const int nxt = s->cur ^ 1;
  void *dst = s->win[nxt];
  // New window = [last `carry` columns of the previous window | chunk].
  const int64_t carry = s->carry * (int64_t)s->in_es / 16, chunk = s->chunk * (int64_t)s->in_es / 16;
  for (int32_t row = 0; row < s->nf; row += 65535) {  // (grid rows)
    const int64_t off = (int64_t)row * (carry + chunk);
    const dim3 grid((unsigned)((carry + chunk + kWindowThreads - 1) / kWindowThreads),
                    (unsigned)std::min<int32_t>(65535, s->nf - row));
    window_kernel<<<grid, kWindowThreads, 0, cs>>>(
        static_cast<const int4 *>(s->win[s->cur]) + off,
        static_cast<const int4 *>(in) + (int64_t)row * chunk, static_cast<int4 *>(dst) + off, carry, chunk);
  }
  if (cudaGetLastError() != cudaSuccess) return FDMT_ERR_CUDA;
  // The window's last `chunk` output columns are the stream's output.
  if (s->fused) {
    const int st = fdmt::execute_view(s->plan, dst, out, s->ws, s->ws_bytes, fdmt::OutView{s->carry, s->chunk}, cs);
    if (st != FDMT_OK) return st;
  } else {
    const int st = fdmt_execute(s->plan, dst, nullptr, s->wout, s->ws, s->ws_bytes, stream);
    if (st != FDMT_OK) return st;
    if (cudaMemcpy2DAsync(out, (size_t)s->chunk * 4, static_cast<char *>(s->wout) + (size_t)s->carry * 4,
                          (size_t)s->window * 4, (size_t)s->chunk * 4, s->nd, cudaMemcpyDeviceToDevice,
                          cs) != cudaSuccess) {
      cudaGetLastError();
      return FDMT_ERR_CUDA;
    }
  }
  s->cur = nxt;
  return FDMT_OK;
}

int fdmt_stream_reset(fdmt_stream_t s, void *stream) {
  if (s == nullptr) return FDMT_ERR_INVALID_ARG;
  // The carry of zeros, in stream order (a captured reset or push replays
  // as it ran): the last columns of the window that the next push reads.
  const size_t pitch = (size_t)s->window * s->in_es;
  if (s->carry > 0 && cudaMemset2DAsync(static_cast<char *>(s->win[0]) + (size_t)s->chunk * s->in_es, pitch, 0,
                                        (size_t)s->carry * s->in_es, (size_t)s->nf,
                                        static_cast<cudaStream_t>(stream)) != cudaSuccess) {
    cudaGetLastError();
    return FDMT_ERR_CUDA;
  }
  s->cur = 0;
  return FDMT_OK;
}

void fdmt_stream_destroy(fdmt_stream_t s) { release(s); }

}  // extern "C"
