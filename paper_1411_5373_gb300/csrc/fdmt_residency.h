// How many blocks of a kernel the current device holds at once.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>

namespace fdmt {

// *blocks = the blocks of `kernel` (threads per block, dynamic shared memory
// in bytes) resident on the current device at once, at least one (an error
// otherwise).  Also allows the kernel up to 227 KiB of shared memory.
// Any thread; results are kept per device.
cudaError_t resident_blocks(const void *kernel, int threads, size_t smem, int *blocks);

}  // namespace fdmt
