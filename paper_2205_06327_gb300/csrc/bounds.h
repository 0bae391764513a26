// Arithmetic that keeps the kernels inside their buffers and limits, in plain
// C++, so that it can be checked on the host without a GPU.
#pragma once

#include <stddef.h>
#include <stdint.h>

#ifdef __CUDACC__
#define PTYCHO_HD __host__ __device__
#else
#define PTYCHO_HD
#endif

namespace ptycho {

// Offset of element (y, x) from a window's corner in an object W pixels wide.
// 64 bits: objects hold up to 2^34 pixels, and 4095 rows of more than 524416
// pixels already pass 2^31.
PTYCHO_HD constexpr int64_t window_at(int y, int x, int W) { return (int64_t)y * W + x; }

// An SM's tensor-memory columns, its shared memory, and what of it every
// resident block takes beside its own.
constexpr int kTmemColumns = 512;
constexpr size_t kSmShared = 228 << 10, kBlockShared = 1 << 10;

// The dynamic shared memory a kernel that needs `need` bytes asks for so that
// at most `blocks` of its blocks are resident on an SM (in whole 128 bytes).
constexpr size_t smem_for_at_most(int blocks, size_t need) {
  const size_t least = (kSmShared / (blocks + 1) - kBlockShared) / 128 * 128 + 128;
  return need > least ? need : least;
}

}  // namespace ptycho
