// Arithmetic that keeps the kernels inside their buffers and limits, in plain
// C++, so that it can be checked on the host without a GPU.
#pragma once

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

}  // namespace ptycho
