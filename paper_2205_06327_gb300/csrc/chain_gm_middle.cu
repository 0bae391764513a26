// Compile-time line-pass instances: windows of two larger radices.
//
// Shapes <R1, R2, R3, lines, threads, blocks per SM>, the fastest of six to
// ten tried for each; us of one evaluation, Stockham passes -> these:
//   144: 400 positions, 8 slices 4995 -> 1066
//   192: 506, 12: 7115 -> 3335 (256 threads at 64 / 80 registers 3974 / 3794,
//        16 x 12 3782, 64 threads 3704)
//   256: 1024, 8: 14317 -> 8094 (256 threads 8715, 64 threads 9586)
#include "chain_gm_line.cuh"

namespace ptycho {

const GmInstance kGmMiddle[] = {
    gm_instance<GmShape<12, 1, 12, 16, 96, 8>>(),   // 144
    gm_instance<GmShape<12, 1, 16, 16, 128, 5>>(),  // 192
    gm_instance<GmShape<16, 1, 16, 16, 128, 4>>(),  // 256
};
const int kGmMiddleCount = sizeof(kGmMiddle) / sizeof(kGmMiddle[0]);

}  // namespace ptycho
