// Compile-time line-pass instances: windows of three radices.
//
// Shapes <R1, R2, R3, lines, threads, blocks per SM>, the fastest of four to
// ten tried for each; us of one evaluation, Stockham passes -> these:
//   162: 256 positions, 8 slices 4781 -> 1346    384: 42, 8: 3574 -> 1085
//   216: 196, 8: 5570 -> 2007                    512: 20, 8: 2550 -> 946
//   288: 100, 8: 4510 -> 1375                   1024: 4, 100: 30427 -> 14253
// For 512: 16 lines in 512 threads 1116, 4 x 8 x 16 975; for 1024: 4 lines
// 14745, 512 threads 16184, 128 threads 18467, 4 x 16 x 16 16035.
#include "chain_gm_line.cuh"

namespace ptycho {

const GmInstance kGmLarge[] = {
    gm_instance<GmShape<6, 3, 9, 18, 128, 5>>(),    // 162
    gm_instance<GmShape<6, 4, 9, 18, 128, 5>>(),    // 216
    gm_instance<GmShape<6, 3, 16, 16, 128, 5>>(),   // 288
    gm_instance<GmShape<6, 4, 16, 16, 256, 3>>(),   // 384
    gm_instance<GmShape<8, 4, 16, 8, 256, 3>>(),    // 512
    gm_instance<GmShape<8, 8, 16, 8, 256, 2>>(),    // 1024
};
const int kGmLargeCount = sizeof(kGmLarge) / sizeof(kGmLarge[0]);

}  // namespace ptycho
