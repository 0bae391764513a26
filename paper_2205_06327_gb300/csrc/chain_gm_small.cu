// Compile-time line-pass instances: windows of two radices.
//
// Shapes <R1, R2, R3, lines, threads, blocks per SM>, the fastest of four to
// ten tried for each; us of one evaluation, Stockham passes -> these:
//   16: 930 positions, 8 slices 671 -> 161    72: 625, 8: 2243 -> 567
//   24: 930, 8: 843 -> 227                    81: 400, 8: 2061 -> 464
//   32: 930, 8: 1009 -> 280                   96: 930, 11: 3151 -> 1601
//   48: 930, 8: 1738 -> 375                  108: 400, 8: 2951 -> 764
//   54: 625, 8: 1850 -> 384
// For 96, at the same time: 8 x 12 in 192 threads 1826, 6 x 16 2092, 12 x 8 in 192
// threads 1727; with dependent launches and one chunk (1601 -> 1386): 8 blocks
// per SM 1386, 6 (more registers) 1356.
#include "chain_gm_line.cuh"

namespace ptycho {

const GmInstance kGmSmall[] = {
    gm_instance<GmShape<4, 1, 4, 16, 64, 8>>(),     // 16
    gm_instance<GmShape<4, 1, 6, 24, 128, 6>>(),    // 24
    gm_instance<GmShape<4, 1, 8, 32, 256, 4>>(),    // 32
    gm_instance<GmShape<6, 1, 8, 16, 128, 4>>(),    // 48
    gm_instance<GmShape<6, 1, 9, 18, 96, 8>>(),     // 54
    gm_instance<GmShape<8, 1, 9, 18, 96, 8>>(),     // 72
    gm_instance<GmShape<9, 1, 9, 27, 128, 8>>(),    // 81
    gm_instance<GmShape<12, 1, 8, 16, 96, 6>>(),    // 96
    gm_instance<GmShape<12, 1, 9, 18, 224, 3>>(),   // 108
};
const int kGmSmallCount = sizeof(kGmSmall) / sizeof(kGmSmall[0]);

}  // namespace ptycho
