// Compile-time line-pass instances: windows of two radices.
#include "chain_gm_line.cuh"

namespace ptycho {

const GmInstance kGmSmall[] = {
    gm_instance<GmShape<6, 1, 8, 16, 128, 4>>(),    // 48
    gm_instance<GmShape<8, 1, 9, 18, 160, 4>>(),    // 72
    gm_instance<GmShape<9, 1, 9, 9, 96, 4>>(),      // 81
    gm_instance<GmShape<8, 1, 12, 16, 192, 4>>(),   // 96
    gm_instance<GmShape<12, 1, 9, 12, 128, 4>>(),   // 108
};
const int kGmSmallCount = sizeof(kGmSmall) / sizeof(kGmSmall[0]);

}  // namespace ptycho
