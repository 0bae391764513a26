// Compile-time line-pass instances: windows of three radices.
#include "chain_gm_line.cuh"

namespace ptycho {

const GmInstance kGmLarge[] = {
    gm_instance<GmShape<6, 4, 16, 8, 256, 4>>(),    // 384
    gm_instance<GmShape<8, 4, 16, 8, 256, 4>>(),    // 512
    gm_instance<GmShape<8, 8, 16, 8, 256, 3>>(),    // 1024
};
const int kGmLargeCount = sizeof(kGmLarge) / sizeof(kGmLarge[0]);

}  // namespace ptycho
