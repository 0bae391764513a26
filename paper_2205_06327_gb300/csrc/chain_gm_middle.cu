// Compile-time line-pass instances: windows of two larger radices.
#include "chain_gm_line.cuh"

namespace ptycho {

const GmInstance kGmMiddle[] = {
    gm_instance<GmShape<12, 1, 12, 16, 192, 4>>(),  // 144
    gm_instance<GmShape<12, 1, 16, 16, 256, 4>>(),  // 192
    gm_instance<GmShape<16, 1, 16, 16, 256, 3>>(),  // 256
};
const int kGmMiddleCount = sizeof(kGmMiddle) / sizeof(kGmMiddle[0]);

}  // namespace ptycho
