// xform_mid_3.cu — instances of the compile-time line transforms (xform_mid.cuh).
#include "xform_mid.cuh"

namespace ps {
PS_MID_INST(72)
PS_MID_INST(81)
PS_MID_INST(96)
}  // namespace ps
