// xform_mid_2.cu — instances of the compile-time line transforms (xform_mid.cuh).
#include "xform_mid.cuh"

namespace ps {
PS_MID_INST(32)
PS_MID_INST(36)
PS_MID_INST(48)
PS_MID_INST(54)
}  // namespace ps
