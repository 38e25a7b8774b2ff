// xform_mid_1.cu — instances of the compile-time line transforms (xform_mid.cuh).
#include "xform_mid.cuh"

namespace ps {
PS_MID_INST(16)
PS_MID_INST(18)
PS_MID_INST(24)
PS_MID_INST(27)
}  // namespace ps
