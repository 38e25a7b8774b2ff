// xform_mid_6.cu — instances of the compile-time line transforms (xform_mid.cuh).
#include "xform_mid.cuh"

namespace ps {
PS_MID_INST(288)
PS_MID_INST(324)
}  // namespace ps
