// xform_mid_5.cu — instances of the compile-time line transforms (xform_mid.cuh).
#include "xform_mid.cuh"

namespace ps {
PS_MID_INST(192)
PS_MID_INST(216)
PS_MID_INST(243)
}  // namespace ps
