// xform_mid_4.cu — instances of the compile-time line transforms (xform_mid.cuh).
#include "xform_mid.cuh"

namespace ps {
PS_MID_INST(108)
PS_MID_INST(144)
PS_MID_INST(162)
}  // namespace ps
