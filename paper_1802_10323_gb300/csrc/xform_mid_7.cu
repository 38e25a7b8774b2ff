// xform_mid_7.cu — instances of the compile-time line transforms (xform_mid.cuh).
#include "xform_mid.cuh"

namespace ps {
PS_MID_INST(384)
PS_MID_INST(432)
PS_MID_INST(486)
}  // namespace ps
