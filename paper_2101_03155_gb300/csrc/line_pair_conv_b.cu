// Axis-1 pass of the line-pair chain for the axis lengths of group B (pair_chain.cuh).
#include "line_pair_kernels.cuh"

namespace ace {
ACE_DEFINE_LP_CONV(b, ACE_LENGTHS_B)
}  // namespace ace
