// Axis-1 pass of the line-pair chain for the axis lengths of group A (pair_chain.cuh).
#include "line_pair_kernels.cuh"

namespace ace {
ACE_DEFINE_LP_CONV(a, ACE_LENGTHS_A)
}  // namespace ace
