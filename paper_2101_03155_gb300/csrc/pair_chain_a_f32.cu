// Pencil-pass kernels (float) for the axis lengths of group A (pair_chain.cuh).
#include "pair_chain.cuh"

namespace ace {
ACE_DEFINE_GROUP(a_f32, float, ACE_LENGTHS_A, ACE_NO_LENGTHS)
}  // namespace ace
