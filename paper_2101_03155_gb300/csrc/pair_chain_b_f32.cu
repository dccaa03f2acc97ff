// Pencil-pass kernels (float) for the axis lengths of group B (pair_chain.cuh).
#include "pair_chain.cuh"

namespace ace {
ACE_DEFINE_GROUP(b_f32, float, ACE_LENGTHS_B, ACE_NO_LENGTHS)
}  // namespace ace
