// line_pair_plane.cu -- the plane passes of the line-pair chain for one length of axis 2 (ACE_LP_N2, set
// by the build: one object per length of line_pair_shapes.h).
#include "line_pair_kernels.cuh"
#include "line_pair_shapes.h"

#ifndef ACE_LP_N2
#define ACE_LP_N2 96
#endif

namespace ace {
namespace {
template <int N2, int N3>
bool plane_ops(PlaneOps<float> *out) {
  if constexpr (((2 * N3 <= 3 * N2 && 2 * N2 <= 3 * N3) || (N2 <= 32 && N3 <= 32)) && lp_plane_smem(N2, N3) <= 227 * 1024) {
    out->fwd = &LpLaunch<N2, N3>::fwd;
    out->inv = &LpLaunch<N2, N3>::inv;
    return true;
  }
  return false;
}
}  // namespace

#define ACE_NAME2(N) line_pair_plane_##N
#define ACE_NAME(N) ACE_NAME2(N)
bool ACE_NAME(ACE_LP_N2)(int n3, PlaneOps<float> *out) {
  switch (n3) {
#define ACE_CASE(N) case N: return plane_ops<ACE_LP_N2, N>(out);
    ACE_LP_PLANE_LENGTHS(ACE_CASE)
#undef ACE_CASE
    default: return false;
  }
}
}  // namespace ace
