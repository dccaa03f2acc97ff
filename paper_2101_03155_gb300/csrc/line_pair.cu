// line_pair.cu -- selection of the line-pair chain's kernels for a grid, and its Coulomb table.
#include "line_pair_kernels.cuh"
#include "line_pair_shapes.h"

namespace ace {
namespace {

// R1, R2 of an axis length in this chain
void lp_factors(int L, int *r1, int *r2) {
  switch (L) {
#define ACE_CASE(L_)         \
  case L_:                   \
    *r1 = LFactor<L_>::R1;   \
    *r2 = LFactor<L_>::R2;   \
    return;
    ACE_PASS_LENGTHS(ACE_CASE)
#undef ACE_CASE
    default: *r1 = *r2 = 0;
  }
}

// Coulomb table in the scratch's layout: [m1][p3][rp] pairs for the rows 2 rp, 2 rp + 1 of the
// permuted axis 2 (0 for the row past an odd N2)
__global__ void lp_table_kernel(const float *K, int n1, int n2, int n3, int a2, int b2, int a3, int b3, float2 *out) {
  const int rps = (n2 + 1) / 2;
  const long long total = (long long)n1 * n3 * rps;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const int rp = (int)(e % rps), p3 = (int)(e / rps % n3);
    const long long m1 = e / ((long long)rps * n3);
    const int k3 = p3 / b3 + a3 * (p3 % b3);
    float v[2] = {0.f, 0.f};
    for (int h = 0; h < 2; ++h) {
      const int p2 = 2 * rp + h;
      if (p2 < n2) v[h] = K[(m1 * n2 + (p2 / b2 + a2 * (p2 % b2))) * n3 + k3];
    }
    out[e] = make_float2(v[0], v[1]);
  }
}

}  // namespace

#define ACE_DECLARE(N) bool line_pair_plane_##N(int n3, PlaneOps<float> *out);
ACE_LP_PLANE_LENGTHS(ACE_DECLARE)
#undef ACE_DECLARE

bool line_pair_ops(int n1, int n2, int n3, PlaneOps<float> *out) {
  if (!pass_length_supported(n1)) return false;
  switch (n2) {
#define ACE_CASE(N) case N: return line_pair_plane_##N(n3, out);
    ACE_LP_PLANE_LENGTHS(ACE_CASE)
#undef ACE_CASE
    default: return false;
  }
}

cudaError_t launch_line_pair_table(const float *K, int n1, int n2, int n3, float *out, cudaStream_t st) {
  int a2, b2, a3, b3;
  lp_factors(n2, &a2, &b2);
  lp_factors(n3, &a3, &b3);
  lp_table_kernel<<<1024, 256, 0, st>>>(K, n1, n2, n3, a2, b2, a3, b3, reinterpret_cast<float2 *>(out));
  return cudaGetLastError();
}

bool lp_conv_a(int L, const PairPassArgs<float> &a, int npacks, cudaStream_t st, cudaError_t *e);
bool lp_conv_b(int L, const PairPassArgs<float> &a, int npacks, cudaStream_t st, cudaError_t *e);
bool lp_conv_c(int L, const PairPassArgs<float> &a, int npacks, cudaStream_t st, cudaError_t *e);
bool lp_conv_d(int L, const PairPassArgs<float> &a, int npacks, cudaStream_t st, cudaError_t *e);

cudaError_t launch_line_pair_conv(const PairPassArgs<float> &a, int npacks, cudaStream_t st) {
  cudaError_t e = cudaErrorInvalidValue;
  if (lp_conv_a(a.n1, a, npacks, st, &e) || lp_conv_b(a.n1, a, npacks, st, &e) ||
      lp_conv_c(a.n1, a, npacks, st, &e) || lp_conv_d(a.n1, a, npacks, st, &e))
    return e;
  return cudaErrorInvalidValue;
}

}  // namespace ace
