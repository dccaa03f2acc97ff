// Dispatch of the pair-potential chain's pencil kernels (double, plain form) over the length groups.
#include "pair_chain.cuh"

namespace ace {
#define ACE_DECLARE_GROUP(G)                                                                             \
  bool pass_##G##_f64(int L, int mode, const PairPassArgs<double> &a, int npacks, cudaStream_t st, cudaError_t *e); \
  bool conv_##G##_f64(int L, const PairPassArgs<double> &a, int npacks, cudaStream_t st, cudaError_t *e);
ACE_DECLARE_GROUP(a)
ACE_DECLARE_GROUP(b)
ACE_DECLARE_GROUP(c)
ACE_DECLARE_GROUP(d)
#undef ACE_DECLARE_GROUP

template <>
cudaError_t launch_pair_pass<double>(int mode, const PairPassArgs<double> &a, int npacks, cudaStream_t st) {
  const int L = (mode == PASS_FWD3_PAIR || mode == PASS_INV3_ACC || mode == PASS_INV3) ? a.n3 : (mode == PASS_CONV1 ? a.n1 : a.n2);
  cudaError_t e = cudaErrorInvalidValue;
  if (pass_a_f64(L, mode, a, npacks, st, &e) || pass_b_f64(L, mode, a, npacks, st, &e) ||
      pass_c_f64(L, mode, a, npacks, st, &e) || pass_d_f64(L, mode, a, npacks, st, &e))
    return e;
  return cudaErrorInvalidValue;
}

template <>
cudaError_t launch_conv_pass<double>(const PairPassArgs<double> &a, int npacks, cudaStream_t st) {
  cudaError_t e = cudaErrorInvalidValue;
  if (conv_a_f64(a.n1, a, npacks, st, &e) || conv_b_f64(a.n1, a, npacks, st, &e) ||
      conv_c_f64(a.n1, a, npacks, st, &e) || conv_d_f64(a.n1, a, npacks, st, &e))
    return e;
  return cudaErrorInvalidValue;
}

// One point per thread; the packs of a batch one after the other.  The terms of an element are added in pack
// order whatever the launch: the FP64 form repeats bit for bit without the rounds of packs on disjoint
// orbitals that its atomic form needed (12 orbitals on 40x45x48 ran 13 rounds of three packs).  It moves 88
// bytes per point and pack beside transforms that wait for the FP64 pipe, so it runs in their shadow.
template <typename T>
__global__ void __launch_bounds__(256) pair_accumulate_kernel(const T *__restrict__ phi, T *W, const cpx<T> *__restrict__ z,
                                                              const int4 *__restrict__ packs, int npacks, long long N) {
  const long long e = blockIdx.x * 256ll + threadIdx.x;
  if (e >= N) return;
  for (int p = 0; p < npacks; ++p) {
    const int4 pk = packs[p];
    const cpx<T> v = z[(long long)p * N + e];
    T *wa = W + (long long)pk.x * N + e, *wb = W + (long long)pk.y * N + e;
    const T fa = phi[(long long)pk.x * N + e], fb = phi[(long long)pk.y * N + e];
    if (pk.z == pk.x && pk.y != pk.x && pk.w != pk.x) {
      // (a, b), (a, d): three different orbitals
      T *wd = W + (long long)pk.w * N + e;
      const T fd = phi[(long long)pk.w * N + e];
      const T a = *wa, b = *wb, d = *wd;
      *wa = a + (v.x * fb + v.y * fd);
      *wb = b + v.x * fa;
      *wd = d + v.y * fa;
    } else {
      *wa += v.x * fb;
      if (pk.y != pk.x) *wb += v.x * fa;
      if (pk.z >= 0) {
        const T fc = phi[(long long)pk.z * N + e], fd = phi[(long long)pk.w * N + e];
        W[(long long)pk.z * N + e] += v.y * fd;
        if (pk.w != pk.z) W[(long long)pk.w * N + e] += v.y * fc;
      }
    }
  }
}

template <typename T>
cudaError_t launch_pair_accumulate(const T *phi, T *W, const cpx<T> *z, const int4 *packs, int npacks, long long N,
                                   cudaStream_t st) {
  pair_accumulate_kernel<T><<<(unsigned)((N + 255) / 256), 256, 0, st>>>(phi, W, z, packs, npacks, N);
  return cudaGetLastError();
}
template cudaError_t launch_pair_accumulate<double>(const double *, double *, const cpx<double> *, const int4 *, int,
                                                    long long, cudaStream_t);
}  // namespace ace
