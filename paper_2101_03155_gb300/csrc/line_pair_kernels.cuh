// line_pair_kernels.cuh -- the kernels of the line-pair chain (line_pair.cuh) and their launchers.
#pragma once

#include "line_pair.cuh"
#include "pair_chain.cuh"
#include "plane_chain.cuh"

namespace ace {

// ---------------------------------------------------------------------------------------
// Plane passes of the compiled shapes: one CTA per (plane i1, pack).
// ---------------------------------------------------------------------------------------
// Threads per SM the plane kernels aim at (about 100 registers each), and CTAs per SM: what shared
// memory allows, held to that many threads.
constexpr int kLpThreads = 640;
template <int N2, int N3>
using PlaneOf = PlaneFix<N2, N3, lp_lines(N2, N3), lp_group(N2, N3),
                         lp_pick_nt(N2, LFactor<N2>::R1, LFactor<N2>::R2, N3, LFactor<N3>::R1, LFactor<N3>::R2, kLpThreads)>;
template <int N2, int N3>
constexpr int lp_min_blocks() {
  constexpr int nt = PlaneOf<N2, N3>::NT;
  constexpr int fit = (228 * 1024) / (lp_plane_smem(N2, N3) + 1024), thr = kLpThreads / nt < 1 ? 1 : kLpThreads / nt;
  return fit < 1 ? 1 : (fit < thr ? fit : thr);
}

template <int N2, int N3>
__global__ void __launch_bounds__((PlaneOf<N2, N3>::NT), (lp_min_blocks<N2, N3>())) lp_fwd_kernel(PlaneArgs<float> a) {
  using G = PlaneOf<N2, N3>;
  const G g;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unit *s = reinterpret_cast<unit *>(smem_raw), *tw2 = s + lp_plane_units(N2, N3), *tw3 = N3 == N2 ? tw2 : tw2 + N2;
  const int i1 = blockIdx.x, pidx = a.pack0 + blockIdx.y;
  const int4 pk = a.packs[pidx];
  unit *dst = reinterpret_cast<unit *>(a.scratch) + ((long long)(pidx - a.batch0) * a.n1 + i1) * (G::RP * N3);
  if (a.skip_rel > 0.f && fwd_plane_negligible(a.pmax, a.gmax, a.n1, i1, pk, a.skip_rel)) {
    lp_zero(g, dst);
    return;
  }
  lp_tables(N2, N3, G::NT, a.tw2, a.tw3, tw2, tw3);
  const PlanePtrs q = lp_ptrs(a, pk, (long long)i1 * (N2 * N3));
  __syncthreads();
  if (q.same_a)
    lp_fwd_load<N2, true>(g, q.fa, q.fb, q.fc, q.fd, true, s, tw2);
  else
    lp_fwd_load<N2, false>(g, q.fa, q.fb, q.fc, q.fd, q.two, s, tw2);
  lp_sync(g);
  lp_fwd_cols2<N2>(g, s);
  __syncthreads();
  if constexpr (N2 % 2 != 0) {
    lp_swap_plane<true>(g, s);
    __syncthreads();
  }
  lp_stage_strided<N3, -1>(g, s, tw3, G::RP, 1, G::P);
  lp_sync(g);
  lp_fwd_rows2<N3>(g, s, dst);
}

template <int N2, int N3>
__global__ void __launch_bounds__((PlaneOf<N2, N3>::NT), (lp_min_blocks<N2, N3>())) lp_inv_kernel(PlaneArgs<float> a) {
  using G = PlaneOf<N2, N3>;
  const G g;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unit *s = reinterpret_cast<unit *>(smem_raw), *tw2 = s + lp_plane_units(N2, N3), *tw3 = N3 == N2 ? tw2 : tw2 + N2;
  const int i1 = blockIdx.x, pidx = a.pack0 + blockIdx.y;
  const int4 pk = a.packs[pidx];
  unit *src = reinterpret_cast<unit *>(a.scratch) + ((long long)(pidx - a.batch0) * a.n1 + i1) * (G::RP * N3);
  if (!(a.skip_rel > 0.f && inv_plane_negligible(a.pmax, a.gmax, a.n1, i1, pk, a.skip_rel))) {
    lp_tables(N2, N3, G::NT, a.tw2, a.tw3, tw2, tw3);
    const PlanePtrs q = lp_ptrs(a, pk, (long long)i1 * (N2 * N3));
    lp_prefetch(q, N2 * N3, a.hints);
    __syncthreads();
    lp_inv_rowsA<N3>(g, src, s, tw3);
    lp_sync(g);
    lp_stage_strided<N3, +1>(g, s, tw3, G::RP, 1, G::P);
    __syncthreads();
    if constexpr (N2 % 2 != 0) {
      lp_swap_plane<false>(g, s);
      __syncthreads();
    }
    lp_inv_colsA<N2>(g, s, tw2);
    lp_sync(g);
    lp_inv_acc<N2>(g, s, q);
  }
  // the spectrum plane was this pack's last use of it: its lines leave L2 without a write-back
  if (a.hints & 1) l2_discard<G::NT>(src, sizeof(unit) * G::RP * N3);
}

template <int N2, int N3>
struct LpLaunch {
  static constexpr int NT = PlaneOf<N2, N3>::NT;
  static cudaError_t fwd(const PlaneArgs<float> &a, int npacks, cudaStream_t st) {
    static unsigned long long done = 0;
    const cudaError_t e = smem_attr_once(lp_fwd_kernel<N2, N3>, lp_plane_smem(N2, N3), done);
    if (e != cudaSuccess) return e;
    lp_fwd_kernel<N2, N3><<<dim3(a.n1, npacks), NT, lp_plane_smem(N2, N3), st>>>(a);
    return cudaGetLastError();
  }
  static cudaError_t inv(const PlaneArgs<float> &a, int npacks, cudaStream_t st) {
    static unsigned long long done = 0;
    const cudaError_t e = smem_attr_once(lp_inv_kernel<N2, N3>, lp_plane_smem(N2, N3), done);
    if (e != cudaSuccess) return e;
    lp_inv_kernel<N2, N3><<<dim3(a.n1, npacks), NT, lp_plane_smem(N2, N3), st>>>(a);
    return cudaGetLastError();
  }
};

// ---------------------------------------------------------------------------------------
// Axis-1 pass: forward transform, Coulomb table, inverse transform.  A warp owns T neighbouring line
// pairs of one pack, in its own part of shared memory ([n][T] units: consecutive units per task row),
// and needs no barrier with the CTA's other warps.  The first stage reads the scratch and the last one
// writes it, 16 T contiguous bytes per row.
// ---------------------------------------------------------------------------------------
template <int L, int V>
struct LpConvShape {
  static constexpr int T = V == 2 ? 4 : 8;         // line pairs of a warp
  static constexpr int WARPS = V == 1 ? 4 : 2;     // warps of a CTA
  static constexpr int ROWS = 32 / T, NT = 32 * WARPS;
  static constexpr int smem = 16 * (WARPS * T * L + L);
  static constexpr int fit = (228 * 1024) / (smem + 1024), thr = 640 / NT;
  static constexpr int minb = fit < thr ? fit : thr;
};

template <int L, int V>
__global__ void __launch_bounds__((LpConvShape<L, V>::NT), (LpConvShape<L, V>::minb)) lp_conv_kernel(PairPassArgs<float> a) {
  using S = LpConvShape<L, V>;
  constexpr int R1 = LFactor<L>::R1, R2 = LFactor<L>::R2, T = S::T, ROWS = S::ROWS, NT = S::NT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int tid = threadIdx.x, w = tid >> 5, t = tid % T, row = (tid & 31) / T;
  unit *tw = reinterpret_cast<unit *>(smem_raw), *s = tw + L + w * (T * L);
  for (int e = tid; e < L; e += NT) tw[e] = {f2bc(a.tw[e].x), f2bc(a.tw[e].y)};
  const int nl = (a.n2 + 1) / 2 * a.n3;  // line pairs of a plane
  const int l = (blockIdx.x * S::WARPS + w) * T + t;
  const bool valid = l < nl;
  char *zc = reinterpret_cast<char *>(reinterpret_cast<unit *>(a.scratch) + (long long)blockIdx.y * L * nl + l);
  const char *kc = reinterpret_cast<const char *>(a.kernel + 2 * l);
  __syncthreads();
  // rows are reached by adding byte strides: the row count of a plane is a launch argument, and
  // products with it per access made a quarter of this kernel's instructions
  const long long zs = (long long)nl * (int)sizeof(unit), ks = (long long)nl * (int)sizeof(float2);
  // forward stage 1: tasks (t, n2)
#pragma unroll 1
  for (int n2 = row; n2 < R2; n2 += ROWS) {
    if (valid) {
      unit x[R1];
      const char *p = zc + n2 * zs;
#pragma unroll
      for (int n1 = 0; n1 < R1; ++n1, p += R2 * zs) x[n1] = ldcg_unit(reinterpret_cast<const unit *>(p));
      UDft<R1, -1>::run(x);
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1)
        s[(k1 * R2 + n2) * T + t] = k1 ? tw_mul<-1>(x[k1], tw_load(tw, n2 * k1)) : x[0];
    }
  }
  __syncwarp();
  // forward stage 2, Coulomb table, inverse stage A: tasks (t, k1)
#pragma unroll 1
  for (int k1 = row; k1 < R1; k1 += ROWS) {
    if (valid) {
      unit *p = s + k1 * R2 * T + t;
      const char *kp = kc + k1 * ks;
      unit x[R2];
      f2 kv[R2];
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2, kp += R1 * ks) kv[k2] = ld2(reinterpret_cast<const float *>(kp));
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) x[n2] = p[n2 * T];
      UDft<R2, -1>::run(x);
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) x[k2] = {x[k2].x * kv[k2], x[k2].y * kv[k2]};
      UDft<R2, +1>::run(x);
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) p[n2 * T] = n2 ? tw_mul<+1>(x[n2], tw_load(tw, n2 * k1)) : x[0];
    }
  }
  __syncwarp();
  // inverse stage B: tasks (t, n2), natural order i1 = n1 R2 + n2 straight to the scratch
#pragma unroll 1
  for (int n2 = row; n2 < R2; n2 += ROWS) {
    if (valid) {
      unit x[R1];
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) x[k1] = s[(k1 * R2 + n2) * T + t];
      UDft<R1, +1>::run(x);
      char *p = zc + n2 * zs;
#pragma unroll
      for (int n1 = 0; n1 < R1; ++n1, p += R2 * zs) *reinterpret_cast<unit *>(p) = x[n1];
    }
  }
}

template <int L, int V>
cudaError_t launch_lp_conv_LV(const PairPassArgs<float> &a, int npacks, cudaStream_t st) {
  using S = LpConvShape<L, V>;
  static unsigned long long done = 0;
  const cudaError_t e = smem_attr_once(lp_conv_kernel<L, V>, S::smem, done);
  if (e != cudaSuccess) return e;
  const int nl = (a.n2 + 1) / 2 * a.n3;
  lp_conv_kernel<L, V><<<dim3((nl + S::T * S::WARPS - 1) / (S::T * S::WARPS), npacks), S::NT, S::smem, st>>>(a);
  return cudaGetLastError();
}
// The axis-1 pass in the pencil tile a.conv_tile selects.
template <int L>
cudaError_t launch_lp_conv_L(const PairPassArgs<float> &a, int npacks, cudaStream_t st) {
  if (a.conv_tile == 1) return launch_lp_conv_LV<L, 1>(a, npacks, st);
  if (a.conv_tile == 2) return launch_lp_conv_LV<L, 2>(a, npacks, st);
  return launch_lp_conv_LV<L, 0>(a, npacks, st);
}

#define ACE_LP_CONV_CASE(L_)                      \
  case L_:                                        \
    *e = launch_lp_conv_L<L_>(a, npacks, st);     \
    return true;
#define ACE_DEFINE_LP_CONV(NAME, LIST)                                                                  \
  bool lp_conv_##NAME(int L, const PairPassArgs<float> &a, int npacks, cudaStream_t st, cudaError_t *e) { \
    switch (L) {                                                                                        \
      LIST(ACE_LP_CONV_CASE)                                                                            \
      default: return false;                                                                            \
    }                                                                                                   \
  }

}  // namespace ace
