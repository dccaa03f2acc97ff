// scdm.cu -- SCDM localisation (selected columns of the density matrix), the unitary change of
// basis of section II (Eq. unit) that turns canonical orbitals into the localized orbitals the pair
// screen needs:
//   1. greedy column-pivoted QR of Psi^T (norb x N, column r = psi(r)): step k takes the grid point
//      of largest residual norm d(r) = |psi(r)|^2 - sum_{j<k} (u_j . psi(r))^2 (first index on
//      ties) and extends the orthonormal basis u_j of the chosen columns;
//   2. M[i][j] = psi_i(c_j), the selected columns of the density matrix P = Psi Psi^T;
//   3. symmetric orthonormalisation: U = M (M^T M)^{-1/2}, phi_k = sum_i psi_i U[i][k].
// The inverse square root is the coupled Newton-Schulz iteration (Higham, "Functions of Matrices",
// 2008, section 6.3) on A = S / |S|_F: Y0 = A, Z0 = I, T = (3 I - Z Y) / 2, Y <- Y T, Z <- T Z, with
// Z -> A^{-1/2} quadratically once |I - Z Y| < 1.  Only FP64 and FP32 ALU arithmetic is used: the
// contractions are n x n, far too small for the tensor cores to matter.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstdlib>

#include "ace_internal.h"
#include "residual_key.h"

namespace ace {
namespace {

constexpr int kUpdNT = 256;  // threads of the streaming selection kernels
constexpr int kUpdBlocks = 1024;  // most blocks of a selection pass (sizes the block-maximum arrays)
constexpr int kNsMax = 64;          // Newton-Schulz iterations at most
constexpr int kNsChunk = 16;        // iterations launched between host checks of convergence
constexpr double kNsStop = 1e-12;   // max |T - I| below which the following iterations are skipped
constexpr int kBlk = 8;             // points of a block of the FP32 selection
constexpr long long kLeft = -1;
constexpr int kSeedLag = 16;        // most vectors a threshold block may be behind
constexpr int kChunk = 8;           // products summed in the working type before the FP64 add
constexpr double kDependent = 1e-24;    // |residual|^2 / |psi(c)|^2 below which a column is dependent
constexpr double kDependent32 = 1e-10;  // the same with FP32 Gram-Schmidt

// Order key of an FP64 residual norm: the bits of a double compare like the values for non-negative ones,
// with chosen points (-1) below them and NaN (never chosen) at kNone.  Comparisons of FP64 values would run
// on the FP64 pipe, which issues one warp instruction per 64 cycles.
__device__ __forceinline__ long long res_key(double v) {
  const long long b = __double_as_longlong(v);
  return (b & 0x7fffffffffffffffll) > 0x7ff0000000000000ll ? kNone : b;
}

// (key, index) maximum, the smaller index winning ties
__device__ __forceinline__ void amax(long long &v, long long &i, long long v2, long long i2) {
  if (v2 > v || (v2 == v && v2 != kNone && i2 < i)) {
    v = v2;
    i = i2;
  }
}

// over the lanes of a warp (in lane 0)
__device__ __forceinline__ void warp_amax(long long &v, long long &i) {
  for (int o = 16; o > 0; o >>= 1) {
    const long long v2 = __shfl_down_sync(0xffffffffu, v, o);
    const long long i2 = __shfl_down_sync(0xffffffffu, i, o);
    amax(v, i, v2, i2);
  }
}
// over the points of a block (lane >> 2; in every lane)
__device__ __forceinline__ long long blk_max(long long v) {
  for (int o = 16; o > 2; o >>= 1) {
    const long long v2 = __shfl_xor_sync(0xffffffffu, v, o);
    v = v2 > v ? v2 : v;
  }
  return v;
}

// State of the greedy selection passed to the streaming kernels.  Each pass publishes one
// (maximum, index) per block; the block that publishes last takes the pivot step of the pass, so
// that no separate launch (and no waiting) sits between the passes.
struct SelArgs {
  long long *bval;       // [gridDim.x] keys of the block maxima of the residual norms
  long long *bidx;       // [gridDim.x] their grid indices
  unsigned int *count;   // blocks of the current pass that have published (the last one resets it)
  void *Ub;              // [n][ldu] of the working type, row j = u_j, row stride ldu
                         // (basis_ld; the padding is zero)
  int *piv;              // [n]
  int *dependent;        // set when a chosen column lies in the span of the earlier ones
  int k;                 // step whose pivot this pass selects
  // FP32 selection: per block of kBlk points, an upper bound of its residual norms and the number of
  // basis vectors its residuals account for; per step, the largest up-to-date residual seen so far
  // and per CTA of a pass the largest bound over its blocks (as they stand at its end), with its block
  long long *tval, *tidx;   // [gridDim.x]
  long long *bmax;       // [blocks]
  int *bcnt;             // [blocks]
  long long *thr;        // [n + 1], from 0 (kLeft: the steps over bounds have been left)
  // clock cycles: the longest CTA of the current pass, and by how much the last passes have cost more than
  // passes over every point would have; then 0, or the step from which on every point is updated
  int *work;
  long long *excess;
  int *left;
  int full_cost, leave_cost, leave_step;
};

template <typename T>
struct Vec2;
template <>
struct Vec2<float> {
  using type = float2;
};
template <>
struct Vec2<double> {
  using type = double2;
};

// Row stride of the basis u_j: whole float4 rows for FP32, even for FP64 (the padding is zero)
template <typename T>
__host__ __device__ constexpr int basis_ld(int n) {
  return sizeof(T) == 4 ? (n + 3) & ~3 : (n + 1) & ~1;
}

// Shared memory of a streaming block: u_{k-1} while streaming, the pivot step's vectors afterwards.
template <typename T>
struct __align__(16) ScdmSmem {
  struct {
    T u[1024], c[1024], red2[1024];
  } sel;
  T us[1024];
  double rv[kUpdNT / 32], rv0[kUpdNT / 32];
  long long rk[kUpdNT / 32], ri[kUpdNT / 32], tk[kUpdNT / 32], ti[kUpdNT / 32];
  long long chosen, top;
  int last, leave;
};

__device__ __forceinline__ float dot4(float4 a, float4 b) {
  return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, a.x * b.x)));
}

// A block's 8 points as a warp holds them: lane 4 p + c has point p and the orbital quads l = c, c + 4, ...,
// c + 28 (orbitals 4 l .. 4 l + 3), x[4 i + t] orbital 4 (c + 4 i) + t (+ 128 f0 with more than 128 orbitals).
__device__ __forceinline__ void load_block(const float *__restrict__ psi, int n, long long N, long long r0, int lim,
                                           int f0, float (&x)[32]) {
  const int lane = threadIdx.x & 31, p = lane >> 2, c = lane & 3;
  const float *q = psi + (long long)(4 * (f0 + c)) * N + r0 + p;
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int orb = 4 * (f0 + c + 4 * i) + t;
      x[4 * i + t] = orb < n && p < lim ? __ldg(q + (long long)(16 * i + t) * N) : 0.f;
    }
}

// pm[q] = u_{j+q} . psi(point lane >> 2) for q < 4 (from the row k - 1 on: any value).  The quads' sums are
// added in FP32 by a pairwise tree over l (l ^ 16, 8, 4 inside the lane, then l ^ 2, 1 over the four lanes of
// a point): two shuffles per vector for 8 points, where a lane per quad needed 23.
__device__ __forceinline__ void project4(const float *__restrict__ psi, int n, long long N, const float *Ub, long long r0,
                                         int lim, int j, int k, float (&x)[32], float (&pm)[4]) {
  const int c = threadIdx.x & 3, nf = (n + 3) / 4;
  const unsigned full = 0xffffffffu;
  const float4 *u4 = reinterpret_cast<const float4 *>(Ub);
  float acc[4][8];
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[q][i] = 0.f;
  for (int f0 = 0; f0 < nf; f0 += 32) {
    if (nf > 32) load_block(psi, n, N, r0, lim, f0, x);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 *u = u4 + (long long)min(j + q, k - 1) * nf + f0 + c;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 w = f0 + c + 4 * i < nf ? u[4 * i] : make_float4(0.f, 0.f, 0.f, 0.f);
        acc[q][i] += dot4(w, make_float4(x[4 * i], x[4 * i + 1], x[4 * i + 2], x[4 * i + 3]));
      }
    }
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
#pragma unroll
    for (int o = 4; o > 0; o >>= 1)
#pragma unroll
      for (int i = 0; i < o; ++i) acc[q][i] += acc[q][i + o];
    float t = acc[q][0];
    t += __shfl_xor_sync(full, t, 2);
    t += __shfl_xor_sync(full, t, 1);
    pm[q] = t;
  }
}

// End of a block's update (a warp): residuals dr of point lane & 7, up to date with j of k vectors.
__device__ __forceinline__ void store_block(long long *d, const SelArgs &s, long long blk, long long r0, int lim, int j_in,
                                            int j, int k, long long dr, long long mx, long long &best, long long &bi) {
  const int lane = threadIdx.x & 31, p = lane >> 2;
  const bool mine = (lane & 3) == 0 && p < lim;
  if (j != j_in && mine) d[r0 + p] = dr;
  if (lane == 0) {
    s.bmax[blk] = mx;
    s.bcnt[blk] = j;
  }
  if (j == k) {
    if (mine) amax(best, bi, dr, r0 + p);
    if (lane == 0 && mx > 0) atomicMax(s.thr + k, mx);
  }
}

// A block's residuals (point lane >> 2, as stored), count and points, for refresh_loaded.  Residuals and
// counts are read through L2: in the pivot step other CTAs of the pass wrote them.
__device__ __forceinline__ void load_state(const float *__restrict__ psi, int n, long long N, const long long *d,
                                           const SelArgs &s, long long blk, long long &r0, int &lim, int &j,
                                           long long &dr, float (&x)[32]) {
  const int p = (threadIdx.x & 31) >> 2;
  r0 = blk * kBlk;
  lim = (int)min((long long)kBlk, N - r0);
  dr = p < lim ? __ldcg(d + r0 + p) : -1;
  j = __ldcg(s.bcnt + blk);
  if (n <= 128) load_block(psi, n, N, r0, lim, 0, x);
}

// Basis rows j .. j + 7 (rows past `upto` repeat the last one) into a warp's staging buffer, asynchronously;
// quads past the orbitals are zero.
constexpr int kRows = 8;                                  // rows of a buffer
constexpr int kStage = 2 * kRows * 32;                    // float4 per warp: two buffers
constexpr int kStageBytes = 16 * kStage * (kUpdNT / 32);
__device__ __forceinline__ void stage_rows(const float *Ub, int nf, int j, int upto, float4 *buf) {
  const int lane = threadIdx.x & 31;
  const float4 *u4 = reinterpret_cast<const float4 *>(Ub);
#pragma unroll
  for (int q = 0; q < kRows; ++q) {
    const unsigned dst = (unsigned)__cvta_generic_to_shared(buf + q * 32 + lane);
    const float4 *src = u4 + (long long)min(j + q, upto - 1) * nf + (lane < nf ? lane : 0);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(lane < nf ? 16 : 0) : "memory");
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// Applies the basis vectors j .. upto - 1 (upto <= k) to one block (a warp): its residuals lose
// (u_j . psi(r))^2 in order of j.  With `stop` it ends early once every residual is below the largest
// up-to-date one: the residuals only fall, so the block cannot hold the pivot.  A block that gets to k adds
// its maximum to (best, bi) and to the threshold.  Returns the block's new bound.
//   Up to 128 orbitals (MANY = false) the rows of the basis come through the warp's staging buffers, eight ahead of
// their use (loads from L2 one vector at a time took most of a long catch-up).
template <bool MANY>
__device__ __forceinline__ long long refresh_loaded(const float *__restrict__ psi, int n, long long N, long long *d,
                                                    const SelArgs &s, long long blk, long long r0, int lim, int j, int k,
                                                    int upto, bool stop, long long dr, float (&x)[32],
                                                    float4 *stage,
                                                    long long &best, long long &bi) {
  const int j_in = j;
  const long long thr = stop ? __ldcg(s.thr + k) : kNone;
  const float *Ub = static_cast<const float *>(s.Ub);
  long long mx = blk_max(dr);
  if (!MANY) {
    const int c = threadIdx.x & 3, nf = (n + 3) / 4;
    int buf = 0;
    if (j < upto) stage_rows(Ub, nf, j, upto, stage);
    while (j < upto && mx >= thr) {
      if (j + kRows < upto) {
        stage_rows(Ub, nf, j + kRows, upto, stage + (buf ^ 1) * (kRows * 32));
        asm volatile("cp.async.wait_group 1;" ::: "memory");
      } else {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
      }
      __syncwarp();
      const int m = min(kRows, upto - j);
      float pm[kRows];
#pragma unroll
      for (int q = 0; q < kRows; ++q) {
        const float4 *u = stage + (buf * kRows + q) * 32 + c;
        float acc[8];
#pragma unroll
        for (int i = 0; i < 8; ++i)
          acc[i] = dot4(u[4 * i], make_float4(x[4 * i], x[4 * i + 1], x[4 * i + 2], x[4 * i + 3]));
#pragma unroll
        for (int o = 4; o > 0; o >>= 1)
#pragma unroll
          for (int i = 0; i < o; ++i) acc[i] += acc[i + o];
        float t = acc[0];
        t += __shfl_xor_sync(0xffffffffu, t, 2);
        pm[q] = t + __shfl_xor_sync(0xffffffffu, t, 1);
      }
      KeySquare sq[kRows];
#pragma unroll
      for (int q = 0; q < kRows; ++q) sq[q] = key_square(__float_as_uint(pm[q]));
      dr = key_close(key_less_all<kRows>(key_open(dr), sq, m), dr);
      j += m;
      mx = blk_max(dr);
      buf ^= 1;
      __syncwarp();
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncwarp();
  } else {
    while (j < upto && mx >= thr) {
      float pm[4];
      project4(psi, n, N, Ub, r0, lim, j, upto, x, pm);
      const int m = min(4, upto - j);
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (q < m) dr = key_downdate(dr, __float_as_uint(pm[q]));
      j += m;
      mx = blk_max(dr);
    }
  }
  store_block(d, s, blk, r0, lim, j_in, j, k, dr, mx, best, bi);
  return mx;
}
template <bool MANY>
__device__ __forceinline__ long long refresh_block(const float *__restrict__ psi, int n, long long N, long long *d,
                                                   const SelArgs &s, long long blk, int k, int upto, bool stop,
                                                   float4 *stage, long long &best, long long &bi) {
  long long r0, dr;
  int lim, j;
  float x[32];
  load_state(psi, n, N, d, s, blk, r0, lim, j, dr, x);
  return refresh_loaded<MANY>(psi, n, N, d, s, blk, r0, lim, j, k, upto, stop, dr, x, stage, best, bi);
}

// Stored residuals: FP64 values, or the keys of the FP32 selection (residual_key.h)
template <typename T>
struct Resid {
  using type = double;
};
template <>
struct Resid<float> {
  using type = long long;
};

// Pivot step k, run by the whole last block of a pass: the pivot c_k from the block maxima (it
// leaves the candidate set), then u_k = psi(c_k) orthogonalised against u_0..u_{k-1} by classical
// Gram-Schmidt applied twice and normalised, in the working type T.  The basis u_j only steers the
// choice of the pivots (U and Phi are computed from the pivots and Psi alone).  A column whose
// residual is at the rounding level of T (|residual|^2 below kDependent(T) |psi(c_k)|^2) gives
// u_k = 0 and sets *dependent.
template <typename T, bool LAZY, bool MANY>
__device__ void pivot_step(const T *__restrict__ psi, long long si, long long sr, int n, long long N, int nblk,
                           typename Resid<T>::type *__restrict__ d, const SelArgs &s, ScdmSmem<T> &sm,
                           float4 *stage) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int kWarps = kUpdNT / 32;
  using V2 = typename Vec2<T>::type;
  T *u = sm.sel.u, *c = sm.sel.c;
  const T *Ub = static_cast<const T *>(s.Ub);
  const int k = s.k;
  long long best = kNone, bi = N;
  for (int b = tid; b < nblk; b += kUpdNT) amax(best, bi, __ldcg(s.bval + b), __ldcg(s.bidx + b));
  warp_amax(best, bi);
  if (lane == 0) {
    sm.rk[warp] = best;
    sm.ri[warp] = bi;
  }
  __syncthreads();
  if (warp == 0) {
    best = lane < kWarps ? sm.rk[lane] : kNone;
    bi = lane < kWarps ? sm.ri[lane] : N;
    warp_amax(best, bi);
    if (lane == 0) {
      sm.chosen = bi < N ? bi : 0;
      s.piv[k] = (int)sm.chosen;
      d[sm.chosen] = -1;
    }
  }
  __syncthreads();
  const long long cr = sm.chosen;
  // LAZY: the next step's threshold comes from the blocks with the largest bounds, one per warp from its
  // share of the CTAs, brought up to date with u_k at the end of this step.  Away from c_k bounds near the
  // top hardly change, so one of these is the next pivot's block, or close to it in value.  Their points are
  // loaded here, ahead of the basis vector.
  long long seed = N, sr0 = 0;
  int slim = 0, sj = 0;
  long long seed_d = -1;
  float sv[32];
  if constexpr (LAZY) {
    if (k + 1 < n) {
      long long tb = kNone, tbi = N;
      for (int b = warp + kWarps * lane; b < nblk; b += kWarps * 32) amax(tb, tbi, __ldcg(s.tval + b), __ldcg(s.tidx + b));
      warp_amax(tb, tbi);
      seed = __shfl_sync(0xffffffffu, tbi, 0);
      if (seed < N && k + 1 - __ldcg(s.bcnt + seed) > kSeedLag) {
        // too far behind: the best point of the share that this pass brought up to date instead
        tb = kNone;
        tbi = N;
        for (int b = warp + kWarps * lane; b < nblk; b += kWarps * 32) amax(tb, tbi, __ldcg(s.bval + b), __ldcg(s.bidx + b));
        warp_amax(tb, tbi);
        tbi = __shfl_sync(0xffffffffu, tbi, 0);
        seed = tbi < N ? tbi / kBlk : N;
      }
      if (seed < N) load_state(psi, n, N, d, s, seed, sr0, slim, sj, seed_d, sv);
    }
  }
  const int ldu = basis_ld<T>(n), np = ldu / 2;
  T part0 = (T)0;
  for (int i = tid; i < ldu; i += kUpdNT) {
    u[i] = i < n ? psi[(long long)i * si + cr * sr] : (T)0;
    part0 += u[i] * u[i];
  }
  __syncthreads();
  const V2 *u2 = reinterpret_cast<const V2 *>(u);
  const int S = np <= 64 ? 4 : (np <= 128 ? 2 : 1);  // row slices of the u update (S ldu <= 1024)
  for (int pass = 0; pass < 2; ++pass) {
    // c_j = u_j . u: 16 lanes per row over consecutive double2, four rows per thread per round
    {
      const int seg = tid & 15, rg = tid >> 4;
      for (int j0 = 0; j0 < k; j0 += 64) {  // same trip count for every thread of the block
        const V2 *q[4];
        T a[4] = {(T)0, (T)0, (T)0, (T)0};
#pragma unroll
        for (int t = 0; t < 4; ++t)
          q[t] = reinterpret_cast<const V2 *>(Ub + (long long)min(j0 + rg + 16 * t, k - 1) * ldu);
#pragma unroll 2
        for (int p = seg; p < np; p += 16) {
          const V2 w = u2[p];
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            const V2 x = q[t][p];
            a[t] += x.x * w.x + x.y * w.y;
          }
        }
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          for (int o = 8; o > 0; o >>= 1) a[t] += __shfl_xor_sync(0xffffffffu, a[t], o);
          if (seg == 0 && j0 + rg + 16 * t < k) c[j0 + rg + 16 * t] = a[t];
        }
      }
    }
    __syncthreads();
    // u -= sum_j c_j u_j: S slices of the rows x (256 / S) threads over pairs of u; the slices'
    // partial sums are added in a fixed order
    {
      const int tps = kUpdNT / S, sl = tid / tps, e0 = tid % tps;
      for (int p = e0; p < np; p += tps) {
        T ax = (T)0, ay = (T)0;
#pragma unroll 8
        for (int j = sl; j < k; j += S) {
          const V2 x = reinterpret_cast<const V2 *>(Ub + (long long)j * ldu)[p];
          const T cj = c[j];
          ax += cj * x.x;
          ay += cj * x.y;
        }
        sm.sel.red2[sl * ldu + 2 * p] = ax;
        sm.sel.red2[sl * ldu + 2 * p + 1] = ay;
      }
    }
    __syncthreads();
    for (int i = tid; i < n; i += kUpdNT) {
      T t = (T)0;
      for (int s2 = 0; s2 < S; ++s2) t += sm.sel.red2[s2 * ldu + i];
      u[i] -= t;
    }
    __syncthreads();
  }
  T part = (T)0;
  for (int i = tid; i < n; i += kUpdNT) part += u[i] * u[i];
  for (int o = 16; o > 0; o >>= 1) {
    part += __shfl_down_sync(0xffffffffu, part, o);
    part0 += __shfl_down_sync(0xffffffffu, part0, o);
  }
  if (lane == 0) {
    sm.rv[warp] = (double)part;
    sm.rv0[warp] = (double)part0;
  }
  __syncthreads();
  if (tid == 0) {
    double t = 0.0, t0 = 0.0;
    for (int w = 0; w < kWarps; ++w) {
      t += sm.rv[w];
      t0 += sm.rv0[w];
    }
    // the chosen column lies in the span of the earlier ones (to rounding): Psi has rank < n
    const bool dep = !(t > (sizeof(T) == 4 ? kDependent32 : kDependent) * t0);
    if (dep) *s.dependent = 1;
    c[0] = dep ? (T)0 : (T)(1.0 / sqrt(t));
  }
  __syncthreads();
  const T inv = c[0];
  T *Uw = static_cast<T *>(s.Ub);
  for (int i = tid; i < ldu; i += kUpdNT) Uw[(long long)k * ldu + i] = i < n ? u[i] * inv : (T)0;
  if constexpr (LAZY) {
    if (k + 1 < n) {
      __threadfence();
      __syncthreads();  // u_k for the CTA, in L2
      if (seed < N) {
        if (sr0 + (lane >> 2) == cr) seed_d = -1;
        refresh_loaded<MANY>(psi, n, N, d, s, seed, sr0, slim, sj, k + 1, k + 1, true, seed_d, sv,
                             stage + warp * kStage, best, bi);
      }
    }
  }
}

// End of a pass for one block: publish the block maximum; the last block to publish takes the
// pivot step and resets the counter for the next pass (true for that block).  Orbital i at point r is psi[i si + r sr].
template <typename T, bool LAZY, bool MANY = false>
__device__ bool finish_pass(long long best, long long bi, long long top, long long ti, long long start,
                            const T *__restrict__ psi, long long si, long long sr, int n, long long N,
                            typename Resid<T>::type *__restrict__ d, const SelArgs &s, ScdmSmem<T> &sm, float4 *stage) {
  const int tid = threadIdx.x;
  constexpr int kWarps = kUpdNT / 32;
  warp_amax(best, bi);
  if constexpr (LAZY) warp_amax(top, ti);
  if ((tid & 31) == 0) {
    sm.rk[tid >> 5] = best;
    sm.ri[tid >> 5] = bi;
    sm.tk[tid >> 5] = top;
    sm.ti[tid >> 5] = ti;
  }
  __syncthreads();
  if (tid < 32) {
    best = tid < kWarps ? sm.rk[tid] : kNone;
    bi = tid < kWarps ? sm.ri[tid] : N;
    warp_amax(best, bi);
    if constexpr (LAZY) {
      top = tid < kWarps ? sm.tk[tid] : kNone;
      ti = tid < kWarps ? sm.ti[tid] : N;
      warp_amax(top, ti);
      if (tid == 0) {
        s.tval[blockIdx.x] = top;
        s.tidx[blockIdx.x] = ti;
        sm.top = ti;
        if (s.k > 0) atomicMax(s.work, (int)min(clock64() - start, 1LL << 30));
      }
    }
    if (tid == 0) {
      s.bval[blockIdx.x] = best;
      s.bidx[blockIdx.x] = bi;
      __threadfence();  // the maximum (and this block's residual norms) before the count
      sm.last = atomicAdd(s.count, 1u) == gridDim.x - 1;
    }
  }
  __syncthreads();
  if (!sm.last) return false;
  __threadfence();
  if (tid == kUpdNT - 1) {  // in the shadow of the pivot step's first loads
    *s.count = 0u;
    if constexpr (LAZY) {
      sm.leave = 0;
      if (s.k > 0) {
        const long long x = max(0ll, __ldcg(s.excess) + __ldcg(s.work) - s.full_cost);
        *s.excess = x;
        *s.work = 0;
        // not past a quarter of the steps: what does not localise shows early, and the blocks' catch-up grows with k
        sm.leave = (x > s.leave_cost && 4 * s.k < n) || s.k == s.leave_step;
      }
    }
  }
  pivot_step<T, LAZY, MANY>(psi, si, sr, n, N, gridDim.x, d, s, sm, stage);
  if constexpr (LAZY) {
    if (sm.leave) {
      __syncthreads();  // the pivot step's own entry of thr
      for (int i = s.k + 1 + tid; i <= n; i += kUpdNT) s.thr[i] = kLeft;
      if (tid == 0) *s.left = s.k + 1;
    }
  }
  return true;
}

// One selection pass of the FP64 form (one point per thread per iteration):
//   NORM: d[r] = |psi(r)|^2 (the start);
//   else: d[r] -= (u_{k-1} . psi(r))^2 for every column still a candidate (d[r] >= 0), u_{k-1} = row
//         k-1 of Ub.
// Products are summed in T in chunks of kChunk, the chunks in FP64.
template <typename T, bool NORM>
__global__ void __launch_bounds__(kUpdNT) scdm_pass_kernel(const T *__restrict__ psi, int n, long long N,
                                                           double *__restrict__ d, SelArgs s) {
  __shared__ ScdmSmem<T> sm;
  if (!NORM)
    for (int i = threadIdx.x; i < n; i += kUpdNT)
      sm.us[i] = static_cast<const T *>(s.Ub)[(long long)(s.k - 1) * basis_ld<T>(n) + i];
  __syncthreads();
  long long best = kNone, bi = N;
  for (long long r = blockIdx.x * (long long)kUpdNT + threadIdx.x; r < N; r += (long long)gridDim.x * kUpdNT) {
    double dr = NORM ? 0.0 : d[r];
    if (NORM || dr >= 0.0) {
      double p = 0.0;
      for (int i0 = 0; i0 < n; i0 += kChunk) {
        const int i1 = min(n, i0 + kChunk);
        T part = (T)0;
        for (int i = i0; i < i1; ++i) {
          const T v = psi[(long long)i * N + r];
          part += (NORM ? v : sm.us[i]) * v;
        }
        p += (double)part;
      }
      dr = NORM ? p : fmax(dr - p * p, 0.0);
      d[r] = dr;
    }
    amax(best, bi, res_key(dr), r);
  }
  finish_pass<T, false>(best, bi, kNone, N, 0, psi, N, 1, n, N, d, s, sm, nullptr);
}

// The FP32 selection.  The residual norms only fall from step to step, so the residual a point had when
// it was last brought up to date bounds its present one: a step has to look only at the blocks whose
// bound reaches the largest up-to-date residual.  For 128 orbitals on 96^3 that is 27,000 block visits in
// all 128 steps, a quarter of the blocks once, where passes over every point (the plain greedy selection)
// read Psi 128 times: 12.3 ms per call, bound by HBM at 0.8 of its bandwidth; now 4.1-4.9 ms, most of it the
// chain of the 127 steps (launch, look at the bounds, visits, pivot step: about 30 us each).
//   Orbitals that no rotation localises (plane waves of a metal) flatten the residuals, and the visits of a step
// then cost more than a pass over every point: the steps measure themselves, and when the last ones have lost
// about what changing over costs, the rest are passes over every point.  64 such orbitals on 72^3: 5.8 ms on
// bounds alone, 3.4 with passes alone, 3.8 with the change; 200 on 64^3: 32, 13.4 and 14.2 ms.
//   Every residual goes through the same operations in the same order in all of these, so the pivots are the
// same whichever way a step goes.

// d[r] = |psi(r)|^2 (FP32), one point per thread; the sum has the order of refresh_block's (32 partial sums over
// orbitals 4 l .. 4 l + 3 (+ 128 f), then the pairwise tree).
template <bool LAZY, bool MANY>
__global__ void __launch_bounds__(kUpdNT) scdm_norm_kernel(const float *__restrict__ psi, int n, long long N,
                                                           long long *__restrict__ d, SelArgs s) {
  __shared__ __align__(16) ScdmSmem<float> sm;
  extern __shared__ float4 stage_all[];  // kStage per warp
  const int nf = (n + 3) / 4;
  long long best = kNone, bi = N;
  const long long step = (long long)gridDim.x * kUpdNT;
  for (long long r0 = blockIdx.x * (long long)kUpdNT; r0 < N; r0 += step) {  // same trip count for the CTA
    const long long r = r0 + threadIdx.x;
    float acc[32];
#pragma unroll
    for (int l = 0; l < 32; ++l) acc[l] = 0.f;
    for (int f0 = 0; f0 < nf; f0 += 32) {
#pragma unroll
      for (int l = 0; l < 32; ++l) {
        float x[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const int i = 4 * (f0 + l) + t;
          x[t] = (i < n && r < N) ? __ldcs(psi + (long long)i * N + r) : 0.f;
        }
        const float4 v = make_float4(x[0], x[1], x[2], x[3]);
        acc[l] += dot4(v, v);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int l = 0; l < o; ++l) acc[l] += acc[l + o];
    const long long dr = r < N ? key_of_bits(__float_as_uint(acc[0])) : -1;
    long long mx = dr;  // over the 8 lanes of a block
    for (int o = kBlk / 2; o > 0; o >>= 1) {
      const long long v = __shfl_xor_sync(0xffffffffu, mx, o);
      mx = v > mx ? v : mx;
    }
    if (r < N) {
      d[r] = dr;
      amax(best, bi, dr, r);
    }
    if (LAZY && r < N && r % kBlk == 0) {
      s.bmax[r / kBlk] = mx;
      s.bcnt[r / kBlk] = 0;
    }
  }
  finish_pass<float, LAZY, MANY>(best, bi, best, bi < N ? bi / kBlk : N, 0, psi, N, 1, n, N, d, s, sm, stage_all);
}

// Few points (see launch_scdm): step k >= 1 over every point, one per thread.  u_{k-1} . psi(r) is summed in the order
// of refresh_block's.
__global__ void __launch_bounds__(kUpdNT) scdm_full_kernel(const float *__restrict__ psi, int n, long long N,
                                                           long long *__restrict__ d, SelArgs s) {
  __shared__ __align__(16) ScdmSmem<float> sm;
  const int tid = threadIdx.x, nf = (n + 3) / 4;
  for (int i = tid; i < (nf + 31) / 32 * 128; i += kUpdNT)
    sm.us[i] = i < 4 * nf ? static_cast<const float *>(s.Ub)[(long long)(s.k - 1) * (4 * nf) + i] : 0.f;
  __syncthreads();
  const float4 *u4 = reinterpret_cast<const float4 *>(sm.us);
  long long best = kNone, bi = N;
  for (long long r = blockIdx.x * (long long)kUpdNT + tid; r < N; r += (long long)gridDim.x * kUpdNT) {
    float acc[32];
#pragma unroll
    for (int l = 0; l < 32; ++l) acc[l] = 0.f;
    for (int f0 = 0; f0 < nf; f0 += 32) {
#pragma unroll
      for (int l8 = 0; l8 < 32; l8 += 8) {
        if (f0 + l8 >= nf) break;
#pragma unroll
        for (int l = l8; l < l8 + 8; ++l) {
          float x[4];
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            const int i = 4 * (f0 + l) + t;
            x[t] = i < n ? __ldg(psi + (long long)i * N + r) : 0.f;
          }
          acc[l] += dot4(u4[f0 + l], make_float4(x[0], x[1], x[2], x[3]));
        }
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int l = 0; l < o; ++l) acc[l] += acc[l + o];
    const long long dr = key_downdate(d[r], __float_as_uint(acc[0]));
    d[r] = dr;
    amax(best, bi, dr, r);
  }
  finish_pass<float, false>(best, bi, kNone, N, 0, psi, N, 1, n, N, d, s, sm, nullptr);
}

// Point-major copy pt[r][i] = psi[i][r] for i < n, zero for n <= i < ld: 32 points x 32 orbitals per block.
__global__ void scdm_points_copy_kernel(const float *__restrict__ psi, int n, long long N, int ld,
                                        float *__restrict__ pt) {
  __shared__ float tile[32][33];
  const long long r0 = blockIdx.x * 32ll;
  const int i0 = blockIdx.y * 32;
  for (int y = threadIdx.y; y < 32; y += 8) {
    const int i = i0 + y;
    tile[y][threadIdx.x] = i < n && r0 + threadIdx.x < N ? psi[(long long)i * N + r0 + threadIdx.x] : 0.f;
  }
  __syncthreads();
  for (int y = threadIdx.y; y < 32; y += 8)
    if (r0 + y < N && i0 + threadIdx.x < ld) pt[(r0 + y) * ld + i0 + threadIdx.x] = tile[threadIdx.x][y];
}

// Every block up to date with u_0 .. u_{k-2}.
template <bool MANY>
__global__ void __launch_bounds__(kUpdNT, 2) scdm_catch_up_kernel(const float *__restrict__ psi, int n, long long N,
                                                                  long long *__restrict__ d, SelArgs s) {
  extern __shared__ float4 stage_all[];  // kStage per warp
  const long long nb = (N + kBlk - 1) / kBlk, nwarps = (long long)gridDim.x * (kUpdNT / 32);
  long long best = kNone, bi = N;
  for (long long b = (long long)blockIdx.x * (kUpdNT / 32) + (threadIdx.x >> 5); b < nb; b += nwarps)
    if (s.bcnt[b] < s.k - 1)
      refresh_block<MANY>(psi, n, N, d, s, b, s.k, s.k - 1, false, stage_all + (threadIdx.x >> 5) * kStage, best, bi);
}

// Step k >= 1 over every point, from the point-major copy pt.  Every warp takes an equal share of the blocks, 32
// points at a time in four blocks: lane l loads the float4 of orbitals 4 l .. 4 l + 3 (+ 128 f) of a block's points
// (whole rows; 128-byte pieces of 128 rows of Psi run at 2.1 TB/s), the lanes' sums are added by refresh_block's
// pairwise tree, and lane l keeps point l of the 32.  In the first such step (FIRST) the blocks that the last
// pivot step looked at have u_{k-1} already.
template <bool FIRST>
__global__ void __launch_bounds__(kUpdNT, 3) scdm_points_kernel(const float *__restrict__ psi,
                                                                const float *__restrict__ pt, int n, long long N,
                                                                long long *__restrict__ d, SelArgs s) {
  __shared__ __align__(16) ScdmSmem<float> sm;
  const int tid = threadIdx.x, lane = tid & 31, nf = (n + 3) / 4, k = s.k;
  const unsigned full = 0xffffffffu;
  const float4 *ub = static_cast<const float4 *>(s.Ub), *pt4 = reinterpret_cast<const float4 *>(pt);
  for (int i = tid; i < nf; i += kUpdNT) reinterpret_cast<float4 *>(sm.us)[i] = ub[(long long)(k - 1) * nf + i];
  __syncthreads();
  const float4 *us = reinterpret_cast<const float4 *>(sm.us);
  const long long nb = (N + kBlk - 1) / kBlk, nwarps = (long long)gridDim.x * (kUpdNT / 32);
  const long long w = (long long)blockIdx.x * (kUpdNT / 32) + (tid >> 5);
  const long long ra = nb * w / nwarps * kBlk, rb = min(N, nb * (w + 1) / nwarps * kBlk);
  long long best = kNone, bi = N;
  for (long long r0 = ra; r0 < rb; r0 += 32) {
    const long long r = r0 + lane;
    long long dr = r < rb ? d[r] : -1;
    const bool done = FIRST && r < rb && s.bcnt[r / kBlk] == k;
    float mine = 0.f;
#pragma unroll 1
    for (int grp = 0; grp < 4; ++grp) {
      const long long rg = r0 + kBlk * grp;
      float acc[kBlk] = {};
#pragma unroll 1
      for (int f0 = 0; f0 < nf; f0 += 32) {
        const int f = f0 + lane, lim = f < nf ? (int)min((long long)kBlk, rb - rg) : 0;
        const float4 uu = f < nf ? us[f] : make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 *base = pt4 + rg * nf + f;
        float4 v[kBlk];
#pragma unroll
        for (int p = 0; p < kBlk; ++p) v[p] = p < lim ? __ldcs(base + p * nf) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int p = 0; p < kBlk; ++p) acc[p] += dot4(uu, v[p]);
      }
#pragma unroll
      for (int p = 0; p < kBlk; ++p) {
        acc[p] += __shfl_xor_sync(full, acc[p], 16);
        acc[p] += __shfl_xor_sync(full, acc[p], 8);
      }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int p = 0; p < o; ++p) {
          const float send = up ? acc[p] : acc[p + o], keep = up ? acc[p + o] : acc[p];
          acc[p] = keep + __shfl_xor_sync(full, send, o);
        }
      }
      if ((lane >> 3) == grp) mine = acc[0];
    }
    if (!done) dr = key_downdate(dr, __float_as_uint(mine));
    if (r < rb) {
      d[r] = dr;
      amax(best, bi, dr, r);
    }
  }
  finish_pass<float, false>(best, bi, kNone, N, 0, psi, N, 1, n, N, d, s, sm, nullptr);
}

// Step k >= 1: the warps look through the blocks' bounds, 32 at a time (neighbouring blocks belong to
// different warps), and bring those that reach the threshold up to date.
//   While the last CTA takes the pivot step, the others move blocks forward whose bound is not far below the
// threshold and which a later step will need: without it the longest catch-up of a step was 57 vectors on
// average (128 orbitals on 96^3), a chain of dependent FP64 updates (8.0 ms per call).  A CTA leaves out the
// block with its largest bound, which the pivot step may be working on.
//   One CTA per SM: a step is a chain of latencies, and held to 128 registers for two it spills on it (ms per
// call with two / one: 128 orbitals on 96^3 5.4 / 4.9, 256 on 64^3 17.4 / 14.5).
constexpr int kAhead = 8;      // vectors per step and block
constexpr int kAheadMost = 4;  // blocks per warp and step
template <bool MANY>
__global__ void __launch_bounds__(kUpdNT, 1) scdm_step_kernel(const float *__restrict__ psi, int n, long long N,
                                                              long long *__restrict__ d, SelArgs s) {
  __shared__ __align__(16) ScdmSmem<float> sm;
  extern __shared__ float4 stage_all[];  // kStage per warp
  float4 *stage = stage_all + (threadIdx.x >> 5) * kStage;
  const int lane = threadIdx.x & 31;
  const unsigned full = 0xffffffffu;
  const long long start = clock64(), nb = (N + kBlk - 1) / kBlk;
  const long long nwarps = (long long)gridDim.x * (kUpdNT / 32);
  const long long w = (long long)blockIdx.x * (kUpdNT / 32) + (threadIdx.x >> 5);
  long long thr = __ldcg(s.thr + s.k);
  const long long soon = key_somewhat_below(thr);
  long long best = kNone, bi = N, top = kNone, ti = N;
  if (thr == kLeft) return;
  for (long long b0 = w; b0 < nb; b0 += 32 * nwarps) {
    const long long b = b0 + lane * nwarps;
    long long bound = b < nb ? s.bmax[b] : kNone;
    unsigned left = __ballot_sync(full, bound >= 0 && bound >= thr);
    while (left) {
      const int src = __ffs(left) - 1;
      left &= left - 1;
      const long long blk = __shfl_sync(full, b, src);
      const long long mx = refresh_block<MANY>(psi, n, N, d, s, blk, s.k, s.k, true, stage, best, bi);
      if (lane == src) bound = mx;
      if (left) {
        thr = __ldcg(s.thr + s.k);
        left &= __ballot_sync(full, bound >= thr);
      }
    }
    amax(top, ti, bound, b);
  }
  if (finish_pass<float, true, MANY>(best, bi, top, ti, start, psi, N, 1, n, N, d, s, sm, stage_all)) return;
  int most = kAheadMost;
  for (long long b0 = w; b0 < nb && most > 0; b0 += 32 * nwarps) {
    const long long b = b0 + lane * nwarps;
    const long long bound = b < nb ? s.bmax[b] : kNone;
    const int cnt = bound >= 0 && bound >= soon && b != sm.top ? s.bcnt[b] : s.k;
    for (unsigned ahead = __ballot_sync(full, cnt < s.k); ahead && most > 0; ahead &= ahead - 1, --most) {
      const int src = __ffs(ahead) - 1;
      const int upto = min(s.k, __shfl_sync(full, cnt, src) + kAhead);
      refresh_block<MANY>(psi, n, N, d, s, __shfl_sync(full, b, src), s.k, upto, false, stage, best, bi);
    }
  }
}

// sum_l a[l sa] b[l sb] over l < n, in eight interleaved partial sums: with one output per thread these
// products wait for the FP64 pipe's latency (four sums: 18 us per 128 x 128 product, its issue rate is 4 us)
__device__ __forceinline__ double strided_dot(const double *__restrict__ a, long long sa, const double *__restrict__ b,
                                              long long sb, int n) {
  double s[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  int l = 0;
  for (; l + 8 <= n; l += 8) {
#pragma unroll
    for (int q = 0; q < 8; ++q) s[q] += a[(l + q) * sa] * b[(l + q) * sb];
  }
  for (; l < n; ++l) s[0] += a[l * sa] * b[l * sb];
  return ((s[0] + s[1]) + (s[2] + s[3])) + ((s[4] + s[5]) + (s[6] + s[7]));
}

// M[i][j] = psi_i(c_j)
template <typename T>
__global__ void scdm_gather_kernel(const T *__restrict__ psi, int n, long long N, const int *__restrict__ piv,
                                   double *__restrict__ M) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n * n) return;
  const int i = e / n, j = e % n;
  M[e] = (double)psi[(long long)i * N + piv[j]];
}

// S = M^T M
__global__ void gram_t_kernel(const double *__restrict__ M, int n, double *__restrict__ S) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n * n) return;
  const int i = e / n, j = e % n;
  double s = strided_dot(M + i, n, M + j, n, n);
  S[e] = s;
}

// f = |S|_F (one CTA of 1024 threads)
__global__ void __launch_bounds__(1024) frob_kernel(const double *__restrict__ S, int n, double *__restrict__ f) {
  __shared__ double rv[32];
  double p0 = 0.0, p1 = 0.0;
  for (int e = threadIdx.x; e < n * n; e += 2048) {
    p0 += S[e] * S[e];
    if (e + 1024 < n * n) p1 += S[e + 1024] * S[e + 1024];
  }
  double part = p0 + p1;
  for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o);
  if ((threadIdx.x & 31) == 0) rv[threadIdx.x >> 5] = part;
  __syncthreads();
  if (threadIdx.x < 32) {
    double s = rv[threadIdx.x];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) *f = sqrt(s);
  }
}

// Y0 = S / f, Z0 = I
__global__ void ns_start_kernel(const double *__restrict__ S, int n, const double *__restrict__ f,
                                double *__restrict__ Y, double *__restrict__ Z) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n * n) return;
  const double inv = *f > 0.0 ? 1.0 / *f : 0.0;
  Y[e] = S[e] * inv;
  Z[e] = (e / n == e % n) ? 1.0 : 0.0;
}

// Whether iteration `it` is skipped: an earlier one reached kNsStop, or stopped converging at the
// rounding level (below 1e-8 and not even a quarter of its predecessor, where quadratic convergence
// would have squared it).  Skipped iterations leave dev[it] = 0, so the later ones skip as well.
__device__ __forceinline__ bool ns_done(const double *__restrict__ dev, int it) {
  if (it == 0) return false;
  const double x = dev[it - 1];
  if (x < kNsStop) return true;
  return it >= 2 && x < 1e-8 && x > 0.25 * dev[it - 2];
}

// Iteration `it`: T = (3 I - Z Y) / 2 and dev[it] = max |T - I|, unless ns_done.
__global__ void ns_t_kernel(const double *__restrict__ Y, const double *__restrict__ Z, int n,
                            double *__restrict__ Tm, double *__restrict__ dev, int it) {
  if (ns_done(dev, it)) return;
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  double x = 0.0;
  if (e < n * n) {
    const int i = e / n, j = e % n;
    const double s = strided_dot(Z + (long long)i * n, 1, Y + j, n, n);
    const double t = -0.5 * s + (i == j ? 1.5 : 0.0);
    Tm[e] = t;
    x = fabs(t - (i == j ? 1.0 : 0.0));
    if (!(x == x)) x = 1e300;  // NaN: never converged
  }
  for (int o = 16; o > 0; o >>= 1) x = fmax(x, __shfl_down_sync(0xffffffffu, x, o));
  // non-negative doubles order like their bit patterns
  if ((threadIdx.x & 31) == 0 && x > 0.0)
    atomicMax(reinterpret_cast<unsigned long long *>(dev + it), (unsigned long long)__double_as_longlong(x));
}

// Y' = Y T and Z' = T Z (threads [0, n^2) and [n^2, 2 n^2)); a skipped iteration copies Y and Z.
__global__ void ns_yz_kernel(const double *__restrict__ Y, const double *__restrict__ Z,
                             const double *__restrict__ Tm, int n, double *__restrict__ Y2, double *__restrict__ Z2,
                             const double *__restrict__ dev, int it) {
  const bool skip = ns_done(dev, it);
  const int nn = n * n;
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= 2 * nn) return;
  const bool isz = e >= nn;
  const int f = isz ? e - nn : e;
  if (skip) {
    (isz ? Z2 : Y2)[f] = (isz ? Z : Y)[f];
    return;
  }
  const int i = f / n, j = f % n;
  double s = 0.0;
  if (!isz)
    s = strided_dot(Y + (long long)i * n, 1, Tm + j, n, n);
  else
    s = strided_dot(Tm + (long long)i * n, 1, Z + j, n, n);
  (isz ? Z2 : Y2)[f] = s;
}

// U = M Z / sqrt(f) (Z = (S/f)^{-1/2}) in FP64, and its transpose in the working type
template <typename T>
__global__ void scdm_factor_kernel(const double *__restrict__ M, const double *__restrict__ Z, int n,
                                   const double *__restrict__ f, double *__restrict__ U, T *__restrict__ Ut) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n * n) return;
  const int i = e / n, j = e % n;
  double s = strided_dot(M + (long long)i * n, 1, Z + j, n, n);
  s /= sqrt(*f);
  U[e] = s;
  Ut[(long long)j * n + i] = (T)s;
}

struct Layout {
  size_t d, bval, bidx, tval, tidx, Ub, M, S, Y0, Y1, Z0, Z1, Tm, U, Ut, f, dev, piv, dependent, count;
  size_t bmax, bcnt, thr, work, excess, left, total;
};

Layout layout(int n, long long N, size_t elem) {
  Layout L{};
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t at = off;
    off += (bytes + 255) / 256 * 256;
    return at;
  };
  const size_t nn = (size_t)n * n;
  L.d = take(sizeof(double) * (size_t)N);
  L.bval = take(sizeof(long long) * kUpdBlocks);
  L.bidx = take(sizeof(long long) * kUpdBlocks);
  L.tval = take(sizeof(long long) * kUpdBlocks);
  L.tidx = take(sizeof(long long) * kUpdBlocks);
  L.Ub = take(elem * (size_t)n * (n + 3));
  L.M = take(sizeof(double) * nn);
  L.S = take(sizeof(double) * nn);
  L.Y0 = take(sizeof(double) * nn);
  L.Y1 = take(sizeof(double) * nn);
  L.Z0 = take(sizeof(double) * nn);
  L.Z1 = take(sizeof(double) * nn);
  L.Tm = take(sizeof(double) * nn);
  L.U = take(sizeof(double) * nn);
  L.Ut = take(elem * nn);
  L.f = take(sizeof(double));
  L.dev = take(sizeof(double) * kNsMax);
  L.piv = take(sizeof(int) * (size_t)n);
  L.dependent = take(sizeof(int));
  L.count = take(sizeof(unsigned int));
  // FP32: the block bounds and the steps' thresholds
  const size_t nb = elem == 4 ? ((size_t)N + kBlk - 1) / kBlk : 0;
  L.bmax = take(sizeof(long long) * nb);
  L.bcnt = take(sizeof(int) * nb);
  L.thr = take(sizeof(long long) * (n + 1));
  L.work = take(sizeof(int));
  L.excess = take(sizeof(long long));
  L.left = take(sizeof(int));
  L.total = off;
  return L;
}

}  // namespace

int scdm_max_iterations() { return kNsMax; }

static int env_value(const char *name, int dflt) {
  const char *v = std::getenv(name);
  return v && *v ? std::atoi(v) : dflt;
}

size_t scdm_workspace_bytes(int n, long long N, size_t elem) { return layout(n, N, elem).total; }

template <typename T>
cudaError_t launch_scdm(const T *psi, int n, long long N, void *ws, cudaStream_t st, long *launches, ScdmResult *res) {
  const Layout L = layout(n, N, sizeof(T));
  char *w = static_cast<char *>(ws);
  auto *d = reinterpret_cast<typename Resid<T>::type *>(w + L.d);
  long long *bval = reinterpret_cast<long long *>(w + L.bval);
  long long *bidx = reinterpret_cast<long long *>(w + L.bidx);
  void *Ub = w + L.Ub;
  double *M = reinterpret_cast<double *>(w + L.M);
  double *S = reinterpret_cast<double *>(w + L.S);
  double *Y[2] = {reinterpret_cast<double *>(w + L.Y0), reinterpret_cast<double *>(w + L.Y1)};
  double *Z[2] = {reinterpret_cast<double *>(w + L.Z0), reinterpret_cast<double *>(w + L.Z1)};
  double *Tm = reinterpret_cast<double *>(w + L.Tm);
  double *f = reinterpret_cast<double *>(w + L.f);
  unsigned int *count = reinterpret_cast<unsigned int *>(w + L.count);
  res->piv = reinterpret_cast<int *>(w + L.piv);
  res->U = reinterpret_cast<double *>(w + L.U);
  res->Ut = w + L.Ut;
  res->dev = reinterpret_cast<double *>(w + L.dev);
  res->dependent = reinterpret_cast<int *>(w + L.dependent);
  cudaError_t e = cudaMemsetAsync(res->dev, 0, sizeof(double) * kNsMax, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(res->dependent, 0, sizeof(int), st);
  if (e != cudaSuccess) return e;
  // column selection: n passes; the last block of each pass takes the pivot step
  SelArgs sa{bval, bidx, count, Ub, res->piv, res->dependent, 0, reinterpret_cast<long long *>(w + L.tval),
             reinterpret_cast<long long *>(w + L.tidx), reinterpret_cast<long long *>(w + L.bmax),
             reinterpret_cast<int *>(w + L.bcnt), reinterpret_cast<long long *>(w + L.thr),
             reinterpret_cast<int *>(w + L.work), reinterpret_cast<long long *>(w + L.excess),
             reinterpret_cast<int *>(w + L.left), 0, 0, 0};
  int dev = 0, sms = 0;
  e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaMemsetAsync(count, 0, sizeof(unsigned int), st);
  if (e != cudaSuccess) return e;
  // at most one resident wave of blocks, with at least `least` points each
  auto blocks = [&](auto kernel, size_t smem, long long least, unsigned *grid) {
    int per_sm = 0;
    // shared memory above 48 KB, asked for once per call (a driver call of a microsecond)
    cudaError_t q = cudaSuccess;
    if (smem) q = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (q == cudaSuccess) q = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kUpdNT, smem);
    *grid = (unsigned)std::max<long long>(1, std::min({(long long)std::max(per_sm, 1) * sms, (long long)kUpdBlocks,
                                                       (N + least - 1) / least}));
    return q;
  };
  unsigned first = 1, next = 1;
  auto steps = [&](auto kernel, size_t smem, int k0, int k1) {
    for (sa.k = k0; sa.k < k1; ++sa.k) kernel<<<next, kUpdNT, smem, st>>>(psi, n, N, d, sa);
    return cudaGetLastError();
  };
  if constexpr (sizeof(T) == 8) {
    e = blocks(scdm_pass_kernel<T, true>, 0, kUpdNT, &first);
    if (e == cudaSuccess) e = blocks(scdm_pass_kernel<T, false>, 0, kUpdNT, &next);
    if (e != cudaSuccess) return e;
    scdm_pass_kernel<T, true><<<first, kUpdNT, 0, st>>>(psi, n, N, d, sa);
    e = steps(scdm_pass_kernel<T, false>, 0, 1, n);
  } else if (4.0 * n * N < 1e6 * env_value("ACE_SCDM_BOUNDS_MB", 60)) {
    // Psi stays in L2 and a pass over every point is cheaper than the bounds (ms per call, with them / without:
    // 64 orbitals on 48^3 1.9 / 1.65, 32 on 64^3 1.35 / 1.09; from 60 MB on the bounds win: 64 on 64^3 2.01 / 2.10,
    // on 72^3 1.97 / 3.2)
    e = blocks(scdm_norm_kernel<false, false>, 0, kUpdNT, &first);
    if (e == cudaSuccess) e = blocks(scdm_full_kernel, 0, kUpdNT, &next);
    if (e != cudaSuccess) return e;
    scdm_norm_kernel<false, false><<<first, kUpdNT, 0, st>>>(psi, n, N, d, sa);
    e = steps(scdm_full_kernel, 0, 1, n);
  } else {
    // a pass over every point reads Psi at about 6.5 TB/s (at 1.9 GHz); leaving takes the point-major copy, the
    // vectors that the blocks miss, about three passes' time
    sa.full_cost = (int)std::min(5e8, 4.0 * n * N / 3400.0);
    sa.leave_cost = 3 * sa.full_cost + 114000;
    sa.leave_step = env_value("ACE_SCDM_LEAVE_STEP", 0);
    // thresholds, clocks and the step of leaving (neighbours in the workspace)
    e = cudaMemsetAsync(sa.thr, 0, L.total - L.thr, st);
    const auto catch_up = n > 128 ? scdm_catch_up_kernel<true> : scdm_catch_up_kernel<false>;
    const auto norm = n > 128 ? scdm_norm_kernel<true, true> : scdm_norm_kernel<true, false>;
    const auto step = n > 128 ? scdm_step_kernel<true> : scdm_step_kernel<false>;
    if (e == cudaSuccess) e = blocks(norm, kStageBytes, kUpdNT, &first);
    if (e == cudaSuccess) e = blocks(catch_up, kStageBytes, kUpdNT, &next);
    if (e == cudaSuccess) e = blocks(step, kStageBytes, kBlk * kUpdNT, &next);  // a block per lane
    if (e != cudaSuccess) return e;
    norm<<<first, kUpdNT, kStageBytes, st>>>(psi, n, N, d, sa);
    // the host looks every 64 steps whether the steps over bounds were left (each look idles the device for
    // about 15 us, a step that returns at once takes 2.5)
    int left = 0;
    for (int k = 1; k < n && left == 0; k += 64) {
      e = steps(step, kStageBytes, k, std::min(n, k + 64));
      if (e == cudaSuccess) e = cudaMemcpyAsync(&left, sa.left, sizeof(int), cudaMemcpyDeviceToHost, st);
      if (e == cudaSuccess) e = cudaStreamSynchronize(st);
      if (e != cudaSuccess) return e;
    }
    if (left > 0 && left < n) {
      const int ld = basis_ld<float>(n);
      float *pt = nullptr;
      e = cudaMallocAsync(&pt, sizeof(float) * (size_t)N * ld, st);
      if (e != cudaSuccess) return e;
      const dim3 tiles((unsigned)((N + 31) / 32), (unsigned)((ld + 31) / 32));
      scdm_points_copy_kernel<<<tiles, dim3(32, 8), 0, st>>>(psi, n, N, ld, pt);
      sa.k = left;
      catch_up<<<next, kUpdNT, kStageBytes, st>>>(psi, n, N, d, sa);
      *launches += 2;
      e = blocks(scdm_points_kernel<false>, 0, kUpdNT, &next);
      for (sa.k = left; sa.k < n && e == cudaSuccess; ++sa.k) {
        if (sa.k == left)
          scdm_points_kernel<true><<<next, kUpdNT, 0, st>>>(psi, pt, n, N, d, sa);
        else
          scdm_points_kernel<false><<<next, kUpdNT, 0, st>>>(psi, pt, n, N, d, sa);
        e = cudaGetLastError();
      }
      cudaFreeAsync(pt, st);
    }
  }
  if (e != cudaSuccess) return e;
  *launches += n;
  // Loewdin factor.  The n x n FP64 products run as one output per thread in 64-thread blocks, so
  // that they spread over most SMs (FP64 throughput per SM is low).
  const int nn = n * n;
  constexpr int kSmallNT = 64;
  const unsigned g1 = (unsigned)((nn + kSmallNT - 1) / kSmallNT), g2 = (unsigned)((2 * nn + kSmallNT - 1) / kSmallNT);
  scdm_gather_kernel<T><<<g1, kSmallNT, 0, st>>>(psi, n, N, res->piv, M);
  gram_t_kernel<<<g1, kSmallNT, 0, st>>>(M, n, S);
  frob_kernel<<<1, 1024, 0, st>>>(S, n, f);
  ns_start_kernel<<<g1, kSmallNT, 0, st>>>(S, n, f, Y[0], Z[0]);
  *launches += 4;
  // Newton-Schulz in chunks of kNsChunk iterations; between chunks the host reads the last two
  // deviations and stops launching once the next iteration would be skipped
  int it = 0;
  while (it < kNsMax) {
    for (const int stop = std::min(kNsMax, it + kNsChunk); it < stop; ++it) {
      const int a = it & 1;
      ns_t_kernel<<<g1, kSmallNT, 0, st>>>(Y[a], Z[a], n, Tm, res->dev, it);
      ns_yz_kernel<<<g2, kSmallNT, 0, st>>>(Y[a], Z[a], Tm, n, Y[a ^ 1], Z[a ^ 1], res->dev, it);
      *launches += 2;
    }
    if (it >= kNsMax) break;
    double h[2];
    e = cudaMemcpyAsync(h, res->dev + it - 2, sizeof(h), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return e;
    if (h[1] < kNsStop || (h[1] < 1e-8 && h[1] > 0.25 * h[0])) break;  // the test of ns_done
  }
  scdm_factor_kernel<T><<<g1, kSmallNT, 0, st>>>(M, Z[it & 1], n, f, res->U, reinterpret_cast<T *>(res->Ut));
  *launches += 1;
  return cudaGetLastError();
}

template cudaError_t launch_scdm<float>(const float *, int, long long, void *, cudaStream_t, long *, ScdmResult *);
template cudaError_t launch_scdm<double>(const double *, int, long long, void *, cudaStream_t, long *, ScdmResult *);

}  // namespace ace
