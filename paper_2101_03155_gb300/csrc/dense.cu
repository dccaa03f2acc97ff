// dense.cu -- CUDA-core dense steps of the ACE build and application.
//
//   gram:      G[i][j] = scale * sum_r f(X_i(r)) f(Y_j(r)),  f = |.| for the pair screen
//              (section II: int |phi_i phi_j| dr) or identity for M = -dV Phi^T W (App. A) and
//              C = dV xi^T psi.  Products and the sum inside one 4096-point chunk are in T; the
//              chunks are added into the FP64 result.
//   left_mul:  Z = A Y with A small (m x n) and Y (n x K): xi = L^-1 W (xi = W L^-T, App. A) and
//              the ACE application out = -C^T xi (section II).
//   cholesky:  M = (M_raw + M_raw^T)/2; -M = L L^T; L^-1; E_x = (f/2) tr M, all FP64 (App. A).
//   compact:   pair list of the screen (i <= j, sorted) and packs of two pairs.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>

#include <cstdint>
#include <cstdlib>

#include "ace_internal.h"
#include "f32x2.cuh"
#include "fft.cuh"

namespace ace {

// ----------------------------------------------------------------------------------------
// General Gram (the FP64 form, and FP32 point counts off the 16-byte grid): BM x BM output tile per CTA
// (BM 16 or 32, in FP32 also 64), 16 x 16 threads with (BM / 16)^2 outputs each, one chunk of K per CTA.
//   FP64 is bound by its pipe (2 multiply-adds per cycle and SM), so what counts is that no output of a tile
// is padding and that every SM has the same number of chunks: 64 x 64 tiles of 4096-point chunks left 12
// orbitals at 28 times the work on 21 SMs (4.8 ms for 86,400 points), and 64 orbitals on 72^3 on 91 of
// 152 SMs (5.3 ms).  Small tiles cost loads (each row is read once per tile of the other operand), which
// stay below 2% of the FP64 time.  FP32 is bound by its shared-memory loads, 2 BM / 16 for (BM / 16)^2
// multiply-adds, and takes tiles of 64 where they add at most half as much again in padding: 128 orbitals on
// 125^3 in tiles of 32 / 64: M 4.15 / 2.53 ms, screen 2.79 / 2.19 ms.
// ----------------------------------------------------------------------------------------
constexpr int GR_BK = 32, GR_NT = 256;
constexpr long long GR_LONGEST = 1ll << 17;  // FP64 (FP32 sums go to FP64 every 4096 points)

struct GramPlan {
  int bm, nbx, tiles;
  long long chunk, chunks;
};
// Chunks of K, at most GR_LONGEST points (FP32: 4096), such that tiles x chunks CTAs spread evenly over the SMs (four to
// sixteen per SM).
static GramPlan gram_plan(int nx, int ny, long long K, bool upper_only, bool fp64) {
  const long long longest = fp64 ? GR_LONGEST : 4096;
  auto padded = [](int n, int b) { return (double)((n + b - 1) / b * b); };
  GramPlan p;
  p.bm = nx <= 16 && ny <= 16 ? 16 : 32;
  if (!fp64 && padded(nx, 64) * padded(ny, 64) <= 1.5 * padded(nx, 32) * padded(ny, 32)) p.bm = 64;
  p.nbx = (nx + p.bm - 1) / p.bm;
  const int nby = (ny + p.bm - 1) / p.bm;
  p.tiles = upper_only ? p.nbx * (p.nbx + 1) / 2 : p.nbx * nby;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      sms < 1)
    sms = 152;
  const long long least = std::max(1ll, (4ll * sms + p.tiles - 1) / p.tiles);
  const long long most = std::max(1ll, std::min(65535ll, (K + 2 * GR_BK - 1) / (2 * GR_BK)));
  long long best = std::min(least, most);
  double fill = 0.0;
  for (long long c = best; c <= std::min(most, 4 * least); ++c) {
    const long long ctas = c * p.tiles, waves = (ctas + sms - 1) / sms;
    const double f = (double)ctas / (double)(waves * sms);
    if (f > fill + 0.01) {
      fill = f;
      best = c;
    }
  }
  p.chunk = std::min(longest, ((K + best - 1) / best + GR_BK - 1) / GR_BK * GR_BK);
  p.chunks = (K + p.chunk - 1) / p.chunk;
  return p;
}

// With `partial` non-null the CTA of chunk c writes its scaled tile sums to partial[c] (no
// atomics) and gram_chunks_reduce_kernel adds the chunks in a fixed order: the result is then
// the same bit for bit on every run.
template <typename T, bool ABS, int BM>
__global__ void __launch_bounds__(GR_NT) gram_kernel(const T *__restrict__ X, int nx, const T *__restrict__ Y, int ny,
                                                     long long K, long long chunk, double scale, bool upper_only, int nbx,
                                                     double *__restrict__ G, double *__restrict__ partial) {
  constexpr int RT = BM / 16;
  __shared__ T xs[GR_BK][BM + 1];
  __shared__ T ys[GR_BK][BM + 1];
  int bi, bj;
  if (upper_only) {
    // blockIdx.x enumerates tile pairs (bi <= bj) row by row
    int idx = blockIdx.x;
    bi = 0;
    while (idx >= nbx - bi) {
      idx -= nbx - bi;
      ++bi;
    }
    bj = bi + idx;
  } else {
    bi = blockIdx.x % nbx;
    bj = blockIdx.x / nbx;
  }
  const int i0 = bi * BM, j0 = bj * BM;
  const long long k0 = (long long)blockIdx.y * chunk;
  const long long k1 = min(K, k0 + chunk);
  const int tid = threadIdx.x;
  const int ty = tid / 16, tx = tid % 16;
  // acc + comp is a compensated (Kahan) running sum of the 32-point partial sums of each tile
  T acc[RT][RT], comp[RT][RT];
#pragma unroll
  for (int a = 0; a < RT; ++a)
#pragma unroll
    for (int b = 0; b < RT; ++b) acc[a][b] = comp[a][b] = (T)0;

  // the next step's rows are loaded into registers while this step multiplies (coalesced along k)
  constexpr int NE = BM * GR_BK / GR_NT;
  T xn[NE], yn[NE];
  auto fetch = [&](long long kk) {
#pragma unroll
    for (int q = 0; q < NE; ++q) {
      const int e = tid + q * GR_NT, r = e / GR_BK, c = e % GR_BK;
      const long long k = kk + c;
      T xv = (T)0, yv = (T)0;
      if (k < k1) {
        if (i0 + r < nx) xv = X[(long long)(i0 + r) * K + k];
        if (j0 + r < ny) yv = Y[(long long)(j0 + r) * K + k];
      }
      if (ABS) {
        xv = xv < (T)0 ? -xv : xv;
        yv = yv < (T)0 ? -yv : yv;
      }
      xn[q] = xv;
      yn[q] = yv;
    }
  };
  fetch(k0);
  for (long long kk = k0; kk < k1; kk += GR_BK) {
#pragma unroll
    for (int q = 0; q < NE; ++q) {
      const int e = tid + q * GR_NT, r = e / GR_BK, c = e % GR_BK;
      xs[c][r] = xn[q];
      ys[c][r] = yn[q];
    }
    __syncthreads();
    if (kk + GR_BK < k1) fetch(kk + GR_BK);
    T part[RT][RT];
#pragma unroll
    for (int a = 0; a < RT; ++a)
#pragma unroll
      for (int b = 0; b < RT; ++b) part[a][b] = (T)0;
#pragma unroll 8
    for (int c = 0; c < GR_BK; ++c) {
      T xr[RT], yr[RT];
#pragma unroll
      for (int a = 0; a < RT; ++a) xr[a] = xs[c][ty + 16 * a];
#pragma unroll
      for (int b = 0; b < RT; ++b) yr[b] = ys[c][tx + 16 * b];
#pragma unroll
      for (int a = 0; a < RT; ++a)
#pragma unroll
        for (int b = 0; b < RT; ++b) part[a][b] += xr[a] * yr[b];
    }
#pragma unroll
    for (int a = 0; a < RT; ++a)
#pragma unroll
      for (int b = 0; b < RT; ++b) {
        const T y = part[a][b] - comp[a][b];
        const T t = acc[a][b] + y;
        comp[a][b] = (t - acc[a][b]) - y;
        acc[a][b] = t;
      }
    __syncthreads();
  }
#pragma unroll
  for (int a = 0; a < RT; ++a)
#pragma unroll
    for (int b = 0; b < RT; ++b) {
      const int i = i0 + ty + 16 * a, j = j0 + tx + 16 * b;
      if (i < nx && j < ny) {
        if (partial)
          partial[((long long)blockIdx.y * nx + i) * ny + j] = scale * (double)acc[a][b];
        else
          atomicAdd(G + (long long)i * ny + j, scale * (double)acc[a][b]);
      }
    }
}

// G_ij = sum over the chunks of partial[c]_ij in a fixed order (eight interleaved sums; upper_only: j >= i
// only)
__global__ void gram_chunks_reduce_kernel(const double *__restrict__ partial, long long chunks, int nx, int ny,
                                          bool upper_only, double *__restrict__ G) {
  const long long ne = (long long)nx * ny;
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= ne || (upper_only && e % ny < e / ny)) return;
  double s[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  long long c = 0;
  for (; c + 8 <= chunks; c += 8) {
#pragma unroll
    for (int q = 0; q < 8; ++q) s[q] += partial[(c + q) * ne + e];
  }
  for (; c < chunks; ++c) s[0] += partial[c * ne + e];
  G[e] = ((s[0] + s[1]) + (s[2] + s[3])) + ((s[4] + s[5]) + (s[6] + s[7]));
}

size_t gram_chunks_bytes(int nx, int ny, long long K) {
  const long long c = std::max(gram_plan(nx, ny, K, false, true).chunks,
                               nx == ny ? gram_plan(nx, ny, K, true, true).chunks : 0);
  return sizeof(double) * (size_t)c * nx * ny;
}

// FP32 operands: 128 x 64 output tile, 256 threads with 8 x 4 outputs each, k-tiles of 16 staged
// in shared memory (double-buffered, next tile prefetched into registers), FP32 partial sums of 32
// points added into a Kahan-compensated FP32 accumulator, FP64 atomics across 4096-point chunks.
constexpr int G2_BM = 128, G2_BN = 64, G2_BK = 16, G2_NT = 256, G2_CHUNK = 4096;

template <bool ABS>
__global__ void __launch_bounds__(G2_NT, 2) gram_f32_kernel(const float *__restrict__ X, int nx,
                                                            const float *__restrict__ Y, int ny, long long K,
                                                            double scale, bool upper_only, int tiles_i,
                                                            double *__restrict__ G) {
  __shared__ __align__(16) float xs[2][G2_BK][G2_BM + 4];
  __shared__ __align__(16) float ys[2][G2_BK][G2_BN + 4];
  const int ti = blockIdx.x % tiles_i, tj = blockIdx.x / tiles_i;
  const int i0 = ti * G2_BM, j0 = tj * G2_BN;
  if (upper_only && j0 + G2_BN - 1 < i0) return;  // tile entirely below the diagonal
  const long long kb = (long long)blockIdx.y * G2_CHUNK;
  const long long ke = min(K, kb + G2_CHUNK);
  const int ntiles = (int)((ke - kb + G2_BK - 1) / G2_BK);
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  float acc[8][4], comp[8][4], part[8][4];
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = comp[a][b] = part[a][b] = 0.f;

  float4 rx[2], ry;
  auto load = [&](int t) {
    const long long k0 = kb + (long long)t * G2_BK;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int f = tid + G2_NT * q, row = f >> 2, kq = (f & 3) * 4;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (i0 + row < nx && k0 + kq < ke) v = __ldg(reinterpret_cast<const float4 *>(X + (long long)(i0 + row) * K + k0 + kq));
      rx[q] = v;
    }
    {
      const int row = tid >> 2, kq = (tid & 3) * 4;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (j0 + row < ny && k0 + kq < ke) v = __ldg(reinterpret_cast<const float4 *>(Y + (long long)(j0 + row) * K + k0 + kq));
      ry = v;
    }
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int f = tid + G2_NT * q, row = f >> 2, kq = (f & 3) * 4;
      const float v[4] = {rx[q].x, rx[q].y, rx[q].z, rx[q].w};
#pragma unroll
      for (int c = 0; c < 4; ++c) xs[buf][kq + c][row] = ABS ? fabsf(v[c]) : v[c];
    }
    const int row = tid >> 2, kq = (tid & 3) * 4;
    const float v[4] = {ry.x, ry.y, ry.z, ry.w};
#pragma unroll
    for (int c = 0; c < 4; ++c) ys[buf][kq + c][row] = ABS ? fabsf(v[c]) : v[c];
  };
  if (ntiles > 0) {
    load(0);
    store(0);
  }
  __syncthreads();
  for (int t = 0; t < ntiles; ++t) {
    const int buf = t & 1;
    if (t + 1 < ntiles) load(t + 1);
#pragma unroll
    for (int k = 0; k < G2_BK; ++k) {
      const float4 a0 = *reinterpret_cast<const float4 *>(&xs[buf][k][ty * 4]);
      const float4 a1 = *reinterpret_cast<const float4 *>(&xs[buf][k][64 + ty * 4]);
      const float4 b = *reinterpret_cast<const float4 *>(&ys[buf][k][tx * 4]);
      const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const float bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) part[r][c] = fmaf(av[r], bv[c], part[r][c]);
    }
    if ((t & 1) || t + 1 == ntiles) {
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float y = part[r][c] - comp[r][c];
          const float s = acc[r][c] + y;
          comp[r][c] = (s - acc[r][c]) - y;
          acc[r][c] = s;
          part[r][c] = 0.f;
        }
    }
    if (t + 1 < ntiles) store(buf ^ 1);
    __syncthreads();
  }
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const int i = i0 + (r < 4 ? ty * 4 + r : 64 + ty * 4 + (r - 4));
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int j = j0 + tx * 4 + c;
      if (i < nx && j < ny && !(upper_only && j < i)) atomicAdd(G + (long long)i * ny + j, scale * (double)acc[r][c]);
    }
  }
}

// ----------------------------------------------------------------------------------------
// Symmetric FP32 Gram (the screen, X = Y, upper triangle): 64 x 64 tiles enumerated over the
// upper triangle of 64-row blocks only, 256 threads with 4 x 4 outputs each, k-step 16, chunks of
// ACE_GS_CHUNK points per CTA.  Products run as packed f32x2 FMAs: the row operand is stored twice in
// shared memory ((a, a) pairs) so that a pair of outputs (c, c + 1) takes one instruction.
// Within a chunk, 32-point FP32 partials are added with Kahan compensation; chunks meet in FP64
// atomics.
// ----------------------------------------------------------------------------------------
// points per CTA and CTAs per SM of the symmetric kernel (the register budget follows)
#ifndef ACE_GS_CHUNK
#define ACE_GS_CHUNK 2048
#endif
#ifndef ACE_GS_MINB
#define ACE_GS_MINB 2
#endif
constexpr int GS_B = 64, GS_BK = 16, GS_NT = 256, GS_CHUNK = ACE_GS_CHUNK;

template <bool ABS>
__global__ void __launch_bounds__(GS_NT, ACE_GS_MINB) gram_sym_f32_kernel(const float *__restrict__ X, int n, long long ld,
                                                                        long long K, double scale,
                                                                        double *__restrict__ G) {
  // (a, a) pairs of the row block and plain values of the column block, double-buffered
  __shared__ __align__(16) float2 xs[2][GS_BK][GS_B + 2];
  __shared__ __align__(16) float ys[2][GS_BK][GS_B + 4];
  // tile t of the upper triangle of nb x nb blocks: row-major over bi <= bj
  int bi = 0, t = blockIdx.x;
  {
    const int nb = (n + GS_B - 1) / GS_B;
    while (t >= nb - bi) {
      t -= nb - bi;
      ++bi;
    }
  }
  const int bj = bi + t;
  const int i0 = bi * GS_B, j0 = bj * GS_B;
  const long long kb = (long long)blockIdx.y * GS_CHUNK;
  const long long ke = min(K, kb + GS_CHUNK);
  const int ntiles = (int)((ke - kb + GS_BK - 1) / GS_BK);
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  unsigned long long acc[4][2], comp[4][2], part[4][2];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) acc[a][b] = comp[a][b] = part[a][b] = 0ull;

  // each thread stages one float4 (4 consecutive points) of one row of each block; the global
  // loads run two k-tiles ahead (register sets 0 and 1 alternate)
  const int lrow = tid >> 2, lk = (tid & 3) * 4;
  float4 rx[2], ry[2];
  auto load = [&](int tt, float4 &vx, float4 &vy) {
    const long long k0 = kb + (long long)tt * GS_BK + lk;
    vx = make_float4(0.f, 0.f, 0.f, 0.f);
    vy = vx;
    if (tt < ntiles && k0 < ke) {
      if (i0 + lrow < n) vx = __ldg(reinterpret_cast<const float4 *>(X + (long long)(i0 + lrow) * ld + k0));
      if (j0 + lrow < n) vy = __ldg(reinterpret_cast<const float4 *>(X + (long long)(j0 + lrow) * ld + k0));
    }
  };
  auto store = [&](int buf, const float4 &ux, const float4 &uy) {
    const float vx[4] = {ux.x, ux.y, ux.z, ux.w}, vy[4] = {uy.x, uy.y, uy.z, uy.w};
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float a = ABS ? fabsf(vx[c]) : vx[c];
      xs[buf][lk + c][lrow] = make_float2(a, a);
      ys[buf][lk + c][lrow] = ABS ? fabsf(vy[c]) : vy[c];
    }
  };
  auto compute = [&](int buf, int tt) {
#pragma unroll
    for (int k = 0; k < GS_BK; ++k) {
      const ulonglong2 a01 = *reinterpret_cast<const ulonglong2 *>(&xs[buf][k][ty * 4]);
      const ulonglong2 a23 = *reinterpret_cast<const ulonglong2 *>(&xs[buf][k][ty * 4 + 2]);
      const ulonglong2 b = *reinterpret_cast<const ulonglong2 *>(&ys[buf][k][tx * 4]);
      const unsigned long long av[4] = {a01.x, a01.y, a23.x, a23.y};
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        part[r][0] = f2fma(av[r], b.x, part[r][0]);
        part[r][1] = f2fma(av[r], b.y, part[r][1]);
      }
    }
    if ((tt & 1) || tt + 1 == ntiles) {
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const unsigned long long y = f2sub(part[r][c], comp[r][c]);
          const unsigned long long sm = f2add(acc[r][c], y);
          comp[r][c] = f2sub(f2sub(sm, acc[r][c]), y);
          acc[r][c] = sm;
          part[r][c] = 0ull;
        }
    }
  };
  load(0, rx[0], ry[0]);
  store(0, rx[0], ry[0]);
  load(1, rx[1], ry[1]);
  __syncthreads();
  // tile tt sits in shared buffer tt & 1; tile tt + 1 in register set (tt + 1) & 1
  for (int tt = 0; tt < ntiles; tt += 2) {
    load(tt + 2, rx[0], ry[0]);
    compute(0, tt);
    store(1, rx[1], ry[1]);
    __syncthreads();
    if (tt + 1 >= ntiles) break;
    load(tt + 3, rx[1], ry[1]);
    compute(1, tt + 1);
    store(0, rx[0], ry[0]);
    __syncthreads();
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int i = i0 + ty * 4 + r;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const float2 v = f2up(acc[r][c]);
      const int j = j0 + tx * 4 + 2 * c;
      if (i < n && j < n && j >= i) atomicAdd(G + (long long)i * n + j, scale * (double)v.x);
      if (i < n && j + 1 < n && j + 1 >= i) atomicAdd(G + (long long)i * n + j + 1, scale * (double)v.y);
    }
  }
}

// Screen contribution of the columns [0, K) of X (rows of stride ld): G += scale * |X| |X|^T on the
// upper triangle (G is not cleared; columns must start on a 16-byte boundary, K % 4 == 0).
cudaError_t launch_screen_cols(const float *X, int n, long long ld, long long K, double scale, double *G,
                               cudaStream_t st) {
  if (K % 4 != 0 || ld % 4 != 0 || (reinterpret_cast<uintptr_t>(X) & 15)) return cudaErrorInvalidValue;
  const int nb = (n + GS_B - 1) / GS_B;
  const long long chunks = (K + GS_CHUNK - 1) / GS_CHUNK;
  if (chunks > 65535) return cudaErrorInvalidValue;
  gram_sym_f32_kernel<true><<<dim3(nb * (nb + 1) / 2, (unsigned)chunks), GS_NT, 0, st>>>(X, n, ld, K, scale, G);
  return cudaGetLastError();
}

// Screen values within band * rho_cut of the threshold, recomputed from phi so that the pair
// decision does not rest on the tensor-core products (BF16x3: up to 3 * 2^-16 relative error per
// product): O_ij = dV sum_r |phi_i(r) phi_j(r)| with FP32 products summed per thread with Kahan
// compensation in FP32, then across the block's threads in FP64 in a fixed order.  Off-diagonal
// upper-triangle entries only (the diagonal is always kept).  One block per candidate pair.
constexpr int RF_NT = 256;
__global__ void __launch_bounds__(RF_NT) screen_refine_kernel(const float *__restrict__ phi, int n, long long N,
                                                              double dV, double rho_cut, double band,
                                                              double *__restrict__ O) {
  __shared__ double red[RF_NT / 32];
  const long long ne = (long long)n * n;
  for (long long e = blockIdx.x; e < ne; e += gridDim.x) {
    const int i = (int)(e / n), j = (int)(e % n);
    if (i >= j) continue;
    const double o = O[e];  // the same value for every thread: the branch is uniform
    if (!(fabs(o - rho_cut) <= band * rho_cut)) continue;
    const float *a = phi + (long long)i * N, *b = phi + (long long)j * N;
    float sum = 0.f, comp = 0.f;
    for (long long r = threadIdx.x; r < N; r += RF_NT) {
      const float y = fabsf(a[r] * b[r]) - comp;
      const float t = sum + y;
      comp = (t - sum) - y;
      sum = t;
    }
    double v = (double)sum - (double)comp;
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int w = 0; w < RF_NT / 32; ++w) t += red[w];
      O[e] = dV * t;
    }
    __syncthreads();
  }
}

cudaError_t launch_screen_refine(const float *phi, int n, long long N, double dV, double rho_cut, double band,
                                 double *O, cudaStream_t st) {
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const long long ne = (long long)n * n;
  const unsigned grid = (unsigned)std::max<long long>(1, std::min<long long>(ne, 2LL * sms));
  screen_refine_kernel<<<grid, RF_NT, 0, st>>>(phi, n, N, dV, rho_cut, band, O);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_gram(const T *X, int nx, const T *Y, int ny, long long K, double scale, bool abs_values,
                        bool upper_only, double *G, cudaStream_t st, double *partial) {
  if constexpr (sizeof(T) == 4) {
    if (K % 4 == 0 && X == Y && nx == ny && upper_only) {
      const int nb = (nx + GS_B - 1) / GS_B;
      const long long chunks = (K + GS_CHUNK - 1) / GS_CHUNK;
      if (chunks > 65535) return cudaErrorInvalidValue;
      cudaError_t e = cudaMemsetAsync(G, 0, sizeof(double) * (size_t)nx * ny, st);
      if (e != cudaSuccess) return e;
      dim3 grid(nb * (nb + 1) / 2, (unsigned)chunks);
      if (abs_values)
        gram_sym_f32_kernel<true><<<grid, GS_NT, 0, st>>>(X, nx, K, K, scale, G);
      else
        gram_sym_f32_kernel<false><<<grid, GS_NT, 0, st>>>(X, nx, K, K, scale, G);
      return cudaGetLastError();
    }
    if (K % 4 == 0) {
      const int tiles_i = (nx + G2_BM - 1) / G2_BM, tiles_j = (ny + G2_BN - 1) / G2_BN;
      const long long chunks = (K + G2_CHUNK - 1) / G2_CHUNK;
      if (chunks > 65535) return cudaErrorInvalidValue;
      cudaError_t e = cudaMemsetAsync(G, 0, sizeof(double) * (size_t)nx * ny, st);
      if (e != cudaSuccess) return e;
      dim3 grid(tiles_i * tiles_j, (unsigned)chunks);
      if (abs_values)
        gram_f32_kernel<true><<<grid, G2_NT, 0, st>>>(X, nx, Y, ny, K, scale, upper_only, tiles_i, G);
      else
        gram_f32_kernel<false><<<grid, G2_NT, 0, st>>>(X, nx, Y, ny, K, scale, upper_only, tiles_i, G);
      return cudaGetLastError();
    }
  }
  const GramPlan p = gram_plan(nx, ny, K, upper_only, sizeof(T) == 8);
  if (p.chunks > 65535) return cudaErrorInvalidValue;
  cudaError_t e = cudaMemsetAsync(G, 0, sizeof(double) * (size_t)nx * ny, st);
  if (e != cudaSuccess) return e;
  const dim3 grid(p.tiles, (unsigned)p.chunks);
  auto run = [&](auto kernel) {
    kernel<<<grid, GR_NT, 0, st>>>(X, nx, Y, ny, K, p.chunk, scale, upper_only, p.nbx, G, partial);
  };
  if (p.bm == 16)
    abs_values ? run(gram_kernel<T, true, 16>) : run(gram_kernel<T, false, 16>);
  else if (p.bm == 64) {
    if constexpr (sizeof(T) == 4) abs_values ? run(gram_kernel<T, true, 64>) : run(gram_kernel<T, false, 64>);
  } else
    abs_values ? run(gram_kernel<T, true, 32>) : run(gram_kernel<T, false, 32>);
  e = cudaGetLastError();
  if (e != cudaSuccess || !partial) return e;
  const long long ne = (long long)nx * ny;
  gram_chunks_reduce_kernel<<<(unsigned)((ne + 63) / 64), 64, 0, st>>>(partial, p.chunks, nx, ny, upper_only, G);
  return cudaGetLastError();
}
template cudaError_t launch_gram<float>(const float *, int, const float *, int, long long, double, bool, bool,
                                        double *, cudaStream_t, double *);
template cudaError_t launch_gram<double>(const double *, int, const double *, int, long long, double, bool, bool,
                                         double *, cudaStream_t, double *);

// ----------------------------------------------------------------------------------------
// FP32 products with at most 8 rows on one side (a few vectors against the stored xi, builds of a
// few orbitals).  Both are bound by reading the large operand once: 95.5 MB at 64 rows of 72^3, where
// 4 vectors take 21 us for the coefficients (5.0 TB/s) and a call of ace_apply went from 197 to 86 us.
// The tensor-core tiles, which take 9 rows and more, pad the short side to 128 and convert every point
// to BF16 pairs for it; these kernels' FP32 products are also the more exact ones.
// ----------------------------------------------------------------------------------------
constexpr int SK_NT = 128;        // threads of both kernels
constexpr int SK_ROWS = 8;        // large-side rows per warp of the Gram
constexpr int SK_FOLD = 16;       // 128-point steps summed in FP32 (16 x 4 products per lane) before the FP64 sum
constexpr int SK_WARPS = 12;      // Gram warps per SM that the split aims at (the 8-row form's residency)

// G_ab = scale * sum_k L_ak S_bk over L of nl rows and S of ns <= MS rows.  A warp takes 8 rows of
// L and one run of columns; its lanes hold all 8 x MS sums, reading 16 bytes of every row per step.
// Lane sums are folded into FP64 every SK_FOLD steps; the runs' sums are added by
// skinny_gram_reduce_kernel in run order.
template <int MS>
__global__ void __launch_bounds__(SK_NT, 3) skinny_gram_kernel(const float *__restrict__ L, int nl,
                                                               const float *__restrict__ S, int ns, long long K,
                                                               long long run, int groups, int runs,
                                                               double *__restrict__ partial) {
  constexpr int NV = SK_ROWS * MS, KEEP = NV >= 32 ? NV / 32 : 1;
  const int lane = threadIdx.x & 31;
  const long long task = (long long)blockIdx.x * (SK_NT / 32) + (threadIdx.x >> 5);
  if (task >= (long long)groups * runs) return;
  const int g = (int)(task % groups), c = (int)(task / groups);
  const long long k0 = (long long)c * run, ke = min(K, k0 + run);
  // rows past the end repeat the last one; their sums are not stored
  const float *lp[SK_ROWS], *sp[MS];
#pragma unroll
  for (int r = 0; r < SK_ROWS; ++r) lp[r] = L + (long long)min(g * SK_ROWS + r, nl - 1) * K;
#pragma unroll
  for (int q = 0; q < MS; ++q) sp[q] = S + (long long)min(q, ns - 1) * K;
  double sum[KEEP];
#pragma unroll
  for (int i = 0; i < KEEP; ++i) sum[i] = 0.0;
  int first = 0;  // index (row * MS + q) of the first value this lane keeps
  for (long long kb = k0; kb < ke; kb += 128 * SK_FOLD) {
    float v[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = 0.f;
    const long long kend = min(ke, kb + 128 * SK_FOLD);
    for (long long k = kb + 4 * lane; k < kend; k += 128) {
      float4 s[MS], l[SK_ROWS];
#pragma unroll
      for (int r = 0; r < SK_ROWS; ++r) l[r] = __ldg(reinterpret_cast<const float4 *>(lp[r] + k));
#pragma unroll
      for (int q = 0; q < MS; ++q) s[q] = __ldg(reinterpret_cast<const float4 *>(sp[q] + k));
#pragma unroll
      for (int r = 0; r < SK_ROWS; ++r)
#pragma unroll
        for (int q = 0; q < MS; ++q) {
          float &a = v[r * MS + q];
          a = fmaf(l[r].x, s[q].x, a);
          a = fmaf(l[r].y, s[q].y, a);
          a = fmaf(l[r].z, s[q].z, a);
          a = fmaf(l[r].w, s[q].w, a);
        }
    }
    __syncwarp();
    // halving exchange: each step adds the partner's half of the values and keeps the own half
    first = 0;
#pragma unroll
    for (int off = 16, h = NV / 2; off > 0; off >>= 1, h >>= 1) {
      if (h > 0) {
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int i = 0; i < h; ++i) {
          const float send = up ? v[i] : v[i + h];
          v[i] = (up ? v[i + h] : v[i]) + __shfl_xor_sync(0xffffffffu, send, off);
        }
        if (up) first += h;
      } else {
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
      }
    }
#pragma unroll
    for (int i = 0; i < KEEP; ++i) sum[i] += (double)v[i];
  }
  double *dst = partial + ((long long)c * groups + g) * NV;
  if (NV < 32 && (lane & (32 / NV - 1))) return;  // lanes that hold the same value
#pragma unroll
  for (int i = 0; i < KEEP; ++i) dst[first + i] = sum[i];
}

// G from the runs' sums: 32 slices of the runs per value (runs of up to 228 at 64 rows: eight loads
// in flight per thread and one round trip), the slices added in a fixed order.
constexpr int SKR_SLICES = 32;
__global__ void __launch_bounds__(32 * SKR_SLICES) skinny_gram_reduce_kernel(const double *__restrict__ partial,
                                                                             int runs, int groups, int MS, int nl,
                                                                             int ns, int sl, int ss, double scale,
                                                                             double *__restrict__ G) {
  __shared__ double part[SKR_SLICES][33];
  const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5;
  const int nv = groups * SK_ROWS * MS, e = blockIdx.x * 32 + lane;
  double s = 0.0;
  if (e < nv) {
#pragma unroll 8
    for (int c = slice; c < runs; c += SKR_SLICES) s += partial[(long long)c * nv + e];
  }
  part[slice][lane] = s;
  __syncthreads();
  if (slice != 0 || e >= nv) return;
  s = 0.0;
#pragma unroll
  for (int i = 0; i < SKR_SLICES; ++i) s += part[i][lane];
  const int a = e / MS, b = e % MS;
  if (a < nl && b < ns) G[(long long)a * sl + (long long)b * ss] = scale * s;
}

struct SkinnyPlan {
  int ms, groups, runs;
  long long run;
};
static SkinnyPlan skinny_gram_plan(int nl, int ns, long long K) {
  SkinnyPlan p;
  p.ms = ns <= 1 ? 1 : ns <= 2 ? 2 : ns <= 4 ? 4 : 8;
  p.groups = (nl + SK_ROWS - 1) / SK_ROWS;
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const long long want = std::max(1, sms * SK_WARPS / p.groups);
  p.run = std::max(128LL, ((K + want - 1) / want + 127) / 128 * 128);
  p.runs = (int)((K + p.run - 1) / p.run);
  return p;
}

bool skinny_gram_ok(const float *X, int nx, const float *Y, int ny, long long K) {
  return std::min(nx, ny) <= 8 && K % 4 == 0 &&
         ((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(Y)) & 15) == 0;
}

size_t skinny_gram_bytes(int nx, int ny, long long K) {
  const SkinnyPlan p = skinny_gram_plan(std::max(nx, ny), std::min(nx, ny), K);
  return sizeof(double) * (size_t)p.runs * p.groups * SK_ROWS * p.ms;
}

// G (nx x ny) = scale X Y^T with min(nx, ny) <= 8 (skinny_gram_ok); ws of skinny_gram_bytes
cudaError_t launch_skinny_gram(const float *X, int nx, const float *Y, int ny, long long K, double scale, double *G,
                               void *ws, cudaStream_t st) {
  const bool ysmall = ny <= nx;
  const float *L = ysmall ? X : Y, *S = ysmall ? Y : X;
  const int nl = ysmall ? nx : ny, ns = ysmall ? ny : nx;
  const SkinnyPlan p = skinny_gram_plan(nl, ns, K);
  double *partial = static_cast<double *>(ws);
  const long long tasks = (long long)p.groups * p.runs;
  const unsigned grid = (unsigned)((tasks + SK_NT / 32 - 1) / (SK_NT / 32));
  auto run = [&](auto kernel) {
    kernel<<<grid, SK_NT, 0, st>>>(L, nl, S, ns, K, p.run, p.groups, p.runs, partial);
  };
  if (p.ms == 1) run(skinny_gram_kernel<1>);
  else if (p.ms == 2) run(skinny_gram_kernel<2>);
  else if (p.ms == 4) run(skinny_gram_kernel<4>);
  else run(skinny_gram_kernel<8>);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int nv = p.groups * SK_ROWS * p.ms;
  skinny_gram_reduce_kernel<<<(nv + 31) / 32, 32 * SKR_SLICES, 0, st>>>(partial, p.runs, p.groups, p.ms, nl, ns,
                                                            ysmall ? ny : 1, ysmall ? 1 : ny, scale, G);
  return cudaGetLastError();
}

// Z (m x K) = A (m x n) Y (n x K) for m <= M: a thread holds the m sums of V neighbouring points
// and reads Y once, eight rows in flight; A passes through shared memory 256 columns at a time.
template <int M, int V>
__global__ void __launch_bounds__(SK_NT) skinny_left_mul_kernel(const float *__restrict__ A, int m, int n,
                                                                const float *__restrict__ Y, long long K,
                                                                float *__restrict__ Z) {
  constexpr int COLS = 256, RB = 8;
  __shared__ __align__(16) float as[COLS][M];
  const long long k = ((long long)blockIdx.x * SK_NT + threadIdx.x) * V;
  float acc[M][V];
  auto load = [](const float *src, float (&yv)[V]) {
    if constexpr (V == 4) {
      const float4 t = __ldg(reinterpret_cast<const float4 *>(src));
      yv[0] = t.x, yv[1] = t.y, yv[2] = t.z, yv[3] = t.w;
    } else {
      yv[0] = __ldg(src);
    }
  };
  auto add = [&](int l, const float (&yv)[V]) {
#pragma unroll
    for (int r = 0; r < M; ++r)
#pragma unroll
      for (int v = 0; v < V; ++v) acc[r][v] = fmaf(as[l][r], yv[v], acc[r][v]);
  };
#pragma unroll
  for (int r = 0; r < M; ++r)
#pragma unroll
    for (int v = 0; v < V; ++v) acc[r][v] = 0.f;
  for (int l0 = 0; l0 < n; l0 += COLS) {
    const int nl = min(COLS, n - l0);
    __syncthreads();
    for (int e = threadIdx.x; e < nl * M; e += SK_NT) {
      const int r = e / nl, c = e % nl;
      as[c][r] = r < m ? A[(long long)r * n + l0 + c] : 0.f;
    }
    __syncthreads();
    if (k < K) {
      const float *y = Y + (long long)l0 * K + k;
      int l = 0;
      for (; l + RB <= nl; l += RB) {
        float yv[RB][V];
#pragma unroll
        for (int b = 0; b < RB; ++b) load(y + (long long)(l + b) * K, yv[b]);
#pragma unroll
        for (int b = 0; b < RB; ++b) add(l + b, yv[b]);
      }
      for (; l < nl; ++l) {
        float yv[V];
        load(y + (long long)l * K, yv);
        add(l, yv);
      }
    }
  }
  if (k >= K) return;
#pragma unroll
  for (int r = 0; r < M; ++r) {
    if (r >= m) break;
    if constexpr (V == 4)
      *reinterpret_cast<float4 *>(Z + (long long)r * K + k) = make_float4(acc[r][0], acc[r][1], acc[r][2], acc[r][3]);
    else
      Z[(long long)r * K + k] = acc[r][0];
  }
}

// Left multiply with m <= 8 rows of A.  Four points per thread where that still gives every SM
// 512 threads and the rows lie on 16-byte boundaries; else one point per thread.
cudaError_t launch_skinny_left_mul(const float *A, int m, int n, const float *Y, long long K, float *Z,
                                   cudaStream_t st) {
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const bool wide = K % 4 == 0 && K / 4 >= 512LL * sms &&
                    ((reinterpret_cast<uintptr_t>(Y) | reinterpret_cast<uintptr_t>(Z)) & 15) == 0;
  const long long threads = wide ? K / 4 : K;
  const unsigned grid = (unsigned)((threads + SK_NT - 1) / SK_NT);
  auto run = [&](auto kernel) { kernel<<<grid, SK_NT, 0, st>>>(A, m, n, Y, K, Z); };
  if (m <= 1) wide ? run(skinny_left_mul_kernel<1, 4>) : run(skinny_left_mul_kernel<1, 1>);
  else if (m <= 2) wide ? run(skinny_left_mul_kernel<2, 4>) : run(skinny_left_mul_kernel<2, 1>);
  else if (m <= 4) wide ? run(skinny_left_mul_kernel<4, 4>) : run(skinny_left_mul_kernel<4, 1>);
  else wide ? run(skinny_left_mul_kernel<8, 4>) : run(skinny_left_mul_kernel<8, 1>);
  return cudaGetLastError();
}

// ----------------------------------------------------------------------------------------
// Left multiply Z (m x K) = A (m x n) * Y (n x K); 16 R x 64 tile, k-step 16, R x 4 per thread.
// Bound by the FP64 pipe (two FMA per clock and SM) in double, so rows of padding cost their full
// time: the launcher takes as few row blocks as tiles of 64 rows would need and the smallest R that
// covers m with them (12 rows: a tile of 16, not 64; 70 rows: two of 48, not of 64).  With a lower
// triangular A (m = n) a row block stops at its last diagonal element, and blocks are 16 rows: at 64 rows
// that leaves 5/8 of the products.  FP32 is bound by its shared-memory loads (R + 4 for 4 R multiply-adds) and
// keeps the tall blocks for a triangular A too: 128 rows of 125^3 take 3.33 ms in blocks of 16 rows, 2.03 in
// blocks of 64.
// Every output adds its terms in the same order whatever R is.
// xi in FP64: 12 rows of 40x45x48 149 -> 37 us, 64 rows of 72^3 2.49 -> 1.55 ms.
// ----------------------------------------------------------------------------------------
constexpr int LM_BN = 64, LM_BK = 16, LM_NT = 256, LM_RMAX = 4;

template <typename T, int R>
__global__ void __launch_bounds__(LM_NT) left_mul_kernel(const T *__restrict__ A, int m, int n,
                                                         const T *__restrict__ Y, long long K, T *__restrict__ Z,
                                                         bool lower) {
  constexpr int LM_BM = 16 * R;
  __shared__ T as[LM_BK][LM_BM + 1];
  __shared__ T ys[LM_BK][LM_BN];
  const int i0 = blockIdx.y * LM_BM;
  const long long c0 = (long long)blockIdx.x * LM_BN;
  const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16;
  T acc[R][4];
#pragma unroll
  for (int a = 0; a < R; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = (T)0;
  const int le = lower ? min(n, i0 + LM_BM) : n;  // columns of A past here are zero
  for (int l0 = 0; l0 < le; l0 += LM_BK) {
    for (int e = tid; e < LM_BM * LM_BK; e += LM_NT) {
      const int r = e / LM_BK, c = e % LM_BK;
      as[c][r] = (i0 + r < m && l0 + c < le) ? A[(long long)(i0 + r) * n + l0 + c] : (T)0;
    }
    for (int e = tid; e < LM_BK * LM_BN; e += LM_NT) {
      const int r = e / LM_BN, c = e % LM_BN;
      ys[r][c] = (l0 + r < le && c0 + c < K) ? Y[(long long)(l0 + r) * K + c0 + c] : (T)0;
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < LM_BK; ++c) {
      if (sizeof(T) == 8 && l0 + c >= le) break;  // in FP32 the test costs more than the zeros
      T ar[R], yr[4];
#pragma unroll
      for (int a = 0; a < R; ++a) ar[a] = as[c][ty + 16 * a];
#pragma unroll
      for (int b = 0; b < 4; ++b) yr[b] = ys[c][tx + 16 * b];
#pragma unroll
      for (int a = 0; a < R; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] += ar[a] * yr[b];
    }
    __syncthreads();
  }
#pragma unroll
  for (int a = 0; a < R; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int i = i0 + ty + 16 * a;
      const long long c = c0 + tx + 16 * b;
      if (i < m && c < K) Z[(long long)i * K + c] = acc[a][b];
    }
}

template <typename T>
cudaError_t launch_left_mul(const T *A, int m, int n, const T *Y, long long K, T *Z, cudaStream_t st, bool lower) {
  const int rmax = lower && sizeof(T) == 8 ? 1 : LM_RMAX;
  const int blocks = (m + 16 * rmax - 1) / (16 * rmax), R = ((m + blocks - 1) / blocks + 15) / 16;
  const dim3 grid((unsigned)((K + LM_BN - 1) / LM_BN), (unsigned)blocks);
  auto run = [&](auto kernel) { kernel<<<grid, LM_NT, 0, st>>>(A, m, n, Y, K, Z, lower); };
  if (R <= 1) run(left_mul_kernel<T, 1>);
  else if (R == 2) run(left_mul_kernel<T, 2>);
  else if (R == 3) run(left_mul_kernel<T, 3>);
  else run(left_mul_kernel<T, 4>);
  return cudaGetLastError();
}
template cudaError_t launch_left_mul<float>(const float *, int, int, const float *, long long, float *, cudaStream_t,
                                            bool);
template cudaError_t launch_left_mul<double>(const double *, int, int, const double *, long long, double *,
                                             cudaStream_t, bool);

// ----------------------------------------------------------------------------------------
// Cholesky of -M, L^-1 and E_x in one CTA (FP64).  A = -M lives in shared memory when n <= 128
// (n^2 doubles), else in a global workspace.  Right-looking factorisation, then the in-place
// inversion of the lower triangle column by column from the last (each column is a triangular
// matrix-vector product with the already inverted trailing block).
// status: 0 ok; 1000000 + j: pivot j of -M not positive; 2000000: non-finite entry in M.
// ----------------------------------------------------------------------------------------
constexpr int CH_NT = 1024;
constexpr int CH_SMEM_MAX_N = 128;

__global__ void __launch_bounds__(CH_NT) cholesky_kernel(const double *__restrict__ M_raw, int n, double spin_factor,
                                                         double *__restrict__ M, double *__restrict__ L,
                                                         double *__restrict__ Linv, double *__restrict__ energy,
                                                         int *__restrict__ status, double *__restrict__ gwork) {
  extern __shared__ double dyn[];
  __shared__ int bad;
  __shared__ double red[CH_NT / 32];
  const bool in_smem = n <= CH_SMEM_MAX_N;
  double *A = in_smem ? dyn : gwork;                       // n * n
  double *tmp = in_smem ? dyn + n * n : gwork + n * n;     // n
  const int tid = threadIdx.x;
  if (tid == 0) bad = 0;
  __syncthreads();
  for (int e = tid; e < n * n; e += CH_NT) {
    const int i = e / n, j = e % n;
    const double v = 0.5 * (M_raw[(long long)i * n + j] + M_raw[(long long)j * n + i]);
    M[e] = v;
    A[e] = -v;
    if (!isfinite(v)) bad = 2000000;
  }
  __syncthreads();
  double part = 0.0;
  for (int k = tid; k < n; k += CH_NT) part += M[(long long)k * n + k];
  for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o);
  if ((tid & 31) == 0) red[tid >> 5] = part;
  __syncthreads();
  if (tid == 0) {
    double s = 0.0;
    for (int w = 0; w < CH_NT / 32; ++w) s += red[w];
    *energy = 0.5 * spin_factor * s;
  }
  if (bad) {
    if (tid == 0) *status = bad;
    return;
  }
  // Right-looking factorisation of the lower triangle, two barriers per step:
  //   (a) column j scaled by 1/L_jj (and copied to col[] for conflict-free reads), L_jj stored;
  //   (b) trailing update A_ik -= L_ij L_kj over the triangle j < k <= i < n, flattened over all
  //       threads; the thread that finishes A_{j+1,j+1} (element 0) takes its square root and
  //       reciprocal for the next step, so no thread waits on a serial pivot computation.
  // The pivot test reads A_jj after the barrier, so every thread takes the same branch.
  double *col = tmp;                       // n: scaled column j
  double *rinv = tmp + n;                  // n: 1 / L_jj
  __shared__ double piv[2];                // sqrt and reciprocal of the next pivot
  if (tid == 0) {
    const double d0 = A[0];
    piv[0] = sqrt(d0);
    piv[1] = 1.0 / piv[0];
  }
  __syncthreads();
  for (int j = 0; j < n; ++j) {
    const double d = A[j * n + j];
    if (!(d > 0.0) || !isfinite(d)) {
      if (tid == 0) *status = 1000000 + j;
      return;
    }
    const double r = piv[0], ri = piv[1];
    for (int i = j + 1 + tid; i < n; i += CH_NT) {
      const double v = A[i * n + j] * ri;
      A[i * n + j] = v;
      col[i] = v;
    }
    if (tid == 0) rinv[j] = ri;
    __syncthreads();
    if (tid == 0) A[j * n + j] = r;  // after the barrier: every thread has read the pivot d
    const int m = n - 1 - j;  // trailing rows j+1 .. n-1
    const int T = m * (m + 1) / 2;
    for (int e = tid; e < T; e += CH_NT) {
      // row q of the trailing triangle starts at q (q + 1) / 2
      int q = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
      while (q * (q + 1) / 2 > e) --q;
      while ((q + 1) * (q + 2) / 2 <= e) ++q;
      const int i = j + 1 + q, k = j + 1 + (e - q * (q + 1) / 2);
      const double v = A[i * n + k] - col[i] * col[k];
      A[i * n + k] = v;
      if (e == 0 && v > 0.0 && isfinite(v)) {  // i == k == j + 1: the next pivot
        piv[0] = sqrt(v);
        piv[1] = 1.0 / piv[0];
      }
    }
    __syncthreads();
  }
  for (int e = tid; e < n * n; e += CH_NT) {
    const int i = e / n, j = e % n;
    L[e] = (j <= i) ? A[e] : 0.0;
  }
  // Inverse: L = U D with U = L D^-1 unit lower (U_ik = L_ik / L_kk) and D = diag(L), so
  // L^-1 = D^-1 Y with Y = U^-1.  Y by right-looking forward substitution from Y = I:
  //   step k: Y_ic -= U_ik Y_kc  for i > k, c <= k   (Y_kk = 1; Y_kc final after step k - 1).
  // Y_ic (c < i) lives in the unused upper triangle at A[c][i]; column k of U is staged in a
  // double buffer during the previous step, so one barrier per step suffices.
  double *ucol = tmp + 2 * n;              // 2 n: columns k (even / odd) of U
  for (int i = 1 + tid; i < n; i += CH_NT) ucol[i] = A[i * n] * rinv[0];
  for (int e = tid; e < n * n; e += CH_NT) {
    const int i = e / n, c = e % n;
    if (c > i) A[e] = 0.0;                 // Y starts at the identity (unit diagonal implicit)
  }
  __syncthreads();
  for (int k = 0; k < n; ++k) {
    const double *u = ucol + (k & 1) * n;
    double *unext = ucol + ((k + 1) & 1) * n;
    if (k + 1 < n)
      for (int i = k + 2 + tid; i < n; i += CH_NT) unext[i] = A[i * n + k + 1] * rinv[k + 1];
    // rectangle i in (k, n), c in [0, k]: lanes along i (contiguous in the upper triangle)
    const int rows = n - 1 - k, cols = k + 1;
    for (int e = tid; e < rows * cols; e += CH_NT) {
      const int c = e / rows, i = k + 1 + (e - c * rows);
      const double ykc = (c == k) ? 1.0 : A[c * n + k];
      A[c * n + i] -= u[i] * ykc;
    }
    __syncthreads();
  }
  for (int e = tid; e < n * n; e += CH_NT) {
    const int i = e / n, c = e % n;
    Linv[e] = (c < i) ? A[c * n + i] * rinv[i] : (c == i ? rinv[i] : 0.0);
  }
  if (tid == 0) *status = 0;
}

// ----------------------------------------------------------------------------------------
// The same factorisation on a cluster of CHC_C CTAs, for n <= CHC_MAX_N.  This GPU retires about
// two FP64 FMA per clock per SM, so the one-CTA kernel above is bound by one SM's FP64 pipe; here
// the work is spread over CHC_C SMs.
//   - Every CTA holds the whole symmetrised -M in shared memory (row stride lda = n | 1, odd, so
//     that a column walk does not hit one bank).  Each CTA symmetrises an eighth of the elements
//     and writes them into every CTA's copy (distributed shared memory) and into M.
//   - Columns are dealt in panels of CHC_B, panel p owned by CTA p % CHC_C.  After panel p is
//     published (a cluster barrier), every other CTA copies it from the owner's shared memory and
//     applies its rank-CHC_B update to the columns it owns.
//   - Look-ahead: the owner of panel p + 1 first updates only that panel's columns, factors it with
//     four warps (the panel in registers, one row group per warp and SM sub-partition, r and L_kj
//     published by warp 0 through shared memory) and arrives at the cluster barrier; its other
//     columns are updated after the arrival.
//     Every other CTA arrives right after its copy and updates its columns before it waits, so the
//     chain from one panel to the next is a copy, an 8-column update and the panel factorisation.
//   - Afterwards every CTA holds all of L; the columns of L^-1 are dealt in pairs, two per warp,
//     in an order that balances the FP64 work over the CTAs.  A warp holds its two columns in
//     registers (lane l: rows l, l + 32, l + 64, l + 96) and runs forward substitution: at step k
//     X_kc (final) is broadcast by a shuffle, the rows i > k take X_ic -= L_ik X_kc (only the row
//     groups below k), and row k + 1, then final, is scaled by 1 / L_(k+1)(k+1).
//   - A non-positive or non-finite pivot is written into every CTA's flag before the barrier, so all
//     CTAs leave the panel loop at the same point; the outputs then carry the same status codes as
//     above.
// Every element's arithmetic is fixed by the algorithm, not by the schedule: the panel updates of an
// element are applied in panel order (each a sum over the panel's columns in order, then one
// subtraction), and the substitution takes the steps k in order, so the result repeats bit for bit.
// All waits are hardware barriers (CTA and cluster); no CTA reads another's shared memory after the
// cluster barrier that follows the last panel.
// ----------------------------------------------------------------------------------------
namespace cg = cooperative_groups;
constexpr int CHC_NT = 256;
constexpr int CHC_C = 8;
constexpr int CHC_B = 8;
constexpr int CHC_MAX_N = 128;
constexpr int CHC_OWN = 16;  // columns a CTA owns at most: 128 / (8 x 8) panels of 8
static_assert(CHC_MAX_N <= CHC_C * CHC_B * (CHC_OWN / CHC_B), "own columns per CTA");
static_assert(CHC_MAX_N <= 2 * CHC_C * (CHC_NT / 32), "two columns of L^-1 per warp");
static_assert(CHC_MAX_N <= 128, "four rows per lane, four row groups in the panel factorisation");
static_assert(CHC_NT >= 128, "four warps factor a panel");

__device__ __forceinline__ void cluster_arrive_release() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait_acquire() {
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ bool finite_bits(double v) {
  return ((__double_as_longlong(v) >> 52) & 0x7ff) != 0x7ff;
}

// Panel (columns c0 .. c0 + w - 1, rows c0 .. n - 1, stored at columns s0 .. s0 + w - 1 of A) factored
// right-looking by the CTA's first NW warps, spread over the SM sub-partitions: an FP64 warp
// instruction issues once per about 64 cycles on a sub-partition, so one warp holding all rows would
// serialise several times the instructions.  Warp m holds rows c0 + lane + 32 m in registers.  For column j, warp 0 takes the pivot d (lane j),
// r = 1 / sqrt(d), scales its rows, and publishes r and the panel rows' scaled L_kj (k < CHC_B)
// through xch (double-buffered by column parity, so one named barrier per column suffices); then
// every warp scales its rows and updates the panel's later columns.  The arithmetic of every
// element is that of a one-warp right-looking factorisation.  Returns 0, or 1000000 + the column of
// a non-positive or non-finite pivot (the same in all NW warps).  Call with threads 0 .. 32 NW - 1;
// the panel must have at most 32 NW rows.
template <int NW>
__device__ __forceinline__ int chc_factor_panel(double *A, int lda, int n, int c0, int s0, int w, double *xch,
                                                int *xflag) {
  const int lane = threadIdx.x & 31, wm = threadIdx.x >> 5, h = n - c0, i = lane + 32 * wm;
  double a[CHC_B];
#pragma unroll
  for (int j = 0; j < CHC_B; ++j) a[j] = (i < h && j < w) ? A[(c0 + i) * lda + s0 + j] : 0.0;
  int status = 0;
#pragma unroll
  for (int j = 0; j < CHC_B; ++j) {
    if (j < w && status == 0) {
      double *buf = xch + (j & 1) * (CHC_B + 1);  // [k]: scaled L_(c0+k)(c0+j), [CHC_B]: r
      if (wm == 0) {
        const double d = __shfl_sync(0xffffffffu, a[j], j);  // row c0 + j: lane j of warp 0
        const long long bits = __double_as_longlong(d);
        const bool ok = bits > 0 && ((bits >> 52) & 0x7ff) != 0x7ff;  // d > 0 and finite
        double r = 0.0;
        if (ok) {
          r = rsqrt(d);
          if (lane > j) a[j] *= r;
          else if (lane == j) a[j] = d * r;
        }
        if (lane < CHC_B) buf[lane] = a[j];
        if (lane == 0) {
          buf[CHC_B] = r;
          xflag[j & 1] = ok ? 0 : 1000000 + c0 + j;
        }
      }
      asm volatile("bar.sync 1, %0;" ::"n"(32 * NW) : "memory");
      status = xflag[j & 1];
      if (status == 0) {
        if (wm > 0) a[j] *= buf[CHC_B];  // rows c0 + 32 and below, all past the pivot
#pragma unroll
        for (int k = j + 1; k < CHC_B; ++k) {
          if (k < w) {
            const double lkj = buf[k];
            if (wm > 0 || lane >= k) a[k] -= a[j] * lkj;
          }
        }
      }
    }
  }
  if (i < h) {
#pragma unroll
    for (int j = 0; j < CHC_B; ++j)
      if (j < w) A[(c0 + i) * lda + s0 + j] = a[j];
  }
  return status;
}

__global__ void __cluster_dims__(CHC_C, 1, 1) __launch_bounds__(CHC_NT)
    cholesky_cluster_kernel(const double *__restrict__ M_raw, int n, double spin_factor, double *__restrict__ M,
                            double *__restrict__ L, double *__restrict__ Linv, double *__restrict__ energy,
                            int *__restrict__ status) {
  cg::cluster_group cluster = cg::this_cluster();
  extern __shared__ double dyn[];
  __shared__ int bad;   // non-finite input: written into every CTA before the first barrier
  __shared__ int pf;    // pivot failure met by this CTA while it factors a panel
  __shared__ int fail;  // pivot failure of a panel's owner, written into every CTA before the
                        // cluster barrier and read only after it
  __shared__ int own[CHC_OWN];  // the columns this CTA owns, ascending (-1: none)
  __shared__ double red[CHC_NT / 32];
  __shared__ double xch[2 * (CHC_B + 1)];  // panel factorisation: r and the scaled panel rows
  __shared__ int xflag[2];
  const int rank = (int)cluster.block_rank(), tid = threadIdx.x;
  const int lda = n | 1;
  double *A = dyn;                          // n x lda
  double *rinv = dyn + (size_t)n * lda;     // n: 1 / L_kk
  const int P = (n + CHC_B - 1) / CHC_B;
  if (tid == 0) {
    bad = 0;
    pf = 0;
    fail = 0;
    int m = 0;
    for (int p = rank; p < P; p += CHC_C)
      for (int c = p * CHC_B; c < min(n, (p + 1) * CHC_B); ++c) own[m++] = c;
    for (; m < CHC_OWN; ++m) own[m] = -1;
  }
  cluster.sync();  // every CTA has started and cleared its flags before any write across CTAs
  // -M symmetrised: this CTA's eighth of the elements, M_sym = (M_raw + M_raw^T) / 2 written to M
  // and its negative into every CTA's A
  {
    double *Aq[CHC_C];
#pragma unroll
    for (int q = 0; q < CHC_C; ++q) Aq[q] = cluster.map_shared_rank(A, q);
    constexpr int U = CHC_MAX_N * CHC_MAX_N / (CHC_NT * CHC_C);  // elements per thread at n = 128
    const int nn = n * n;
    double s[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = (u * CHC_C + rank) * CHC_NT + tid;
      s[u] = 0.0;
      if (e < nn) {
        const int i = e / n, j = e - (e / n) * n;
        s[u] = i == j ? M_raw[e] : 0.5 * (M_raw[e] + M_raw[j * n + i]);
      }
    }
    bool ok = true;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = (u * CHC_C + rank) * CHC_NT + tid;
      if (e < nn) {
        const int i = e / n, j = e - (e / n) * n;
        M[e] = s[u];
        ok = ok && finite_bits(s[u]);
        const double v = __longlong_as_double(__double_as_longlong(s[u]) ^ (long long)0x8000000000000000ull);
#pragma unroll
        for (int q = 0; q < CHC_C; ++q) Aq[q][i * lda + j] = v;
      }
    }
    if (!ok)
      for (int q = 0; q < CHC_C; ++q) *cluster.map_shared_rank(&bad, q) = 2000000;  // every CTA sees it
  }
  if (rank == 0) {
    double part = 0.0;
    for (int k = tid; k < n; k += CHC_NT) part += M_raw[k * n + k];
    for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o);
    if ((tid & 31) == 0) red[tid >> 5] = part;
    __syncthreads();
    if (tid == 0) {
      double t = 0.0;
      for (int w = 0; w < CHC_NT / 32; ++w) t += red[w];
      *energy = 0.5 * spin_factor * t;
    }
  }
  cluster.sync();  // A complete in every CTA, bad the same everywhere
  // panel 0 by its owner
  if (!bad && rank == 0) {
    if (tid < 128) {
      const int r = chc_factor_panel<4>(A, lda, n, 0, 0, min(n, CHC_B), xch, xflag);
      if (tid == 0) pf = r;
    }
    __syncthreads();
    if (pf && tid < CHC_C) *cluster.map_shared_rank(&fail, tid) = pf;
  }
  cluster.sync();  // panel 0 final in its owner's shared memory (or the failure announced)
  const int lane16 = tid & 15, row16 = tid >> 4;  // (own column, row) lanes of the column-parallel update
  for (int p = 0; p < P; ++p) {
    if (bad || fail) break;  // the same in every CTA after the barrier
    const int c0 = p * CHC_B, c1 = min(n, c0 + CHC_B), w = c1 - c0, owner = p % CHC_C;
    if (rank != owner) {  // rows c0.. of the panel's columns from the owner, four loads in flight
      const double *src = cluster.map_shared_rank(A, owner);
      const int ne = (n - c0) * CHC_B;
      for (int base = tid; base < ne; base += 4 * CHC_NT) {
        double v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int e = base + u * CHC_NT, c = e & (CHC_B - 1);
          v[u] = (e < ne && c < w) ? src[(c0 + (e >> 3)) * lda + c0 + c] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int e = base + u * CHC_NT, c = e & (CHC_B - 1);
          if (e < ne && c < w) A[(c0 + (e >> 3)) * lda + c0 + c] = v[u];
        }
      }
    }
    __syncthreads();  // the panel, and the previous panel's updates of this CTA's columns, complete
    const bool ahead = p + 1 < P && rank == (p + 1) % CHC_C;
    const int c2 = min(n, c1 + CHC_B);
    if (ahead) {
      // rank-w update of the next panel's columns k in [c1, c2), rows i >= k, then its factorisation
      const int col = tid & (CHC_B - 1), rl = tid >> 3, k = c1 + col;
      if (k < c2)
        for (int i = c1 + rl; i < n; i += CHC_NT / CHC_B) {
          if (i < k) continue;
          double acc = 0.0;
          for (int j = c0; j < c1; ++j) acc += A[i * lda + j] * A[k * lda + j];
          A[i * lda + k] -= acc;
        }
      __syncthreads();
      if (tid < 128) {
        const int r = chc_factor_panel<4>(A, lda, n, c1, c1, c2 - c1, xch, xflag);
        if (tid == 0) pf = r;
      }
      __syncthreads();
      if (pf && tid < CHC_C) *cluster.map_shared_rank(&fail, tid) = pf;
    }
    cluster_arrive_release();  // the next panel is published once every CTA has arrived
    // rank-w update of this CTA's other columns k >= c1 (k >= c2 for the look-ahead owner), rows i >= k
    {
      const int k = own[lane16];
      if (k >= (ahead ? c2 : c1))
        for (int i = k + row16; i < n; i += CHC_NT / 16) {
          double acc = 0.0;
          for (int j = c0; j < c1; ++j) acc += A[i * lda + j] * A[k * lda + j];
          A[i * lda + k] -= acc;
        }
    }
    cluster_wait_acquire();
  }
  cluster.sync();  // no CTA reads another's shared memory past this point
  if (bad || fail) {
    if (rank == 0 && tid == 0) *status = bad ? bad : fail;
    return;
  }
  for (int e = tid; e < n * CHC_OWN; e += CHC_NT) {
    const int i = e / CHC_OWN, cc = e % CHC_OWN, c = own[cc];
    if (c < 0) continue;
    L[(long long)i * n + c] = (i >= c) ? A[i * lda + c] : 0.0;
  }
  for (int k = tid; k < n; k += CHC_NT) rinv[k] = 1.0 / A[k * lda + k];
  __syncthreads();
  {
    const int lane = tid & 31, wp = tid >> 5;
    // column pairs (2t, 2t + 1), dealt so that every CTA gets early and late columns alike
    const int t = CHC_C * wp + ((wp & 1) ? CHC_C - 1 - rank : rank);
    const int ca = 2 * t < n ? 2 * t : -1, cb = 2 * t + 1 < n ? 2 * t + 1 : -1;
    double xa[4], xb[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int i = lane + 32 * m;
      xa[m] = (ca >= 0 && i == ca) ? rinv[ca] : 0.0;
      xb[m] = (cb >= 0 && i == cb) ? rinv[cb] : 0.0;
    }
    if (ca >= 0) {
#pragma unroll
      for (int kb = 0; kb < 4; ++kb) {
        // steps k in this row group; the last step, n - 2, makes row n - 1 final
        const int kbeg = max(ca, 32 * kb), kend = min(n - 1, 32 * kb + 32);
        for (int k = kbeg; k < kend; ++k) {
          const int lk = k & 31;
          const double xka = __shfl_sync(0xffffffffu, xa[kb], lk), xkb = __shfl_sync(0xffffffffu, xb[kb], lk);
          const bool ub = cb >= 0 && k >= cb;
#pragma unroll
          for (int m = kb; m < 4; ++m) {
            const int i = lane + 32 * m;
            if (i > k && i < n) {
              const double lik = A[i * lda + k];
              xa[m] -= lik * xka;
              if (ub) xb[m] -= lik * xkb;
            }
          }
          // row k + 1 is final: lane (k + 1) & 31 of row group kb, or lane 0 of group kb + 1
          if (lk != 31) {
            if (lane == lk + 1) {
              const double s = rinv[k + 1];
              xa[kb] *= s;
              if (ub) xb[kb] *= s;
            }
          } else if (kb < 3) {
            if (lane == 0) {
              const double s = rinv[k + 1];
              xa[kb + 1] *= s;
              if (ub) xb[kb + 1] *= s;
            }
          }
        }
      }
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int i = lane + 32 * m;
      if (i < n) {
        if (ca >= 0) Linv[(long long)i * n + ca] = i >= ca ? xa[m] : 0.0;
        if (cb >= 0) Linv[(long long)i * n + cb] = i >= cb ? xb[m] : 0.0;
      }
    }
  }
  if (rank == 0 && tid == 0) *status = 0;
}

// ----------------------------------------------------------------------------------------
// The factorisation for CHC_MAX_N < n <= CHW_MAX_N on a cluster of CHC_C CTAs whose shared memory
// holds only their own columns: all of -M does not fit one SM at these sizes.
//   - Panel p (8 columns) is owned by CTA p % CHC_C, which keeps its panels' columns, all rows,
//     in `own` (local column 8 (p / CHC_C) + j, odd row stride).  Each CTA symmetrises its own
//     columns straight from M_raw and writes them to M.
//   - The panel loop is that of the kernel above: after panel p is published, every CTA copies it
//     (rows c0..n-1) from its owner into its panel buffer p & 1; the owner of panel p + 1 updates that
//     panel's columns, factors it (eight warps, one row group each) and arrives at the cluster
//     barrier; every CTA updates its other columns before it waits.
//   - Afterwards each CTA writes its columns of L, and of L^T into the workspace (row c of L^T is
//     column c of L); after a cluster barrier, the columns of L^-1 are dealt in groups of four, one
//     group per warp, in an order that balances the FP64 work over the CTAs.  Forward substitution
//     holds a warp's four columns in registers (lane l: rows l + 32 m) and reads column k of L from
//     shared memory, where 32 rows of L^T at a time are staged (in the space of `own`).
// Status codes as above.
// ----------------------------------------------------------------------------------------
constexpr int CHW_MAX_N = 256;
constexpr int CHW_LDO = 33;  // own-column block: up to 32 columns per CTA, odd row stride
constexpr int CHW_LDP = 9;   // panel buffer row stride
static_assert(CHW_MAX_N <= CHC_C * CHC_B * 4, "four panels per CTA at most");
static_assert(CHW_MAX_N <= 4 * CHC_C * (CHC_NT / 32), "four columns of L^-1 per warp");
static_assert(CHW_MAX_N <= 32 * (CHC_NT / 32), "one row group per warp in the panel factorisation");
static_assert(32 * CHW_MAX_N <= CHW_MAX_N * CHW_LDO, "a 32-row slab of L^T fits in the own-column block");

__global__ void __cluster_dims__(CHC_C, 1, 1) __launch_bounds__(CHC_NT)
    cholesky_cluster_wide_kernel(const double *__restrict__ M_raw, int n, double spin_factor, double *__restrict__ M,
                                 double *__restrict__ L, double *__restrict__ Linv, double *__restrict__ energy,
                                 int *__restrict__ status, double *__restrict__ Lt) {
  cg::cluster_group cluster = cg::this_cluster();
  extern __shared__ double dyn[];
  __shared__ int bad, pf, fail;
  __shared__ double red[CHC_NT / 32];
  __shared__ double xch[2 * (CHC_B + 1)];
  __shared__ int xflag[2];
  const int rank = (int)cluster.block_rank(), tid = threadIdx.x;
  double *own = dyn;                              // n x CHW_LDO
  // two n x CHW_LDP panel buffers, panel p in buffer p & 1: after arriving at the barrier a thread
  // still reads panel p while a faster one, past the wait, may already copy panel p + 1
  double *pbuf = own + (size_t)n * CHW_LDO;
  double *rinv = pbuf + 2 * (size_t)n * CHW_LDP;  // n
  const int P = (n + CHC_B - 1) / CHC_B;
  if (tid == 0) {
    bad = 0;
    pf = 0;
    fail = 0;
  }
  cluster.sync();  // every CTA has started and cleared its flags before any write across CTAs
  // own columns of -M_sym (all rows), M_sym written to M: local column lc = 8 t + j holds column
  // c = 8 (rank + CHC_C t) + j
  {
    bool ok = true;
    for (int e = tid; e < n * 32; e += CHC_NT) {
      const int i = e >> 5, lc = e & 31, c = CHC_B * (rank + CHC_C * (lc >> 3)) + (lc & 7);
      if (c >= n) continue;
      const double v = i == c ? M_raw[(long long)c * n + c]
                              : 0.5 * (M_raw[(long long)i * n + c] + M_raw[(long long)c * n + i]);
      M[(long long)i * n + c] = v;
      ok = ok && finite_bits(v);
      own[i * CHW_LDO + lc] = __longlong_as_double(__double_as_longlong(v) ^ (long long)0x8000000000000000ull);
    }
    if (!ok)
      for (int q = 0; q < CHC_C; ++q) *cluster.map_shared_rank(&bad, q) = 2000000;
  }
  if (rank == 0) {
    double part = 0.0;
    for (int k = tid; k < n; k += CHC_NT) part += M_raw[(long long)k * n + k];
    for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o);
    if ((tid & 31) == 0) red[tid >> 5] = part;
    __syncthreads();
    if (tid == 0) {
      double t = 0.0;
      for (int w = 0; w < CHC_NT / 32; ++w) t += red[w];
      *energy = 0.5 * spin_factor * t;
    }
  }
  cluster.sync();  // own columns complete, bad the same everywhere
  if (!bad && rank == 0) {
    const int r = chc_factor_panel<CHC_NT / 32>(own, CHW_LDO, n, 0, 0, min(n, CHC_B), xch, xflag);
    if (tid == 0) pf = r;
    __syncthreads();
    if (pf && tid < CHC_C) *cluster.map_shared_rank(&fail, tid) = pf;
  }
  cluster.sync();  // panel 0 final in its owner's shared memory (or the failure announced)
  for (int p = 0; p < P; ++p) {
    if (bad || fail) break;  // the same in every CTA after the barrier
    const int c0 = p * CHC_B, c1 = min(n, c0 + CHC_B), w = c1 - c0, owner = p % CHC_C;
    const int s_p = CHC_B * (p / CHC_C);  // the panel's columns in its owner's block
    double *pb = pbuf + (size_t)(p & 1) * n * CHW_LDP;
    {
      // rows c0.. of the panel into the panel buffer (from the owner's block; the owner's own copy
      // is local), four loads in flight
      const double *src = rank == owner ? own : cluster.map_shared_rank(own, owner);
      const int ne = (n - c0) * CHC_B;
      for (int base = tid; base < ne; base += 4 * CHC_NT) {
        double v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int e = base + u * CHC_NT, c = e & (CHC_B - 1);
          v[u] = (e < ne && c < w) ? src[(c0 + (e >> 3)) * CHW_LDO + s_p + c] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int e = base + u * CHC_NT, c = e & (CHC_B - 1);
          if (e < ne && c < w) pb[(c0 + (e >> 3)) * CHW_LDP + c] = v[u];
        }
      }
    }
    __syncthreads();  // the panel copied, and the previous panel's updates of this CTA's columns done
    const bool ahead = p + 1 < P && rank == (p + 1) % CHC_C;
    const int c2 = min(n, c1 + CHC_B);
    if (ahead) {
      const int s_n = CHC_B * ((p + 1) / CHC_C);
      const int col = tid & (CHC_B - 1), rl = tid >> 3, k = c1 + col;
      if (k < c2)
        for (int i = c1 + rl; i < n; i += CHC_NT / CHC_B) {
          if (i < k) continue;
          double acc = 0.0;
          for (int j = 0; j < w; ++j) acc += pb[i * CHW_LDP + j] * pb[k * CHW_LDP + j];
          own[i * CHW_LDO + s_n + col] -= acc;
        }
      __syncthreads();
      const int r = chc_factor_panel<CHC_NT / 32>(own, CHW_LDO, n, c1, s_n, c2 - c1, xch, xflag);
      if (tid == 0) pf = r;
      __syncthreads();
      if (pf && tid < CHC_C) *cluster.map_shared_rank(&fail, tid) = pf;
    }
    cluster_arrive_release();  // the next panel is published once every CTA has arrived
    {
      // rank-w update of this CTA's other columns k >= c1 (k >= c2 for the look-ahead owner), rows i >= k
      const int lc = tid & 31, rl = tid >> 5;
      const int k = CHC_B * (rank + CHC_C * (lc >> 3)) + (lc & 7);
      if (k < n && k >= (ahead ? c2 : c1))
        for (int i = k + rl; i < n; i += CHC_NT / 32) {
          double acc = 0.0;
          for (int j = 0; j < w; ++j) acc += pb[i * CHW_LDP + j] * pb[k * CHW_LDP + j];
          own[i * CHW_LDO + lc] -= acc;
        }
    }
    cluster_wait_acquire();
  }
  cluster.sync();  // no CTA reads another's shared memory past this point
  if (bad || fail) {
    if (rank == 0 && tid == 0) *status = bad ? bad : fail;
    return;
  }
  // this CTA's columns of L (row-major, zeros above the diagonal) and of L^T (row c = column c of L)
  for (int e = tid; e < n * 32; e += CHC_NT) {
    const int i = e >> 5, lc = e & 31, c = CHC_B * (rank + CHC_C * (lc >> 3)) + (lc & 7);
    if (c >= n) continue;
    const double v = own[i * CHW_LDO + lc];
    L[(long long)i * n + c] = i >= c ? v : 0.0;
    if (i >= c) Lt[(long long)c * n + i] = v;
  }
  __threadfence();
  cluster.sync();  // every column of L^T written
  for (int k = tid; k < n; k += CHC_NT) rinv[k] = 1.0 / __ldcg(Lt + (long long)k * n + k);
  {
    double *S = own;  // 32 rows of L^T at a time
    const int lane = tid & 31, wp = tid >> 5;
    const int t = CHC_C * wp + ((wp & 1) ? CHC_C - 1 - rank : rank);  // group of columns 4t .. 4t + 3
    int cq[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) cq[q] = 4 * t + q < n ? 4 * t + q : -1;
    __syncthreads();  // rinv complete
    double x[4][8];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int m = 0; m < 8; ++m) x[q][m] = (cq[q] >= 0 && lane + 32 * m == cq[q]) ? rinv[cq[q]] : 0.0;
#pragma unroll
    for (int kb = 0; kb < 8; ++kb) {
      const int k_lo = 32 * kb, k_hi = min(n, 32 * kb + 32);
      if (k_lo >= n) break;  // the same in every thread
      __syncthreads();      // the previous slab is no longer read
      for (int e = tid; e < (k_hi - k_lo) * n; e += CHC_NT) {
        const int kk = e / n, i = e - kk * n;
        S[e] = i > k_lo + kk ? __ldcg(Lt + (long long)(k_lo + kk) * n + i) : 0.0;
      }
      __syncthreads();
      if (cq[0] >= 0) {
        // steps k in this slab; the last step, n - 2, makes row n - 1 final
        for (int k = max(cq[0], k_lo); k < min(n - 1, k_hi); ++k) {
          const int lk = k & 31;
          double xk[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) xk[q] = __shfl_sync(0xffffffffu, x[q][kb], lk);
          const double *Sk = S + (k - k_lo) * n;
#pragma unroll
          for (int m = kb; m < 8; ++m) {
            const int i = lane + 32 * m;
            if (i > k && i < n) {
              const double lik = Sk[i];
#pragma unroll
              for (int q = 0; q < 4; ++q)
                if (cq[q] >= 0 && k >= cq[q]) x[q][m] -= lik * xk[q];
            }
          }
          // row k + 1 is final: lane (k + 1) & 31 of row group kb, or lane 0 of group kb + 1
          if (lk != 31) {
            if (lane == lk + 1) {
              const double sc = rinv[k + 1];
#pragma unroll
              for (int q = 0; q < 4; ++q)
                if (cq[q] >= 0 && k >= cq[q]) x[q][kb] *= sc;
            }
          } else if (kb < 7) {
            if (lane == 0) {
              const double sc = rinv[k + 1];
#pragma unroll
              for (int q = 0; q < 4; ++q)
                if (cq[q] >= 0 && k >= cq[q]) x[q][kb + 1] *= sc;
            }
          }
        }
      }
    }
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const int i = lane + 32 * m;
      if (i < n) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (cq[q] >= 0) Linv[(long long)i * n + cq[q]] = i >= cq[q] ? x[q][m] : 0.0;
      }
    }
  }
  if (rank == 0 && tid == 0) *status = 0;
}

// ----------------------------------------------------------------------------------------
// The same for n <= 32 in one CTA.  A chain of n pivots bounds it: each FP64 instruction of the chain takes
// a scheduler about 64 cycles, and the cluster form adds its barriers and panel copies (26 us at n = 16,
// this one 19).
//   - Lane i of every warp is row i; warp w holds the columns k = w, w + 8, ... of -M and of Y in
//     registers.  Elimination in LDL^T form: column j, published in shared memory by its warp, gives
//     t_i = A_ij / d_j = U_ij, then A_ik -= t_i A_kj (k > j) and Y_ic -= t_i Y_jc (c <= j), so that
//     Y = U^-1 grows along with U and only one reciprocal per column is on the chain.
//   - The warp that owns column j + 1 updates it first and publishes it before the rest of its work.
//   - At the end L = U sqrt(D) and L^-1 = D^-1/2 Y, all square roots side by side.
// Every element's arithmetic is fixed, so the result repeats bit for bit.  Same status codes as above.
// ----------------------------------------------------------------------------------------
constexpr int CHS_MAX_N = 32, CHS_W = 8, CHS_NT = CHS_W * 32, CHS_S = CHS_MAX_N / CHS_W;

__global__ void __launch_bounds__(CHS_NT) cholesky_small_kernel(const double *__restrict__ M_raw, int n,
                                                                double spin_factor, double *__restrict__ M,
                                                                double *__restrict__ L, double *__restrict__ Linv,
                                                                double *__restrict__ energy,
                                                                int *__restrict__ status) {
  __shared__ double col[2][CHS_MAX_N], diag[CHS_MAX_N], U[CHS_MAX_N][CHS_MAX_N + 1];
  const int tid = threadIdx.x, i = tid & 31, w = tid >> 5;
  double a[CHS_S], y[CHS_S];
  bool ok = true;
#pragma unroll
  for (int s = 0; s < CHS_S; ++s) {
    const int k = s * CHS_W + w;
    a[s] = 0.0;
    y[s] = 0.0;
    if (i < n && k < n) {
      const double v = i == k ? M_raw[i * n + i] : 0.5 * (M_raw[i * n + k] + M_raw[k * n + i]);
      M[i * n + k] = v;
      ok = ok && finite_bits(v);
      a[s] = -v;
    }
  }
  if (w == 0) {
    double part = i < n ? M_raw[i * n + i] : 0.0;
    for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o);
    if (i == 0) *energy = 0.5 * spin_factor * part;
    col[0][i] = a[0];
  }
  if (__syncthreads_or(!ok)) {
    if (tid == 0) *status = 2000000;
    return;
  }
#pragma unroll
  for (int jb = 0; jb < CHS_S; ++jb) {
    for (int jw = 0; jw < CHS_W; ++jw) {
      const int j = jb * CHS_W + jw;
      if (j >= n) break;
      if (j > 0) __syncthreads();
      const double *c = col[j & 1];
      const double d = c[j];
      if (__double_as_longlong(d) <= 0 || !finite_bits(d)) {  // the same value in every thread
        if (tid == 0) *status = 1000000 + j;
        return;
      }
      // a division would cost the chain 1 us per column more (the reciprocal and the product round twice, as
      // scaling by rsqrt does in the cluster form); it is taken where the reciprocal is not a normal number
      const int dh = __double2hiint(d);
      const double t = i > j ? (dh >= 0x00200000 && dh < 0x7fd00000 ? c[i] * __drcp_rn(d) : c[i] / d) : 0.0;
      bool first = w == ((j + 1) & (CHS_W - 1));  // owner of column j + 1, not published yet
#pragma unroll
      for (int s = jb; s < CHS_S; ++s) {
        const int k = s * CHS_W + w;
        if (k > j && k < n) {
          a[s] = fma(-t, c[k], a[s]);
          if (first) {
            col[(j + 1) & 1][i] = a[s];
            first = false;
          }
        }
      }
      if (w == jw) U[j][i] = t;
      if (tid == 0) diag[j] = d;
#pragma unroll
      for (int s = 0; s <= jb; ++s) {
        const int cc = s * CHS_W + w;
        const double yj = __shfl_sync(0xffffffffu, y[s], j);
        if (cc <= j) y[s] = fma(-t, cc == j ? 1.0 : yj, y[s]);
      }
    }
  }
  __syncthreads();
  const double di = i < n ? diag[i] : 1.0;
  const double root = sqrt(di), inv = 1.0 / root;
  if (w == 0) col[0][i] = root;
  __syncthreads();
#pragma unroll
  for (int s = 0; s < CHS_S; ++s) {
    const int k = s * CHS_W + w;
    if (i < n && k < n) {
      L[i * n + k] = k < i ? U[k][i] * col[0][k] : k == i ? root : 0.0;
      Linv[i * n + k] = k < i ? y[s] * inv : k == i ? inv : 0.0;
    }
  }
  if (tid == 0) *status = 0;
}

static bool cluster_cholesky_off() {
  static const bool off = [] {
    const char *v = std::getenv("ACE_CHOLESKY_ONE_CTA");
    return v && *v && *v != '0';
  }();
  return off;
}

// Once per device and kernel: the shared-memory limit for the largest n, and whether such a cluster
// fits (state[dev]: 0 unknown, 1 usable, -1 not).
template <typename K>
static bool cluster_ready(K kernel, size_t smax, int *state, cudaStream_t st) {
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) return false;
  if (state[dev] == 0) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smax);
    int clusters = 0;
    if (e == cudaSuccess) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(CHC_C);
      cfg.blockDim = dim3(CHC_NT);
      cfg.dynamicSmemBytes = smax;
      cfg.stream = st;
      e = cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg);
    }
    cudaGetLastError();
    state[dev] = (e == cudaSuccess && clusters > 0) ? 1 : -1;
  }
  return state[dev] == 1;
}

cudaError_t launch_cholesky(const double *M_raw, int n, double spin_factor, double *M, double *L, double *Linv,
                            double *energy, int *status, double *gwork, cudaStream_t st) {
  // up to 32 rows (one lane each) in one CTA; stage times, small against cluster: 14 and 23 us at n = 12, 19
  // and 26 at 16, 27 and 37 at 24
  if (!cluster_cholesky_off() && n <= CHS_MAX_N) {
    cholesky_small_kernel<<<1, CHS_NT, 0, st>>>(M_raw, n, spin_factor, M, L, Linv, energy, status);
    return cudaGetLastError();
  }
  if (!cluster_cholesky_off() && n <= CHC_MAX_N) {
    static int state[64] = {};
    const size_t smax = sizeof(double) * ((size_t)CHC_MAX_N * (CHC_MAX_N | 1) + (size_t)CHC_MAX_N);
    if (cluster_ready(cholesky_cluster_kernel, smax, state, st)) {
      const size_t smem = sizeof(double) * ((size_t)n * (n | 1) + (size_t)n);
      cholesky_cluster_kernel<<<CHC_C, CHC_NT, smem, st>>>(M_raw, n, spin_factor, M, L, Linv, energy, status);
      return cudaGetLastError();
    }
  }
  if (!cluster_cholesky_off() && n > CHC_MAX_N && n <= CHW_MAX_N && gwork != nullptr) {
    // columns spread over the cluster; gwork (n x n doubles at least) holds L^T
    static int state[64] = {};
    const size_t smax = sizeof(double) * (size_t)CHW_MAX_N * (CHW_LDO + 2 * CHW_LDP + 1);
    if (cluster_ready(cholesky_cluster_wide_kernel, smax, state, st)) {
      const size_t smem = sizeof(double) * (size_t)n * (CHW_LDO + 2 * CHW_LDP + 1);
      cholesky_cluster_wide_kernel<<<CHC_C, CHC_NT, smem, st>>>(M_raw, n, spin_factor, M, L, Linv, energy, status,
                                                                 gwork);
      return cudaGetLastError();
    }
  }
  const size_t smem = n <= CH_SMEM_MAX_N ? sizeof(double) * ((size_t)n * n + 4 * n) : 0;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(cholesky_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  if (n > CH_SMEM_MAX_N && gwork == nullptr) return cudaErrorInvalidValue;
  cholesky_kernel<<<1, CH_NT, smem, st>>>(M_raw, n, spin_factor, M, L, Linv, energy, status, gwork);
  return cudaGetLastError();
}

// ----------------------------------------------------------------------------------------
// Screen compaction (one CTA): keep (i <= j) iff i == j or rho_cut <= 0 or O_ij >= rho_cut,
// in lexicographic order; packs = consecutive pairs two at a time.  Also writes the symmetric O.
// ----------------------------------------------------------------------------------------
constexpr int CP_NT = 1024;

__global__ void __launch_bounds__(CP_NT) compact_kernel(const double *__restrict__ O, int n, double rho_cut,
                                                        int2 *__restrict__ pairs, int4 *__restrict__ packs,
                                                        int *__restrict__ count, double *__restrict__ O_sym) {
  __shared__ int warp_sums[CP_NT / 32];
  __shared__ int running;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (tid == 0) running = 0;
  for (int base = tid; base < n * n; base += 4 * CP_NT) {  // four loads in flight per thread
    double v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = base + u * CP_NT, i = e / n, j = e % n;
      v[u] = e < n * n ? ((i <= j) ? O[e] : O[(long long)j * n + i]) : 0.0;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (base + u * CP_NT < n * n) O_sym[base + u * CP_NT] = v[u];
  }
  __syncthreads();
  const long long total = (long long)n * (n + 1) / 2;
  for (long long base = 0; base < total; base += CP_NT) {
    const long long e = base + tid;
    int keep = 0, i = 0, j = 0;
    if (e < total) {
      // row-major enumeration of the upper triangle: row i holds n - i entries
      // row i starts at s(i) = i (2n - i + 1) / 2; take the largest i with s(i) <= e (an FP32
      // estimate, made exact by the integer corrections below; FP64 is slow on this GPU)
      const float b = 2.0f * (float)n + 1.0f;
      i = (int)((b - sqrtf(fmaxf(b * b - 8.0f * (float)e, 0.0f))) * 0.5f);
      if (i < 0) i = 0;
      if (i > n - 1) i = n - 1;
      while (i > 0 && (long long)i * (2 * n - i + 1) / 2 > e) --i;
      while ((long long)(i + 1) * (2 * n - i) / 2 <= e) ++i;
      j = i + (int)(e - (long long)i * (2 * n - i + 1) / 2);
      const double o = O[(long long)i * n + j];
      keep = (i == j) || (rho_cut <= 0.0) || (o >= rho_cut);
    }
    const unsigned ballot = __ballot_sync(0xffffffffu, keep);
    const int prefix = __popc(ballot & ((1u << lane) - 1u));
    if (lane == 0) warp_sums[wid] = __popc(ballot);
    __syncthreads();
    int off = running;
    for (int w = 0; w < wid; ++w) off += warp_sums[w];
    if (keep) pairs[off + prefix] = make_int2(i, j);
    __syncthreads();
    if (tid == 0) {
      int s = 0;
      for (int w = 0; w < CP_NT / 32; ++w) s += warp_sums[w];
      running += s;
    }
    __syncthreads();
  }
  const int np = running;
  const int nk = (np + 1) / 2;
  for (int p = tid; p < nk; p += CP_NT) {
    const int2 a = pairs[2 * p];
    const int2 b = (2 * p + 1 < np) ? pairs[2 * p + 1] : make_int2(-1, -1);
    packs[p] = make_int4(a.x, a.y, b.x, b.y);
  }
  if (tid == 0) *count = np;
}

cudaError_t launch_screen_compact(const double *O, int n, double rho_cut, int2 *pairs, int4 *packs, int *count,
                                  double *O_sym, cudaStream_t st) {
  compact_kernel<<<1, CP_NT, 0, st>>>(O, n, rho_cut, pairs, packs, count, O_sym);
  return cudaGetLastError();
}

// ----------------------------------------------------------------------------------------
// Queue assembly: the pack lists of several builds, concatenated in build order.  Every CTA forms
// the prefix of the pack counts (nb is small) and copies a grid-strided share of the packs.
// ----------------------------------------------------------------------------------------
constexpr int QA_NT = 256;

__global__ void __launch_bounds__(QA_NT) queue_assemble_kernel(const QueueSrc *__restrict__ src, int nb,
                                                               int4 *__restrict__ out, int *__restrict__ pack_build,
                                                               int *__restrict__ np_out) {
  __shared__ int off[kQueueMaxBuilds + 1];
  if (threadIdx.x == 0) {
    int o = 0;
    for (int b = 0; b < nb; ++b) {
      off[b] = o;
      o += (__ldcg(src[b].count) + 1) / 2;
    }
    off[nb] = o;
    if (blockIdx.x == 0) *np_out = o;
  }
  __syncthreads();
  const int total = off[nb];
  for (int q = blockIdx.x * QA_NT + threadIdx.x; q < total; q += gridDim.x * QA_NT) {
    int lo = 0, hi = nb - 1;  // the last build whose list starts at or before q (never an empty one)
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (off[mid] <= q)
        lo = mid;
      else
        hi = mid - 1;
    }
    out[q] = src[lo].packs[q - off[lo]];
    pack_build[q] = lo;
  }
}

// One CTA per (plane i1, orbital a): the plane's max |phi|, and the orbital's max by an atomic max
// on the bit pattern (non-negative floats order as their bits do).
constexpr int PM_NT = 256;
__global__ void __launch_bounds__(PM_NT) plane_max_kernel(const float *__restrict__ phi, int n1, long long npl,
                                                         float *__restrict__ pmax, float *__restrict__ gmax) {
  __shared__ float red[PM_NT / 32];
  const int i1 = blockIdx.x, a = blockIdx.y;
  const float *p = phi + ((long long)a * n1 + i1) * npl;
  float m = 0.f;
  if ((npl & 3) == 0 && (reinterpret_cast<uintptr_t>(p) & 15) == 0) {
    const float4 *q = reinterpret_cast<const float4 *>(p);
    for (long long e = threadIdx.x; e < npl / 4; e += PM_NT) {
      const float4 v = __ldg(q + e);
      m = fmaxf(m, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
    }
  } else {
    for (long long e = threadIdx.x; e < npl; e += PM_NT) m = fmaxf(m, fabsf(__ldg(p + e)));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < PM_NT / 32; ++w) m = fmaxf(m, red[w]);
    pmax[(long long)a * n1 + i1] = m;
    atomicMax(reinterpret_cast<int *>(gmax + a), __float_as_int(m));
  }
}

cudaError_t launch_plane_max(const float *phi, int norb, int n1, long long npl, float *pmax, float *gmax,
                             cudaStream_t st) {
  if (norb < 1 || norb > 65535) return cudaErrorInvalidValue;
  plane_max_kernel<<<dim3(n1, norb), PM_NT, 0, st>>>(phi, n1, npl, pmax, gmax);
  return cudaGetLastError();
}

__global__ void flag_fanout_kernel(const int *src, int *const *dst, int n) {
  if (__ldcg(src) == 0) return;
  for (int i = threadIdx.x; i < n; i += blockDim.x) *dst[i] = 1;
}

cudaError_t launch_flag_fanout(const int *src, int *const *dst, int n, cudaStream_t st) {
  flag_fanout_kernel<<<1, 128, 0, st>>>(src, dst, n);
  return cudaGetLastError();
}

cudaError_t launch_queue_assemble(const QueueSrc *src, int nb, int4 *packs_out, int *pack_build, int *np_out,
                                  cudaStream_t st) {
  if (nb < 1 || nb > kQueueMaxBuilds) return cudaErrorInvalidValue;
  queue_assemble_kernel<<<2 * 152, QA_NT, 0, st>>>(src, nb, packs_out, pack_build, np_out);
  return cudaGetLastError();
}

// ----------------------------------------------------------------------------------------
// Elementwise precision conversion with scale.
// ----------------------------------------------------------------------------------------
template <typename Tin, typename Tout>
__global__ void convert_kernel(const Tin *__restrict__ in, Tout *__restrict__ out, long long count, double scale) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count;
       i += (long long)gridDim.x * blockDim.x)
    out[i] = (Tout)(scale * (double)in[i]);
}

template <typename Tin, typename Tout>
cudaError_t launch_convert(const Tin *in, Tout *out, long long count, double scale, cudaStream_t st) {
  const int nt = 256;
  const long long blocks = min((count + nt - 1) / nt, (long long)152 * 16);
  if (count == 0) return cudaSuccess;
  convert_kernel<Tin, Tout><<<(unsigned)blocks, nt, 0, st>>>(in, out, count, scale);
  return cudaGetLastError();
}
template cudaError_t launch_convert<double, float>(const double *, float *, long long, double, cudaStream_t);
template cudaError_t launch_convert<float, double>(const float *, double *, long long, double, cudaStream_t);
template cudaError_t launch_convert<double, double>(const double *, double *, long long, double, cudaStream_t);
template cudaError_t launch_convert<float, float>(const float *, float *, long long, double, cudaStream_t);

}  // namespace ace

namespace ace {
// A[c][k] = scale * C[k][c] (C is n x m FP64, A is m x n in T)
template <typename T>
__global__ void transpose_scale_kernel(const double *__restrict__ C, int n, int m, double scale, T *__restrict__ A) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n * m; e += gridDim.x * blockDim.x) {
    const int c = e / n, k = e % n;
    A[e] = (T)(scale * C[(long long)k * m + c]);
  }
}
template <typename T>
cudaError_t launch_transpose_scale(const double *C, int n, int m, double scale, T *A, cudaStream_t st) {
  const int nt = 256;
  const int blocks = (int)min((long long)(n * m + nt - 1) / nt, 4096LL);
  transpose_scale_kernel<T><<<blocks > 0 ? blocks : 1, nt, 0, st>>>(C, n, m, scale, A);
  return cudaGetLastError();
}
template cudaError_t launch_transpose_scale<float>(const double *, int, int, double, float *, cudaStream_t);
template cudaError_t launch_transpose_scale<double>(const double *, int, int, double, double *, cudaStream_t);
}  // namespace ace
