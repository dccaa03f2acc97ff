// line_pair.cuh -- the FP32 pair-potential chain in three passes (plane, pencil, plane), two
// neighbouring lines per thread.
//
// Every transform stage runs on two lines at once: an element is a "unit" of 16 bytes,
// {re of line A, re of line B, im of line A, im of line B}, held as two f32x2 register pairs.  All
// complex arithmetic is then packed FP32 (one instruction per two points for an add, two for half a
// twiddle multiply), multiplication by +-i is a renaming, index arithmetic and twiddle loads are
// shared by both lines, and shared memory moves in 16-byte accesses.  The chain this replaces kept
// (re, im) in a register pair: 189 warp instructions and 46 shared-memory wavefronts per 32 points
// of a pack on 96^3; see the figures at the kernels.
//
// Plane layout in shared memory (N2 x N3 points, RP = ceil(N2/2) row pairs, CP = ceil(N3/2) column
// pairs, pitch P = CP rounded up to odd): two slots of RP x P units.
//   column form  U(r, cp): slot r & 1, index (r >> 1) P + cp, lines = columns 2 cp, 2 cp + 1 at row r
//   row form     V(rp, c): slot c & 1, index rp P + (c >> 1), lines = rows 2 rp, 2 rp + 1 at column c
// The 2 x 2 points (rp, cp) occupy the same two units in both forms, so the change of form is in
// place.  Lanes run over cp in the column stages (consecutive units) and over rp in the row stages
// (odd pitch): both free of bank conflicts.  An odd N2 (N3) leaves a zero line in the last pair.
//
// Scratch spectrum of a pack: [i1][p3][rp] units (lines 2 rp, 2 rp + 1 of the permuted axis 2 at
// position p3 of the permuted axis 3): contiguous over rp, which the lanes of the row stages and of
// the axis-1 pass run over.  Positions: natural index k = k1 + R1 k2 sits at p = k1 R2 + k2.
#pragma once

#include "ace_internal.h"
#include "fft.cuh"

namespace ace {

// ---------------------------------------------------------------------------------------
// f2: one FP32 value of each of two lines.
// ---------------------------------------------------------------------------------------
struct alignas(8) f2 {
  float2 v;
};
__device__ __forceinline__ f2 f2bc(float c) { return {make_float2(c, c)}; }
__device__ __forceinline__ f2 f2mk(float a, float b) { return {make_float2(a, b)}; }
__device__ __forceinline__ f2 operator+(f2 a, f2 b) { return {__fadd2_rn(a.v, b.v)}; }
__device__ __forceinline__ f2 operator*(f2 a, f2 b) { return {__fmul2_rn(a.v, b.v)}; }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) { return {__ffma2_rn(a.v, b.v, c.v)}; }
// a difference is a packed multiply-add by -1: exact, one instruction
__device__ __forceinline__ f2 operator-(f2 a, f2 b) { return {__ffma2_rn(b.v, make_float2(-1.f, -1.f), a.v)}; }
__device__ __forceinline__ f2 operator-(f2 a) { return {make_float2(-a.v.x, -a.v.y)}; }

using unit = cpx<f2>;

__device__ __forceinline__ void red2(float *p, f2 v) { atomicAdd(reinterpret_cast<float2 *>(p), v.v); }
__device__ __forceinline__ f2 ld2(const float *p) { return {__ldg(reinterpret_cast<const float2 *>(p))}; }

// a + D i b
template <int D>
__device__ __forceinline__ unit addrot(unit a, unit b) {
  return D > 0 ? unit{a.x - b.y, a.y + b.x} : unit{a.x + b.y, a.y - b.x};
}
// (a) (c + i s), c and s compile-time or loaded, both lines alike
__device__ __forceinline__ unit mulcs(unit a, f2 c, f2 s, f2 ns) {
  return {fma2(a.x, c, a.y * ns), fma2(a.y, c, a.x * s)};
}

// w_R^{D E} a with compile-time constants
template <int R, int E, int D>
__device__ __forceinline__ unit twu(unit a) {
  constexpr int e = E % R;
  if constexpr (e == 0) {
    return a;
  } else if constexpr (4 * e == R) {
    return D < 0 ? unit{a.y, -a.x} : unit{-a.y, a.x};
  } else {
    return mulcs(a, f2bc((float)Tw<R, e, D>::re), f2bc((float)Tw<R, e, D>::im), f2bc((float)-Tw<R, e, D>::im));
  }
}

// Small transforms on units: natural order in, natural order out.
template <int R, int D>
struct UDft;
template <int D>
struct UDft<1, D> {
  static __device__ __forceinline__ void run(unit *) {}
};
template <int D>
struct UDft<2, D> {
  static __device__ __forceinline__ void run(unit *x) {
    const unit a = x[0], b = x[1];
    x[0] = a + b;
    x[1] = a - b;
  }
};
template <int D>
struct UDft<3, D> {
  static __device__ __forceinline__ void run(unit *x) {
    constexpr float s3 = 0.8660254037844386467637231707529361834714;  // sin(2 pi / 3)
    const unit t = x[1] + x[2], d = x[1] - x[2];
    const f2 h = f2bc(-0.5f), p = f2bc(D * s3), n = f2bc(-D * s3);
    const unit m = {fma2(t.x, h, x[0].x), fma2(t.y, h, x[0].y)};
    x[0] = x[0] + t;
    x[1] = {fma2(d.y, n, m.x), fma2(d.x, p, m.y)};
    x[2] = {fma2(d.y, p, m.x), fma2(d.x, n, m.y)};
  }
};
template <int D>
struct UDft<4, D> {
  static __device__ __forceinline__ void run(unit *x) {
    const unit a = x[0] + x[2], b = x[0] - x[2], c = x[1] + x[3], d = x[1] - x[3];
    x[0] = a + c;
    x[2] = a - c;
    x[1] = addrot<D>(b, d);
    x[3] = addrot<-D>(b, d);
  }
};
template <int D>
struct UDft<5, D> {
  static __device__ __forceinline__ void run(unit *x) {
    const f2 c1 = f2bc((float)ct_cos2pi(1, 5)), c2 = f2bc((float)ct_cos2pi(2, 5));
    const f2 s1 = f2bc((float)(D * ct_sin2pi(1, 5))), s2 = f2bc((float)(D * ct_sin2pi(2, 5)));
    const f2 m1 = f2bc((float)(-D * ct_sin2pi(1, 5)));
    const unit a1 = x[1] + x[4], b1 = x[1] - x[4], a2 = x[2] + x[3], b2 = x[2] - x[3], x0 = x[0];
    const unit p1 = {fma2(a2.x, c2, fma2(a1.x, c1, x0.x)), fma2(a2.y, c2, fma2(a1.y, c1, x0.y))};
    const unit p2 = {fma2(a2.x, c1, fma2(a1.x, c2, x0.x)), fma2(a2.y, c1, fma2(a1.y, c2, x0.y))};
    // q1 = D (s1 b1 + s2 b2), q2 = D (s2 b1 - s1 b2); x1, x4 = p1 +- i q1, x2, x3 = p2 +- i q2
    const unit q1 = {fma2(b1.x, s1, b2.x * s2), fma2(b1.y, s1, b2.y * s2)};
    const unit q2 = {fma2(b1.x, s2, b2.x * m1), fma2(b1.y, s2, b2.y * m1)};
    x[0] = x0 + (a1 + a2);
    x[1] = addrot<1>(p1, q1);
    x[4] = addrot<-1>(p1, q1);
    x[2] = addrot<1>(p2, q2);
    x[3] = addrot<-1>(p2, q2);
  }
};
// 8 points: two 4-point transforms and the eighth roots of one as (1 +- i) / sqrt 2, so that the
// scaling is part of the last additions
template <int D>
struct UDft<8, D> {
  static __device__ __forceinline__ void run(unit *x) {
    unit e[4] = {x[0], x[2], x[4], x[6]}, o[4] = {x[1], x[3], x[5], x[7]};
    UDft<4, D>::run(e);
    UDft<4, D>::run(o);
    constexpr float r = 0.7071067811865475244008443621048490392848;
    const f2 c = f2bc(r), n = f2bc(-r);
    x[0] = e[0] + o[0];
    x[4] = e[0] - o[0];
    x[2] = addrot<D>(e[2], o[2]);
    x[6] = addrot<-D>(e[2], o[2]);
    const unit u = addrot<D>(o[1], o[1]);   // (1 + D i) o1
    const unit w = addrot<-D>(o[3], o[3]);  // (1 - D i) o3; w8^{3D} o3 = -w / sqrt 2
    x[1] = {fma2(u.x, c, e[1].x), fma2(u.y, c, e[1].y)};
    x[5] = {fma2(u.x, n, e[1].x), fma2(u.y, n, e[1].y)};
    x[3] = {fma2(w.x, n, e[3].x), fma2(w.y, n, e[3].y)};
    x[7] = {fma2(w.x, c, e[3].x), fma2(w.y, c, e[3].y)};
  }
};
// R = P Q by one Cooley-Tukey step, or without twiddles (prime-factor mapping) for coprime factors;
// the index maps are those of DftCT and DftPFA
template <int P, int Q, int D>
struct UDftCT {
  static __device__ __forceinline__ void run(unit *x) {
    constexpr int R = P * Q;
    unit y[R];
    static_for<Q>([&](auto n2c) {
      constexpr int n2 = decltype(n2c)::value;
      unit t[P];
      static_for<P>([&](auto n1c) { t[decltype(n1c)::value] = x[Q * decltype(n1c)::value + n2]; });
      UDft<P, D>::run(t);
      static_for<P>([&](auto k1c) {
        constexpr int k1 = decltype(k1c)::value;
        y[n2 * P + k1] = twu<R, n2 * k1, D>(t[k1]);
      });
    });
    static_for<P>([&](auto k1c) {
      constexpr int k1 = decltype(k1c)::value;
      unit t[Q];
      static_for<Q>([&](auto n2c) { t[decltype(n2c)::value] = y[decltype(n2c)::value * P + k1]; });
      UDft<Q, D>::run(t);
      static_for<Q>([&](auto k2c) { x[k1 + P * decltype(k2c)::value] = t[decltype(k2c)::value]; });
    });
  }
};
template <int P, int Q, int D>
struct UDftPFA {
  static constexpr int R = P * Q, A = ct_inv_mod(Q % P, P), B = ct_inv_mod(P % Q, Q);
  static __device__ __forceinline__ void run(unit *x) {
    unit y[R];
    static_for<Q>([&](auto n2c) {
      constexpr int n2 = decltype(n2c)::value;
      unit t[P];
      static_for<P>([&](auto n1c) { t[decltype(n1c)::value] = x[(Q * decltype(n1c)::value + P * n2) % R]; });
      UDft<P, D>::run(t);
      static_for<P>([&](auto k1c) { y[n2 * P + decltype(k1c)::value] = t[decltype(k1c)::value]; });
    });
    static_for<P>([&](auto k1c) {
      constexpr int k1 = decltype(k1c)::value;
      unit t[Q];
      static_for<Q>([&](auto n2c) { t[decltype(n2c)::value] = y[decltype(n2c)::value * P + k1]; });
      UDft<Q, D>::run(t);
      static_for<Q>([&](auto k2c) { x[(Q * A * k1 + P * B * decltype(k2c)::value) % R] = t[decltype(k2c)::value]; });
    });
  }
};
template <int D> struct UDft<6, D> : UDftPFA<2, 3, D> {};
template <int D> struct UDft<9, D> : UDftCT<3, 3, D> {};
template <int D> struct UDft<10, D> : UDftPFA<2, 5, D> {};
template <int D> struct UDft<12, D> : UDftPFA<3, 4, D> {};
template <int D> struct UDft<15, D> : UDftPFA<3, 5, D> {};
template <int D> struct UDft<16, D> : UDftCT<4, 4, D> {};
template <int D> struct UDft<18, D> : UDftPFA<2, 9, D> {};
template <int D> struct UDft<20, D> : UDftPFA<4, 5, D> {};
template <int D> struct UDft<25, D> : UDftCT<5, 5, D> {};
template <int D> struct UDft<27, D> : UDftCT<3, 9, D> {};

// ---------------------------------------------------------------------------------------
// Factorisations L = R1 R2 of this chain: those of Factor, except that an even L has an even R2 (the
// column stage that changes the form then owns whole 2 x 2 tiles).
// ---------------------------------------------------------------------------------------
template <int L>
struct LFactor {
  static constexpr int R1 = Factor<L>::R1, R2 = Factor<L>::R2;
};
#define ACE_LFACTOR(L_, A_, B_)             \
  template <>                               \
  struct LFactor<L_> {                      \
    static constexpr int R1 = A_, R2 = B_;  \
    static_assert(A_ * B_ == L_, "factor"); \
  };
ACE_LFACTOR(2, 1, 2)
ACE_LFACTOR(4, 2, 2)
ACE_LFACTOR(12, 3, 4)
ACE_LFACTOR(18, 3, 6)
ACE_LFACTOR(30, 5, 6)
ACE_LFACTOR(40, 5, 8)
ACE_LFACTOR(50, 5, 10)
ACE_LFACTOR(60, 6, 10)
ACE_LFACTOR(72, 9, 8)
ACE_LFACTOR(80, 10, 8)
ACE_LFACTOR(90, 9, 10)
ACE_LFACTOR(108, 9, 12)
ACE_LFACTOR(162, 9, 18)
ACE_LFACTOR(240, 15, 16)
#undef ACE_LFACTOR

// ---------------------------------------------------------------------------------------
// Plane geometry (compile-time).
//
// Work split.  Large planes (LW = 0): the CTA's threads walk the tasks (line, task row) of a stage with
// the line fastest, so that a warp reads and adds 256-byte runs, and a CTA barrier ends every stage.
// Small planes: a group of GT threads owns LW neighbouring lines in the column stages and LW in the row
// stages and runs both stages of its lines, so that only the change from columns to rows (or back) needs
// the CTA's barrier and the groups drift apart.  Measured per pack on one box (linear / groups): 32^3
// 0.49 / 0.43 us, 48^3 1.45 / 0.98 us, 64^3 2.85 / 2.35 us; 72^3 4.68 / 4.60, 96^3 9.3 / 9.5, 108^3
// 16.8 / 19.1, 128^3 25.4 / 27.4 us (shorter runs cost more than the barriers there).
// ---------------------------------------------------------------------------------------
template <int N2_, int N3_, int LW_, int GT_, int NT_>
struct PlaneFix {
  static constexpr int N2 = N2_, N3 = N3_, CP = (N3 + 1) / 2, RP = (N2 + 1) / 2, P = CP | 1, H = RP * P;
  static constexpr bool even3 = N3 % 2 == 0;
  static constexpr int LW = LW_, GT = GT_, NT = NT_;
  __device__ __forceinline__ int nt() const { return NT; }
};
// Barrier of the threads that share the calling thread's lines (barrier 0 is the CTA's).
template <typename G>
__device__ __forceinline__ void lp_sync(const G &g) {
  if (g.LW == 0)
    __syncthreads();
  else if (g.GT == 32)
    __syncwarp();
  else
    asm volatile("bar.sync %0, %1;" ::"r"(1 + (int)threadIdx.x / g.GT), "r"(g.GT) : "memory");
}

// Tasks (l, m), l < nl, m < nm, of one stage: f(l, m).
template <typename G, typename F>
__device__ __forceinline__ void lp_tasks(const G &g, int nl, int nm, F &&f) {
  if (g.LW == 0) {
#pragma unroll 1
    for (int t = threadIdx.x; t < nl * nm; t += g.nt()) {
      const int m = t / nl;
      f(t - m * nl, m);
    }
  } else {
    const int grp = threadIdx.x / g.GT, lane = threadIdx.x - grp * g.GT;
#pragma unroll 1
    for (int l = grp * g.LW + (lane & (g.LW - 1)); l < nl; l += g.nt() / g.GT * g.LW) {
#pragma unroll 1
      for (int m = lane / g.LW; m < nm; m += g.GT / g.LW) f(l, m);
    }
  }
}
// Every task (l, m) over the whole CTA (no line ownership).
template <typename G, typename F>
__device__ __forceinline__ void lp_all(const G &g, int nl, int nm, F &&f) {
#pragma unroll 1
  for (int t = threadIdx.x; t < nl * nm; t += g.nt()) {
    const int m = t / nl;
    f(t - m * nl, m);
  }
}

// Twiddle m of an axis from the table in shared memory, {c, c, s, s}
__device__ __forceinline__ unit tw_load(const unit *tw, int m) { return tw[m]; }
template <int D>
__device__ __forceinline__ unit tw_mul(unit a, unit w) {  // w = e^{-i..}: D < 0 as is, D > 0 conjugate
  return D < 0 ? mulcs(a, w.x, w.y, -w.y) : mulcs(a, w.x, -w.y, w.y);
}

// Base unit of element a R2 + b of a line (a compile-time in the callers' loops): element e sits at
// slot e & 1, index (e >> 1) ST.  For an even R2 the slot depends on b only.
template <int R2>
__device__ __forceinline__ int lp_elem(int a, int b, int ST, int H) {
  if constexpr (R2 % 2 == 0) {
    return (a * (R2 / 2)) * ST + (b >> 1) * ST + (b & 1) * H;
  } else {
    const int e = a * R2 + b;
    return (e >> 1) * ST + (e & 1) * H;
  }
}

// Stage with stride R2 (elements n1 R2 + n2, n2 fixed) of lines l, in place; D = -1: forward stage 1
// (twiddled), D = +1: inverse stage B.  ST/LST: units between element pairs / lines.
template <int L, int D, typename G>
__device__ __forceinline__ void lp_stage_strided(const G &g, unit *s, const unit *tw, int nl, int ST, int LST) {
  constexpr int R1 = LFactor<L>::R1, R2 = LFactor<L>::R2;
  lp_tasks(g, nl, R2, [&](int l, int n2) {
    unit *p = s + l * LST;
    unit x[R1];
#pragma unroll
    for (int n1 = 0; n1 < R1; ++n1) x[n1] = p[lp_elem<R2>(n1, n2, ST, g.H)];
    UDft<R1, D>::run(x);
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) {
      unit v = x[k1];
      if (D < 0 && k1 > 0) v = tw_mul<-1>(v, tw_load(tw, n2 * k1));
      p[lp_elem<R2>(k1, n2, ST, g.H)] = v;
    }
  });
}

// Change of form of one 2 x 2 tile: units (A, B) of two rows over two columns <-> of two columns over
// two rows (its own inverse).
__device__ __forceinline__ void tile_swap(unit &A, unit &B) {
  const float2 ax = A.x.v, ay = A.y.v, bx = B.x.v, by = B.y.v;
  A = {f2mk(ax.x, bx.x), f2mk(ay.x, by.x)};
  B = {f2mk(ax.y, bx.y), f2mk(ay.y, by.y)};
}

// ---- axis 2 (columns), forward stage 1 straight from the orbitals: the densities of the pack,
// z = phi_a phi_b + i phi_c phi_d, are formed on the way into registers ----
template <int L2, bool ROWPACK, typename G>
__device__ __forceinline__ void lp_fwd_load(const G &g, const float *__restrict__ pa, const float *__restrict__ pb,
                                            const float *__restrict__ pc, const float *__restrict__ pd, bool two,
                                            unit *s, const unit *tw) {
  constexpr int R1 = LFactor<L2>::R1, R2 = LFactor<L2>::R2;
  lp_tasks(g, g.CP, R2, [&](int cp, int n2) {
    unit x[R1];
    const int e0 = n2 * g.N3 + 2 * cp;
    if (g.even3) {
// every load of the task is in flight before the first product
      f2 a[R1];
#pragma unroll
      for (int n1 = 0; n1 < R1; ++n1) {
        const int e = e0 + n1 * R2 * g.N3;
        a[n1] = ld2(pa + e);
        x[n1] = {ld2(pb + e), ld2(pd + e)};
      }
      if constexpr (ROWPACK) {
#pragma unroll
        for (int n1 = 0; n1 < R1; ++n1) x[n1] = {a[n1] * x[n1].x, a[n1] * x[n1].y};
      } else {
#pragma unroll
        for (int n1 = 0; n1 < R1; ++n1) {
          const f2 c = ld2(pc + e0 + n1 * R2 * g.N3);
          x[n1] = {a[n1] * x[n1].x, two ? c * x[n1].y : f2bc(0.f)};
        }
      }
    } else {
      const bool in = 2 * cp + 1 < g.N3;  // the last column of an odd row has no neighbour
      const int o = in ? 1 : 0;
#pragma unroll
      for (int n1 = 0; n1 < R1; ++n1) {
        const int e = e0 + n1 * R2 * g.N3;
        const float re0 = __ldg(pa + e) * __ldg(pb + e), im0 = __ldg(pc + e) * __ldg(pd + e);
        const float re1 = __ldg(pa + e + o) * __ldg(pb + e + o), im1 = __ldg(pc + e + o) * __ldg(pd + e + o);
        x[n1] = {f2mk(re0, in ? re1 : 0.f), f2mk(two ? im0 : 0.f, two && in ? im1 : 0.f)};
      }
    }
    UDft<R1, -1>::run(x);
    unit *p = s + cp;
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) {
      unit v = x[k1];
      if (k1 > 0) v = tw_mul<-1>(v, tw_load(tw, n2 * k1));
      p[lp_elem<R2>(k1, n2, g.P, g.H)] = v;
    }
  });
}

// ---- axis 2, forward stage 2 (rows k1 R2 + k2); for an even N2 the results leave in row form ----
template <int L2, typename G>
__device__ __forceinline__ void lp_fwd_cols2(const G &g, unit *s) {
  constexpr int R1 = LFactor<L2>::R1, R2 = LFactor<L2>::R2;
  lp_tasks(g, g.CP, R1, [&](int cp, int k1) {
    unit *p = s + cp;
    unit x[R2];
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) x[n2] = p[lp_elem<R2>(k1, n2, g.P, g.H)];
    UDft<R2, -1>::run(x);
    if constexpr (L2 % 2 == 0) {
#pragma unroll
      for (int j = 0; j < R2; j += 2) tile_swap(x[j], x[j + 1]);
    }
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) p[lp_elem<R2>(k1, n2, g.P, g.H)] = x[n2];
  });
}

// Change of form of the whole plane (odd N2, where no column task owns whole tiles).
template <bool FWD, typename G>
__device__ __forceinline__ void lp_swap_plane(const G &g, unit *s) {
  lp_all(g, g.CP, g.RP, [&](int cp, int rp) {
    unit *p = s + rp * g.P + cp;
    unit A = p[0], B = p[g.H];
    if (FWD && 2 * rp + 1 >= g.N2) B = {f2bc(0.f), f2bc(0.f)};
    tile_swap(A, B);
    p[0] = A;
    p[g.H] = B;
  });
}

// ---- axis 3 (rows), forward stage 2: results straight to the scratch plane [p3][rp] ----
template <int L3, typename G>
__device__ __forceinline__ void lp_fwd_rows2(const G &g, const unit *s, unit *dst) {
  constexpr int R1 = LFactor<L3>::R1, R2 = LFactor<L3>::R2;
  lp_tasks(g, g.RP, R1, [&](int rp, int k1) {
    const unit *p = s + rp * g.P;
    unit x[R2];
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) x[n2] = p[lp_elem<R2>(k1, n2, 1, g.H)];
    UDft<R2, -1>::run(x);
    unit *q = dst + k1 * R2 * g.RP + rp;
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) q[k2 * g.RP] = x[k2];
  });
}

__device__ __forceinline__ unit ldcg_unit(const unit *p) {
  const float4 q = __ldcg(reinterpret_cast<const float4 *>(p));
  return {f2mk(q.x, q.y), f2mk(q.z, q.w)};
}

// ---- axis 3, inverse stage A straight from the scratch plane ----
template <int L3, typename G>
__device__ __forceinline__ void lp_inv_rowsA(const G &g, const unit *src, unit *s, const unit *tw) {
  constexpr int R1 = LFactor<L3>::R1, R2 = LFactor<L3>::R2;
  lp_tasks(g, g.RP, R1, [&](int rp, int k1) {
    const unit *q = src + k1 * R2 * g.RP + rp;
    unit x[R2];
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) x[k2] = ldcg_unit(q + k2 * g.RP);
    UDft<R2, +1>::run(x);
    unit *p = s + rp * g.P;
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) {
      unit v = x[n2];
      if (n2 > 0) v = tw_mul<+1>(v, tw_load(tw, n2 * k1));
      p[lp_elem<R2>(k1, n2, 1, g.H)] = v;
    }
  });
}

// ---- axis 2, inverse stage A (permuted rows k1 R2 + k2), from row form for an even N2 ----
template <int L2, typename G>
__device__ __forceinline__ void lp_inv_colsA(const G &g, unit *s, const unit *tw) {
  constexpr int R1 = LFactor<L2>::R1, R2 = LFactor<L2>::R2;
  lp_tasks(g, g.CP, R1, [&](int cp, int k1) {
    unit *p = s + cp;
    unit x[R2];
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) x[k2] = p[lp_elem<R2>(k1, k2, g.P, g.H)];
    if constexpr (L2 % 2 == 0) {
#pragma unroll
      for (int j = 0; j < R2; j += 2) tile_swap(x[j], x[j + 1]);
    }
    UDft<R2, +1>::run(x);
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) {
      unit v = x[n2];
      if (n2 > 0) v = tw_mul<+1>(v, tw_load(tw, n2 * k1));
      p[lp_elem<R2>(k1, n2, g.P, g.H)] = v;
    }
  });
}

struct PlanePtrs {
  const float *fa, *fb, *fc, *fd;
  float *wa, *wb, *wc, *wd;
  bool rowpack;  // (a, b), (a, d) with b, d != a
  bool two, same_a, diag1, diag2;
};

// ---- axis 2, inverse stage B with the accumulation of W from registers (Eq. vx): v = v_ab + i v_cd
// at the natural rows n1 R2 + n2 of columns 2 cp, 2 cp + 1 ----
template <int L2, typename G>
__device__ __forceinline__ void lp_inv_acc(const G &g, const unit *s, const PlanePtrs &q) {
  constexpr int R1 = LFactor<L2>::R1, R2 = LFactor<L2>::R2;
  lp_tasks(g, g.CP, R2, [&](int cp, int n2) {
    const unit *p = s + cp;
    unit x[R1];
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) x[k1] = p[lp_elem<R2>(k1, n2, g.P, g.H)];
    UDft<R1, +1>::run(x);
    const int e0 = n2 * g.N3 + 2 * cp;
    if (g.even3) {
      if (q.rowpack) {
// the loads of GR rows are in flight together
        constexpr int GR = R1 % 4 == 0 ? 4 : (R1 % 3 == 0 ? 3 : (R1 % 5 == 0 ? 5 : 1));
#pragma unroll
        for (int m = 0; m < R1; m += GR) {
          f2 a[GR], b[GR], d[GR];
#pragma unroll
          for (int j = 0; j < GR; ++j) {
            const int e = e0 + (m + j) * R2 * g.N3;
            a[j] = ld2(q.fa + e);
            b[j] = ld2(q.fb + e);
            d[j] = ld2(q.fd + e);
          }
#pragma unroll
          for (int j = 0; j < GR; ++j) {
            const int e = e0 + (m + j) * R2 * g.N3;
            red2(q.wa + e, fma2(x[m + j].x, b[j], x[m + j].y * d[j]));
            red2(q.wb + e, x[m + j].x * a[j]);
            red2(q.wd + e, x[m + j].y * a[j]);
          }
        }
      } else {
#pragma unroll
        for (int n1 = 0; n1 < R1; ++n1) {
          const int e = e0 + n1 * R2 * g.N3;
          const f2 a = ld2(q.fa + e), b = ld2(q.fb + e), c = ld2(q.fc + e), d = ld2(q.fd + e);
          const f2 ad = q.same_a ? fma2(x[n1].x, b, x[n1].y * d) : x[n1].x * b;
          red2(q.wa + e, ad);
          if (q.two && !q.same_a) red2(q.wc + e, x[n1].y * d);
          if (!q.diag1) red2(q.wb + e, x[n1].x * a);
          if (q.two && !q.diag2) red2(q.wd + e, x[n1].y * c);
        }
      }
    } else {
#pragma unroll
      for (int n1 = 0; n1 < R1; ++n1) {
        const float2 re = x[n1].x.v, im = x[n1].y.v;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (2 * cp + h >= g.N3) break;
          const int e = e0 + n1 * R2 * g.N3 + h;
          const float u = h ? re.y : re.x, w = h ? im.y : im.x;
          const float a = __ldg(q.fa + e), b = __ldg(q.fb + e), c = __ldg(q.fc + e), d = __ldg(q.fd + e);
          atomicAdd(q.wa + e, q.same_a ? u * b + w * d : u * b);
          if (q.two && !q.same_a) atomicAdd(q.wc + e, w * d);
          if (!q.diag1) atomicAdd(q.wb + e, u * a);
          if (q.two && !q.diag2) atomicAdd(q.wd + e, w * c);
        }
      }
    }
  });
}

// Asks L2 for the 16-byte lines wholly inside [base, base + bytes) (one thread; no wait).
__device__ __forceinline__ void l2_prefetch(const void *base, int bytes) {
  const unsigned long long b = reinterpret_cast<unsigned long long>(base);
  const unsigned long long first = (b + 15) & ~15ull;
  const unsigned n = (unsigned)(((b + bytes) & ~15ull) - first);
  if (n) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(first), "r"(n) : "memory");
}
// The orbital and W planes that the accumulation will touch, fetched while the transforms run (ACE_L2_HINTS bits 1
// and 2, off by default: within 2% either way).  Taking the call out changes the inverse kernel's schedule: 128
// orbitals on 96^3 11.63 -> 11.80 ms, 96 on 100x108x90 10.75 -> 10.86.
__device__ __forceinline__ void lp_prefetch(const PlanePtrs &q, int npts, int mode) {
  const int t = threadIdx.x;
  if ((mode & 2) && t < 4 && !(t == 2 && q.same_a)) l2_prefetch(t == 0 ? q.fa : t == 1 ? q.fb : t == 2 ? q.fc : q.fd, 4 * npts);
  if ((mode & 4) && t >= 4 && t < 8 && !(t == 6 && q.same_a))
    l2_prefetch(t == 4 ? q.wa : t == 5 ? q.wb : t == 6 ? q.wc : q.wd, 4 * npts);
}

// Twiddle tables of both axes in shared memory as {c, c, s, s} units (shared when N2 = N3).
__device__ __forceinline__ void lp_tables(int n2, int n3, int nt, const cpx<float> *t2, const cpx<float> *t3, unit *tw2,
                                          unit *tw3) {
  for (int e = threadIdx.x; e < n2; e += nt) tw2[e] = {f2bc(t2[e].x), f2bc(t2[e].y)};
  if (tw3 != tw2)
    for (int e = threadIdx.x; e < n3; e += nt) tw3[e] = {f2bc(t3[e].x), f2bc(t3[e].y)};
}

__host__ __device__ constexpr int lp_plane_units(int n2, int n3) {
  return 2 * ((n2 + 1) / 2) * (((n3 + 1) / 2) | 1);
}
// dynamic shared memory of a plane CTA: the plane and the twiddle tables
__host__ __device__ constexpr int lp_plane_smem(int n2, int n3) {
  return 16 * (lp_plane_units(n2, n3) + n2 + (n3 == n2 ? 0 : n3));
}

// The pack's orbital and W planes at plane offset off.
__device__ __forceinline__ PlanePtrs lp_ptrs(const PlaneArgs<float> &a, int4 pk, long long off) {
  PlanePtrs q;
  q.two = pk.z >= 0;
  q.same_a = q.two && pk.z == pk.x;
  q.diag1 = pk.x == pk.y;
  q.diag2 = pk.z == pk.w;
  q.rowpack = q.same_a && !q.diag1 && !q.diag2;
  const long long ia = (long long)pk.x * a.N + off, ib = (long long)pk.y * a.N + off;
  const long long ic = q.two ? (long long)pk.z * a.N + off : ia, id = q.two ? (long long)pk.w * a.N + off : ib;
  q.fa = a.phi + ia;
  q.fb = a.phi + ib;
  q.fc = a.phi + ic;
  q.fd = a.phi + id;
  q.wa = a.W + ia;
  q.wb = a.W + ib;
  q.wc = a.W + ic;
  q.wd = a.W + id;
  return q;
}

// The split of a plane: groups for planes of which six or more fit on an SM (up to 64 x 64), 64 threads
// on 16 lines where the line counts are multiples of 16, else a warp on 8; larger planes linear.
__host__ __device__ constexpr int lp_lines(int n2, int n3) {
  if (6 * (lp_plane_smem(n2, n3) + 1024) > 228 * 1024) return 0;
  return (n2 + 1) / 2 % 16 == 0 && (n3 + 1) / 2 % 16 == 0 ? 16 : 8;
}
__host__ __device__ constexpr int lp_group(int n2, int n3) { return lp_lines(n2, n3) == 16 ? 64 : 32; }

// Threads of a plane CTA.  Groups: enough for every line.  Linear: the count (a multiple of 32) with the
// least serial work per SM, i.e. the sum over the four stages of task rounds x radix, divided by the
// CTAs that shared memory and `threads` threads per SM allow; the smaller count on ties.
__host__ __device__ constexpr int lp_rounds(int tasks, int nt) { return (tasks + nt - 1) / nt; }
__host__ __device__ constexpr int lp_pick_nt(int n2, int a2, int b2, int n3, int a3, int b3, int threads) {
  const int cp = (n3 + 1) / 2, rp = (n2 + 1) / 2, lines = cp > rp ? cp : rp;
  if (const int lw = lp_lines(n2, n3)) return (lines + lw - 1) / lw * lp_group(n2, n3);
  const int fit = (228 * 1024) / (lp_plane_smem(n2, n3) + 1024);
  int best = 64;
  double cost = 1e30;
  for (int nt = 64; nt <= threads && nt <= 1024; nt += 32) {
    int ctas = threads / nt < fit ? threads / nt : fit;
    if (ctas < 1) ctas = 1;
    const double work = lp_rounds(cp * b2, nt) * a2 + lp_rounds(cp * a2, nt) * b2 + lp_rounds(rp * b3, nt) * a3 +
                        lp_rounds(rp * a3, nt) * b3;
    if (work / ctas < cost - 1e-9) {
      cost = work / ctas;
      best = nt;
    }
  }
  return best;
}

template <typename G>
__device__ __forceinline__ void lp_zero(const G &g, unit *dst) {
  for (int e = threadIdx.x; e < g.RP * g.N3; e += g.nt()) dst[e] = {f2bc(0.f), f2bc(0.f)};
}

}  // namespace ace
