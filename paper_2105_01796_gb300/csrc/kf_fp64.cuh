// kf_fp64.cuh -- double-precision building blocks shared by the FP64 fit
// kernel and the method-variant kernel: the transport Jacobian layout, the
// per-state workspace record, the gain-matrix update with the Joseph form and
// the fixed-point form of the smoother (paper Sect. 2).
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "kf_device.cuh"
#include "kf_internal.h"

namespace kfgb {
namespace dev {

// 1/sqrt(x) (x > 0) and 1/x (x != 0) for the whole double range: the
// argument is scaled by a power of two into [1, 4) (resp. [1, 2)) on the
// integer pipe, the third-order Newton form runs there, and the result is
// scaled back.  Arguments with extreme exponents (zero, subnormal, Inf, NaN)
// take CUDA's double operations, so NaN and Inf propagate as usual; out of
// line, since a copy of them at every use lengthens bodies that fetch their
// instructions from far (97 tracks 207.5 -> 200.4 us, autograd of 2000 tracks
// 1902 -> 1860: more than the innovation's second reciprocal costs).
static __device__ __noinline__ double rsqrt_call(double x) { return 1.0 / sqrt(x); }
static __device__ __noinline__ double rcp_call(double x) { return 1.0 / x; }

__device__ __forceinline__ double rsqrt_any(double x) {
  const int hi = __double2hiint(x);
  const int e = ((hi >> 20) & 0x7ff) - 1023;
  if (e < -1000 || e > 1000) return rsqrt_call(x);
  const int k = e >> 1;
  const double r = rsqrt_nr<2>(__hiloint2double(hi - (k << 21), __double2loint(x)));
  return __hiloint2double(__double2hiint(r) - (k << 20), __double2loint(r));
}

__device__ __forceinline__ double rcp_any(double x) {
  const int hi = __double2hiint(x);
  const int e = ((hi >> 20) & 0x7ff) - 1023;
  if (e < -1000 || e > 1000) return rcp_call(x);
  const double r = rcp_nr<2>(__hiloint2double(hi - (e << 20), __double2loint(x)));
  return __hiloint2double(__double2hiint(r) - (e << 20), __double2loint(r));
}

// ---------------------------------------------------------------------------
// transport Jacobian F of one transition: rows 0..3 and 5 over columns 0..4
// are stored; row 4 (q/p) is e4 times the energy-loss factor, column 5 is e5.
// ---------------------------------------------------------------------------
template <typename R>
struct Jac {
  R f[4][5];   // rows loc0, loc1, phi, theta over columns 0..4
  R ft[5];     // time row over columns 0..4 (column 5 of that row is 1)
};

// element (r, c) of F for r in {0..3, 5}, c in 0..4 (a value select, so the
// struct stays in registers when r and c are compile-time constants)
template <typename R>
__device__ __forceinline__ R jf(const Jac<R>& J, int r, int c) { return r == 5 ? J.ft[c] : J.f[r][c]; }

// ---------------------------------------------------------------------------
// workspace access: record element e of state k for chunk track i
// ---------------------------------------------------------------------------
struct WS {
  double* w64;
  float* w32;
  size_t nt;
  int rec64, rec32;
  int i;
  __device__ __forceinline__ double& d(int k, int e) const { return w64[((size_t)k * rec64 + e) * nt + i]; }
  __device__ float& f(int k, int e) const { return w32[((size_t)k * rec32 + e) * nt + i]; }
};

// Row r of B = G F C, and element (r, c) of B F^T G from that row: F(r, c) by
// f for rows 0..3 and 5 over columns 0..4 (row 4 = e4, column 5 = e5),
// G = diag(1, 1, 1, 1, g, 1).  Written as FMA chains: the kernels that share
// them give the same bits.
//
// N here and below: 6, or 5 for the parameters without the time (the last one;
// the packed elements 0..14 are the leading 5x5 block).  Nothing else depends
// on the time: it is not measured and moves no other parameter.
template <int N, class FE>
__device__ __forceinline__ void fc_row(const FE& f, int r, double g, const double C[21], double b[6]) {
#pragma unroll
  for (int j = 0; j < N; ++j) {
    if (r == 4) {
      b[j] = g * C[sym(4, j)];
      continue;
    }
    double v = f(r, 0) * C[sym(0, j)];
#pragma unroll
    for (int q = 1; q < 5; ++q) v = fma(f(r, q), C[sym(q, j)], v);
    b[j] = r == 5 ? v + C[sym(5, j)] : v;
  }
}
template <class FE>
__device__ __forceinline__ double fcf_element(const FE& f, int c, double g, const double b[6]) {
  if (c == 4) return g * b[4];
  double v = b[0] * f(c, 0);
#pragma unroll
  for (int q = 1; q < 5; ++q) v = fma(b[q], f(c, q), v);
  return c == 5 ? v + b[5] : v;
}

// C <- G F C F^T G
template <int N>
__device__ __forceinline__ void cov_transport(const Jac<double>& J, double g, double C[21]) {
  const auto f = [&](int r, int c) { return jf(J, r, c); };
  double Cp[21];
#pragma unroll
  for (int a = 0; a < N; ++a) {
    double b[6];
    fc_row<N>(f, a, g, C, b);
#pragma unroll
    for (int c = 0; c < N; ++c)
      if (c <= a) Cp[sy(a, c)] = fcf_element(f, c, g, b);
  }
#pragma unroll
  for (int e = 0; e < sy(N, 0); ++e) C[e] = Cp[e];
}

// ---------------------------------------------------------------------------
// gain-matrix update with the Joseph covariance form
//   S = V + H Cp H^T, K = Cp H^T S^-1, xf = xp + K r
//   Cf = (I-KH) Cp (I-KH)^T + K V K^T
//      = Cp + K W - (H Cp)^T K^T,  W = S K^T - H Cp   (expanded, exact for any K)
// Cp, Cf packed lower triangles.
// ---------------------------------------------------------------------------
// (k0, k1) = (h0, h1) S^-1 with the factors of S = L D L^T, L = (1, 0; l, 1):
// f = (1 / S00, l = S01 / S00, 1 / (S11 - l S01)).
//
// The gains are solved for, not formed with S^-1.  A loose prior and a precise
// hit make S ill-conditioned (a direction that both coordinates of a tilted
// plane see: 81 mm^2 against 1e-4), and an explicit inverse leaves a residual
// K S - H C of that condition times the rounding.  The Joseph form takes such an
// error to second order, the smoother's P_0 -= K0 h^T and S -= h K^T to first:
// smoothed variances of such tracks were off by up to 2 % of themselves.  The
// factors leave a residual at rounding level whatever the condition, for the
// same four instructions a row: 100k tracks of 31 states 4902 -> 4884 us, 97
// tracks 205 -> 208 us (a longer chain), whole-fit gradient of 100k tracks of
// 21 states 12.65 -> 12.97 ms.
__device__ __forceinline__ void innovation_solve(const double f[3], double h0, double h1, double& k0, double& k1) {
  k1 = fma(-f[1], h0, h1) * f[2];
  k0 = fma(-f[1], k1, h0 * f[0]);
}

// x > 0 and finite, decided on the integer pipe
__device__ __forceinline__ bool dpos_finite(double x) {
  const long long b = __double_as_longlong(x);
  return b > 0 && b < 0x7ff0000000000000LL;
}

// Gain, increments and chi2 of the gain-matrix update: S = V + H Cp H^T (its
// factors in f), K = Cp H^T S^-1, r the predicted residual, dx = K r.
template <int N>
__device__ __forceinline__ int kalman_gain(const double xp[6], const double Cp[21], const double m[2],
                                           const double V[3], double K[6][2], double f[3], double r[2],
                                           double dx[6], double& chi2) {
  const double S00 = V[0] + Cp[sy(0, 0)], S01 = V[1] + Cp[sy(1, 0)], S11 = V[2] + Cp[sy(1, 1)];
  f[0] = rcp_any(S00);
  f[1] = S01 * f[0];
  const double d1 = fma(-f[1], S01, S11);
  if (!dpos_finite(S00) || !dpos_finite(d1)) return dpos(S00) && dpos(d1) ? ST_NONFINITE : ST_NON_SPD;
  f[2] = rcp_any(d1);
  r[0] = m[0] - xp[0];
  r[1] = m[1] - xp[1];
  const double q = fma(-f[1], r[0], r[1]);
  chi2 = fma(r[0] * f[0], r[0], (q * f[2]) * q);
#pragma unroll
  for (int i = 0; i < N; ++i) {
    innovation_solve(f, Cp[sym(i, 0)], Cp[sym(i, 1)], K[i][0], K[i][1]);
    dx[i] = fma(K[i][0], r[0], K[i][1] * r[1]);
  }
  return ST_OK;
}

// C <- Cp + K W - (H Cp)^T K^T, W = S K^T - H Cp (the Joseph form, expanded)
template <int N>
__device__ __forceinline__ void joseph_update(double C[21], const double V[3], const double K[6][2]) {
  const double S00 = V[0] + C[sy(0, 0)], S01 = V[1] + C[sy(1, 0)], S11 = V[2] + C[sy(1, 1)];
  double h0[6], h1[6], W0[6], W1[6];
#pragma unroll
  for (int j = 0; j < N; ++j) {
    h0[j] = C[sym(0, j)];
    h1[j] = C[sym(1, j)];
    W0[j] = fma(S00, K[j][0], fma(S01, K[j][1], -h0[j]));
    W1[j] = fma(S01, K[j][0], fma(S11, K[j][1], -h1[j]));
  }
#pragma unroll
  for (int i = 0; i < N; ++i)
#pragma unroll
    for (int j = 0; j < N; ++j) if (j <= i) {
      double v = C[sy(i, j)];
      v = fma(K[i][0], W0[j], v);
      v = fma(K[i][1], W1[j], v);
      v = fma(-h0[i], K[j][0], v);
      v = fma(-h1[i], K[j][1], v);
      C[sy(i, j)] = v;
    }
}

// ---------------------------------------------------------------------------
// positive definiteness of a predicted covariance
// ---------------------------------------------------------------------------

// All Cholesky pivots of the leading n x n block positive, in double precision.
static __device__ __noinline__ bool spd_pivots_fp64(const double C[21], int n) {
  double L[21];
  bool ok = true;
  for (int e = 0; e < sy(n, 0); ++e) L[e] = C[e];
  for (int j = 0; j < n; ++j) {
    double dj = L[sy(j, j)];
    for (int q = 0; q < j; ++q) dj -= L[sy(j, q)] * L[sy(j, q)];
    if (!(dj > 0.0)) ok = false;
    const double idg = rsqrt_any(dj);
    L[sy(j, j)] = dj * idg;
    for (int r = j + 1; r < n; ++r) {
      double v = L[sy(r, j)];
      for (int q = 0; q < j; ++q) v -= L[sy(r, q)] * L[sy(j, q)];
      L[sy(r, j)] = v * idg;
    }
  }
  return ok;
}

// The same verdict without FP64 work in the usual case: a float LDL^T of C
// with its diagonal lowered by 1e-5 of itself.  If its pivots are positive,
// the smallest eigenvalue of the Jacobi-scaled C exceeds 1e-5 less the
// rounding errors (conversion 6 x 6e-8, factorisation 7 x 6e-8 x 6 = 2.5e-6:
// Rump's verification by a shifted floating-point Cholesky, BIT 46, 2006), so
// the double-precision factorisation cannot fail.  Otherwise (or with a
// diagonal near the ends of the float range) the FP64 pivots decide.  The
// predicted covariances of the telescope fits have a smallest scaled
// eigenvalue of 0.02 and more.
template <int N>
__device__ __forceinline__ bool spd_certificate(const double C[21]) {
  float U[21], L[21], iD[6];
#pragma unroll
  for (int e = 0; e < sy(N, 0); ++e) U[e] = d2f(C[e]);
  bool ok = true;
#pragma unroll
  for (int j = 0; j < N; ++j) {
    const float cjj = U[sy(j, j)];
    ok = ok && cjj > 1e-30f && cjj < 1e30f;
    float dj = cjj * (1.0f - 1e-5f);
#pragma unroll
    for (int q = 0; q < N; ++q)
      if (q < j) dj = fmaf(-U[sy(j, q)], L[sy(j, q)], dj);
    ok = ok && dj > 0.0f;
    iD[j] = 1.0f / dj;
#pragma unroll
    for (int r = 0; r < N; ++r)
      if (r > j) {
        float u = U[sy(r, j)];
#pragma unroll
        for (int q = 0; q < N; ++q)
          if (q < j) u = fmaf(-U[sy(r, q)], L[sy(j, q)], u);
        U[sy(r, j)] = u;
        L[sy(r, j)] = u * iD[j];
      }
  }
  return ok;
}

template <int N>
__device__ __forceinline__ bool spd_check(const double C[21]) {
  if (spd_certificate<N>(C)) return true;
  double t[21];
#pragma unroll
  for (int e = 0; e < sy(N, 0); ++e) t[e] = C[e];
  return spd_pivots_fp64(t, N);
}

// Whether the time's pivot can be taken as positive in every prediction of a
// track that starts from C, so that the other five parameters decide.  The
// time of state k is the part of t_0 that is independent of the other
// parameters (of variance at least 1e-5 C_tt once C is certified) plus a
// function of the path: its pivot never falls below the former, and fails in
// double precision only if the path's contribution to its variance is some
// 1e8 times C_tt.  That contribution is about the position's variance over
// c^2; the bound allows positions uncertain by the seed's widths over 10 m of
// path, a thousandfold.
__device__ __forceinline__ bool time_is_settled(const double C[21]) {
  const double path = (C[sy(0, 0)] + C[sy(1, 1)]) + 1e8 * (C[sy(2, 2)] + C[sy(3, 3)]);
  return spd_certificate<6>(C) && C[sy(5, 5)] > 1e-6 * (kInvC * kInvC) * path;
}

// ---------------------------------------------------------------------------
// fixed-point smoother
//
// The RTS smoother's state 0 (its parameters and covariance are the fit's
// result) equals the estimate of the state x_0 by a filter of the augmented
// state (x_0, x_k), which runs along with the forward filter:
//   predict  S = S F^T       (S = Cov(x_0, x_k), 6x5: x_k's time is not needed)
//   update   h = S H^T, K0 = h (V + H Cp H^T)^-1,
//            x_0 += K0 r, P_0 -= K0 h^T, S -= h K^T
// with F, K, r, V the forward filter's.  It takes about 250 FP64 instructions
// per state where the backward recursion with stored Jacobians (a Cholesky
// factorisation, six pairs of triangular solves and A (Cs' - Cp') A^T) takes
// 735, needs no inverse of Cp, and no record of the forward pass is written
// to memory (720 B per state before).  Against an evaluation of the whole fit
// in 80 bits (27 shapes of 1000 tracks over 5 to 30 planes) the rms errors of
// parameters, covariances and chi2 are 0.10 to 0.33, 0.26 to 0.56 and 0.41 to
// 0.89 of those of the backward recursion in plain double precision.
// ---------------------------------------------------------------------------

// row (v0..v4) -> row F^T over the columns 0..4, with F row 4 = g e4
template <class FE>
__device__ __forceinline__ void row_times_ft(const FE& f, double g, double v[5]) {
  double o[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    double a = f(r, 0) * v[0];
#pragma unroll
    for (int c = 1; c < 5; ++c) a = fma(f(r, c), v[c], a);
    o[r] = a;
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) v[r] = o[r];
  v[4] = g * v[4];
}

// Measurement update of row i of S, x_0[i] and row i of P_0 (lower part);
// h of the other rows comes in hall (rows 0..i are used).
__device__ __forceinline__ void fixed_point_row(int i, double S[5], const double K[6][2], const double f[3],
                                                const double r[2], const double hall[6][2], double& x0,
                                                double P0[21]) {
  const double h0 = hall[i][0], h1 = hall[i][1];
  double k0, k1;
  innovation_solve(f, h0, h1, k0, k1);
  x0 = fma(k0, r[0], fma(k1, r[1], x0));
#pragma unroll
  for (int c = 0; c < 6; ++c)
    if (c <= i) P0[sy(i, c)] = fma(-k0, hall[c][0], fma(-k1, hall[c][1], P0[sy(i, c)]));
#pragma unroll
  for (int c = 0; c < 5; ++c) S[c] = fma(-h0, K[c][0], fma(-h1, K[c][1], S[c]));
}

// Per-state record for the smoothed parameters of every state (written only
// when they are wanted): F 25 | K 12 | S^-1 r 2 | x_f 6 | C_f 21 | g, the
// factor of F's q/p row (with energy loss only).
struct StateRec {
  static constexpr int F = 0, K = 25, IR = 37, XF = 39, CF = 45, G = 66;
};
static_assert(StateRec::G + 1 <= kRec64Fp64, "record size");

// Smoothed parameters of states n-1 .. 1 from the records, by the adjoint
// form of the smoother (Bryson and Frazier): x_s,k = x_f,k - C_f,k l_k with
//   l~ = l - H^T (K^T l + S^-1 r),  l_{k-1} = F_k^T l~.
__device__ __forceinline__ void smooth_states(const WS& ws, int n, double* out_states, int64_t n_states, int64_t o0,
                                              bool with_g = false) {
  double l[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  for (int k = n - 1; k >= 1; --k) {
#pragma unroll
    for (int r = 0; r < 6; ++r) {
      double v = ws.d(k, StateRec::XF + r);
#pragma unroll
      for (int c = 0; c < 6; ++c) v = fma(-ws.d(k, StateRec::CF + sym(r, c)), l[c], v);
      out_states[r * n_states + o0 + k] = v;
    }
    double a0 = ws.d(k, StateRec::IR), a1 = ws.d(k, StateRec::IR + 1);
#pragma unroll
    for (int r = 0; r < 6; ++r) {
      a0 = fma(ws.d(k, StateRec::K + 2 * r), l[r], a0);
      a1 = fma(ws.d(k, StateRec::K + 2 * r + 1), l[r], a1);
    }
    l[0] -= a0;
    l[1] -= a1;
    double m[6];
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      double v = c == 4 ? (with_g ? ws.d(k, StateRec::G) * l[4] : l[4]) : 0.0;
#pragma unroll
      for (int r = 0; r < 5; ++r) v = fma(ws.d(k, StateRec::F + r * 5 + c), l[r == 4 ? 5 : r], v);
      m[c] = v;
    }
    m[5] = l[5];
#pragma unroll
    for (int c = 0; c < 6; ++c) l[c] = m[c];
  }
}

}  // namespace dev
}  // namespace kfgb
