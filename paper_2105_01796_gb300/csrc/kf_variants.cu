// kf_variants.cu -- FP64 kernel of the method variants the paper describes
// besides its baseline fit (arXiv 2105.01796), one track per thread, fused
// filter + smoother like the FP64 path:
//   * smoother by a backward Kalman filter (Sect. 2, Fig. 2): a second filter
//     runs from the last state to the first with its own RKN propagation,
//     and its prediction onto each state is combined with the forward
//     filter's state by the weighted mean;
//   * energy loss in the surface material (Sect. 1): the mean (Bethe) loss
//     moves q/p at every surface with material, its Jacobian factor enters
//     the transport, and a straggling variance is added to q/p;
//   * a position-dependent field given as a grid map (Sect. 4.3): the RKN
//     stages take the trilinearly interpolated field at their own points.
// Any combination of the three runs here; the baseline method keeps its own
// tuned FP64 and mixed kernels.
//
// The bound is the FP64 pipe, as for the FP64 fit, and the constant-field
// variants share its transport and its fixed-point smoother (one kernel per
// kind of field).  In a map the field of every stage is another, so the steps
// stay stage by stage; the corrections after the first are tiny and take
// their leading terms.  The backward filter's weighted mean (a 6x6
// factorisation and six solves) is formed on the states that are output.
// 50k tracks of 21 states with energy loss 7.54 -> 2.16 ms; 30k tracks of 31
// states with map, energy loss and backward filter 16.9 -> 9.43 ms (4286 FP64
// instructions per state; the 938 warps run as one wave of 7 per SM).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "kf_device.cuh"
#include "kf_filter.cuh"
#include "kf_fp64.cuh"
#include "kf_internal.h"
#include "kf_transport.cuh"

namespace kfgb {
namespace {
using namespace dev;

// ---------------------------------------------------------------------------
// field
// ---------------------------------------------------------------------------

// Offset in the grid cell and the cell of one axis, for any u (clamped onto
// the grid; NaN: 0).
static __device__ __noinline__ double2 clamped_cell(double u, int n) {
  u = fmin(fmax(u, 0.0), (double)(n - 1));
  int c = (int)u;
  c = c > n - 2 ? n - 2 : c;
  return make_double2(u - (double)c, (double)c);
}

// Field at r: the trilinear interpolation of the map's 8 grid points around r
// (r clamped onto the grid; every index stays inside [0, n-1], also for a
// non-finite r).  Inside the grid the cell index is the low word of u + 1.5 x
// 2^52 rounded down: 4 FP64 instructions per axis where conversions, minimum
// and maximum take about 12 slots.
__device__ __forceinline__ void field_at(const FitParams& p, const double r[3], double B[3]) {
  int idx[3];
  double w[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    constexpr double kMagic = 6755399441055744.0;
    const double u = fma(r[a], p.map_inv_spacing[a], p.map_off[a]);
    const double s = __dadd_rd(u, kMagic);
    idx[a] = __double2loint(s);
    w[a] = u - (s - kMagic);
    if (__double2hiint(s) != 0x43380000 || (unsigned)idx[a] > (unsigned)(p.map_n[a] - 2)) {
      const double2 c = clamped_cell(u, p.map_n[a]);
      w[a] = c.x;
      idx[a] = (int)c.y;
    }
  }
  const size_t sx = 3, sy_ = (size_t)p.map_n[0] * 3, sz = sy_ * (size_t)p.map_n[1];
  const double* base = p.map_b + (size_t)idx[2] * sz + (size_t)idx[1] * sy_ + (size_t)idx[0] * sx;
  const double v[3] = {1.0 - w[0], 1.0 - w[1], 1.0 - w[2]};
  const double yz[4] = {v[1] * v[2], w[1] * v[2], v[1] * w[2], w[1] * w[2]};
  B[0] = B[1] = B[2] = 0.0;
#pragma unroll
  for (int c8 = 0; c8 < 4; ++c8) {
    const double* q = base + (c8 >> 1) * sz + (c8 & 1) * sy_;
    const double w0 = v[0] * yz[c8], w1 = w[0] * yz[c8];
#pragma unroll
    for (int c = 0; c < 3; ++c) B[c] = fma(w1, __ldg(q + sx + c), fma(w0, __ldg(q + c), B[c]));
  }
}

__device__ __forceinline__ void cross3(const double a[3], const double b[3], double o[3]) {
  o[0] = a[1] * b[2] - a[2] * b[1];
  o[1] = a[2] * b[0] - a[0] * b[2];
  o[2] = a[0] * b[1] - a[1] * b[0];
}

// ---------------------------------------------------------------------------
// RKN step with the field at the stage points
// ---------------------------------------------------------------------------

// free-state accumulators plus the varying columns of G = D J_bf
// (columns: 0 phi, 1 theta, 2 q/p)
struct GProp {
  double r[3], T[3], lam, len;
  double gr[3][3], gT[3][3];
};

// One 4-stage Nystrom step of length h:
//   k1 = a(r, T), k2 = a(r + h/2 T + h^2/8 k1, T + h/2 k1),
//   k3 = a(same point, T + h/2 k2), k4 = a(r + h T + h^2/2 k3, T + h k3),
//   a(r, T) = (q/p) kappa T x B(r),
//   r' = r + h T + h^2/6 (k1 + k2 + k3),  T' = T + h/6 (k1 + 2 k2 + 2 k3 + k4).
// G advances by the derivative of this map with the three stage fields held
// fixed (exact for a uniform field).
// v x b (+ t)
__device__ __forceinline__ void cross_add(const double v[3], const double b[3], const double t[3], double o[3]) {
  o[0] = fma(v[1], b[2], fma(-v[2], b[1], t[0]));
  o[1] = fma(v[2], b[0], fma(-v[0], b[2], t[1]));
  o[2] = fma(v[0], b[1], fma(-v[1], b[0], t[2]));
}

__device__ __forceinline__ void rkn_step_field(const FitParams& p, GProp& s, double h) {
  const double hh = 0.5 * h, h6 = h * (1.0 / 6.0), hh6 = h * h6;
  double k1[3], k2[3], k4[3];  // kappa B of the stages, then (q/p) kappa B
  double t1[3], t2[3], t3[3], t4[3];  // kappa T_s x B_s
  double T2[3], T3[3], T4[3], pt[3];
  field_at(p, s.r, k1);
#pragma unroll
  for (int i = 0; i < 3; ++i) k1[i] *= kKappa;
  cross3(s.T, k1, t1);
  const double hl = hh * s.lam;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    T2[i] = fma(hl, t1[i], s.T[i]);
    pt[i] = fma(0.5 * hh, s.T[i] + T2[i], s.r[i]);  // r + h/2 T + h^2/8 a1
  }
  field_at(p, pt, k2);
#pragma unroll
  for (int i = 0; i < 3; ++i) k2[i] *= kKappa;
  cross3(T2, k2, t2);
#pragma unroll
  for (int i = 0; i < 3; ++i) T3[i] = fma(hl, t2[i], s.T[i]);
  cross3(T3, k2, t3);
  const double fl = h * s.lam;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    T4[i] = fma(fl, t3[i], s.T[i]);
    pt[i] = fma(hh, s.T[i] + T4[i], s.r[i]);  // r + h T + h^2/2 a3
  }
  field_at(p, pt, k4);
#pragma unroll
  for (int i = 0; i < 3; ++i) k4[i] *= kKappa;
  cross3(T4, k4, t4);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const double m = t2[i] + t3[i];
    s.r[i] = fma(hh6 * s.lam, t1[i] + m, fma(h, s.T[i], s.r[i]));
    s.T[i] = fma(h6 * s.lam, fma(2.0, m, t1[i] + t4[i]), s.T[i]);
    k1[i] *= s.lam;
    k2[i] *= s.lam;
    k4[i] *= s.lam;
  }
  // Jacobian columns
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double g[3] = {s.gT[0][c], s.gT[1][c], s.gT[2][c]};
    double d1[3], d2[3], d3[3], d4[3], v[3];
    if (c == 2) cross_add(g, k1, t1, d1); else cross3(g, k1, d1);
#pragma unroll
    for (int i = 0; i < 3; ++i) v[i] = fma(hh, d1[i], g[i]);
    if (c == 2) cross_add(v, k2, t2, d2); else cross3(v, k2, d2);
#pragma unroll
    for (int i = 0; i < 3; ++i) v[i] = fma(hh, d2[i], g[i]);
    if (c == 2) cross_add(v, k2, t3, d3); else cross3(v, k2, d3);
#pragma unroll
    for (int i = 0; i < 3; ++i) v[i] = fma(h, d3[i], g[i]);
    if (c == 2) cross_add(v, k4, t4, d4); else cross3(v, k4, d4);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const double m = d2[i] + d3[i];
      s.gr[i][c] = fma(hh6, d1[i] + m, fma(h, g[i], s.gr[i][c]));
      s.gT[i][c] = fma(h6, fma(2.0, m, d1[i] + d4[i]), g[i]);
    }
  }
  s.len += h;
}

// The same step for a tiny h, to the order that double precision resolves:
//   r += h T + h^2/2 a, T += h a, a = lk T x B(r)
// and its derivative.  What it leaves out is (h lk B)^2 / 2 of the direction
// (below 1e-17 under the caller's bound) and h^2 / 2 of the field's change
// along the step (1e-16 for a field that changes by its own size over one
// 25 mm grid cell at h = 2e-6 mm).  One field lookup instead of three and
// about 60 FP64 instructions instead of 350; B is the field at r.
__device__ __forceinline__ void tiny_step_field(GProp& s, double h, const double B[3]) {
  const double hl = h * s.lam * kKappa, hk = h * kKappa;
  double TB[3];
  cross3(s.T, B, TB);
#pragma unroll
  for (int i = 0; i < 3; ++i) s.gr[i][2] = fma(h, fma(0.5 * hk, TB[i], s.gT[i][2]), s.gr[i][2]);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double g[3] = {s.gT[0][c], s.gT[1][c], s.gT[2][c]};
    double x[3];
    cross3(g, B, x);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      if (c < 2) s.gr[i][c] = fma(h, g[i], s.gr[i][c]);
      s.gT[i][c] = fma(hl, x[i], g[i]) + (c == 2 ? hk * TB[i] : 0.0);
    }
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    s.r[i] = fma(h, fma(0.5 * hl, TB[i], s.T[i]), s.r[i]);
    s.T[i] = fma(hl, TB[i], s.T[i]);
  }
  s.len += h;
}

__device__ __forceinline__ bool plane_distance(const GProp& s, const Surf& sb, double& out) {
  const double d = sb.n(0) * (sb.c(0) - s.r[0]) + sb.n(1) * (sb.c(1) - s.r[1]) + sb.n(2) * (sb.c(2) - s.r[2]);
  const double nT = sb.n(0) * s.T[0] + sb.n(1) * s.T[1] + sb.n(2) * s.T[2];
  if (!(fabs(nT) > 1e-9)) return false;
  out = d * rcp_any(nT);
  return true;
}

// Propagation to plane b through the field map (see propagate_to_plane for
// the constant field); Be receives the field at the end point.  The first
// correction is a full step; the second (below 2e-6 mm) takes its leading
// terms and one lookup; the third (rounding of the position) only moves the
// point along T.  With the cell lookup in 4 instructions per axis and kappa B
// premultiplied once per stage, 12.8 -> 11.0 ms on the 30k tracks above.
__device__ __forceinline__ int propagate_map(const FitParams& p, const Surf& sb, const double r0[3], const Angles& a0,
                                             double lam, End& o, Cols64& g, double Be[3]) {
  GProp s;
#pragma unroll
  for (int i = 0; i < 3; ++i) s.r[i] = r0[i];
  s.T[0] = a0.cp * a0.st;
  s.T[1] = a0.sp * a0.st;
  s.T[2] = a0.ct;
  s.lam = lam;
  s.len = 0.0;
  s.gT[0][0] = -s.T[1]; s.gT[1][0] = s.T[0]; s.gT[2][0] = 0.0;
  s.gT[0][1] = a0.cp * a0.ct;  s.gT[1][1] = a0.sp * a0.ct; s.gT[2][1] = -a0.st;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    s.gT[i][2] = 0.0;
    s.gr[i][0] = s.gr[i][1] = s.gr[i][2] = 0.0;
  }
  double s0;
  if (!plane_distance(s, sb, s0)) return ST_NO_INTERSECTION;
  int nsub = 1;
  double h = s0;
  if (!(fabs(s0) <= p.h_max)) {
    const double nsub_d = ceil(fabs(s0) / p.h_max);
    if (!(nsub_d <= 64.0)) return ST_NO_INTERSECTION;
    nsub = nsub_d < 1.0 ? 1 : (int)nsub_d;
    h = s0 / nsub;
  }
  // one loop over main steps and corrections (one copy of the long step)
  bool have_B = false;
  double x1 = 0.0;  // (h lk B)^2 / h^2 of the last tiny step
  int j = 0;
  for (;;) {
    if (j >= nsub) {
      if (j == nsub + p.n_iter) break;
      if (!plane_distance(s, sb, h)) return ST_NO_INTERSECTION;
    }
    ++j;
    if (j > nsub && fabs(h) <= 2e-6) {
      if (x1 > 0.0 && fabs(h) <= 1e-12 && h * h * x1 <= 1e-34) {
        // a standing point: the turn is below 1e-17
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          s.r[i] = fma(h, s.T[i], s.r[i]);
#pragma unroll
          for (int c = 0; c < 3; ++c) s.gr[i][c] = fma(h, s.gT[i][c], s.gr[i][c]);
        }
        s.len += h;
        continue;
      }
      field_at(p, s.r, Be);
      const double lk = lam * kKappa;
      const double q = lk * lk * fma(Be[0], Be[0], fma(Be[1], Be[1], Be[2] * Be[2]));
      if (h * h * q <= 2e-17) {
        x1 = q;
        have_B = fabs(h) <= 1e-12;  // the end point's field too
        tiny_step_field(s, h, Be);
        continue;
      }
    }
    have_B = false;
    x1 = 0.0;
    rkn_step_field(p, s, h);
  }
  if (!have_B) field_at(p, s.r, Be);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    o.r[i] = s.r[i];
    o.T[i] = s.T[i];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      g.gr[i][c] = s.gr[i][c];
      g.gT[i][c] = s.gT[i][c];
    }
  }
  const double mass = p.mass;
  o.g2 = fma(mass * mass * lam, lam, 1.0);
  const double igam = rsqrt_any(o.g2);
  o.dtds = o.g2 * igam * kInvC;
  o.dt = s.len * o.dtds;
  g.gtl = s.len * (mass * mass * lam * kInvC) * igam;
  return ST_OK;
}

// FIELD: 0 constant along z, 1 constant, 2 map.
// Transport x (bound, surface a, angles ang) to surface b in either direction
// (the path length comes out negative when b lies behind): x becomes the
// prediction but for its angles, which stay in ang and o.
template <int FIELD>
__device__ __forceinline__ int transport_variant(const FitParams& p, const Surf& sa, const Surf& sb, double x[6],
                                                 const Angles& ang, End& o, Jac<double>& J) {
  double r0[3], B[3] = {p.bfield[0], p.bfield[1], p.bfield[2]};
#pragma unroll
  for (int e = 0; e < 3; ++e) r0[e] = fma(x[0], sa.u(e), fma(x[1], sa.v(e), sa.c(e)));
  Cols64 g;
  const int st = FIELD == 2
                     ? propagate_map(p, sb, r0, ang, x[4], o, g, B)
                     : propagate_to_plane<FIELD == 0, 7>(sb, r0, ang, x[4], B, p.mass, p.h_max, p.n_iter, o, g);
  if (st != ST_OK) return st;
  double inv_nT;
  end_frame(sb, o, inv_nT);
  jacobian_columns<FIELD == 0, 31>(sa, sb, o, g, x[4], B, inv_nT, [&](int r, int c, double v) {
    if (r == 5) J.ft[c] = v; else J.f[r][c] = v;
  });
  const double d0 = o.r[0] - sb.c(0), d1 = o.r[1] - sb.c(1), d2 = o.r[2] - sb.c(2);
  x[0] = fma(d0, sb.u(0), fma(d1, sb.u(1), d2 * sb.u(2)));
  x[1] = fma(d0, sb.v(0), fma(d1, sb.v(1), d2 * sb.v(2)));
  x[5] += o.dt;
  return ST_OK;
}

// ---------------------------------------------------------------------------
// energy loss
// ---------------------------------------------------------------------------

// Sternheimer density effect, X = log10(beta gamma):
//   X >= x1: 2 ln10 X - Cbar;  x0 <= X < x1: that + a (x1 - X)^k;
//   X < x0: delta0 10^(2 (X - x0))
// ln_bg = ln(beta gamma).  (x1 - X)^k as exp(k ln(x1 - X)): the general
// pow() costs over twice the FP64 instructions of both.
__device__ __forceinline__ double density_effect(const FitParams& p, double ln_bg) {
  const double X = ln_bg * 0.4342944819032518277;
  const double cbar = p.mat[3], x0 = p.mat[4], x1 = p.mat[5], a = p.mat[6], k = p.mat[7], d0 = p.mat[8];
  if (X >= x1) return fma(2.0, ln_bg, -cbar);
  if (X >= x0) return fma(2.0, ln_bg, -cbar) + a * exp(k * log_df(x1 - X));
  return d0 * pow(10.0, 2.0 * (X - x0));
}

constexpr double kBetheK = 0.307075e-3;  // 4 pi N_A r_e^2 m_e c^2, GeV cm^2/mol
constexpr double kMe = 0.51099895e-3;    // electron mass, GeV

// The mean loss through a surface (dir = +1) or its restoration (dir = -1),
// evaluated at the current momentum; thickness x/X0 * X0rho / cos.  qop
// changes, jac = (p^3 E')/(p'^3 E), var_down = (E_d/p_d^3)^2 sigma_E^2 on the
// downstream side with sigma_E = 4 xi / (2 sqrt(2 ln 2)) (the Gaussian of the
// Landau FWHM).  The stopping power is Bethe's formula with the density
// effect.  ST_NONFINITE if the particle stops.
// FP64 quotients and roots cost ten pipe slots and more each: they are
// Newton-refined reciprocals here (5 to 6), and E, p', 1/p' and 1/E come from
// two reciprocal square roots (about 170 slots per call against 420).
__device__ __forceinline__ int energy_loss(const FitParams& p, double& qop, double xx0, double inv_cos, int dir,
                                           double& jac, double& var_down) {
  const double mass = p.mass, im = rcp_any(mass);
  const double thick = xx0 * p.mat[2] * fabs(inv_cos);
  const double iq = fabs(qop), pm = rcp_any(iq);
  const double bg = pm * im, bg2 = bg * bg;
  const double Esq = fma(pm, pm, mass * mass), iE = rsqrt_any(Esq), E = Esq * iE;
  const double ib2 = Esq * (iq * iq);  // 1 / beta^2
  const double gam = E * im, r = kMe * im;
  const double wden = fma(r, fma(2.0, gam, r), 1.0);  // wmax = 2 me bg^2 / wden
  const double q = 2.0 * kMe * bg2, iI = rcp_any(p.mat[1]);
  const double arg = (q * iI) * (q * iI) * rcp_any(wden);
  const double b2 = pm * iE * (pm * iE);
  const double dedx = kBetheK * p.mat[0] * ib2 * (0.5 * log_df(arg) - b2 - 0.5 * density_effect(p, log_df(bg)));
  const double dE = dedx * thick;
  const double E2 = dir > 0 ? E - dE : E + dE;
  if (!(E2 > mass)) return ST_NONFINITE;
  const double ip2 = rsqrt_any(fma(E2, E2, -mass * mass));
  const double xi = 0.5 * kBetheK * p.mat[0] * thick * ib2;
  const double sigE = xi * (4.0 / 2.354820045030949327);  // 2 sqrt(2 ln 2)
  const double ip2c = ip2 * ip2 * ip2;
  jac = pm * pm * pm * iE * (E2 * ip2c);
  const double dqdE = dir > 0 ? E2 * ip2c : E * (iq * iq * iq);
  var_down = (dqdE * sigE) * (dqdE * sigE);
  qop = qop > 0.0 ? ip2 : -ip2;
  return ST_OK;
}

// multiple-scattering variances of (phi, theta) for q/p = lam (g2 = 1 + m^2
// lam^2) crossing a surface of x/X0 = xx0 at incidence 1/inv_cos
__device__ __forceinline__ void add_scattering(double lam, double g2, double xx0, double inv_cos, double inv_st,
                                               double C[21]) {
  const double q = highland_sq(lam, g2, xx0, inv_cos);
  C[sy(2, 2)] = fma(q, inv_st * inv_st, C[sy(2, 2)]);
  C[sy(3, 3)] += q;
}

// X = S^-1 B for SPD S (packed) and a symmetric right-hand side B (packed),
// through the Cholesky factor of the Jacobi-scaled D^-1/2 S D^-1/2; K = X^T.
__device__ __forceinline__ int spd_solve_sym(const double S[21], const double B[21], double X[6][6]) {
  double L[21];
  double id[6];  // 1 / sqrt(S_ii), the Jacobi scaling
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    if (!(S[sy(i, i)] > 0.0)) return ST_NON_SPD;
    id[i] = rsqrt_any(S[sy(i, i)]);
  }
#pragma unroll
  for (int i = 0; i < 6; ++i)
#pragma unroll
    for (int j = 0; j < 6; ++j)
      if (j <= i) L[sy(i, j)] = S[sy(i, j)] * (id[i] * id[j]);
  double idg[6];
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    double dj = L[sy(j, j)];
#pragma unroll
    for (int q = 0; q < 6; ++q)
      if (q < j) dj -= L[sy(j, q)] * L[sy(j, q)];
    if (!(dj > 0.0)) return ST_NON_SPD;
    idg[j] = rsqrt_any(dj);
    L[sy(j, j)] = dj * idg[j];
#pragma unroll
    for (int r = 0; r < 6; ++r)
      if (r > j) {
        double v = L[sy(r, j)];
#pragma unroll
        for (int q = 0; q < 6; ++q)
          if (q < j) v -= L[sy(r, q)] * L[sy(j, q)];
        L[sy(r, j)] = v * idg[j];
      }
  }
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    double y[6];
#pragma unroll
    for (int r = 0; r < 6; ++r) {
      double v = B[sym(r, c)] * id[r];
#pragma unroll
      for (int q = 0; q < 6; ++q)
        if (q < r) v -= L[sy(r, q)] * y[q];
      y[r] = v * idg[r];
    }
    double z[6];
#pragma unroll
    for (int r = 5; r >= 0; --r) {
      double v = y[r];
#pragma unroll
      for (int q = 0; q < 6; ++q)
        if (q > r) v -= L[sy(q, r)] * z[q];
      z[r] = v * idg[r];
    }
#pragma unroll
    for (int r = 0; r < 6; ++r) X[r][c] = z[r] * id[r];
  }
  return ST_OK;
}

// ---------------------------------------------------------------------------
// the fused fit
// ---------------------------------------------------------------------------

// records of the backward-filter smoother: the forward-filtered states
struct BackRec {
  static constexpr int XF = 0, CF = 6;
};

// What a launch wants besides the smoothed state 0 by the fixed-point
// smoother: nothing, the smoothed parameters of every state, or the backward
// filter in its place.
enum : int { kState0 = 0, kEveryState = 1, kBackward = 2 };

// States 1 .. n-1 of the forward filter (N as in filter_states).
template <int FIELD, int N, int MODE>
__device__ __forceinline__ int variant_states(const FitParams& p, const double* s_surf, const WS& ws, int64_t o0, int n,
                                              Filter& f) {
  int sid_prev = p.surface_id[o0];
#pragma unroll 1
  for (int k = 1; k < n; ++k) {
    const int sid = p.surface_id[o0 + k];
    const Surf sa{s_surf + sid_prev * kSurfStride}, sb{s_surf + sid * kSurfStride};
    Jac<double> J;
    End o;
    const Angles a0 = f.ang;
    int status = transport_variant<FIELD>(p, sa, sb, f.x, a0, o, J);
    if (status != ST_OK) return status;
    if (MODE == kEveryState || (MODE == kBackward && p.out_states))
      end_angles(f.x[2], f.x[3], a0, o, f.x[2], f.x[3]);
    f.ang = o.a;
    // material of surface k (before the update): scattering with the
    // arriving momentum, then the mean loss and its straggling
    const double xx0 = sb.xx0(), lam = f.x[4];
    double g = 1.0, var_q = 0.0;
    if (p.energy_loss && xx0 > 0.0) {
      status = energy_loss(p, f.x[4], xx0, o.inv_cos, +1, g, var_q);
      if (status != ST_OK) return status;
    }
    cov_transport<N>(J, g, f.C);
    if (xx0 > 0.0) add_scattering(lam, o.g2, xx0, o.inv_cos, o.inv_st, f.C);
    f.C[sy(4, 4)] += var_q;
    if (MODE != kBackward) {
      f.spd = f.spd && spd_check<N>(f.C);
      const auto fe = [&](int r, int c) { return jf(J, r, c); };
#pragma unroll
      for (int r = 0; r < 6; ++r) row_times_ft(fe, g, f.S[r]);
    }
    if (MODE == kEveryState) {
#pragma unroll
      for (int e = 0; e < 25; ++e) ws.d(k, StateRec::F + e) = e < 20 ? J.f[e / 5][e % 5] : J.ft[e % 5];
      ws.d(k, StateRec::G) = g;
    }
    double K[6][2], ir[2] = {0.0, 0.0};
    if (!p.is_hole[o0 + k]) {
      double m[2], V[3], fs[3], r[2], dx[6], c2;
      hit_of(p, o0 + k, m, V);
      status = kalman_gain<N>(f.x, f.C, m, V, K, fs, r, dx, c2);
      if (status != ST_OK) return status;
      joseph_update<N>(f.C, V, K);
      f.chi2 += c2;
      ++f.nmeas;
#pragma unroll
      for (int e = 0; e < N; ++e) f.x[e] += dx[e];
      innovation_solve(fs, r[0], r[1], ir[0], ir[1]);
      if (MODE != kBackward) {
        double hall[6][2];
#pragma unroll
        for (int e = 0; e < 6; ++e) {
          hall[e][0] = f.S[e][0];
          hall[e][1] = f.S[e][1];
        }
#pragma unroll
        for (int e = 0; e < 6; ++e) fixed_point_row(e, f.S[e], K, fs, r, hall, f.xs[e], f.P0);
      }
      turn(f.ang.cp, f.ang.sp, dx[2]);
      turn(f.ang.ct, f.ang.st, dx[3]);
    } else {
#pragma unroll
      for (int e = 0; e < 6; ++e) K[e][0] = K[e][1] = 0.0;
    }
    if (MODE == kBackward) {
#pragma unroll
      for (int e = 0; e < 6; ++e) ws.d(k, BackRec::XF + e) = f.x[e];
#pragma unroll
      for (int e = 0; e < 21; ++e) ws.d(k, BackRec::CF + e) = f.C[e];
    } else if (MODE == kEveryState) {
#pragma unroll
      for (int e = 0; e < 6; ++e) {
        ws.d(k, StateRec::K + 2 * e) = K[e][0];
        ws.d(k, StateRec::K + 2 * e + 1) = K[e][1];
        ws.d(k, StateRec::XF + e) = f.x[e];
      }
      ws.d(k, StateRec::IR) = ir[0];
      ws.d(k, StateRec::IR + 1) = ir[1];
#pragma unroll
      for (int e = 0; e < 21; ++e) ws.d(k, StateRec::CF + e) = f.C[e];
    }
    sid_prev = sid;
  }
  return ST_OK;
}

// The same with the time, out of line (see filter_states_with_time).
template <int FIELD>
__device__ __noinline__ int variant_states_with_time(const FitParams& p, const double* s_surf, const WS& ws, int64_t o0,
                                                     int n, Filter* f) {
  Filter t = *f;
  const int st = variant_states<FIELD, 6, kState0>(p, s_surf, ws, o0, n, t);
  *f = t;
  return st;
}

template <int FIELD, int MODE>
__device__ __forceinline__ void fit_one_variants(const FitParams& p, const double* s_surf, int i) {
  const int t = track_of(p, i);
  const size_t TT = (size_t)p.n_tracks_total;
  const WS ws{p.ws64, p.ws32, (size_t)p.n_tracks, kRec64Fp64, 0, i};
  int64_t o0, o1;
  int n;
  int status = track_input(p, t, o0, o1, n);
  const bool states = p.out_states != nullptr;
  double xs[6], P0[21];
  double chi2sum = 0.0;
  int nmeas = 0;
  if (status == ST_OK) {
    Filter f;
    status = filter_first(p, t, o0, f);
    if (status == ST_OK) {
      if (MODE == kBackward) {
#pragma unroll
        for (int e = 0; e < 6; ++e) ws.d(0, BackRec::XF + e) = f.x[e];
#pragma unroll
        for (int e = 0; e < 21; ++e) ws.d(0, BackRec::CF + e) = f.C[e];
        status = variant_states<FIELD, 6, MODE>(p, s_surf, ws, o0, n, f);
      } else if (MODE == kEveryState) {
        status = variant_states<FIELD, 6, MODE>(p, s_surf, ws, o0, n, f);
      } else if (time_is_settled(f.C)) {
        status = variant_states<FIELD, 5, kState0>(p, s_surf, ws, o0, n, f);
      } else {
        Filter q = f;
        status = variant_states_with_time<FIELD>(p, s_surf, ws, o0, n, &q);
        f = q;
      }
    }
    chi2sum = f.chi2;
    nmeas = f.nmeas;
#pragma unroll
    for (int e = 0; e < 6; ++e) xs[e] = f.xs[e] + p.seed_params[e * TT + t];
#pragma unroll
    for (int e = 0; e < 21; ++e) P0[e] = f.P0[e];
    if (MODE != kBackward) {
      if (status == ST_OK && !f.spd) status = ST_NON_SPD;
      if (MODE == kEveryState && status == ST_OK) {
        smooth_states(ws, n, p.out_states, p.n_states, o0, true);
#pragma unroll
        for (int e = 0; e < 6; ++e) p.out_states[e * p.n_states + o0] = xs[e];
      }
    } else if (status == ST_OK) {
      double (&x)[6] = f.x;
      double (&C)[21] = f.C;
      Angles& ang = f.ang;
      // ------------------------------------------------ backward filter
      // starts at the last state from the forward-filtered parameters with
      // bf_scale times their covariance; the last state keeps the forward
      // filtered state.  x, C and ang are the backward state from here on.
      if (states)
#pragma unroll
        for (int e = 0; e < 6; ++e) p.out_states[e * p.n_states + o0 + n - 1] = x[e];
#pragma unroll
      for (int e = 0; e < 21; ++e) C[e] *= p.bf_scale;
      for (int k = n - 1; k >= 1; --k) {
        if (!p.is_hole[o0 + k]) {
          const double m[2] = {p.loc[o0 + k], p.loc[p.n_states + o0 + k]};
          const double V[3] = {p.cov[o0 + k], p.cov[p.n_states + o0 + k], p.cov[2 * p.n_states + o0 + k]};
          double c2, K[6][2], fs[3], r[2], dx[6];
          status = kalman_gain<6>(x, C, m, V, K, fs, r, dx, c2);
          if (status != ST_OK) break;
          joseph_update<6>(C, V, K);
#pragma unroll
          for (int e = 0; e < 6; ++e) x[e] += dx[e];
          turn(ang.cp, ang.sp, dx[2]);
          turn(ang.ct, ang.st, dx[3]);
        }
        // material of surface k at the backward state: its scattering noise,
        // then the mean loss restored (straggling on the downstream side)
        const Surf sk{s_surf + p.surface_id[o0 + k] * kSurfStride};
        const Surf sj{s_surf + p.surface_id[o0 + k - 1] * kSurfStride};
        const double xx0 = sk.xx0();
        if (xx0 > 0.0) {
          const double inv_cos = rcp_any(fma(sk.n(0), ang.cp * ang.st, fma(sk.n(1), ang.sp * ang.st, sk.n(2) * ang.ct)));
          const double lam = x[4];
          add_scattering(lam, fma(p.mass * p.mass * lam, lam, 1.0), xx0, inv_cos, rcp_any(ang.st), C);
          if (p.energy_loss) {
            double g, var_q;
            status = energy_loss(p, x[4], xx0, inv_cos, -1, g, var_q);
            if (status != ST_OK) break;
            C[sy(4, 4)] += var_q;
#pragma unroll
            for (int j = 0; j < 6; ++j) C[sym(4, j)] *= g;
            C[sy(4, 4)] *= g;
          }
        }
        // back-propagation to surface k-1
        Jac<double> J;
        End o;
        status = transport_variant<FIELD>(p, sk, sj, x, ang, o, J);
        if (status != ST_OK) break;
        ang = o.a;
        cov_transport<6>(J, 1.0, C);
        // weighted mean with the forward-filtered state k-1:
        //   K = Cf (Cf + Cb)^-1, xs = xf + K (xb - xf), Cs = Cf - K Cf,
        // on the states that are output; the others only have to be
        // positive definite
        double Cf[21], Ssum[21];
#pragma unroll
        for (int e = 0; e < 21; ++e) {
          Cf[e] = ws.d(k - 1, BackRec::CF + e);
          Ssum[e] = Cf[e] + C[e];
        }
        if (k > 1 && !states) {
          if (!spd_check<6>(Ssum)) {
            status = ST_NON_SPD;
            break;
          }
          continue;
        }
        x[2] = atan2_call(o.T[1], o.T[0]);
        x[3] = atan2_call(fma(o.a.cp, o.T[0], o.a.sp * o.T[1]), o.T[2]);
        double X[6][6], xf[6];  // X = (Cf + Cb)^-1 Cf = K^T
#pragma unroll
        for (int e = 0; e < 6; ++e) xf[e] = ws.d(k - 1, BackRec::XF + e);
        status = spd_solve_sym(Ssum, Cf, X);
        if (status != ST_OK) break;
#pragma unroll
        for (int r = 0; r < 6; ++r) {
          double acc = 0.0;
#pragma unroll
          for (int q = 0; q < 6; ++q) acc += X[q][r] * (x[q] - xf[q]);
          xs[r] = xf[r] + acc;
        }
#pragma unroll
        for (int r = 0; r < 6; ++r)
#pragma unroll
          for (int c = 0; c < 6; ++c)
            if (c <= r) {
              double acc = 0.0;
#pragma unroll
              for (int q = 0; q < 6; ++q) acc += X[q][r] * Cf[sym(q, c)];
              P0[sy(r, c)] = Cf[sy(r, c)] - acc;
            }
        if (states)
#pragma unroll
          for (int e = 0; e < 6; ++e) p.out_states[e * p.n_states + o0 + k - 1] = xs[e];
      }
    }
    if (status == ST_OK) {
      bool fin = isfinite(chi2sum);
#pragma unroll
      for (int e = 0; e < 6; ++e) fin = fin && isfinite(xs[e]);
#pragma unroll
      for (int e = 0; e < 21; ++e) fin = fin && isfinite(P0[e]);
      if (!fin) status = ST_NONFINITE;
    }
  }
  if (status != ST_OK) {
    const double nan = qnan();
#pragma unroll
    for (int e = 0; e < 6; ++e) xs[e] = nan;
#pragma unroll
    for (int e = 0; e < 21; ++e) P0[e] = nan;
    chi2sum = nan;
    nmeas = 0;
    if (p.out_states && n >= 1 && o0 >= 0 && o1 <= p.n_states && n <= p.max_states)
      for (int k = 0; k < n; ++k)
        for (int e = 0; e < 6; ++e) p.out_states[e * p.n_states + o0 + k] = nan;
  }
#pragma unroll
  for (int e = 0; e < 6; ++e) p.out_params[e * TT + t] = xs[e];
#pragma unroll
  for (int e = 0; e < 21; ++e) p.out_cov[e * TT + t] = P0[e];
  p.out_chi2[t] = chi2sum;
  if (p.out_ndf) p.out_ndf[t] = 2 * nmeas;
  if (p.out_status) p.out_status[t] = (uint8_t)status;
}

template <int FIELD, int MODE>
struct VariantBody {
  static constexpr int kStride = kSurfStride;
  static __device__ __forceinline__ void run(const FitParams& p, const double* s_surf, int i) {
    fit_one_variants<FIELD, MODE>(p, s_surf, i);
  }
};

template <int FIELD>
cudaError_t launch_mode(const FitParams& p, int block, cudaStream_t stream, int* launched) {
  if (p.smoother != 0) return launch_body<VariantBody<FIELD, kBackward>, 1>(p, block, stream, launched);
  if (p.out_states) return launch_body<VariantBody<FIELD, kEveryState>, 1>(p, block, stream, launched);
  return launch_body<VariantBody<FIELD, kState0>, 1>(p, block, stream, launched);
}

}  // namespace

cudaError_t launch_fit_variants(const FitParams& p, int block, cudaStream_t stream, int* launched) {
  if (launched) *launched = 0;
  if (p.n_tracks <= 0) return cudaSuccess;
  const int b = block ? block : 128;
  if (p.auto_shape && p.uniform() && !p.order) {
    // waves of one CTA per SM (plan_waves): 30k tracks with map, energy loss
    // and backward filter 10.6 -> 9.58 ms, 50k with energy loss 2.31 -> 2.17 ms
    int dev = 0, nsm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const WavePlan plan = plan_waves(((long long)p.n_tracks + 31) / 32, nsm, false);
    FitParams a = p;
    a.auto_shape = 0;
    a.work_counter = nullptr;
    int l = 0, count = 0;
    if (plan.main > 0) {
      const long long n = plan.main * 32;
      a.n_tracks = (int32_t)(n < p.n_tracks ? n : p.n_tracks);
      e = launch_fit_variants(a, 32 * plan.warps, stream, &l);
      if (e != cudaSuccess) return e;
      count = l;
      a.track0 = p.track0 + a.n_tracks;
      a.n_tracks = p.n_tracks - a.n_tracks;
    }
    e = launch_fit_variants(a, 32 * (plan.last > 0 ? plan.last : 1), stream, &l);
    if (launched) *launched = count + l;
    return e;
  }
  if (p.map_b) return launch_mode<2>(p, b, stream, launched);
  if (p.bfield[0] == 0.0 && p.bfield[1] == 0.0) return launch_mode<0>(p, b, stream, launched);
  return launch_mode<1>(p, b, stream, launched);
}

}  // namespace kfgb
