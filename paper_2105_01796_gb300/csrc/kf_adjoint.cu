// kf_adjoint.cu -- gradients of the Kalman fit with respect to per-surface
// alignment parameters and the seed parameters.
//
// Objective: L = sum_t [ w_t chi2_t + v_t . x_s0,t + W_t . C_s0,t ], chi2 of
// the predicted residuals (paper Sect. 2 filter step list), x_s0 and C_s0 the
// smoothed state 0 (the smoother paragraph).
//
// Method (reverse mode throughout), one thread per track, two passes:
//   F  the filter of the fit kernel with the smoothed state 0 carried along
//      (the fixed-point smoother of kf_fp64.cuh: S = Cov(x_0, x_k) beside x
//      and C); the filtered states (and S, when v or W is given) are written
//      to scratch;
//   B  for k = last .. 1: the transport k-1 -> k is run again from the stored
//      state, then reversed together with the update at k:
//       1. reverse through chi2_k, the gain-matrix update and the smoother's
//          update (exact algebra)
//       2. reverse through C_p = F C_f F^T + Q and S_p = S F^T
//       3. one reverse sweep through the transport gives the adjoints of its
//          18 inputs (x_f,k-1; the alignment of surfaces k-1 and k) for the
//          contraction with the adjoints of (x_p, F, Q): this includes the
//          derivative of F itself, since the sweep runs through the code
//          that forms F.
//     state 0: reverse through its update; x_p,0 is the seed.
// Alignment of a surface (shifts along its local axes, then rotations about
// them):  c' = c + R (du, dv, dn),  R' = R Ru(alpha) Rv(beta) Rn(gamma).  The
// moved surfaces and the derivative of R' are formed once per call
// (align_kernel); the adjoint of each surface's centre and axes is complete
// when both transitions that touch it are reversed, and only then contracted
// with them.
//
// The bound is the FP64 pipe.  The transport enters as the coefficients of
// operators in N v = kappa (v x B) (kf_transport.cuh), so its reverse is dot
// products of the columns' adjoints with N v and N^2 v plus scalar algebra
// per step, instead of a reverse of every RKN stage of every column; the
// smoother's reverse is a few products with S instead of a backward pass of
// its own with its recomputations.  Against the stage-by-stage reverse with
// checkpoints every 5 states and a separate smoother adjoint: chi2 gradient
// of 100k tracks x 21 states 50.3 -> 10.8 ms (9.6 ms without the time row,
// 9.4 ms with the cheaper logarithm), fit and whole gradient of 2000 tracks x
// 21 states 14.8 -> 3.57 ms (there two warps shared 32 tracks; 1.86 ms with
// the team kernel below).
// Storing every filtered state (176 B, whole fit 416 B) costs 0.14 ms of
// memory traffic on the 100k tracks; recomputing them took a quarter of the
// kernel.
// The fused multiply-adds are written out and the compiler contracts nothing
// more (as in kf_kernels.cu and kf_team.cu): the warps of a team agree, and
// both kernels give the same bits and those of the FP64 fit.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "kf_device.cuh"
#include "kf_filter.cuh"
#include "kf_fp64.cuh"
#include "kf_internal.h"
#include "kf_team.cuh"
#include "kf_transport.cuh"

namespace kfgb {
namespace {
using namespace dev;

// scratch per state and track (kf_filter.cuh)
constexpr int kRX = AdjRec::X, kRC = AdjRec::C, kRS = AdjRec::S;
constexpr int kRecFilter = AdjRec::kFilter, kRecWhole = AdjRec::kWhole;
// derivative table per surface: R, then R dM/d(angle) for the three angles
constexpr int kDTab = 36;

// The moved surface table (the fit kernels' layout) and the derivative
// table.  align null: zero alignment.
__global__ void align_kernel(int n, const double* __restrict__ packed, const double* __restrict__ align,
                             double* __restrict__ out, double* __restrict__ dtab) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  const Surf f{packed + (size_t)s * kSurfStride};
  double a[6], cs[3], sn[3];
  for (int e = 0; e < 6; ++e) a[e] = align ? align[(size_t)e * n + s] : 0.0;
  for (int m = 0; m < 3; ++m) sincos(a[3 + m], &sn[m], &cs[m]);
  const double Ru[9] = {1, 0, 0, 0, cs[0], -sn[0], 0, sn[0], cs[0]};
  const double Rv[9] = {cs[1], 0, sn[1], 0, 1, 0, -sn[1], 0, cs[1]};
  const double Rn[9] = {cs[2], -sn[2], 0, sn[2], cs[2], 0, 0, 0, 1};
  const double dRu[9] = {0, 0, 0, 0, -sn[0], -cs[0], 0, cs[0], -sn[0]};
  const double dRv[9] = {-sn[1], 0, cs[1], 0, 0, 0, -cs[1], 0, -sn[1]};
  const double dRn[9] = {-sn[2], -cs[2], 0, cs[2], -sn[2], 0, 0, 0, 0};
  double R[9];
  for (int e = 0; e < 9; ++e) R[e] = f.d[3 + e];
  auto mul = [](const double* X, const double* Y, double* Z) {
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j) Z[3 * i + j] = X[3 * i] * Y[j] + X[3 * i + 1] * Y[3 + j] + X[3 * i + 2] * Y[6 + j];
  };
  double* d = dtab + (size_t)s * kDTab;
  for (int e = 0; e < 9; ++e) d[e] = R[e];
  double x[9], y[9], R2[9];
  mul(Rv, Rn, x);
  mul(Ru, x, y);
  mul(R, y, R2);
  mul(dRu, x, y);
  mul(R, y, d + 9);
  mul(dRv, Rn, x);
  mul(Ru, x, y);
  mul(R, y, d + 18);
  mul(Rv, dRn, x);
  mul(Ru, x, y);
  mul(R, y, d + 27);
  double* o = out + (size_t)s * kSurfStride;
  for (int e = 0; e < kSurfStride; ++e) o[e] = f.d[e];
  for (int i = 0; i < 3; ++i) o[i] = f.d[i] + R[3 * i] * a[0] + R[3 * i + 1] * a[1] + R[3 * i + 2] * a[2];
  for (int e = 0; e < 9; ++e) o[3 + e] = R2[e];
}

__device__ __forceinline__ double dot3(const double a[3], const double b[3]) {
  return fma(a[0], b[0], fma(a[1], b[1], a[2] * b[2]));
}
__device__ __forceinline__ void axpy3(double a, const double x[3], double y[3]) {
#pragma unroll
  for (int i = 0; i < 3; ++i) y[i] = fma(a, x[i], y[i]);
}

// ---------------------------------------------------------------------------
// the transport with what its reverse needs
// ---------------------------------------------------------------------------
constexpr int kMaxSteps = 64 + 16;  // main steps and corrections

// One step of the path: the coefficients before it, its length and the
// Newton iterations summed in it (0: a main step).
struct Step {
  PathG<true> w;
  double s;
  int m;
};

struct Path {
  double T0[3], NT[3], NNT[3];
  double p00, pN, pNN, d0, s0;
  PathG<true> w;  // the whole path
  int nsub, n_steps;
};

// n . N^j T and n . (c - r) where the path has the coefficients w
__device__ __forceinline__ void path_scalars(const Path& p, const PathG<true>& w, double nu2, double& dist, double& p0,
                                             double& p1, double& p2) {
  p0 = p.p00 + fma(w.eb, p.pN, w.eg * p.pNN);
  p1 = fma(w.eb, p.pNN, fma(-nu2 * w.eg, p.pN, p.pN));
  p2 = fma(-nu2 * w.eb, p.pN, fma(-nu2 * w.eg, p.pNN, p.pNN));
  dist = p.d0 - fma(w.len, p.p00, fma(w.rb, p.pN, w.rg * p.pNN));
}

// one Newton iteration at correction length s (see propagate_to_plane)
__device__ __forceinline__ void newton_terms(double s, double lam, double nu2, double dist, double p0, double p1,
                                             double p2, double& di, double& nT, double& inv) {
  const double x = s * lam, y = x * x * nu2;
  const double c24 = fma(y, -1.0 / 24.0, 0.5);
  nT = fma(x, fma(x * c24, p2, fma(y, -1.0 / 6.0, 1.0) * p1), p0);
  di = fma(-s, fma(x, fma(x * (1.0 / 6.0), p2, c24 * p1), p0), dist);
  inv = rcp_nr<1>(nT);
}

// The path from r0 (angles a0) to plane b; tape[j] records step j.  The
// forward pass took this path already, so no step can fail.
template <bool BZ>
__device__ __forceinline__ void path_forward(const Surf& sb, const double r0[3], const Angles& a0, double lam,
                                             const double kB[3], double nu2, double h_max, int n_iter, Path& p,
                                             Step* tape) {
  p.T0[0] = a0.cp * a0.st;
  p.T0[1] = a0.sp * a0.st;
  p.T0[2] = a0.ct;
  applyA<double, BZ>(kB, p.T0, p.NT);
  applyA<double, BZ>(kB, p.NT, p.NNT);
  const double n[3] = {sb.n(0), sb.n(1), sb.n(2)};
  p.p00 = dot3(n, p.T0);
  p.pN = dot3(n, p.NT);
  p.pNN = dot3(n, p.NNT);
  p.d0 = fma(n[0], sb.c(0) - r0[0], fma(n[1], sb.c(1) - r0[1], n[2] * (sb.c(2) - r0[2])));
  p.s0 = p.d0 * rcp_any(p.p00);
  int nsub = 1;
  double h = p.s0;
  if (!(fabs(p.s0) <= h_max)) {
    const double nsub_d = fmin(ceil(fabs(p.s0) / h_max), 64.0);
    nsub = nsub_d < 1.0 ? 1 : (int)nsub_d;
    h = p.s0 / nsub;
  }
  p.nsub = nsub;
  p.w.step(h, lam, nu2, true);
  tape[0].s = h;
  tape[0].m = 0;
  int ns = 1;
  for (; ns < nsub; ++ns) {
    tape[ns].w = p.w;
    tape[ns].s = h;
    tape[ns].m = 0;
    p.w.step(h, lam, nu2, false);
  }
  for (int it = 0; it < n_iter; ++ns) {
    double dist, p0, p1, p2;
    path_scalars(p, p.w, nu2, dist, p0, p1, p2);
    double s = dist * rcp_any(p0);
    const int it0 = it++;
    while (it < n_iter) {
      const double x = s * lam;
      if (!(x * x * nu2 <= 1e-6)) break;
      double di, nT, inv;
      newton_terms(s, lam, nu2, dist, p0, p1, p2, di, nT, inv);
      s = fma(di, inv, s);
      ++it;
    }
    tape[ns].w = p.w;
    tape[ns].s = s;
    tape[ns].m = it - it0;
    p.w.step(s, lam, nu2, false);
  }
  p.n_steps = ns;
}

// adjoints of the coefficients of a path
struct CoefAdj {
  double eb, eg, rb, rg, deb, deg, drb, drg, len;
};

// Reverse of PathG::step(h, lam, nu2): a (adjoints of the coefficients after
// the step) becomes those before it; hb and lamb accumulate.  first: the
// coefficients before the step are zero.
__device__ __forceinline__ void step_reverse(const PathG<true>& w, double h, double lam, double nu2, bool first,
                                             CoefAdj& a, double& hb, double& lamb) {
  const double x = h * lam, x2 = x * x, y = x2 * nu2, hx = h * x, hh = h * h;
  const double t6 = fma(y, -1.0 / 6.0, 1.0), t24 = fma(y, -1.0 / 24.0, 0.5), t8 = fma(y, -0.125, 0.5);
  const double t2 = fma(y, -0.5, 1.0);
  const double b2 = x * t6, g2 = x2 * t24, rb2 = hx * t24, rg2 = hx * x * (1.0 / 6.0);
  const double db2 = h * t2, dg2 = hx * t6, drb2 = hh * t8, drg2 = hh * x * (1.0 / 3.0);
  double b2b, g2b, rb2b, rg2b, db2b, dg2b, drb2b, drg2b;
  hb += a.len;
  if (first) {
    b2b = a.eb; g2b = a.eg; rb2b = a.rb; rg2b = a.rg;
    db2b = a.deb; dg2b = a.deg; drb2b = a.drb; drg2b = a.drg;
  } else {
    const double eb = w.eb, eg1 = fma(-nu2, w.eg, 1.0), neb = -nu2 * w.eb;
    const double d1 = w.deb, d2 = w.deg, nd1 = -nu2 * d1, nd2 = -nu2 * d2;
    b2b = fma(a.eb, eg1, fma(a.eg, eb, fma(a.deb, nd2, a.deg * d1)));
    g2b = fma(a.eb, neb, fma(a.eg, eg1, fma(a.deb, nd1, a.deg * nd2)));
    rb2b = fma(a.rb, eg1, fma(a.rg, eb, fma(a.drb, nd2, a.drg * d1)));
    rg2b = fma(a.rb, neb, fma(a.rg, eg1, fma(a.drb, nd1, a.drg * nd2)));
    db2b = fma(a.deb, eg1, a.deg * eb);
    dg2b = fma(a.deb, neb, a.deg * eg1);
    drb2b = fma(a.drb, eg1, a.drg * eb);
    drg2b = fma(a.drb, neb, a.drg * eg1);
    hb += fma(a.rb, eb, fma(a.rg, w.eg, fma(a.drb, d1, a.drg * d2)));
    const double G1 = fma(-nu2, g2, 1.0), nb = -nu2 * b2, H1 = fma(-nu2, rg2, h), nrb = -nu2 * rb2;
    const double ndg = -nu2 * dg2, ndb = -nu2 * db2, ndrg = -nu2 * drg2, ndrb = -nu2 * drb2;
    CoefAdj o = a;  // rb, rg, drb, drg and len pass through
    o.eb = fma(a.eb, G1, fma(a.eg, b2, fma(a.rb, H1, fma(a.rg, rb2,
           fma(a.deb, ndg, fma(a.deg, db2, fma(a.drb, ndrg, a.drg * drb2)))))));
    o.eg = fma(a.eb, nb, fma(a.eg, G1, fma(a.rb, nrb, fma(a.rg, H1,
           fma(a.deb, ndb, fma(a.deg, ndg, fma(a.drb, ndrb, a.drg * ndrg)))))));
    o.deb = fma(a.deb, G1, fma(a.deg, b2, fma(a.drb, H1, a.drg * rb2)));
    o.deg = fma(a.deb, nb, fma(a.deg, G1, fma(a.drb, nrb, a.drg * H1)));
    a = o;
  }
  // the step's own coefficients as functions of (h, x = h lam)
  const double xb = fma(b2b, t2, fma(g2b, b2, fma(rb2b * h, t8, fma(rg2b, hx * (1.0 / 3.0),
                    fma(db2b, -hx * nu2, fma(dg2b * h, t2, fma(drb2b, -0.25 * hh * x * nu2,
                    drg2b * hh * (1.0 / 3.0))))))));
  hb += fma(rb2b * x, t24, fma(rg2b, x2 * (1.0 / 6.0), fma(db2b, t2, fma(dg2b, b2,
        fma(drb2b, 2.0 * h * t8, fma(drg2b, hx * (2.0 / 3.0), xb * lam))))));
  lamb = fma(xb, h, lamb);
}

// v x B operators transposed: N^T = -N
template <bool BZ>
__device__ __forceinline__ void add_transposed(const double kB[3], const double y1[3], const double y2[3],
                                               double out[3]) {
  // out += N^T y1 + (N^2)^T y2 = -N (y1 - N y2)
  if (BZ) {
    const double z0 = fma(-y2[1], kB[2], y1[0]), z1 = fma(y2[0], kB[2], y1[1]);
    out[0] = fma(-z1, kB[2], out[0]);
    out[1] = fma(z0, kB[2], out[1]);
    return;
  }
  double z[3], q[3];
  applyA<double, false>(kB, y2, z);
#pragma unroll
  for (int i = 0; i < 3; ++i) z[i] = y1[i] - z[i];
  applyA<double, false>(kB, z, q);
#pragma unroll
  for (int i = 0; i < 3; ++i) out[i] -= q[i];
}

// adjoint of a surface's centre and axes
struct PlaneAdj {
  double c[3], u[3], v[3], n[3];
};

// Reverse of a transport.  In: the forward's path, tape, end state, columns
// and inv_nT; lxp (adjoint of x_p), lJ(r, c) (of F, rows 0..3 over columns
// 0..4), lqp, lqt (of the scattering variances).  The objective does not
// depend on the time of any state but the seed's, so nothing here has a time.  Out: lx; the
// adjoints of plane a (c, u, v) in pa, those of plane b added to pb.
template <bool BZ, class LJ>
__device__ __forceinline__ void transport_reverse(const Surf& sa, const Surf& sb, const double x01[2],
                                                  const double r0[3], const Angles& a0, double lam, const double kB[3],
                                                  double nu2, double mass, double xx0, const Path& p, const Step* tape,
                                                  const End& o, const Cols64& g, double inv_nT, const double lxp[5],
                                                  LJ lJ, double lqp, double lqt, double lx[5], PlaneAdj& pa,
                                                  PlaneAdj& pb) {
  const double m2 = mass * mass;
  const double u[3] = {sb.u(0), sb.u(1), sb.u(2)}, v[3] = {sb.v(0), sb.v(1), sb.v(2)}, n[3] = {sb.n(0), sb.n(1), sb.n(2)};
  const double* T = o.T;
  const double is = o.inv_st;
  const double fv[2] = {-o.a.sp * is, o.a.cp * is};
  const double hv[3] = {o.a.cp * o.a.ct, o.a.sp * o.a.ct, -o.a.st};
  double NTe[3], AT[3];
  applyA<double, BZ>(kB, T, NTe);
#pragma unroll
  for (int i = 0; i < 3; ++i) AT[i] = lam * NTe[i];
  const double uT = dot3(u, T), vT = dot3(v, T);
  const double fA = fma(fv[0], AT[0], fv[1] * AT[1]), hA = dot3(hv, AT);

  double Tb[3] = {0.0, 0.0, 0.0}, rb[3], lamb = lxp[4];
  double uTb = 0.0, vTb = 0.0, fAb = 0.0, hAb = 0.0, nTb = 0.0;
  double fvb[2] = {0.0, 0.0}, hvb[3] = {0.0, 0.0, 0.0};
  double pc[5][3], tc[3][3];  // adjoints of the columns
  // x_p = (u . d, v . d), d = r - c
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const double d = o.r[i] - sb.c(i);
    rb[i] = fma(lxp[0], u[i], lxp[1] * v[i]);
    pb.u[i] = fma(lxp[0], d, pb.u[i]);
    pb.v[i] = fma(lxp[1], d, pb.v[i]);
    pb.c[i] -= rb[i];
  }
  // the projections of the columns (see jacobian_columns)
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    const double q[3] = {c == 0 ? sa.u(0) : c == 1 ? sa.v(0) : g.gr[0][c < 2 ? 0 : c - 2],
                         c == 0 ? sa.u(1) : c == 1 ? sa.v(1) : g.gr[1][c < 2 ? 0 : c - 2],
                         c == 0 ? sa.u(2) : c == 1 ? sa.v(2) : g.gr[2][c < 2 ? 0 : c - 2]};
    const double l0 = lJ(0, c), l1 = lJ(1, c), l2 = lJ(2, c), l3 = lJ(3, c);
    const double w = -dot3(n, q) * inv_nT;
    const double wb = fma(l0, uT, fma(l1, vT, fma(l2, fA, l3 * hA)));
    uTb = fma(l0, w, uTb);
    vTb = fma(l1, w, vTb);
    fAb = fma(l2, w, fAb);
    hAb = fma(l3, w, hAb);
    const double wi = -wb * inv_nT;
    nTb = fma(wi, w, nTb);
#pragma unroll
    for (int i = 0; i < 3; ++i) pc[c][i] = fma(l0, u[i], fma(l1, v[i], wi * n[i]));
    axpy3(l0, q, pb.u);
    axpy3(l1, q, pb.v);
    axpy3(wi, q, pb.n);
    if (c >= 2) {
      tc[c - 2][0] = fma(l2, fv[0], l3 * hv[0]);
      tc[c - 2][1] = fma(l2, fv[1], l3 * hv[1]);
      tc[c - 2][2] = l3 * hv[2];
      fvb[0] = fma(l2, g.gT[0][c - 2], fvb[0]);
      fvb[1] = fma(l2, g.gT[1][c - 2], fvb[1]);
#pragma unroll
      for (int i = 0; i < 3; ++i) hvb[i] = fma(l3, g.gT[i][c - 2], hvb[i]);
    }
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    pa.u[i] = pc[0][i];
    pa.v[i] = pc[1][i];
  }
  // Highland noise: q = (0.0136 lam)^2 g2 eps l^2, q_phi = q / sin^2(theta),
  // eps = xx0 |T| / |n.T|, l = 1 + 0.038 ln(eps g2)
  double isb = 0.0, tnb = 0.0;  // tnb: adjoint of ln |T|
  if (xx0 > 0.0) {
    const double eps = xx0 * fabs(o.inv_cos), a = 0.0136 * lam;
    const double l = fma(0.038, log_df(eps * o.g2), 1.0), il = 0.076 * rcp_any(l);
    const double q = a * a * o.g2 * eps * (l * l);
    const double qb = fma(lqp, is * is, lqt) * q;
    isb = 2.0 * lqp * q * is;
    const double ge = qb * (1.0 + il);
    lamb = fma(2.0 * qb, rcp_any(lam), fma(ge, 2.0 * m2 * lam * rcp_any(o.g2), lamb));
    tnb = ge;
    nTb = fma(-ge, inv_nT, nTb);
  }
  // uT = u . T, vT = v . T, fA = f . AT, hA = h . AT, AT = lam N T, nT = n . T
  double ATb[3];
  axpy3(uTb, u, Tb);
  axpy3(vTb, v, Tb);
  axpy3(nTb, n, Tb);
  axpy3(uTb, T, pb.u);
  axpy3(vTb, T, pb.v);
  axpy3(nTb, T, pb.n);
  fvb[0] = fma(fAb, AT[0], fvb[0]);
  fvb[1] = fma(fAb, AT[1], fvb[1]);
  axpy3(hAb, AT, hvb);
  ATb[0] = fma(fAb, fv[0], hAb * hv[0]);
  ATb[1] = fma(fAb, fv[1], hAb * hv[1]);
  ATb[2] = hAb * hv[2];
  lamb += dot3(ATb, NTe);
  {
    double z[3];
    applyA<double, BZ>(kB, ATb, z);
    axpy3(-lam, z, Tb);  // N^T = -N
  }
  // f = (-sin phi, cos phi) / sin theta, h = (cos phi cos theta, sin phi cos
  // theta, -sin theta): through the angles, dphi = f . dT / |T|, dtheta = h . dT / |T|
  {
    const double cpb = fma(fvb[1], is, hvb[0] * o.a.ct), spb = fma(-fvb[0], is, hvb[1] * o.a.ct);
    isb = fma(fvb[1], o.a.cp, fma(-fvb[0], o.a.sp, isb));
    const double ctb = fma(hvb[0], o.a.cp, hvb[1] * o.a.sp);
    const double stb = fma(-isb, is * is, -hvb[2]);
    const double itn = fabs(o.inv_cos) > 0.0 ? inv_nT * rcp_any(o.inv_cos) : 0.0;  // 1 / |T|
    const double phib = (lxp[2] + fma(o.a.cp, spb, -o.a.sp * cpb)) * itn;
    const double thb = (lxp[3] + fma(o.a.ct, stb, -o.a.st * ctb)) * itn;
    const double tt = tnb * (itn * itn);
    Tb[0] += fma(phib, fv[0], fma(thb, hv[0], tt * T[0]));
    Tb[1] += fma(phib, fv[1], fma(thb, hv[1], tt * T[1]));
    Tb[2] += fma(thb, hv[2], tt * T[2]);
  }
  CoefAdj a;
  // the operators on T, the phi and theta columns, and their lam derivatives
  // on T (the q/p column): out = (len + rb N + rg N^2) v to the position,
  // (1 + eb N + eg N^2) v to the direction
  const PathG<true>& w = p.w;
  double Vb[3][3];  // adjoints of T0, v_phi, v_theta
  a.eb = dot3(Tb, p.NT);
  a.eg = dot3(Tb, p.NNT);
  a.rb = dot3(rb, p.NT);
  a.rg = dot3(rb, p.NNT);
  a.len = dot3(rb, p.T0);
  a.deb = dot3(tc[2], p.NT);
  a.deg = dot3(tc[2], p.NNT);
  a.drb = dot3(pc[4], p.NT);
  a.drg = dot3(pc[4], p.NNT);
  {
    double y1[3], y2[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      Vb[0][i] = fma(w.len, rb[i], Tb[i]);
      y1[i] = fma(w.rb, rb[i], fma(w.eb, Tb[i], fma(w.drb, pc[4][i], w.deb * tc[2][i])));
      y2[i] = fma(w.rg, rb[i], fma(w.eg, Tb[i], fma(w.drg, pc[4][i], w.deg * tc[2][i])));
    }
    add_transposed<BZ>(kB, y1, y2, Vb[0]);
  }
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const double vc[3] = {c == 0 ? -p.T0[1] : a0.cp * a0.ct, c == 0 ? p.T0[0] : a0.sp * a0.ct, c == 0 ? 0.0 : -a0.st};
    double Nv[3], NNv[3], y1[3], y2[3];
    applyA<double, BZ>(kB, vc, Nv);
    applyA<double, BZ>(kB, Nv, NNv);
    a.eb += dot3(tc[c], Nv);
    a.eg += dot3(tc[c], NNv);
    a.rb += dot3(pc[2 + c], Nv);
    a.rg += dot3(pc[2 + c], NNv);
    a.len += dot3(pc[2 + c], vc);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      Vb[1 + c][i] = fma(w.len, pc[2 + c][i], tc[c][i]);
      y1[i] = fma(w.rb, pc[2 + c][i], w.eb * tc[c][i]);
      y2[i] = fma(w.rg, pc[2 + c][i], w.eg * tc[c][i]);
    }
    add_transposed<BZ>(kB, y1, y2, Vb[1 + c]);
  }
  // the steps, last first
  double d0b = 0.0, p00b = 0.0, pNb = 0.0, pNNb = 0.0, hmain = 0.0;
#pragma unroll 1
  for (int j = p.n_steps - 1; j >= 0; --j) {
    const Step& st = tape[j];
    double sbar = 0.0;
    step_reverse(st.w, st.s, lam, nu2, j == 0, a, sbar, lamb);
    if (st.m == 0) {
      hmain += sbar;
      continue;
    }
    // the correction's Newton iterations, replayed
    double dist, p0, p1, p2, p0b = 0.0, p1b = 0.0, p2b = 0.0, distb = 0.0;
    path_scalars(p, st.w, nu2, dist, p0, p1, p2);
    const double ip0 = rcp_any(p0);
    double it_s[16], it_di[16], it_inv[16];
    double s = dist * ip0;
    for (int i = 1; i < st.m; ++i) {
      double di, nT, inv;
      newton_terms(s, lam, nu2, dist, p0, p1, p2, di, nT, inv);
      it_s[i & 15] = s;
      it_di[i & 15] = di;
      it_inv[i & 15] = inv;
      s = fma(di, inv, s);
    }
    for (int i = st.m - 1; i >= 1; --i) {
      const double si = it_s[i & 15], inv = it_inv[i & 15];
      const double x = si * lam, y = x * x * nu2, c24 = fma(y, -1.0 / 24.0, 0.5), t6 = fma(y, -1.0 / 6.0, 1.0);
      const double dib = sbar * inv, nTb2 = -dib * (it_di[i & 15] * inv);
      const double gg = fma(x, fma(x * (1.0 / 6.0), p2, c24 * p1), p0), gb = -dib * si;
      distb += dib;
      sbar = fma(-dib, gg, sbar);
      p0b += fma(-dib, si, nTb2);
      p1b = fma(gb, x * c24, fma(nTb2, x * t6, p1b));
      p2b = fma(gb, x * x * (1.0 / 6.0), fma(nTb2, x * x * c24, p2b));
      const double xb = fma(gb, fma(x * (1.0 / 3.0), p2, fma(y, -0.125, 0.5) * p1),
                            nTb2 * fma(x * t6, p2, fma(y, -0.5, 1.0) * p1));
      sbar = fma(xb, lam, sbar);
      lamb = fma(xb, si, lamb);
    }
    {
      const double db = sbar * ip0;
      distb += db;
      p0b = fma(-db, dist * ip0, p0b);
    }
    const double eg1 = fma(-nu2, st.w.eg, 1.0), neb = -nu2 * st.w.eb;
    p00b += fma(-distb, st.w.len, p0b);
    pNb += fma(p0b, st.w.eb, fma(p1b, eg1, fma(p2b, neb, -distb * st.w.rb)));
    pNNb += fma(p0b, st.w.eg, fma(p1b, st.w.eb, fma(p2b, eg1, -distb * st.w.rg)));
    d0b += distb;
    a.eb += fma(p0b, p.pN, fma(p1b, p.pNN, -nu2 * p2b * p.pN));
    a.eg += fma(p0b, p.pNN, -nu2 * fma(p1b, p.pN, p2b * p.pNN));
    a.len = fma(-distb, p.p00, a.len);
    a.rb = fma(-distb, p.pN, a.rb);
    a.rg = fma(-distb, p.pNN, a.rg);
  }
  {
    const double s0b = p.nsub == 1 ? hmain : hmain / (double)p.nsub;
    const double db = s0b * rcp_any(p.p00);
    d0b += db;
    p00b = fma(-db, p.s0, p00b);
  }
  // d0 = n . (c - r0); p00 = n . T0, pN = n . N T0, pNN = n . N^2 T0
  {
    double y1[3], y2[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      pb.n[i] += fma(d0b, sb.c(i) - r0[i], fma(p00b, p.T0[i], fma(pNb, p.NT[i], pNNb * p.NNT[i])));
      pb.c[i] = fma(d0b, n[i], pb.c[i]);
      rb[i] = fma(-d0b, n[i], rb[i]);
      Vb[0][i] = fma(p00b, n[i], Vb[0][i]);
      y1[i] = pNb * n[i];
      y2[i] = pNNb * n[i];
    }
    add_transposed<BZ>(kB, y1, y2, Vb[0]);
  }
  // the start: r0 = c + x0 u + x1 v; T0 and the columns from the angles
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    pa.c[i] = rb[i];
    pa.u[i] = fma(x01[0], rb[i], pa.u[i]);
    pa.v[i] = fma(x01[1], rb[i], pa.v[i]);
    pa.n[i] = 0.0;
  }
  lx[0] = fma(rb[0], sa.u(0), fma(rb[1], sa.u(1), rb[2] * sa.u(2)));
  lx[1] = fma(rb[0], sa.v(0), fma(rb[1], sa.v(1), rb[2] * sa.v(2)));
  const double cpst = p.T0[0], spst = p.T0[1], cpct = a0.cp * a0.ct, spct = a0.sp * a0.ct;
  // v_phi = (-sp st, cp st, 0), v_theta = (cp ct, sp ct, -st)
  lx[2] = fma(Vb[0][1], cpst, -Vb[0][0] * spst) - fma(Vb[1][0], cpst, Vb[1][1] * spst) +
          fma(Vb[2][1], cpct, -Vb[2][0] * spct);
  lx[3] = fma(Vb[0][0], cpct, fma(Vb[0][1], spct, -Vb[0][2] * a0.st)) + fma(Vb[1][1], cpct, -Vb[1][0] * spct) -
          fma(Vb[2][0], cpst, fma(Vb[2][1], spst, Vb[2][2] * a0.ct));
  lx[4] = lamb;
}

// ---------------------------------------------------------------------------
// the update
// ---------------------------------------------------------------------------

// What the smoother adds to the reverse of a transition: with h = Sp H^T
// (Sp = Cov(x_0, x_k) predicted) its update is
//   x0 += h y (weight v), P0 -= h Si h^T (weight W), Sf = Sp - h Si P^T,
// and its prediction Sp = S F^T.  Contributions to the adjoints of y (yb), Si
// (G: 00, 01, 11) and F (lF), and LS^T h for that of P (Z).
struct SmOut {
  double yb[2], G[3], Z[5][2], lF[4][5];
};

// The factors of S at a state's update (innovation_solve: as in the filter, no
// inverse of S is formed) and y = Si r.
struct Innov {
  double f[3], r[2], y[2];
};
__device__ __forceinline__ Innov innovation(const double xp[2], const double Cp[21], const double m[2],
                                            const double V[3]) {
  const double S00 = V[0] + Cp[sy(0, 0)], S01 = V[1] + Cp[sy(1, 0)], S11 = V[2] + Cp[sy(1, 1)];
  Innov q;
  q.f[0] = rcp_any(S00);
  q.f[1] = S01 * q.f[0];
  q.f[2] = rcp_any(fma(-q.f[1], S01, S11));
  q.r[0] = m[0] - xp[0];
  q.r[1] = m[1] - xp[1];
  innovation_solve(q.f, q.r[0], q.r[1], q.y[0], q.y[1]);
  return q;
}

// Reverse through one measured update:
//   P = Cp H^T, S = V + H Cp H^T, Si = S^-1, r = m - H xp, y = Si r,
//   xf = xp + P y, Cf = Cp - P Si P^T, chi2 = r^T y (weight w),
// with the smoother's contributions if SM.  lf, Lf (packed, full-matrix
// convention; adjoints of xf, Cf) become those of xp, Cp.  N: parameters
// (5: without the time).
template <bool SM, int N>
__device__ __forceinline__ void update_reverse(const Innov& q, const double Cp[21], double w, const SmOut& sm,
                                               double lf[6], double Lf[21]) {
  // U = Lf P; yb = P^T lf (+ h^T v); G = adjoint of Si (symmetric)
  const double* r = q.r;
  double Z[6][2], yb[2] = {0.0, 0.0};
  const double wr0 = w * r[0], wr1 = w * r[1];
  double G00, G01, G11;
  if (SM) {
    yb[0] = sm.yb[0];
    yb[1] = sm.yb[1];
    G00 = fma(wr0, r[0], sm.G[0]);
    G01 = fma(wr0, r[1], sm.G[1]);
    G11 = fma(wr1, r[1], sm.G[2]);
  } else {
    G00 = wr0 * r[0];
    G01 = wr0 * r[1];
    G11 = wr1 * r[1];
  }
#pragma unroll
  for (int i = 0; i < N; ++i) {
    double u0 = 0.0, u1 = 0.0;
#pragma unroll
    for (int j = 0; j < N; ++j) {
      u0 = fma(Lf[sym(i, j)], Cp[sym(j, 0)], u0);
      u1 = fma(Lf[sym(i, j)], Cp[sym(j, 1)], u1);
    }
    yb[0] = fma(Cp[sym(i, 0)], lf[i], yb[0]);
    yb[1] = fma(Cp[sym(i, 1)], lf[i], yb[1]);
    G00 = fma(-Cp[sym(i, 0)], u0, G00);
    G01 = fma(-Cp[sym(i, 0)], u1, G01);
    G11 = fma(-Cp[sym(i, 1)], u1, G11);
    Z[i][0] = SM && i < 5 ? fma(2.0, u0, sm.Z[i < 5 ? i : 0][0]) : 2.0 * u0;
    Z[i][1] = SM && i < 5 ? fma(2.0, u1, sm.Z[i < 5 ? i : 0][1]) : 2.0 * u1;
  }
  G00 = fma(yb[0], r[0], G00);
  G11 = fma(yb[1], r[1], G11);
  G01 = fma(0.5, fma(yb[0], r[1], yb[1] * r[0]), G01);
  // adjoint of S: -Si G Si
  double t00, t01, t10, t11, x00, x10, x01, x11;
  innovation_solve(q.f, G00, G01, t00, t01);
  innovation_solve(q.f, G01, G11, t10, t11);
  innovation_solve(q.f, t00, t10, x00, x10);
  innovation_solve(q.f, t01, t11, x01, x11);
  Lf[sy(0, 0)] -= x00;
  Lf[sy(1, 0)] -= x10;
  Lf[sy(1, 1)] -= x11;
  // adjoint of P: lf y^T - Z Si, into columns 0 and 1 (symmetrised)
#pragma unroll
  for (int i = 0; i < N; ++i) {
    double z0, z1;
    innovation_solve(q.f, Z[i][0], Z[i][1], z0, z1);
    const double P0 = fma(lf[i], q.y[0], -z0);
    const double P1 = fma(lf[i], q.y[1], -z1);
    Lf[sym(i, 0)] = i == 0 ? Lf[sym(i, 0)] + P0 : fma(0.5, P0, Lf[sym(i, 0)]);
    Lf[sym(i, 1)] = i == 1 ? Lf[sym(i, 1)] + P1 : fma(0.5, P1, Lf[sym(i, 1)]);
  }
  // adjoint of r: Si (yb + 2 w r)
  double s0, s1;
  innovation_solve(q.f, yb[0], yb[1], s0, s1);
  lf[0] -= fma(2.0 * w, q.y[0], s0);
  lf[1] -= fma(2.0 * w, q.y[1], s1);
}

struct GradParams {
  FitParams f;          // geometry (the moved surfaces), inputs, options
                        // (outputs unused); a launch covers tracks
                        // [track0, track0 + n_tracks) of n_tracks_total
  const double* dtab;        // [S][kDTab] derivative table
  const double* dl_dchi2;    // [T] or null (all ones)
  const double* dl_dparams;  // [6][T] or null: weights of the smoothed state-0 parameters
  const double* dl_dcov;     // [21][T] or null: weights of its packed covariance
  double* chi2;         // [T] or null
  double* out_params;   // [6][T] or null: smoothed parameters of state 0
  double* out_cov;      // [21][T] or null: smoothed covariance of state 0
  double* grad_seed;    // [6][T] or null
  double* grad_align;   // [6][S] or null (accumulated with atomicAdd; zeroed by the host)
  double* rec;          // [max_states][kRecFilter or kRecWhole][n_tracks]
};

// add v[0..5] to grad_align[.][sid] (all 32 lanes of the warp call this
// together; inactive lanes pass act = false).  When every active lane is on
// the same surface the warp adds its sums once, lane e the sum e; otherwise
// each active lane adds.
__device__ __forceinline__ void add_align_grad(double* grad, int n_surf, int sid, const double v[6], bool act) {
  const unsigned full = 0xffffffffu;
  const unsigned any = __ballot_sync(full, act);
  if (any == 0u) return;
  const int lead = __ffs(any) - 1;
  const int sid0 = __shfl_sync(full, sid, lead);
  if (__all_sync(full, !act || sid == sid0)) {
    const int lane = threadIdx.x & 31;
    double mine = 0.0;
#pragma unroll
    for (int e = 0; e < 6; ++e) {
      double sum = act ? v[e] : 0.0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(full, sum, o);
      if (lane == e) mine = sum;
    }
    if (lane < 6) atomicAdd(&grad[(size_t)lane * n_surf + sid0], mine);
  } else if (act) {
#pragma unroll
    for (int e = 0; e < 6; ++e) atomicAdd(&grad[(size_t)e * n_surf + sid], v[e]);
  }
}

// the surface's six alignment derivatives from the adjoint of its centre and axes
__device__ __forceinline__ void plane_gradient(const double* __restrict__ d, const PlaneAdj& a, double out[6]) {
#pragma unroll
  for (int e = 0; e < 3; ++e) out[e] = fma(d[e], a.c[0], fma(d[3 + e], a.c[1], d[6 + e] * a.c[2]));
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    const double* D = d + 9 + 9 * m;
    double v = 0.0;
#pragma unroll
    for (int i = 0; i < 3; ++i) v = fma(a.u[i], D[3 * i], fma(a.v[i], D[3 * i + 1], fma(a.n[i], D[3 * i + 2], v)));
    out[3 + m] = v;
  }
}

// One track of a launch as pass B sees it.
template <bool SM>
struct TrackB {
  const GradParams* g;
  const double* s_surf;
  int64_t o0;
  int tl, tg;
  double kB[3], nu2;
  __device__ __forceinline__ TrackB(const GradParams& gp, const double* surf, int slot, bool bz)
      : g(&gp), s_surf(surf), tl(slot), tg(gp.f.track0 + slot) {
    o0 = gp.f.offsets[tg];
#pragma unroll
    for (int e = 0; e < 3; ++e) kB[e] = kKappa * gp.f.bfield[e];
    nu2 = bz ? kB[2] * kB[2] : dot3(kB, kB);
  }
  __device__ __forceinline__ double rec(int k, int e) const {
    return g->rec[((size_t)k * (SM ? kRecWhole : kRecFilter) + e) * (size_t)g->f.n_tracks + tl];
  }
  __device__ __forceinline__ Surf surf(int k) const { return Surf{s_surf + g->f.surface_id[o0 + k] * kSurfStride}; }
  __device__ __forceinline__ bool hole(int k) const { return g->f.is_hole[o0 + k] != 0; }
};

// the filtered state a transition starts from
struct StartB {
  double x01[2], lam, r0[3];
  Angles a0;
};
template <bool SM>
__device__ __forceinline__ StartB start_of(const TrackB<SM>& t, int k) {
  StartB s;
  s.x01[0] = t.rec(k - 1, kRX + 0);
  s.x01[1] = t.rec(k - 1, kRX + 1);
  s.lam = t.rec(k - 1, kRX + 2);
  s.a0 = {t.rec(k - 1, kRX + 3), t.rec(k - 1, kRX + 4), t.rec(k - 1, kRX + 5), t.rec(k - 1, kRX + 6)};
  const Surf sa = t.surf(k - 1);
#pragma unroll
  for (int e = 0; e < 3; ++e) s.r0[e] = fma(s.x01[0], sa.u(e), fma(s.x01[1], sa.v(e), sa.c(e)));
  return s;
}

// Transition k-1 -> k run again.
struct FwdB {
  Path path;
  End o;
  Cols64 gc;
  double inv_nT, F[4][5], xp[2], Cp[21], hm[6][2];
};

// every double of it that another warp needs (the tape apart)
template <bool SM, class V>
__device__ __forceinline__ void visit(FwdB& f, V v) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    v(f.path.T0[i]); v(f.path.NT[i]); v(f.path.NNT[i]);
    v(f.o.r[i]); v(f.o.T[i]);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      v(f.gc.gr[i][c]);
      v(f.gc.gT[i][c]);
    }
  }
  v(f.path.p00); v(f.path.pN); v(f.path.pNN); v(f.path.d0); v(f.path.s0);
  PathG<true>& w = f.path.w;
  v(w.eb); v(w.eg); v(w.rb); v(w.rg); v(w.deb); v(w.deg); v(w.drb); v(w.drg); v(w.len);
  v(f.o.a.cp); v(f.o.a.sp); v(f.o.a.ct); v(f.o.a.st); v(f.o.inv_st); v(f.o.inv_cos); v(f.o.g2);
  v(f.inv_nT);
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 5; ++c) v(f.F[r][c]);
  v(f.xp[0]); v(f.xp[1]);
#pragma unroll
  for (int e = 0; e < 15; ++e) v(f.Cp[e]);
  if (SM)
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      v(f.hm[i][0]);
      v(f.hm[i][1]);
    }
}

template <bool BZ, bool SM>
__device__ __forceinline__ void forward_part(const TrackB<SM>& t, int k, const StartB& st, FwdB& f, Step* tape) {
  const FitParams& p = t.g->f;
  const Surf sa = t.surf(k - 1), sb = t.surf(k);
  const double Bf[3] = {p.bfield[0], p.bfield[1], p.bfield[2]};
  Path& path = f.path;
  End& o = f.o;
  Cols64& gc = f.gc;
  path_forward<BZ>(sb, st.r0, st.a0, st.lam, t.kB, t.nu2, p.h_max, p.n_iter, path, tape);
  const PathG<true>& q = path.w;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    o.r[i] = st.r0[i] + fma(q.len, path.T0[i], fma(q.rb, path.NT[i], q.rg * path.NNT[i]));
    o.T[i] = path.T0[i] + fma(q.eb, path.NT[i], q.eg * path.NNT[i]);
    gc.gr[i][2] = fma(q.drb, path.NT[i], q.drg * path.NNT[i]);
    gc.gT[i][2] = fma(q.deb, path.NT[i], q.deg * path.NNT[i]);
  }
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const double vc[3] = {c == 0 ? -path.T0[1] : st.a0.cp * st.a0.ct, c == 0 ? path.T0[0] : st.a0.sp * st.a0.ct,
                          c == 0 ? 0.0 : -st.a0.st};
    double Nv[3], NNv[3];
    applyA<double, BZ>(t.kB, vc, Nv);
    applyA<double, BZ>(t.kB, Nv, NNv);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      gc.gr[i][c] = fma(q.len, vc[i], fma(q.rb, Nv[i], q.rg * NNv[i]));
      gc.gT[i][c] = vc[i] + fma(q.eb, Nv[i], q.eg * NNv[i]);
    }
  }
  o.g2 = fma(p.mass * p.mass * st.lam, st.lam, 1.0);
  o.dtds = gc.gtl = 0.0;  // (no time row)
  end_frame(sb, o, f.inv_nT);
  Jac<double> J;
  jacobian_columns<BZ, 31>(sa, sb, o, gc, st.lam, Bf, f.inv_nT, [&](int r, int c, double x) {
    if (r < 4) J.f[r][c] = f.F[r][c] = x;
  });
  if (t.hole(k)) return;
#pragma unroll
  for (int e = 0; e < 15; ++e) f.Cp[e] = t.rec(k - 1, kRC + e);
  cov_transport<5>(J, 1.0, f.Cp);
  const double xx0 = sb.xx0();
  if (xx0 > 0.0) {
    const double z = highland_sq(st.lam, o.g2, xx0, o.inv_cos);
    f.Cp[sy(2, 2)] = fma(z, o.inv_st * o.inv_st, f.Cp[sy(2, 2)]);
    f.Cp[sy(3, 3)] += z;
  }
  if (SM)
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      double h0 = 0.0, h1 = 0.0;
#pragma unroll
      for (int c = 0; c < 5; ++c) {
        const double z = t.rec(k - 1, kRS + 5 * i + c);
        h0 = fma(f.F[0][c], z, h0);
        h1 = fma(f.F[1][c], z, h1);
      }
      f.hm[i][0] = h0;
      f.hm[i][1] = h1;
    }
  const double d0 = o.r[0] - sb.c(0), d1 = o.r[1] - sb.c(1), d2 = o.r[2] - sb.c(2);
  f.xp[0] = fma(d0, sb.u(0), fma(d1, sb.u(1), d2 * sb.u(2)));
  f.xp[1] = fma(d0, sb.v(0), fma(d1, sb.v(1), d2 * sb.v(2)));
}

// the innovation of transition k run again (of a hole: not used)
template <bool SM>
__device__ __forceinline__ Innov innovation_at(const TrackB<SM>& t, int k, const FwdB& f) {
  Innov q;
  if (t.hole(k)) return q;
  double m[2], V[3];
  hit_of(t.g->f, t.o0 + k, m, V);
  return innovation(f.xp, f.Cp, m, V);
}

// The smoother's part of the reverse of transition k: LS (adjoint of S_k)
// becomes that of S_k-1; it depends on nothing else of the reverse.
__device__ __forceinline__ void smoother_part(const TrackB<true>& t, int k, const double F[4][5], const double Cp[21],
                                              const Innov& q, const double hm[6][2], const double v[6],
                                              const double W[21], double LS[6][5], SmOut& o) {
  if (!t.hole(k)) {
    o.yb[0] = o.yb[1] = o.G[0] = o.G[1] = o.G[2] = 0.0;
#pragma unroll
    for (int j = 0; j < 5; ++j) o.Z[j][0] = o.Z[j][1] = 0.0;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      o.yb[0] = fma(hm[i][0], v[i], o.yb[0]);
      o.yb[1] = fma(hm[i][1], v[i], o.yb[1]);
      // row i of W h and of LS P
      double a0 = 0.0, a1 = 0.0, q0 = 0.0, q1 = 0.0;
#pragma unroll
      for (int j = 0; j < 6; ++j) {
        a0 = fma(W[sym(i, j)], hm[j][0], a0);
        a1 = fma(W[sym(i, j)], hm[j][1], a1);
      }
#pragma unroll
      for (int j = 0; j < 5; ++j) {
        q0 = fma(LS[i][j], Cp[sym(j, 0)], q0);
        q1 = fma(LS[i][j], Cp[sym(j, 1)], q1);
        o.Z[j][0] = fma(LS[i][j], hm[i][0], o.Z[j][0]);
        o.Z[j][1] = fma(LS[i][j], hm[i][1], o.Z[j][1]);
      }
      const double b0 = a0 + q0, b1 = a1 + q1;
      o.G[0] = fma(-hm[i][0], b0, o.G[0]);
      o.G[2] = fma(-hm[i][1], b1, o.G[2]);
      o.G[1] = fma(-0.5, fma(hm[i][0], b1, hm[i][1] * b0), o.G[1]);
      const double c0 = fma(2.0, a0, q0), c1 = fma(2.0, a1, q1);
      // adjoint of h: v y^T - (2 W h + LS P) Si
      double s0, s1;
      innovation_solve(q.f, c0, c1, s0, s1);
      LS[i][0] += fma(v[i], q.y[0], -s0);
      LS[i][1] += fma(v[i], q.y[1], -s1);
    }
  }
  // Sp = S F^T
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 5; ++c) o.lF[r][c] = 0.0;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    double s[5], o5[5];
#pragma unroll
    for (int c = 0; c < 5; ++c) s[c] = t.rec(k - 1, kRS + 5 * i + c);
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < 5; ++c) o.lF[r][c] = fma(LS[i][r], s[c], o.lF[r][c]);
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      double q = c == 4 ? LS[i][4] : 0.0;
#pragma unroll
      for (int r = 0; r < 4; ++r) q = fma(LS[i][r], F[r][c], q);
      o5[c] = q;
    }
#pragma unroll
    for (int c = 0; c < 5; ++c) LS[i][c] = o5[c];
  }
}

// The rest of the reverse of transition k: lf, Lf (adjoints of x_f,k and
// C_f,k) become those of k-1; adj enters with what transition k+1 contributed
// to the adjoint of surface k and leaves with what this one contributes to
// that of k-1; ga receives surface k's alignment derivatives.
template <bool BZ, bool SM>
__device__ __forceinline__ void reverse_part(const TrackB<SM>& t, int k, double w, const StartB& st, const FwdB& f,
                                             const Step* tape, const Innov& q, const SmOut& sm, double lf[6],
                                             double Lf[21], PlaneAdj& adj, double ga[6]) {
  const FitParams& p = t.g->f;
  const Surf sa = t.surf(k - 1), sb = t.surf(k);
  if (!t.hole(k)) update_reverse<SM, 5>(q, f.Cp, w, sm, lf, Lf);
  // reverse of Cp = F C F^T + Q (and Sp = S F^T):
  //   l_F = 2 Lp F C (+ LSp^T S), L_C = F^T Lp F
  double lF[4][5];  // rows loc0, loc1, phi, theta
  double LF[5][5];
#pragma unroll
  for (int a = 0; a < 5; ++a)
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      double q = c == 4 ? Lf[sym(a, 4)] : 0.0;
#pragma unroll
      for (int r = 0; r < 4; ++r) q = fma(Lf[sym(a, r)], f.F[r][c], q);
      LF[a][c] = q;
    }
  {
    double Cq[15];
#pragma unroll
    for (int e = 0; e < 15; ++e) Cq[e] = t.rec(k - 1, kRC + e);
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < 5; ++c) {
        double q = 0.0;
#pragma unroll
        for (int j = 0; j < 5; ++j) q = fma(LF[r][j], Cq[sym(j, c)], q);
        lF[r][c] = SM ? fma(2.0, q, sm.lF[r][c]) : 2.0 * q;
      }
  }
  const double lqp = Lf[sy(2, 2)], lqt = Lf[sy(3, 3)];
#pragma unroll
  for (int a = 0; a < 5; ++a)
#pragma unroll
    for (int b = 0; b < 5; ++b)
      if (b <= a) {
        double q = a == 4 ? LF[4][b] : 0.0;
#pragma unroll
        for (int r = 0; r < 4; ++r) q = fma(f.F[r][a], LF[r][b], q);
        Lf[sy(a, b)] = q;
      }
  double lx[5];
  PlaneAdj na;
  transport_reverse<BZ>(sa, sb, st.x01, st.r0, st.a0, st.lam, t.kB, t.nu2, p.mass, sb.xx0(), f.path, tape, f.o, f.gc,
                        f.inv_nT, lf, [&](int r, int c) { return lF[r][c]; }, lqp, lqt, lx, na, adj);
#pragma unroll
  for (int e = 0; e < 5; ++e) lf[e] = lx[e];
  if (t.g->grad_align) plane_gradient(t.g->dtab + (size_t)p.surface_id[t.o0 + k] * kDTab, adj, ga);
  adj = na;
}

// weights of the smoothed state 0 (zero for a track without status ST_OK);
// the weight of a packed element (i, j), i > j, of the covariance stands for
// both C_ij and C_ji in the full-matrix convention: half each
template <bool SM>
__device__ __forceinline__ void smoother_weights(const GradParams& g, int tg, bool ok, double v[6], double W[21]) {
  const size_t TG = (size_t)g.f.n_tracks_total;
#pragma unroll
  for (int e = 0; e < 6; ++e) v[e] = SM && g.dl_dparams && ok ? g.dl_dparams[e * TG + tg] : 0.0;
#pragma unroll
  for (int i = 0; i < 6; ++i)
#pragma unroll
    for (int j = 0; j < 6; ++j)
      if (j <= i) {
        const double q = SM && g.dl_dcov && ok ? g.dl_dcov[sy(i, j) * TG + tg] : 0.0;
        W[sy(i, j)] = i == j ? q : 0.5 * q;
      }
}

// The reverse's own state, and its end: surface and update of state 0.
struct RevB {
  double lf[6], Lf[21];  // adjoints of x_f, C_f (packed, full-matrix convention)
  PlaneAdj adj;
  double w;
};
__device__ __forceinline__ void reverse_begin(const GradParams& g, int tg, bool in_range, RevB& b) {
#pragma unroll
  for (int e = 0; e < 6; ++e) b.lf[e] = 0.0;
#pragma unroll
  for (int e = 0; e < 21; ++e) b.Lf[e] = 0.0;
#pragma unroll
  for (int i = 0; i < 3; ++i) b.adj.c[i] = b.adj.u[i] = b.adj.v[i] = b.adj.n[i] = 0.0;
  b.w = (g.dl_dchi2 && in_range) ? g.dl_dchi2[tg] : 1.0;
}
template <bool SM>
__device__ __forceinline__ void reverse_end(const TrackB<SM>& t, bool in_range, int status, RevB& b,
                                            const double LS[6][5]) {
  const GradParams& g = *t.g;
  const FitParams& p = g.f;
  const size_t TG = (size_t)p.n_tracks_total;
  if (g.grad_align) {
    const bool act = status == ST_OK;
    const int sid = act ? p.surface_id[t.o0] : 0;
    double ga[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    if (act) plane_gradient(g.dtab + (size_t)sid * kDTab, b.adj, ga);
    add_align_grad(g.grad_align, p.n_surfaces, sid, ga, act);
  }
  // state 0: x_s0, P_0 and S start as the filtered state 0 (S = P_0 = C_f,0);
  // reverse through its update; x_p,0 is the seed, which also enters x_s0
  // directly
  if (in_range && g.grad_seed) {
    if (status == ST_OK) {
      double v[6], W[21];
      smoother_weights<SM>(g, t.tg, true, v, W);
#pragma unroll
      for (int e = 0; e < 6; ++e) b.lf[e] += v[e];
      if (!t.hole(0)) {
        if (SM)
#pragma unroll
          for (int i = 0; i < 6; ++i)
#pragma unroll
            for (int j = 0; j <= i; ++j) {
              double q = j < 5 ? LS[i][j] : 0.0;
              if (i < 5) q += LS[j][i];
              b.Lf[sy(i, j)] += fma(0.5, q, W[sy(i, j)]);
            }
        double m[2], V[3], xp0[2], Cp0[21];
        hit_of(p, t.o0, m, V);
        xp0[0] = p.seed_params[t.tg];
        xp0[1] = p.seed_params[TG + t.tg];
#pragma unroll
        for (int e = 0; e < 21; ++e) Cp0[e] = p.seed_cov[e * TG + t.tg];
        SmOut none;
        update_reverse<false, 6>(innovation(xp0, Cp0, m, V), Cp0, b.w, none, b.lf, b.Lf);
      }
    }
#pragma unroll
    for (int e = 0; e < 6; ++e) g.grad_seed[e * TG + t.tg] = status == ST_OK ? b.lf[e] : qnan();
  }
}

// states of a track that pass B reverses, and the most of a warp's tracks: the
// warps step through them together, so that the reduction of the alignment
// gradient sees whole warps
__device__ __forceinline__ int states_of(const FitParams& p, int tg, int status, int& nmax) {
  const int n = status == ST_OK ? (int)(p.offsets[tg + 1] - p.offsets[tg]) : 0;
  nmax = n;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) nmax = max(nmax, __shfl_xor_sync(0xffffffffu, nmax, o));
  return n;
}

// Pass B of track slot tl (in_range: a track of the launch; status: of its
// forward pass).  All 32 lanes of a warp call it together.
template <bool BZ, bool SM>
__device__ __forceinline__ void grad_reverse(const GradParams& g, const double* s_surf, int tl, bool in_range,
                                             int status) {
  const TrackB<SM> t(g, s_surf, tl, BZ);
  RevB b;
  reverse_begin(g, t.tg, in_range, b);
  double LS[6][5], v[6], W[21];  // LS: adjoint of S of state k
  smoother_weights<SM>(g, t.tg, status == ST_OK, v, W);
#pragma unroll
  for (int i = 0; i < 6; ++i)
#pragma unroll
    for (int j = 0; j < 5; ++j) LS[i][j] = 0.0;
  int nmax;
  const int n = states_of(g.f, t.tg, status, nmax);
#pragma unroll 1
  for (int k = nmax - 1; k >= 1; --k) {
    const bool act = k < n;
    double ga[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    if (act) {
      const StartB st = start_of(t, k);
      Step tape[kMaxSteps];
      FwdB f;
      SmOut sm;
      forward_part<BZ, SM>(t, k, st, f, tape);
      const Innov q = innovation_at(t, k, f);
      if constexpr (SM) smoother_part(t, k, f.F, f.Cp, q, f.hm, v, W, LS, sm);
      reverse_part<BZ, SM>(t, k, b.w, st, f, tape, q, sm, b.lf, b.Lf, b.adj, ga);
    }
    if (g.grad_align) add_align_grad(g.grad_align, g.f.n_surfaces, act ? g.f.surface_id[t.o0 + k] : 0, ga, act);
  }
  reverse_end<SM>(t, in_range, status, b, LS);
}

// Pass B of 32 tracks by three warps in a pipeline (two without the
// smoother's adjoint, which has no part in it then): at stage j warp 1 runs
// transition j of the sweep again, warp 2 the smoother's part of transition
// j - 1, and warp 0 the rest of the reverse of j - 2, each from what the
// others left in shared memory; one barrier per stage.  Every value is
// computed as in grad_reverse.
constexpr int kPipeFwd = 92, kPipeHm = 12, kPipeTape = 13, kPipeSm = 35;
constexpr int kPipeFields = 3 * (kPipeFwd + kPipeHm + kPipeTape) + 2 * kPipeSm + 30;
template <bool BZ, bool SM, int w>
__device__ __forceinline__ void grad_reverse_pipe(const GradParams& g, const double* s_surf, double* sh, int tl,
                                                  bool in_range, int status) {
  constexpr int kLag = SM ? 2 : 1, kThreads = SM ? 96 : 64;
  constexpr int kSlot = kPipeFwd + kPipeHm + kPipeTape;
  const int lane = threadIdx.x & 31;
  auto sync = [] {
    __syncwarp();
    asm volatile("barrier.cta.sync 2, %0;" ::"n"(kThreads) : "memory");
  };
  const TrackB<SM> t(g, s_surf, tl, BZ);
  double* slot[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) slot[i] = sh + (size_t)i * kSlot * 32 + lane;
  double* sm_slot = sh + (size_t)3 * kSlot * 32 + lane;
  double* s_LS = sm_slot + (size_t)2 * kPipeSm * 32;
  RevB b;
  double LS[6][5], v[6], W[21];
  if (w == 0) reverse_begin(g, t.tg, in_range, b);
  if (w == 2) {
    smoother_weights<SM>(g, t.tg, status == ST_OK, v, W);
#pragma unroll
    for (int i = 0; i < 6; ++i)
#pragma unroll
      for (int j = 0; j < 5; ++j) LS[i][j] = 0.0;
  }
  int nmax;
  const int n = states_of(g.f, t.tg, status, nmax);
  const int steps = nmax - 1;
#pragma unroll 1
  for (int j = 0; j < steps + kLag; ++j) {
    const int mine = w == 1 ? j : w == 2 ? j - 1 : j - kLag;  // transition of the sweep
    const int k = nmax - 1 - mine;
    const bool go = mine >= 0 && mine < steps, act = go && k < n;
    double* q = slot[0] + (size_t)(mine >= 0 ? mine % 3 : 0) * kSlot * 32;
    double* qs = sm_slot + (size_t)(mine >= 0 ? mine & 1 : 0) * kPipeSm * 32;
    if (w == 1 && act) {
      const StartB st = start_of(t, k);
      Step tape[kMaxSteps];
      FwdB f;
      forward_part<BZ, SM>(t, k, st, f, tape);
      int e = 0;
      visit<SM>(f, [&](double x) { q[(e++) * 32] = x; });
      double* z = q + (size_t)(kPipeFwd + kPipeHm) * 32;
      z[0] = (double)f.path.nsub;
      z[32] = (double)f.path.n_steps;
      if (f.path.n_steps == 2) {
        const Step& s = tape[1];
        z[2 * 32] = s.w.eb; z[3 * 32] = s.w.eg; z[4 * 32] = s.w.rb; z[5 * 32] = s.w.rg;
        z[6 * 32] = s.w.deb; z[7 * 32] = s.w.deg; z[8 * 32] = s.w.drb; z[9 * 32] = s.w.drg;
        z[10 * 32] = s.w.len; z[11 * 32] = s.s; z[12 * 32] = (double)s.m;
      }
    }
    if constexpr (SM && w == 2) {
      if (act) {
        FwdB f;
        SmOut o;
        int e = 0;
        visit<SM>(f, [&](double& x) { x = q[(e++) * 32]; });  // (what is not used is not loaded)
        smoother_part(t, k, f.F, f.Cp, innovation_at(t, k, f), f.hm, v, W, LS, o);
#pragma unroll
        for (int i = 0; i < 2; ++i) qs[i * 32] = o.yb[i];
#pragma unroll
        for (int i = 0; i < 3; ++i) qs[(2 + i) * 32] = o.G[i];
#pragma unroll
        for (int i = 0; i < 10; ++i) qs[(5 + i) * 32] = o.Z[i / 2][i % 2];
#pragma unroll
        for (int i = 0; i < 20; ++i) qs[(15 + i) * 32] = o.lF[i / 5][i % 5];
      }
    }
    if (w == 0) {
      double ga[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
      if (act) {
        const StartB st = start_of(t, k);
        Step tape[kMaxSteps];
        FwdB f;
        SmOut sm;
        int e = 0;
        visit<SM>(f, [&](double& x) { x = q[(e++) * 32]; });
        const double* z = q + (size_t)(kPipeFwd + kPipeHm) * 32;
        f.path.nsub = (int)z[0];
        f.path.n_steps = (int)z[32];
        if (f.path.n_steps <= 2) {
          tape[0].s = f.path.nsub == 1 ? f.path.s0 : f.path.s0 / f.path.nsub;
          tape[0].m = 0;
          Step& s = tape[1];
          s.w.eb = z[2 * 32]; s.w.eg = z[3 * 32]; s.w.rb = z[4 * 32]; s.w.rg = z[5 * 32];
          s.w.deb = z[6 * 32]; s.w.deg = z[7 * 32]; s.w.drb = z[8 * 32]; s.w.drg = z[9 * 32];
          s.w.len = z[10 * 32]; s.s = z[11 * 32]; s.m = f.path.n_steps == 2 ? (int)z[12 * 32] : 0;
        } else {
          Path again;  // more steps: their records are not passed on
          path_forward<BZ>(t.surf(k), st.r0, st.a0, st.lam, t.kB, t.nu2, g.f.h_max, g.f.n_iter, again, tape);
        }
        if (SM) {
#pragma unroll
          for (int i = 0; i < 2; ++i) sm.yb[i] = qs[i * 32];
#pragma unroll
          for (int i = 0; i < 3; ++i) sm.G[i] = qs[(2 + i) * 32];
#pragma unroll
          for (int i = 0; i < 10; ++i) sm.Z[i / 2][i % 2] = qs[(5 + i) * 32];
#pragma unroll
          for (int i = 0; i < 20; ++i) sm.lF[i / 5][i % 5] = qs[(15 + i) * 32];
        }
        reverse_part<BZ, SM>(t, k, b.w, st, f, tape, innovation_at(t, k, f), sm, b.lf, b.Lf, b.adj, ga);
      }
      if (g.grad_align && go)
        add_align_grad(g.grad_align, g.f.n_surfaces, act ? g.f.surface_id[t.o0 + k] : 0, ga, act);
    }
    sync();
  }
  if (SM) {
    if (w == 2)
#pragma unroll
      for (int i = 0; i < 30; ++i) s_LS[i * 32] = LS[i / 5][i % 5];
    sync();
    if (w == 0)
#pragma unroll
      for (int i = 0; i < 30; ++i) LS[i / 5][i % 5] = s_LS[i * 32];
  }
  if (w == 0) reverse_end<SM>(t, in_range, status, b, LS);
}

// outputs of a track whose CTA's staging wait gave up: NaN, and nothing is
// added to the alignment gradient
__device__ __forceinline__ void write_failed_grad(const GradParams& g, int tg) {
  const size_t TG = (size_t)g.f.n_tracks_total;
  if (g.chi2) g.chi2[tg] = qnan();
  if (g.grad_seed)
    for (int e = 0; e < 6; ++e) g.grad_seed[(size_t)e * TG + tg] = qnan();
  if (g.out_params)
    for (int e = 0; e < 6; ++e) g.out_params[(size_t)e * TG + tg] = qnan();
  if (g.out_cov)
    for (int e = 0; e < 21; ++e) g.out_cov[(size_t)e * TG + tg] = qnan();
}

// Register-cap variants as for the fit kernels: MINB 1 may use 255
// registers (up to 8 warps per SM), 3 caps at 168 (12 warps) and 4 at 128
// (16 warps).  SM: with the smoother's adjoint (v or W given).
template <int MINB, bool BZ, bool SM>
__global__ void __launch_bounds__(max_threads_of(MINB), 1) kf_grad_kernel(const GradParams g) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  double* s_surf = reinterpret_cast<double*>(smem_raw);
  __shared__ __align__(8) uint64_t s_mbar;
  const FitParams& p = g.f;
  const bool staged = stage_surfaces(s_surf, p.surf, (uint32_t)(p.n_surfaces * kSurfStride * 8), &s_mbar,
                                     p.error_flag, p.wait_limit, p.skip_stage_copy != 0);
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const bool in_range = t < p.n_tracks;
  const int tl = in_range ? t : 0;
  const int tg = p.track0 + tl;
  const size_t TG = (size_t)p.n_tracks_total, TL = (size_t)p.n_tracks;
  if (!staged) {
    // a bounded wait of this call gave up (the whole CTA returns here, so no
    // warp-wide reduction below is entered)
    if (in_range) write_failed_grad(g, tg);
    return;
  }
  const bool want = g.grad_seed || g.grad_align;
  const bool smooth = SM || g.out_params || g.out_cov;
  int64_t o0, o1;
  int n;
  int status = in_range ? track_input(p, tg, o0, o1, n) : ST_BAD_INPUT;

  // ---------------------------------------------------------- F: forward
  Filter f;
  if (status == ST_OK) status = filter_first(p, tg, o0, f);
  if (status == ST_OK) {
    constexpr int REC = SM ? 2 : 1;
    const WS ws{nullptr, nullptr, TL, 0, 0, tl};
    if (!smooth || time_is_settled(f.C)) {
      status = filter_states<BZ, 5, false, REC>(p, s_surf, ws, o0, n, smooth, g.rec, f);
    } else {
      Filter q = f;
      status = filter_states_with_time<BZ, REC>(p, s_surf, ws, o0, n, smooth, g.rec, &q);
      f = q;
    }
    if (status == ST_OK && !f.spd) status = ST_NON_SPD;
  }
  if (in_range) {
    if (g.chi2) g.chi2[tg] = status == ST_OK ? f.chi2 : qnan();
    if (g.out_params)
#pragma unroll
      for (int e = 0; e < 6; ++e)
        g.out_params[e * TG + tg] = status == ST_OK ? f.xs[e] + p.seed_params[e * TG + tg] : qnan();
    if (g.out_cov)
#pragma unroll
      for (int e = 0; e < 21; ++e) g.out_cov[e * TG + tg] = status == ST_OK ? f.P0[e] : qnan();
  }
  if (!want) return;

  grad_reverse<BZ, SM>(g, s_surf, tl, in_range, status);
}

// The same for batches that leave most sub-partitions idle: a CTA of 4 warps
// per 32 tracks whose forward pass is the team fit's (kf_team.cuh: 0.6 of one
// warp's time) and whose pass B is a pipeline over its warps.  Up to one team
// per SM.  2000 tracks x 21 states, forward and backward of the
// differentiable fit: 3.57 -> 2.98 ms with the team's forward pass (2.66
// without the time row), 1.86 ms with the pipeline.
template <bool BZ, bool SM>
__global__ void __launch_bounds__(128, 1) kf_grad_team_kernel(const GradParams g) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  double* s_surf = reinterpret_cast<double*>(smem_raw);
  __shared__ __align__(8) uint64_t s_mbar;
  const FitParams& p = g.f;
  double* sh = s_surf + (size_t)p.n_surfaces * kSurfStride;
  const bool staged = stage_surfaces(s_surf, p.surf, (uint32_t)(p.n_surfaces * kSurfStride * 8), &s_mbar,
                                     p.error_flag, p.wait_limit, p.skip_stage_copy != 0);
  const int base = blockIdx.x * kTeamTracks, i = base + (int)(threadIdx.x & 31);
  const bool in_range = i < p.n_tracks;
  if (!staged) {
    if (in_range && threadIdx.x < 32) write_failed_grad(g, p.track0 + i);
    return;
  }
  constexpr int REC = SM ? 2 : 1;
  __shared__ int s_status[32];
  const int wid = threadIdx.x >> 5;
  switch (wid) {
    case 0: s_status[threadIdx.x] = fit_team<BZ, 4, 0, REC>(p, s_surf, sh, base, g.rec); break;
    case 1: fit_team<BZ, 4, 1, REC>(p, s_surf, sh, base, g.rec); break;
    case 2: fit_team<BZ, 4, 2, REC>(p, s_surf, sh, base, g.rec); break;
    default: fit_team<BZ, 4, 3, REC>(p, s_surf, sh, base, g.rec); break;
  }
  if (!g.grad_seed && !g.grad_align) return;
  __threadfence_block();
  __syncthreads();  // the records and the verdicts; the exchange buffers are free
  const int status = s_status[threadIdx.x & 31], tl = in_range ? i : 0;
  if (wid == 0) grad_reverse_pipe<BZ, SM, 0>(g, s_surf, sh, tl, in_range, status);
  if (wid == 1) grad_reverse_pipe<BZ, SM, 1>(g, s_surf, sh, tl, in_range, status);
  if constexpr (SM)
    if (wid == 2) grad_reverse_pipe<BZ, SM, 2>(g, s_surf, sh, tl, in_range, status);
}

// dynamic shared memory of one of its CTAs
size_t grad_team_smem_bytes(int n_surfaces) {
  static_assert(kPipeFields >= kShFields, "the exchange buffers are reused");
  static_assert((kMaxSurfaces * kSurfStride + kPipeFields * 32) * 8 + 1024 <= 227 * 1024,
                "fits beside the largest surface table");
  return ((size_t)n_surfaces * kSurfStride + (size_t)kPipeFields * 32) * sizeof(double);
}

template <int MINB, bool BZ, bool SM>
cudaError_t launch_grad_v(const GradParams& g, int block, cudaStream_t stream) {
  const FitParams& f = g.f;
  const size_t smem = (size_t)f.n_surfaces * kSurfStride * sizeof(double);
  auto kern = kf_grad_kernel<MINB, BZ, SM>;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  if (block <= 0) {
    // CTAs of w warps, one per SM per wave, w the smallest count (within the
    // warps this variant's registers allow per SM) that covers the batch's
    // 32-track warp units in r full waves: the last wave is nearly full
    int dev = 0, nsm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const long long wmax = max_threads_of(MINB) / 32;
    const long long units = ((long long)f.n_tracks + 31) / 32;
    long long w = wmax;
    for (long long r = 1; r <= 1024; ++r) {
      w = (units + r * nsm - 1) / (r * nsm);
      if (w <= wmax) break;
    }
    block = 32 * (int)(w < 1 ? 1 : (w > wmax ? wmax : w));
  }
  const int grid = (f.n_tracks + block - 1) / block;
  kern<<<grid, block, smem, stream>>>(g);
  return cudaGetLastError();
}

template <bool BZ, bool SM>
cudaError_t launch_grad_team(const GradParams& g, cudaStream_t stream) {
  const size_t smem = grad_team_smem_bytes(g.f.n_surfaces);
  auto kern = kf_grad_team_kernel<BZ, SM>;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  kern<<<(g.f.n_tracks + kTeamTracks - 1) / kTeamTracks, 128, smem, stream>>>(g);
  return cudaGetLastError();
}

template <int MINB>
cudaError_t launch_grad_m(const GradParams& g, bool sm, int block, cudaStream_t stream) {
  const bool bz = g.f.bfield[0] == 0.0 && g.f.bfield[1] == 0.0;
  if (sm) return bz ? launch_grad_v<MINB, true, true>(g, block, stream) : launch_grad_v<MINB, false, true>(g, block, stream);
  return bz ? launch_grad_v<MINB, true, false>(g, block, stream) : launch_grad_v<MINB, false, false>(g, block, stream);
}

}  // namespace

size_t grad_table_doubles(int n_surfaces) { return (size_t)n_surfaces * (kSurfStride + kDTab); }

cudaError_t launch_align_tables(int n_surfaces, const double* packed, const double* align, double* tables,
                                cudaStream_t stream) {
  align_kernel<<<(n_surfaces + 63) / 64, 64, 0, stream>>>(n_surfaces, packed, align, tables,
                                                          tables + (size_t)n_surfaces * kSurfStride);
  return cudaGetLastError();
}

size_t grad_scratch_doubles(int max_states, bool smoother_adjoint) {
  return (size_t)(smoother_adjoint ? kRecWhole : kRecFilter) * (size_t)max_states;
}

cudaError_t launch_grad(const FitParams& f, const GradArgs& a, const double* tables, double* scratch, int block,
                        int min_blocks, int team_warps, cudaStream_t stream) {
  GradParams g;
  g.f = f;
  g.f.surf = tables;
  g.dtab = tables + (size_t)f.n_surfaces * kSurfStride;
  g.dl_dchi2 = a.dl_dchi2;
  g.dl_dparams = a.dl_dparams;
  g.dl_dcov = a.dl_dcov;
  g.chi2 = a.chi2;
  g.out_params = a.params;
  g.out_cov = a.cov;
  g.grad_seed = a.grad_seed;
  g.grad_align = a.grad_align;
  g.rec = scratch;
  const bool sm = (a.grad_seed || a.grad_align) && (a.dl_dparams || a.dl_dcov);
  // teams where the caller asks for them, and for a batch of at most one team
  // per SM with the launch shape left to the library (above that two teams
  // would share an SM's pipes)
  int dev = 0, nsm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const bool team =
      team_warps == 2 || (team_warps == 0 && block <= 0 && min_blocks <= 1 && f.n_tracks <= 32 * nsm);
  if (team) {
    g.f.out_params = a.params;
    g.f.out_cov = a.cov;
    g.f.out_chi2 = a.chi2;
    const bool bz = f.bfield[0] == 0.0 && f.bfield[1] == 0.0;
    if (sm) return bz ? launch_grad_team<true, true>(g, stream) : launch_grad_team<false, true>(g, stream);
    return bz ? launch_grad_team<true, false>(g, stream) : launch_grad_team<false, false>(g, stream);
  }
  switch (min_blocks) {
    case 4: return launch_grad_m<4>(g, sm, block, stream);
    case 3: return launch_grad_m<3>(g, sm, block, stream);
    default: return launch_grad_m<1>(g, sm, block, stream);
  }
}

}  // namespace kfgb
