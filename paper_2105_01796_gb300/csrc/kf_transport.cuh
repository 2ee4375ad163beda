// kf_transport.cuh -- the FP64 path's RKN propagation to a plane with its
// transport Jacobian (paper Sect. 4.1), shared by the one-thread-per-track
// kernel (kf_kernels.cu) and the track-team kernel (kf_team.cu).
//
// With N v = kappa (v x B) and lam = q/p, dT/ds = lam N T in a constant
// field, and one 4-stage Nystrom step of length h is the polynomial
//   T' = E T, r' = r + R T,  x = h lam,
//   E = 1 + xN + (xN)^2/2 + (xN)^3/6 + (xN)^4/24,
//   R = h (1 + xN/2 + (xN)^2/6 + (xN)^3/24)
// (the classic RKN4 combinations of the stage accelerations).  The same E and
// R carry every Jacobian column, and dE/dlam, dR/dlam acting on T are the q/p
// column.  Since N^3 = -nu^2 N (nu = kappa |B|), each operator is
// a + b N + c N^2: its coefficients are formed once per step and
// applied to the columns, instead of taking every column through the four
// stages.  With the field along z, N turns the (x, y) components by a right
// angle, and E and R become 2x2 rotation-like matrices of the bend plane.
//
// The plane corrections are scalar: along the path n.T and n.r are
// polynomials in the correction length s, so the Newton iterations cost a
// few operations each and one step of their summed length moves the state.
// A sum of steps differs from the steps in turn by the truncation of the
// exponential, (s lam nu)^5 / 120; it is used while |s lam nu| <= 1e-3
// (below 1e-17 of the direction), and longer corrections step in turn.
//
// FP64 instructions per transition (the FP64 pipe is the bound: a warp DFMA
// holds a sub-partition's pipe for 64 cycles): about 320 with the field along
// z against 1170 for the stage-by-stage form (4 RKN steps x 3 columns).
#pragma once
#include <cuda_runtime.h>
#include <math.h>

#include "kf_device.cuh"
#include "kf_df.cuh"
#include "kf_fp64.cuh"

namespace kfgb {
namespace dev {

// sine and cosine of any angle, out of line (seed angles; large turns)
static __device__ __noinline__ double2 sincos_call(double a) {
  double2 r;
  sincos(a, &r.x, &r.y);
  return r;
}
static __device__ __noinline__ double atan2_call(double y, double x) { return atan2(y, x); }

// cosines and sines of the direction's angles
struct Angles {
  double cp, sp, ct, st;
};

__device__ __forceinline__ Angles angles_of(double phi, double theta) {
  const double2 p = sincos_call(phi), t = sincos_call(theta);
  return {p.y, p.x, t.y, t.x};
}

// (c, s) of an angle turned by d: Taylor series of sin d and cos d - 1 up to
// |d| = 1/16 (first omitted terms below 3e-20), else the library's functions.
// A filter increment is almost always in the series' range: about 15 FP64
// instructions against 40 for a fresh sincos.
__device__ __forceinline__ void turn(double& c, double& s, double d) {
  double sd, cm;
  if (fabs(d) <= 0.0625) {
    const double d2 = d * d;
    double v = fma(d2, 1.0 / 362880.0, -1.0 / 5040.0);
    v = fma(d2, v, 1.0 / 120.0);
    v = fma(d2, v, -1.0 / 6.0);
    sd = fma(d * d2, v, d);
    double u = fma(d2, 1.0 / 40320.0, -1.0 / 720.0);
    u = fma(d2, u, 1.0 / 24.0);
    u = fma(d2, u, -0.5);
    cm = d2 * u;
  } else {
    const double2 r = sincos_call(d);
    sd = r.x;
    cm = r.y - 1.0;
  }
  const double c0 = c;
  c = fma(c0, cm, fma(-s, sd, c0));
  s = fma(s, cm, fma(c0, sd, s));
}

// a + atan(num / den) for a quotient up to 1/8 (series: first omitted term
// below 3e-18); false (nothing written) outside that range or when the result
// leaves [lo, hi]: the caller takes atan2.
__device__ __forceinline__ bool add_small_atan(double a, double num, double den, double lo, double hi, double& out) {
  if (!(den > 0.0) || !(fabs(num) <= 0.125 * den)) return false;
  const double q = num * rcp_any(den), z = q * q;
  double v = fma(z, 1.0 / 17.0, -1.0 / 15.0);
  v = fma(z, v, 1.0 / 13.0);
  v = fma(z, v, -1.0 / 11.0);
  v = fma(z, v, 1.0 / 9.0);
  v = fma(z, v, -1.0 / 7.0);
  v = fma(z, v, 1.0 / 5.0);
  v = fma(z, v, -1.0 / 3.0);
  const double r = a + fma(q * z, v, q);
  if (!(r >= lo && r <= hi)) return false;
  out = r;
  return true;
}

// ---------------------------------------------------------------------------
// the path operators, accumulated over steps
// ---------------------------------------------------------------------------

// Field along z: the bend-plane unit vector e, its path integral q, and with
// QP their derivatives with respect to q/p.  J v = (v1, -v0), N = kBz J.
template <bool QP>
struct PathZ {
  double e[2], q[2], de[2], dq[2], len;
  // first: q, de and dq are zero (not set yet)
  __device__ __forceinline__ void step(double h, double lam, double kB, bool first) {
    const double x = h * lam * kB, x2 = x * x;
    const double t6 = fma(x2, -1.0 / 6.0, 1.0);
    const double ec = fma(x2, fma(x2, 1.0 / 24.0, -0.5), 1.0), es = x * t6;
    const double hx = h * x;
    const double rc = h * t6, rs = hx * fma(x2, -1.0 / 24.0, 0.5);
    const double e0 = e[0], e1 = e[1];
    if (QP) {
      const double hk = h * kB, hhk = h * hk;
      const double dec = -hk * es, des = hk * fma(x2, -0.5, 1.0);
      const double drc = hhk * x * (-1.0 / 3.0), drs = hhk * fma(x2, -0.125, 0.5);
      if (first) {
        dq[0] = fma(drc, e0, drs * e1);
        dq[1] = fma(drc, e1, -drs * e0);
        de[0] = fma(dec, e0, des * e1);
        de[1] = fma(dec, e1, -des * e0);
      } else {
        const double g0 = de[0], g1 = de[1];
        dq[0] = fma(drc, e0, fma(drs, e1, fma(rc, g0, fma(rs, g1, dq[0]))));
        dq[1] = fma(drc, e1, fma(-drs, e0, fma(rc, g1, fma(-rs, g0, dq[1]))));
        de[0] = fma(dec, e0, fma(des, e1, fma(ec, g0, es * g1)));
        de[1] = fma(dec, e1, fma(-des, e0, fma(ec, g1, -es * g0)));
      }
    }
    if (first) {
      q[0] = fma(rc, e0, rs * e1);
      q[1] = fma(rc, e1, -rs * e0);
      len = h;
    } else {
      q[0] = fma(rc, e0, fma(rs, e1, q[0]));
      q[1] = fma(rc, e1, fma(-rs, e0, q[1]));
      len += h;
    }
    e[0] = fma(ec, e0, es * e1);
    e[1] = fma(ec, e1, -es * e0);
  }
};

// Any constant field: E = 1 + eb N + eg N^2, R = len + rb N + rg N^2 and with
// QP their derivatives (no constant term); nu2 = nu^2.
template <bool QP>
struct PathG {
  double eb, eg, rb, rg, deb, deg, drb, drg, len;
  __device__ __forceinline__ void step(double h, double lam, double nu2, bool first) {
    const double x = h * lam, x2 = x * x, y = x2 * nu2, hx = h * x;
    const double b2 = x * fma(y, -1.0 / 6.0, 1.0), g2 = x2 * fma(y, -1.0 / 24.0, 0.5);
    const double rb2 = hx * fma(y, -1.0 / 24.0, 0.5), rg2 = hx * x * (1.0 / 6.0);
    const double hh = h * h;
    const double db2 = h * fma(y, -0.5, 1.0), dg2 = h * x * fma(y, -1.0 / 6.0, 1.0);
    const double drb2 = hh * fma(y, -0.125, 0.5), drg2 = hh * x * (1.0 / 3.0);
    if (first) {
      eb = b2; eg = g2; rb = rb2; rg = rg2; len = h;
      if (QP) { deb = db2; deg = dg2; drb = drb2; drg = drg2; }
      return;
    }
    // products mod N^3 = -nu2 N:  (b N + c N^2)(1 + eb N + eg N^2)
    //   = b N + (c + b eb) N^2 - nu2 [(b eg + c eb) N + c eg N^2]
    if (QP) {
      const double d1 = deb, d2 = deg;
      drb = drb + fma(-nu2, fma(drb2, eg, drg2 * eb), drb2) + fma(-nu2, fma(rb2, d2, rg2 * d1), h * d1);
      drg = drg + fma(drb2, eb, fma(-nu2 * drg2, eg, drg2)) + fma(rb2, d1, fma(-nu2 * rg2, d2, h * d2));
      deb = fma(-nu2, fma(db2, eg, dg2 * eb), db2) + fma(-nu2, fma(b2, d2, g2 * d1), d1);
      deg = fma(db2, eb, fma(-nu2 * dg2, eg, dg2)) + fma(b2, d1, fma(-nu2 * g2, d2, d2));
    }
    rb = rb + fma(-nu2, fma(rb2, eg, rg2 * eb), fma(h, eb, rb2));
    rg = rg + fma(rb2, eb, fma(-nu2 * rg2, eg, fma(h, eg, rg2)));
    const double o1 = eb, o2 = eg;
    eb = fma(-nu2, fma(b2, o2, g2 * o1), o1 + b2);
    eg = fma(b2, o1, fma(-nu2 * g2, o2, o2 + g2));
    len += h;
  }
};

// Where a transport ends: the point and direction, the unit direction's
// angles, and what the noise needs.
struct End {
  double r[3], T[3];   // free end point and direction (|T| = 1 up to the steps' truncation)
  Angles a;            // of the unit direction
  double inv_st;       // 1 / sin(theta)
  double inv_cos;      // 1 / cosine of incidence at b (signed)
  double g2, dtds, dt; // 1 + m^2 lam^2; dt/ds; flight time
};

// Columns of D J_bf that vary along the path, at the end point: position and
// direction rows of the phi, theta and q/p columns; CMASK bit c: column c is
// formed.
struct Cols64 {
  double gr[3][3], gT[3][3], gtl;
};

// Propagate the free state r0, direction angles a0, lam = q/p to plane b.
template <bool BZ, int CMASK>
__device__ __forceinline__ int propagate_to_plane(const Surf& sb, const double r0[3], const Angles& a0, double lam,
                                                  const double B[3], double mass, double h_max, int n_iter, End& o,
                                                  Cols64& g) {
  constexpr bool QP = (CMASK & 4) != 0;
  const double T0[3] = {a0.cp * a0.st, a0.sp * a0.st, a0.ct};
  const double n0 = sb.n(0), n1 = sb.n(1), n2 = sb.n(2);
  const double kB[3] = {kKappa * B[0], kKappa * B[1], kKappa * B[2]};
  const double nu2 = BZ ? kB[2] * kB[2] : fma(kB[0], kB[0], fma(kB[1], kB[1], kB[2] * kB[2]));
  // N T0, N^2 T0 (general field) and their components along n
  double NT[3], NNT[3], pN = 0.0, pNN = 0.0;
  const double p00 = fma(n0, T0[0], fma(n1, T0[1], n2 * T0[2]));
  if (!BZ) {
    applyA<double, false>(kB, T0, NT);
    applyA<double, false>(kB, NT, NNT);
    pN = fma(n0, NT[0], fma(n1, NT[1], n2 * NT[2]));
    pNN = fma(n0, NNT[0], fma(n1, NNT[1], n2 * NNT[2]));
  }
  // main steps over the straight-line distance
  const double d0 = fma(n0, sb.c(0) - r0[0], fma(n1, sb.c(1) - r0[1], n2 * (sb.c(2) - r0[2])));
  if (!(fabs(p00) > 1e-9)) return ST_NO_INTERSECTION;
  const double s0 = d0 * rcp_any(p00);
  int nsub = 1;
  double h = s0;
  if (!(fabs(s0) <= h_max)) {
    const double nsub_d = ceil(fabs(s0) / h_max);
    if (!(nsub_d <= 64.0)) return ST_NO_INTERSECTION;
    nsub = nsub_d < 1.0 ? 1 : (int)nsub_d;
    h = s0 / nsub;
  }
  PathZ<QP> z;
  PathG<QP> w;
  if (BZ) {
    z.e[0] = a0.cp;
    z.e[1] = a0.sp;
    z.step(h, lam, kB[2], true);
    for (int k = 1; k < nsub; ++k) z.step(h, lam, kB[2], false);
  } else {
    w.step(h, lam, nu2, true);
    for (int k = 1; k < nsub; ++k) w.step(h, lam, nu2, false);
  }
  // Newton corrections onto the plane: along a correction of length s,
  // x = s lam, y = x^2 nu^2,
  //   n.T = p0 + (x - x y/6) p1 + (x^2/2 - x^2 y/24) p2,
  //   n.(c - r) = dist - s [p0 + (x/2 - x y/24) p1 + x^2/6 p2]
  // with p_j = n . N^j T at the point where the correction starts
  for (int it = 0; it < n_iter;) {
    double dist, p0, p1, p2;
    if (BZ) {
      const double st = a0.st;
      const double zt = n2 * a0.ct;
      const double c0 = fma(n0, z.e[0], n1 * z.e[1]) * st;
      p0 = c0 + zt;
      p1 = (kB[2] * st) * fma(n0, z.e[1], -n1 * z.e[0]);
      p2 = -nu2 * c0;
      dist = d0 - fma(fma(n0, z.q[0], n1 * z.q[1]), st, zt * z.len);
    } else {
      p0 = p00 + fma(w.eb, pN, w.eg * pNN);
      p1 = fma(w.eb, pNN, fma(-nu2 * w.eg, pN, pN));
      p2 = fma(-nu2 * w.eb, pN, fma(-nu2 * w.eg, pNN, pNN));
      dist = d0 - fma(w.len, p00, fma(w.rb, pN, w.rg * pNN));
    }
    double s;
    {
      if (!(fabs(p0) > 1e-9)) return ST_NO_INTERSECTION;
      s = dist * rcp_any(p0);
      ++it;
    }
    // short corrections are summed (see the file comment); the remaining ones
    // are far below the first, so a 1e-13 reciprocal leaves nothing of note
    while (it < n_iter) {
      const double x = s * lam, y = x * x * nu2;
      if (!(y <= 1e-6)) break;
      const double c24 = fma(y, -1.0 / 24.0, 0.5);
      const double nT = fma(x, fma(x * c24, p2, fma(y, -1.0 / 6.0, 1.0) * p1), p0);
      const double di = fma(-s, fma(x, fma(x * (1.0 / 6.0), p2, c24 * p1), p0), dist);
      if (!(fabs(nT) > 1e-9)) return ST_NO_INTERSECTION;
      s = fma(di, rcp_nr<1>(nT), s);
      ++it;
    }
    if (BZ)
      z.step(s, lam, kB[2], false);
    else
      w.step(s, lam, nu2, false);
  }

  // end point, direction and the columns
  double len;
  if (BZ) {
    const double st = a0.st, ct = a0.ct;
    len = z.len;
    const double dr0 = st * z.q[0], dr1 = st * z.q[1];
    o.T[0] = st * z.e[0];
    o.T[1] = st * z.e[1];
    o.T[2] = ct;
    o.r[0] = fma(st, z.q[0], r0[0]);
    o.r[1] = fma(st, z.q[1], r0[1]);
    o.r[2] = fma(len, ct, r0[2]);
    // the phi column turns with the bend plane, the theta column is
    // (ct e, -st); neither needs a pass of its own
    g.gr[0][0] = -dr1; g.gr[1][0] = dr0; g.gr[2][0] = 0.0;
    g.gT[0][0] = -o.T[1]; g.gT[1][0] = o.T[0]; g.gT[2][0] = 0.0;
    g.gr[0][1] = ct * z.q[0]; g.gr[1][1] = ct * z.q[1]; g.gr[2][1] = -len * st;
    g.gT[0][1] = ct * z.e[0]; g.gT[1][1] = ct * z.e[1]; g.gT[2][1] = -st;
    if (QP) {
      g.gr[0][2] = st * z.dq[0]; g.gr[1][2] = st * z.dq[1]; g.gr[2][2] = 0.0;
      g.gT[0][2] = st * z.de[0]; g.gT[1][2] = st * z.de[1]; g.gT[2][2] = 0.0;
    }
  } else {
    len = w.len;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      o.r[i] = r0[i] + fma(len, T0[i], fma(w.rb, NT[i], w.rg * NNT[i]));
      o.T[i] = T0[i] + fma(w.eb, NT[i], w.eg * NNT[i]);
      if (QP) {
        g.gr[i][2] = fma(w.drb, NT[i], w.drg * NNT[i]);
        g.gT[i][2] = fma(w.deb, NT[i], w.deg * NNT[i]);
      }
    }
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      if (!(CMASK & (1 << c))) continue;
      double v[3], Nv[3], NNv[3];
      v[0] = c == 0 ? -T0[1] : a0.cp * a0.ct;
      v[1] = c == 0 ? T0[0] : a0.sp * a0.ct;
      v[2] = c == 0 ? 0.0 : -a0.st;
      if (c == 0) {  // v[2] = 0
        Nv[0] = v[1] * kB[2];
        Nv[1] = -v[0] * kB[2];
        Nv[2] = fma(v[0], kB[1], -v[1] * kB[0]);
      } else {
        applyA<double, false>(kB, v, Nv);
      }
      applyA<double, false>(kB, Nv, NNv);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        g.gr[i][c] = (c == 0 && i == 2) ? fma(w.rb, Nv[i], w.rg * NNv[i])
                                        : fma(len, v[i], fma(w.rb, Nv[i], w.rg * NNv[i]));
        g.gT[i][c] = (c == 0 && i == 2) ? fma(w.eb, Nv[i], w.eg * NNv[i])
                                        : v[i] + fma(w.eb, Nv[i], w.eg * NNv[i]);
      }
    }
  }
  o.g2 = fma(mass * mass * lam, lam, 1.0);
  const double igam = rsqrt_any(o.g2);
  o.dtds = o.g2 * igam * kInvC;
  o.dt = __dmul_rn(len, o.dtds);
  if (QP) g.gtl = len * (mass * mass * lam * kInvC) * igam;
  return ST_OK;
}

// The end frame: angles of the unit direction and the quotients the
// projections and the noise use.
__device__ __forceinline__ void end_frame(const Surf& sb, End& o, double& inv_nT) {
  const double rho2 = fma(o.T[0], o.T[0], o.T[1] * o.T[1]);
  const double irho = rsqrt_any(rho2);
  const double tn2 = fma(o.T[2], o.T[2], rho2);
  const double itn = rsqrt_any(tn2);
  const double tn = tn2 * itn;
  o.a.cp = o.T[0] * irho;
  o.a.sp = o.T[1] * irho;
  o.a.st = rho2 * irho * itn;
  o.a.ct = o.T[2] * itn;
  o.inv_st = tn * irho;
  inv_nT = rcp_any(fma(sb.n(0), o.T[0], fma(sb.n(1), o.T[1], sb.n(2) * o.T[2])));
  o.inv_cos = tn * inv_nT;
}

// The columns of F in FMASK (bit j: 0 loc0, 1 loc1, 2 phi, 3 theta, 4 q/p):
// path correction dfree += F' w, w = -(n . position rows) / (n . T),
// F' = (T, dt/ds, A T, 0) at the end point, then free -> bound.  The
// projections of F' onto b's axes are formed once, so a column costs its own
// projections plus one FMA per row.  put(r, c, v): row r (0 loc0, 1 loc1,
// 2 phi, 3 theta, 5 time).
template <bool BZ, int FMASK, class Put>
__device__ __forceinline__ void jacobian_columns(const Surf& sa, const Surf& sb, const End& o, const Cols64& g,
                                                 double lam, const double B[3], double inv_nT, Put put) {
  const double lk = lam * kKappa;
  const double bs[3] = {lk * B[0], lk * B[1], lk * B[2]};
  double AT[3];
  applyA<double, BZ>(bs, o.T, AT);
  const double m0 = -sb.n(0) * inv_nT, m1 = -sb.n(1) * inv_nT, m2 = -sb.n(2) * inv_nT;
  const double f0 = -o.a.sp * o.inv_st, f1 = o.a.cp * o.inv_st;                       // dphi/dT
  const double h0 = o.a.cp * o.a.ct, h1 = o.a.sp * o.a.ct, h2 = -o.a.st;              // dtheta/dT
  const double u0 = sb.u(0), u1 = sb.u(1), u2 = sb.u(2), v0 = sb.v(0), v1 = sb.v(1), v2 = sb.v(2);
  const double uT = fma(u0, o.T[0], fma(u1, o.T[1], u2 * o.T[2]));
  const double vT = fma(v0, o.T[0], fma(v1, o.T[1], v2 * o.T[2]));
  const double fA = fma(f0, AT[0], f1 * AT[1]);
  const double hA = BZ ? fma(h0, AT[0], h1 * AT[1]) : fma(h0, AT[0], fma(h1, AT[1], h2 * AT[2]));
  const double dtds = o.dtds;
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    if (!(FMASK & (1 << c))) continue;
    // with the field along z the phi and q/p columns stay in the bend plane
    const bool flat = BZ && (c == 2 || c == 4);
    const double p0 = c == 0 ? sa.u(0) : c == 1 ? sa.v(0) : g.gr[0][c - 2 < 0 ? 0 : c - 2];
    const double p1 = c == 0 ? sa.u(1) : c == 1 ? sa.v(1) : g.gr[1][c - 2 < 0 ? 0 : c - 2];
    const double p2 = c == 0 ? sa.u(2) : c == 1 ? sa.v(2) : g.gr[2][c - 2 < 0 ? 0 : c - 2];
    const double w = flat ? fma(m0, p0, m1 * p1) : fma(m0, p0, fma(m1, p1, m2 * p2));
    put(0, c, fma(uT, w, flat ? fma(u0, p0, u1 * p1) : fma(u0, p0, fma(u1, p1, u2 * p2))));
    put(1, c, fma(vT, w, flat ? fma(v0, p0, v1 * p1) : fma(v0, p0, fma(v1, p1, v2 * p2))));
    if (c < 2) {
      put(2, c, fA * w);
      put(3, c, hA * w);
      put(5, c, dtds * w);
    } else {
      const double t0 = g.gT[0][c - 2], t1 = g.gT[1][c - 2], t2 = g.gT[2][c - 2];
      put(2, c, fma(fA, w, fma(f0, t0, f1 * t1)));
      put(3, c, fma(hA, w, flat ? fma(h0, t0, h1 * t1) : fma(h0, t0, fma(h1, t1, h2 * t2))));
      put(5, c, c == 4 ? fma(dtds, w, g.gtl) : dtds * w);
    }
  }
}

// theta0^2 of the Highland width (see highland()): no square root is needed,
// the width enters squared.
__device__ __forceinline__ double highland_sq(double lam, double g2, double xx0, double inv_cos) {
  const double eps = xx0 * fabs(inv_cos);
  const double a = 0.0136 * lam, l = fma(0.038, log_df(eps * g2), 1.0);
  return a * a * g2 * eps * (l * l);
}

// Angles (phi, theta) of the end direction from those of the start direction
// (a0 their cosines and sines): the turn between the two by a short atan
// series, or atan2 where the turn is large or an angle leaves its range.
__device__ __forceinline__ void end_angles(double phi0, double theta0, const Angles& a0, const End& o, double& phi,
                                           double& theta) {
  constexpr double kPi = 3.141592653589793116;
  const double rho2 = fma(o.T[0], o.T[0], o.T[1] * o.T[1]);
  const double rho = fma(o.a.cp, o.T[0], o.a.sp * o.T[1]);
  if (!add_small_atan(phi0, fma(a0.cp, o.T[1], -a0.sp * o.T[0]), fma(a0.cp, o.T[0], a0.sp * o.T[1]), -kPi, kPi, phi))
    phi = atan2_call(o.T[1], o.T[0]);
  if (!add_small_atan(theta0, fma(a0.ct, rho, -a0.st * o.T[2]), fma(a0.st, rho, a0.ct * o.T[2]), 0.0, kPi, theta))
    theta = atan2_call(rho2 > 0.0 ? rho : rho2, o.T[2]);
}

}  // namespace dev
}  // namespace kfgb
