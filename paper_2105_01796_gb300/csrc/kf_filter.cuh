// kf_filter.cuh -- the forward filter of one track in double precision with
// the fixed-point smoother carried along, for one thread per track: the FP64
// fit (kf_kernels.cu) and the adjoint's forward pass (kf_adjoint.cu).
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "kf_device.cuh"
#include "kf_fp64.cuh"
#include "kf_internal.h"
#include "kf_transport.cuh"

namespace kfgb {
namespace dev {

// The filtered states the adjoint's reverse pass starts from, per state and
// track: loc0, loc1, q/p, the direction's cos phi, sin phi, cos theta, sin
// theta, the covariance of the five parameters without the time, and with
// the smoother's adjoint S = Cov(x_0, x_k) (6x5).
struct AdjRec {
  static constexpr int X = 0, C = 7, S = 22, kFilter = 22, kWhole = 52;
};

struct Filter {
  double x[6], C[21];    // filtered state k
  Angles ang;            // of its direction
  double S[6][5];        // Cov(x_0, x_k)
  double xs[6], P0[21];  // the smoothed state 0, as its offset from the seed
                         // (so that the sum over the states rounds at the
                         // offset's size), and its covariance
  double chi2;
  int nmeas;
  bool spd;
};

__device__ __forceinline__ void hit_of(const FitParams& p, int64_t at, double m[2], double V[3]) {
  m[0] = p.loc[at];
  m[1] = p.loc[p.n_states + at];
  V[0] = p.cov[at];
  V[1] = p.cov[p.n_states + at];
  V[2] = p.cov[2 * p.n_states + at];
}

// The seed of track t and the update of state 0, where the smoothed state 0
// starts as the filtered one.
__device__ __forceinline__ int filter_first(const FitParams& p, int t, int64_t o0, Filter& f) {
  const size_t TT = (size_t)p.n_tracks_total;
#pragma unroll
  for (int e = 0; e < 6; ++e) {
    f.x[e] = p.seed_params[e * TT + t];
    f.xs[e] = 0.0;
  }
#pragma unroll
  for (int e = 0; e < 21; ++e) f.C[e] = p.seed_cov[e * TT + t];
  f.chi2 = 0.0;
  f.nmeas = 0;
  f.spd = true;
  if (!p.is_hole[o0]) {
    double m[2], V[3], K[6][2], fs[3], r[2];
    hit_of(p, o0, m, V);
    const int status = kalman_gain<6>(f.x, f.C, m, V, K, fs, r, f.xs, f.chi2);
    if (status != ST_OK) return status;
    joseph_update<6>(f.C, V, K);
    f.nmeas = 1;
#pragma unroll
    for (int e = 0; e < 6; ++e) f.x[e] += f.xs[e];
  }
  f.ang = angles_of(f.x[2], f.x[3]);
#pragma unroll
  for (int e = 0; e < 21; ++e) f.P0[e] = f.C[e];
#pragma unroll
  for (int r = 0; r < 6; ++r)
#pragma unroll
    for (int c = 0; c < 5; ++c) f.S[r][c] = f.C[sym(r, c)];
  return ST_OK;
}

// record of state k for the adjoint (REC 1: the filter's, 2: with S)
template <int REC>
__device__ __forceinline__ void put_adj_record(const Filter& f, int k, double* rec, const WS& ws) {
  constexpr int kRec = REC == 2 ? AdjRec::kWhole : AdjRec::kFilter;
  auto put = [&](int e, double v) { rec[((size_t)k * kRec + e) * ws.nt + ws.i] = v; };
  put(AdjRec::X + 0, f.x[0]);
  put(AdjRec::X + 1, f.x[1]);
  put(AdjRec::X + 2, f.x[4]);
  put(AdjRec::X + 3, f.ang.cp);
  put(AdjRec::X + 4, f.ang.sp);
  put(AdjRec::X + 5, f.ang.ct);
  put(AdjRec::X + 6, f.ang.st);
#pragma unroll
  for (int e = 0; e < 15; ++e) put(AdjRec::C + e, f.C[e]);
  if (REC == 2)
#pragma unroll
    for (int r = 0; r < 6; ++r)
#pragma unroll
      for (int c = 0; c < 5; ++c) put(AdjRec::S + 5 * r + c, f.S[r][c]);
}

// States 1 .. n-1 after filter_first.  N = 6 carries the time as well; N = 5
// leaves out its parameter and covariance row, which neither the results at
// state 0 nor chi2 depend on (about 100 of 1050 FP64 instructions per state),
// where time_is_settled says that they cannot change the verdict on the
// predictions either.  STATES (with N = 6): the records of smooth_states.
// smooth: carry the smoothed state 0 and check the predictions.
template <bool BZ, int N, bool STATES, int REC>
__device__ __forceinline__ int filter_states(const FitParams& p, const double* s_surf, const WS& ws, int64_t o0, int n,
                                             bool smooth, double* rec, Filter& f) {
  if (REC && n > 1) put_adj_record<REC>(f, 0, rec, ws);
  int sid_prev = p.surface_id[o0];
#pragma unroll 1
  for (int k = 1; k < n; ++k) {
    const int sid = p.surface_id[o0 + k];
    const Surf sa{s_surf + sid_prev * kSurfStride}, sb{s_surf + sid * kSurfStride};
    // field copied to registers: taking the address of a kernel parameter
    // would move the parameter block to local memory
    const double Bf[3] = {p.bfield[0], p.bfield[1], p.bfield[2]};
    double r0[3];
#pragma unroll
    for (int e = 0; e < 3; ++e) r0[e] = fma(f.x[0], sa.u(e), fma(f.x[1], sa.v(e), sa.c(e)));
    End o;
    Jac<double> J;
    {
      Cols64 g;
      const int st = propagate_to_plane<BZ, 7>(sb, r0, f.ang, f.x[4], Bf, p.mass, p.h_max, p.n_iter, o, g);
      if (st != ST_OK) return st;
      double inv_nT;
      end_frame(sb, o, inv_nT);
      jacobian_columns<BZ, 31>(sa, sb, o, g, f.x[4], Bf, inv_nT, [&](int r, int c, double v) {
        if (r == 5) J.ft[c] = v; else J.f[r][c] = v;
      });
    }
    const double d0 = o.r[0] - sb.c(0), d1 = o.r[1] - sb.c(1), d2 = o.r[2] - sb.c(2);
    f.x[0] = fma(d0, sb.u(0), fma(d1, sb.u(1), d2 * sb.u(2)));
    f.x[1] = fma(d0, sb.v(0), fma(d1, sb.v(1), d2 * sb.v(2)));
    // the filter needs the angles' cosines and sines only
    if (STATES) end_angles(f.x[2], f.x[3], f.ang, o, f.x[2], f.x[3]);
    if (N == 6) f.x[5] += o.dt;
    f.ang = o.a;
    cov_transport<N>(J, 1.0, f.C);
    // multiple scattering of surface k (added before the update)
    const double xx0 = sb.xx0();
    if (xx0 > 0.0) {
      const double q = highland_sq(f.x[4], o.g2, xx0, o.inv_cos);
      f.C[sy(2, 2)] = fma(q, o.inv_st * o.inv_st, f.C[sy(2, 2)]);
      f.C[sy(3, 3)] += q;
    }
    const auto fe = [&](int r, int c) { return jf(J, r, c); };
    if (smooth) {
      f.spd = f.spd && spd_check<N>(f.C);
#pragma unroll
      for (int r = 0; r < 6; ++r) row_times_ft(fe, 1.0, f.S[r]);
    }
    if (STATES)
#pragma unroll
      for (int e = 0; e < 25; ++e) ws.d(k, StateRec::F + e) = e < 20 ? J.f[e / 5][e % 5] : J.ft[e % 5];
    // update
    double K[6][2], ir[2] = {0.0, 0.0};
    if (!p.is_hole[o0 + k]) {
      double m[2], V[3], fs[3], r[2], dx[6], c2;
      hit_of(p, o0 + k, m, V);
      const int st = kalman_gain<N>(f.x, f.C, m, V, K, fs, r, dx, c2);
      if (st != ST_OK) return st;
      joseph_update<N>(f.C, V, K);
      f.chi2 += c2;
      ++f.nmeas;
#pragma unroll
      for (int e = 0; e < N; ++e) f.x[e] += dx[e];
      innovation_solve(fs, r[0], r[1], ir[0], ir[1]);
      if (smooth) {
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
    if (STATES) {
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
    if (REC && k < n - 1) put_adj_record<REC>(f, k, rec, ws);
    sid_prev = sid;
  }
  return ST_OK;
}

// The same with the time, out of line, for the rare track whose seed leaves
// its pivot open.
template <bool BZ, int REC>
static __device__ __noinline__ int filter_states_with_time(const FitParams& p, const double* s_surf, const WS& ws,
                                                           int64_t o0, int n, bool smooth, double* rec, Filter* f) {
  Filter t = *f;
  const int st = filter_states<BZ, 6, false, REC>(p, s_surf, ws, o0, n, smooth, rec, t);
  *f = t;
  return st;
}

// offsets and surface ids of track t
__device__ __forceinline__ int track_input(const FitParams& p, int t, int64_t& o0, int64_t& o1, int& n) {
  o0 = p.offsets[t];
  o1 = p.offsets[t + 1];
  n = (int)(o1 - o0);
  if (!(o1 > o0) || o0 < 0 || o1 > p.n_states || n > p.max_states) return ST_BAD_INPUT;
  int status = ST_OK;
  for (int k = 0; k < n; ++k) {
    const int sid = p.surface_id[o0 + k];
    if (sid < 0 || sid >= p.n_surfaces) status = ST_BAD_INPUT;
  }
  return status;
}

}  // namespace dev
}  // namespace kfgb
