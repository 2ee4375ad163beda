// kf_team.cuh -- the FP64 fit of 32 tracks by a team of W warps (kf_team.cu
// says why and how), shared by the team fit kernel and the adjoint's kernel
// for small batches (kf_adjoint.cu), whose forward pass it is.
// Each warp runs its own instance of this code on the state and takes the
// discrete decisions (sub-steps, corrections, failures) by itself: the files
// that include it are compiled with -fmad=false, so that every instance does
// the same IEEE operations and all warps agree.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "kf_device.cuh"
#include "kf_filter.cuh"
#include "kf_fp64.cuh"
#include "kf_internal.h"
#include "kf_transport.cuh"

namespace kfgb {
namespace dev {

constexpr int kTeamTracks = 32;
// shared exchange buffers per CTA, [field][32 tracks] doubles
// F 25 | Cp 21 | Cf 21 | the cosines and sines of the next transport's start
// angles 4 | 1/sin^2(theta) and theta0^2 of the scattering 2 | S H^T 12; at the
// end the smoothed state 0 and its covariance take the place of F
constexpr int kShF = 0, kShCp = 25, kShCf = 46, kShTrig = 67, kShQ = 71, kShH = 73, kShFields = 85;
constexpr int kShOut = 0;  // 27 fields

// owner warp of matrix row r of C, and of row r of S; N = 6 or 5 rows of C
// (without the time).  They even out F C F^T + S F^T and the two updates (FP64
// instructions per warp, W = 4, N = 5: 65 / 80 / 75 / 70 and 74 / 50 / 54 / 50).
template <int W, int N>
__host__ __device__ constexpr int row_owner(int r) {
  return N == 5 ? (W == 2 ? ((r == 3 || r == 0) ? 0 : 1) : (r == 3 ? 0 : r == 2 ? 1 : r == 1 ? 2 : 3))
                : (W == 2 ? ((r == 5 || r == 3 || r == 0) ? 0 : 1)
                          : (r == 5 ? 0 : (r == 4 || r == 0) ? 1 : (r == 3 || r == 1) ? 2 : 3));
}
template <int W, int N>
__host__ __device__ constexpr int srow_owner(int r) {
  return N == 5 ? (W == 2 ? 1 - (r & 1) : (r == 5 ? 0 : r < 2 ? 1 : r < 4 ? 2 : 3))
                : (W == 2 ? (r & 1) : (r == 4 ? 0 : r < 2 ? 1 : r == 2 ? 2 : 3));
}
// owner warp of column j of F (0 loc0, 1 loc1, 2 phi, 3 theta, 4 q/p)
template <int W>
__host__ __device__ constexpr int col_owner(int j) {
  return W == 2 ? ((j == 4 || j == 3) ? 0 : 1) : (j == 2 ? 0 : j == 3 ? 1 : j == 4 ? 2 : 3);
}
template <int W>
__host__ __device__ constexpr int col_mask(int w) {
  return (col_owner<W>(0) == w ? 1 : 0) | (col_owner<W>(1) == w ? 2 : 0) | (col_owner<W>(2) == w ? 4 : 0) |
         (col_owner<W>(3) == w ? 8 : 0) | (col_owner<W>(4) == w ? 16 : 0);
}
// the warps that compute the Highland width and turn the direction's angles:
// the ones with the least split work beside them
template <int W>
__host__ __device__ constexpr int noise_owner() { return W == 2 ? 1 : 0; }
template <int W>
__host__ __device__ constexpr int turn_owner() { return W == 2 ? 1 : 3; }

// The team's barrier.  Each warp runs its own instance of the code below, so
// the barrier is the PTX one, which may be reached from different places.
template <int W>
__device__ __forceinline__ void team_sync() {
  __syncwarp();
  asm volatile("barrier.cta.sync 1, %0;" ::"n"(32 * W) : "memory");
}

// One warp's part of a transport: the state in full, the columns of F that
// warp w owns to shared memory (sF[(r * 5 + c) * 32 + lane], time row r = 4).
template <bool BZ, int W, int w>
__device__ __forceinline__ int transport_warp(const Surf& sa, const Surf& sb, const double r0[3], const Angles& ang,
                                              double lam, const double B[3], double mass, double h_max, int n_iter,
                                              End& o, double* sF, double* sQ, int lane) {
  constexpr int fmask = col_mask<W>(w);
  Cols64 g;
  const int st = propagate_to_plane<BZ, (fmask >> 2) & 7>(sb, r0, ang, lam, B, mass, h_max, n_iter, o, g);
  if (st != ST_OK) return st;
  double inv_nT;
  end_frame(sb, o, inv_nT);
  jacobian_columns<BZ, fmask>(sa, sb, o, g, lam, B, inv_nT, [&](int r, int c, double v) {
    sF[((r == 5 ? 4 : r) * 5 + c) * kTeamTracks + lane] = v;
  });
  if (w == noise_owner<W>()) {
    const double xx0 = sb.xx0();
    const double q = xx0 > 0.0 ? highland_sq(lam, o.g2, xx0, o.inv_cos) : 0.0;
    sQ[0 * kTeamTracks + lane] = o.inv_st * o.inv_st;
    sQ[1 * kTeamTracks + lane] = q;
  }
  return ST_OK;
}

// States 1 .. n-1 of the CTA's tracks, in lockstep up to nmax; this is warp w.
// f holds the track's state after filter_first (of S, P0 and xs the rows this
// warp owns are kept up); N and REC as in filter_states.
template <bool BZ, int W, int w, int N, int REC>
__device__ __forceinline__ int team_states(const FitParams& p, const double* s_surf, double* sh, const WS& ws, int lane,
                                           int64_t o0, int n, int nmax, int status, bool smooth, double* rec,
                                           Filter& f) {
  double* sF = sh + kShF * kTeamTracks;
  double* sCp = sh + kShCp * kTeamTracks;
  double* sCf = sh + kShCf * kTeamTracks;
  double* sTrig = sh + kShTrig * kTeamTracks;
  double* sQ = sh + kShQ * kTeamTracks;
  double* sH = sh + kShH * kTeamTracks;
  const bool states = N == 6 && !REC && p.out_states != nullptr;
  const double Bf[3] = {p.bfield[0], p.bfield[1], p.bfield[2]};
  auto put_record = [&](int k, const Angles& ang) {
    constexpr int kRec = REC == 2 ? AdjRec::kWhole : AdjRec::kFilter;
    auto put = [&](int e, double v) { rec[((size_t)k * kRec + e) * ws.nt + ws.i] = v; };
    if (w == 0) {
      put(AdjRec::X + 0, f.x[0]);
      put(AdjRec::X + 1, f.x[1]);
      put(AdjRec::X + 2, f.x[4]);
    }
    if (w == turn_owner<W>()) {
      put(AdjRec::X + 3, ang.cp);
      put(AdjRec::X + 4, ang.sp);
      put(AdjRec::X + 5, ang.ct);
      put(AdjRec::X + 6, ang.st);
    }
    if (w == W / 2)
#pragma unroll
      for (int e = 0; e < 15; ++e) put(AdjRec::C + e, f.C[e]);
    if (REC == 2)
#pragma unroll
      for (int r = 0; r < 6; ++r)
        if (srow_owner<W, N>(r) == w)
#pragma unroll
          for (int c = 0; c < 5; ++c) put(AdjRec::S + 5 * r + c, f.S[r][c]);
  };
  auto put_angles = [&](const Angles& ang) {
    sTrig[0 * kTeamTracks + lane] = ang.cp;
    sTrig[1 * kTeamTracks + lane] = ang.sp;
    sTrig[2 * kTeamTracks + lane] = ang.ct;
    sTrig[3 * kTeamTracks + lane] = ang.st;
  };
  if (status == ST_OK) {
    if (w == turn_owner<W>()) put_angles(f.ang);
    if (REC && n > 1) put_record(0, f.ang);
  }
  team_sync<W>();  // the start angles complete
#pragma unroll 1
  for (int k = 1; k < nmax; ++k) {
    bool act = status == ST_OK && k < n;
    Angles ang = {0.0, 0.0, 0.0, 0.0};  // of the prediction
    if (act) {
      const Surf sa{s_surf + p.surface_id[o0 + k - 1] * kSurfStride}, sb{s_surf + p.surface_id[o0 + k] * kSurfStride};
      const Angles a0 = {sTrig[0 * kTeamTracks + lane], sTrig[1 * kTeamTracks + lane], sTrig[2 * kTeamTracks + lane],
                         sTrig[3 * kTeamTracks + lane]};
      double r0[3];
#pragma unroll
      for (int e = 0; e < 3; ++e) r0[e] = fma(f.x[0], sa.u(e), fma(f.x[1], sa.v(e), sa.c(e)));
      End o;
      status = transport_warp<BZ, W, w>(sa, sb, r0, a0, f.x[4], Bf, p.mass, p.h_max, p.n_iter, o, sF, sQ, lane);
      act = status == ST_OK;
      if (act) {
        const double d0 = o.r[0] - sb.c(0), d1 = o.r[1] - sb.c(1), d2 = o.r[2] - sb.c(2);
        f.x[0] = fma(d0, sb.u(0), fma(d1, sb.u(1), d2 * sb.u(2)));
        f.x[1] = fma(d0, sb.v(0), fma(d1, sb.v(1), d2 * sb.v(2)));
        if (states) end_angles(f.x[2], f.x[3], a0, o, f.x[2], f.x[3]);
        if (N == 6) f.x[5] += o.dt;
        ang = o.a;
      }
    }
    team_sync<W>();  // F and the scattering complete
    if (act) {
      const auto fe = [&](int r, int c) { return sF[((r == 5 ? 4 : r) * 5 + c) * kTeamTracks + lane]; };
      // the rows of F C F^T and of S F^T this warp owns
#pragma unroll
      for (int r = 0; r < N; ++r) {
        if (row_owner<W, N>(r) != w) continue;
        double brow[6];
        fc_row<N>(fe, r, 1.0, f.C, brow);
#pragma unroll
        for (int c = 0; c <= r; ++c) {
          double v = fcf_element(fe, c, 1.0, brow);
          if (r == c && r == 2) v = fma(sQ[1 * kTeamTracks + lane], sQ[0 * kTeamTracks + lane], v);
          if (r == c && r == 3) v += sQ[1 * kTeamTracks + lane];
          sCp[sy(r, c) * kTeamTracks + lane] = v;
        }
      }
#pragma unroll
      for (int r = 0; r < 6; ++r) {
        if (srow_owner<W, N>(r) != w) continue;
        row_times_ft(fe, 1.0, f.S[r]);
        sH[(2 * r) * kTeamTracks + lane] = f.S[r][0];
        sH[(2 * r + 1) * kTeamTracks + lane] = f.S[r][1];
      }
      if (states && w == 0)
#pragma unroll
        for (int e = 0; e < 25; ++e) ws.d(k, StateRec::F + e) = sF[e * kTeamTracks + lane];
    }
    team_sync<W>();  // Cp and S H^T complete
    if (act) {
#pragma unroll
      for (int e = 0; e < sy(N, 0); ++e) f.C[e] = sCp[e * kTeamTracks + lane];
      if (w == 0 && smooth) f.spd = f.spd && spd_check<N>(f.C);
    }
    // update: gain and x_f in every warp, the rows split
    const bool meas = act && !p.is_hole[o0 + k];
    double K[6][2] = {}, ir[2] = {0.0, 0.0}, dx[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    if (meas) {
      double m[2], V[3], fs[3], r[2], c2;
      hit_of(p, o0 + k, m, V);
      status = kalman_gain<N>(f.x, f.C, m, V, K, fs, r, dx, c2);
      if (status == ST_OK) {
        f.chi2 += c2;
        ++f.nmeas;
        double Cf[21];
#pragma unroll
        for (int e = 0; e < sy(N, 0); ++e) Cf[e] = f.C[e];
        joseph_update<N>(Cf, V, K);  // the rows of other warps are not used
#pragma unroll
        for (int q = 0; q < N; ++q) {
          if (row_owner<W, N>(q) != w) continue;
#pragma unroll
          for (int c = 0; c <= q; ++c) sCf[sy(q, c) * kTeamTracks + lane] = Cf[sy(q, c)];
        }
        double hall[6][2];
#pragma unroll
        for (int e = 0; e < 6; ++e) {
          hall[e][0] = sH[(2 * e) * kTeamTracks + lane];
          hall[e][1] = sH[(2 * e + 1) * kTeamTracks + lane];
        }
#pragma unroll
        for (int e = 0; e < 6; ++e)
          if (srow_owner<W, N>(e) == w) fixed_point_row(e, f.S[e], K, fs, r, hall, f.xs[e], f.P0);
#pragma unroll
        for (int e = 0; e < N; ++e) f.x[e] += dx[e];
        innovation_solve(fs, r[0], r[1], ir[0], ir[1]);
      }
    }
    // the start angles' cosines and sines for the next transport
    if (act && status == ST_OK && w == turn_owner<W>()) {
      if (meas) {
        turn(ang.cp, ang.sp, dx[2]);
        turn(ang.ct, ang.st, dx[3]);
      }
      put_angles(ang);
    }
    team_sync<W>();  // Cf and the start angles complete
    if (act && status == ST_OK) {
      if (meas)
#pragma unroll
        for (int e = 0; e < sy(N, 0); ++e) f.C[e] = sCf[e * kTeamTracks + lane];
      if (states && w == W - 1) {
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
      if (REC && k < n - 1) put_record(k, ang);
    }
  }

  // gather the smoothed state 0 (and the records) in warp 0
  double* sOut = sh + kShOut * kTeamTracks;
  if (status == ST_OK) {
#pragma unroll
    for (int r = 0; r < 6; ++r)
      if (srow_owner<W, N>(r) == w) {
        sOut[r * kTeamTracks + lane] = f.xs[r];
#pragma unroll
        for (int c = 0; c <= r; ++c) sOut[(6 + sy(r, c)) * kTeamTracks + lane] = f.P0[sy(r, c)];
      }
  }
  if (states || REC) __threadfence_block();  // the other warps' records, read by warp 0
  team_sync<W>();
  if (w == 0 && status == ST_OK) {
#pragma unroll
    for (int e = 0; e < 6; ++e) f.xs[e] = sOut[e * kTeamTracks + lane];
#pragma unroll
    for (int e = 0; e < 21; ++e) f.P0[e] = sOut[(6 + e) * kTeamTracks + lane];
  }
  return status;
}

// One CTA: the 32 tracks of slots [base, base + 32), W warps; this is warp w.
// REC 1, 2: the filtered states go to rec ([state][kFilter or kWhole][track])
// for the adjoint.  Returns the track's status (complete in warp 0 only).
template <bool BZ, int W, int w, int REC = 0>
__device__ __forceinline__ int fit_team(const FitParams& p, const double* s_surf, double* sh, int base,
                                        double* rec = nullptr) {
  const int lane = threadIdx.x & 31;
  const int i = base + lane;
  const bool valid = i < p.n_tracks;
  const int t = valid ? track_of(p, i) : 0;
  const size_t TT = (size_t)p.n_tracks_total;
  const WS ws{p.ws64, p.ws32, (size_t)p.n_tracks, kRec64Fp64, 0, valid ? i : 0};
  const bool states = !REC && p.out_states != nullptr;
  // the filter alone (chi2 and its gradient) does not ask for positive
  // definite predictions; nor does the adjoint check its results
  const bool smooth = REC != 1 || p.out_params || p.out_cov;
  int64_t o0 = 0, o1 = 0;
  int n = 0;
  int status = valid ? track_input(p, t, o0, o1, n) : ST_BAD_INPUT;
  // the CTA's longest track sets the lockstep count, and one track that needs
  // the time carried makes all carry it (the same in every warp)
  int nmax = status == ST_OK ? n : 0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) nmax = max(nmax, __shfl_xor_sync(0xffffffffu, nmax, o));
  Filter f;
  if (status == ST_OK) status = filter_first(p, t, o0, f);
  const bool five = !states && __all_sync(0xffffffffu, status != ST_OK || !smooth || time_is_settled(f.C));
  status = five ? team_states<BZ, W, w, 5, REC>(p, s_surf, sh, ws, lane, o0, n, nmax, status, smooth, rec, f)
                : team_states<BZ, W, w, 6, REC>(p, s_surf, sh, ws, lane, o0, n, nmax, status, smooth, rec, f);
  if (!valid || w != 0) return status;
  if (status == ST_OK && !f.spd) status = ST_NON_SPD;
  if (status == ST_OK) {
#pragma unroll
    for (int e = 0; e < 6; ++e) f.xs[e] += p.seed_params[e * TT + t];
    if (states) {
      smooth_states(ws, n, p.out_states, p.n_states, o0);
#pragma unroll
      for (int e = 0; e < 6; ++e) p.out_states[e * p.n_states + o0] = f.xs[e];
    }
    bool fin = isfinite(f.chi2);
#pragma unroll
    for (int e = 0; e < 6; ++e) fin = fin && isfinite(f.xs[e]);
#pragma unroll
    for (int e = 0; e < 21; ++e) fin = fin && isfinite(f.P0[e]);
    if (!fin && !REC) status = ST_NONFINITE;
  }
  if (status != ST_OK) {
    const double nan = qnan();
#pragma unroll
    for (int e = 0; e < 6; ++e) f.xs[e] = nan;
#pragma unroll
    for (int e = 0; e < 21; ++e) f.P0[e] = nan;
    f.chi2 = nan;
    f.nmeas = 0;
    if (states && n >= 1 && o0 >= 0 && o1 <= p.n_states && n <= p.max_states)
      for (int k = 0; k < n; ++k)
        for (int e = 0; e < 6; ++e) p.out_states[e * p.n_states + o0 + k] = nan;
  }
  // (the adjoint may want fewer outputs)
  if (p.out_params)
#pragma unroll
    for (int e = 0; e < 6; ++e) p.out_params[e * TT + t] = f.xs[e];
  if (p.out_cov)
#pragma unroll
    for (int e = 0; e < 21; ++e) p.out_cov[e * TT + t] = f.P0[e];
  if (p.out_chi2) p.out_chi2[t] = f.chi2;
  if (p.out_ndf) p.out_ndf[t] = 2 * f.nmeas;
  if (p.out_status) p.out_status[t] = (uint8_t)status;
  return status;
}

}  // namespace dev
}  // namespace kfgb
