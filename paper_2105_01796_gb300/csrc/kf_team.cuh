// kf_team.cuh -- the FP64 fit of 32 tracks by a team of W warps (kf_team.cu
// says why and how), shared by the team fit kernel and the adjoint's kernel
// for small batches (kf_adjoint.cu), whose forward pass it is.
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
// theta, the covariance, and with the smoother's adjoint S = Cov(x_0, x_k).
struct AdjRec {
  static constexpr int X = 0, C = 7, S = 28, kFilter = 28, kWhole = 64;
};

constexpr int kTeamTracks = 32;
// shared exchange buffers per CTA, [field][32 tracks] doubles
// F 25 | Cp 21 | Cf 21 | the cosines and sines of the next transport's start
// angles 4 | 1/sin^2(theta) and theta0^2 of the scattering 2 | S H^T 12; at the
// end the smoothed state 0 and its covariance take the place of F
constexpr int kShF = 0, kShCp = 25, kShCf = 46, kShTrig = 67, kShQ = 71, kShH = 73, kShFields = 85;
constexpr int kShOut = 0;  // 27 fields

// owner warp of matrix row r of C (rows hold 1..6 lower-triangle elements)
template <int W>
__host__ __device__ constexpr int row_owner(int r) {
  return W == 2 ? ((r == 5 || r == 3 || r == 0) ? 0 : 1)
                : (r == 5 ? 0 : (r == 4 || r == 0) ? 1 : (r == 3 || r == 1) ? 2 : 3);
}
// owner warp of row r of S: evens out F C F^T + S F^T and the two updates
// (FP64 instructions per warp, W = 4: 81 / 100 / 105 / 90 and 52 / 66 / 48 / 68)
template <int W>
__host__ __device__ constexpr int srow_owner(int r) {
  return W == 2 ? (r & 1) : (r == 4 ? 0 : r < 2 ? 1 : r == 2 ? 2 : 3);
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
__host__ __device__ constexpr int turn_owner() { return W == 2 ? 1 : 2; }

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
  double* sF = sh + kShF * kTeamTracks;
  double* sCp = sh + kShCp * kTeamTracks;
  double* sCf = sh + kShCf * kTeamTracks;
  double* sTrig = sh + kShTrig * kTeamTracks;
  double* sQ = sh + kShQ * kTeamTracks;
  double* sH = sh + kShH * kTeamTracks;
  double* sOut = sh + kShOut * kTeamTracks;
  const bool states = p.out_states != nullptr;
  int64_t o0 = 0, o1 = 0;
  int n = 0;
  int status = valid ? ST_OK : ST_BAD_INPUT;
  if (valid) {
    o0 = p.offsets[t];
    o1 = p.offsets[t + 1];
    n = (int)(o1 - o0);
    if (!(o1 > o0) || o0 < 0 || o1 > p.n_states || n > p.max_states) status = ST_BAD_INPUT;
    if (status == ST_OK)
      for (int k = 0; k < n; ++k) {
        const int sid = p.surface_id[o0 + k];
        if (sid < 0 || sid >= p.n_surfaces) status = ST_BAD_INPUT;
      }
  }
  // the CTA's longest track sets the lockstep count (the same in every warp)
  int nmax = status == ST_OK ? n : 0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) nmax = max(nmax, __shfl_xor_sync(0xffffffffu, nmax, o));
  const double Bf[3] = {p.bfield[0], p.bfield[1], p.bfield[2]};

  double x[6], C[21];
  double S[6][6], P0[21], xs[6];  // only the rows this warp owns are live
  double chi2sum = 0.0;
  int nmeas = 0;
  bool spd = true;
  // the filter alone (chi2 and its gradient) does not ask for positive
  // definite predictions; nor does the adjoint check its results
  const bool verdict = REC != 1 || p.out_params || p.out_cov;
  if (status == ST_OK) {
#pragma unroll
    for (int e = 0; e < 6; ++e) x[e] = p.seed_params[e * TT + t];
#pragma unroll
    for (int e = 0; e < 21; ++e) C[e] = p.seed_cov[e * TT + t];
  }
  for (int k = 0; k < nmax; ++k) {
    bool act = status == ST_OK && k < n;
    Angles ang = {0.0, 0.0, 0.0, 0.0};  // of the prediction
    if (k > 0) {
      if (act) {
        const Surf sa{s_surf + p.surface_id[o0 + k - 1] * kSurfStride}, sb{s_surf + p.surface_id[o0 + k] * kSurfStride};
        const Angles a0 = {sTrig[0 * kTeamTracks + lane], sTrig[1 * kTeamTracks + lane],
                           sTrig[2 * kTeamTracks + lane], sTrig[3 * kTeamTracks + lane]};
        double r0[3];
#pragma unroll
        for (int e = 0; e < 3; ++e) r0[e] = fma(x[0], sa.u(e), fma(x[1], sa.v(e), sa.c(e)));
        End o;
        status = transport_warp<BZ, W, w>(sa, sb, r0, a0, x[4], Bf, p.mass, p.h_max, p.n_iter, o, sF, sQ, lane);
        act = status == ST_OK;
        if (act) {
          const double d0 = o.r[0] - sb.c(0), d1 = o.r[1] - sb.c(1), d2 = o.r[2] - sb.c(2);
          x[0] = fma(d0, sb.u(0), fma(d1, sb.u(1), d2 * sb.u(2)));
          x[1] = fma(d0, sb.v(0), fma(d1, sb.v(1), d2 * sb.v(2)));
          if (states) end_angles(x[2], x[3], a0, o, x[2], x[3]);
          x[5] += o.dt;
          ang = o.a;
        }
      }
      team_sync<W>();  // F and the scattering complete
      if (act) {
        const auto fe = [&](int r, int c) { return sF[((r == 5 ? 4 : r) * 5 + c) * kTeamTracks + lane]; };
        // the rows of F C F^T and of S F^T this warp owns
#pragma unroll
        for (int r = 0; r < 6; ++r) {
          if (row_owner<W>(r) != w) continue;
          double brow[6];
          fc_row(fe, r, 1.0, C, brow);
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
          if (srow_owner<W>(r) != w) continue;
          double v[6];
#pragma unroll
          for (int c = 0; c < 6; ++c) v[c] = S[r][c];
          row_times_ft(fe, 1.0, v, S[r]);
          sH[(2 * r) * kTeamTracks + lane] = S[r][0];
          sH[(2 * r + 1) * kTeamTracks + lane] = S[r][1];
        }
        if (states && w == 0)
#pragma unroll
          for (int e = 0; e < 25; ++e) ws.d(k, StateRec::F + e) = sF[e * kTeamTracks + lane];
      }
      team_sync<W>();  // Cp and S H^T complete
      if (act) {
#pragma unroll
        for (int e = 0; e < 21; ++e) C[e] = sCp[e * kTeamTracks + lane];
        if (w == 0 && verdict) spd = spd && spd_check(C);
      }
    }
    // update: gain and x_f in every warp, the rows split
    const bool meas = act && !p.is_hole[o0 + k];
    double dx[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    double K[6][2] = {}, ir[2] = {0.0, 0.0};
    if (meas) {
      const double m[2] = {p.loc[o0 + k], p.loc[p.n_states + o0 + k]};
      const double V[3] = {p.cov[o0 + k], p.cov[p.n_states + o0 + k], p.cov[2 * p.n_states + o0 + k]};
      double Si[3], r[2], c2;
      status = kalman_gain(x, C, m, V, K, Si, r, dx, c2);
      if (status == ST_OK) {
        chi2sum += c2;
        ++nmeas;
        double Cf[21];
#pragma unroll
        for (int e = 0; e < 21; ++e) Cf[e] = C[e];
        joseph_update(Cf, V, K);  // the rows of other warps are not used
#pragma unroll
        for (int q = 0; q < 6; ++q) {
          if (row_owner<W>(q) != w) continue;
#pragma unroll
          for (int c = 0; c <= q; ++c) sCf[sy(q, c) * kTeamTracks + lane] = Cf[sy(q, c)];
        }
        if (k > 0) {
          double hall[6][2];
#pragma unroll
          for (int e = 0; e < 6; ++e) {
            hall[e][0] = sH[(2 * e) * kTeamTracks + lane];
            hall[e][1] = sH[(2 * e + 1) * kTeamTracks + lane];
          }
#pragma unroll
          for (int e = 0; e < 6; ++e)
            if (srow_owner<W>(e) == w) fixed_point_row(e, S[e], K, Si, r, hall, xs[e], P0);
        }
#pragma unroll
        for (int e = 0; e < 6; ++e) x[e] += dx[e];
        ir[0] = fma(Si[0], r[0], Si[1] * r[1]);
        ir[1] = fma(Si[1], r[0], Si[2] * r[1]);
      }
    }
    // the start angles' cosines and sines for the next transport
    if (act && status == ST_OK && w == turn_owner<W>()) {
      if (k == 0) {
        ang = angles_of(x[2], x[3]);
      } else if (meas) {
        turn(ang.cp, ang.sp, dx[2]);
        turn(ang.ct, ang.st, dx[3]);
      }
      sTrig[0 * kTeamTracks + lane] = ang.cp;
      sTrig[1 * kTeamTracks + lane] = ang.sp;
      sTrig[2 * kTeamTracks + lane] = ang.ct;
      sTrig[3 * kTeamTracks + lane] = ang.st;
    }
    team_sync<W>();  // Cf and the start angles complete
    if (act && status == ST_OK) {
      if (meas)
#pragma unroll
        for (int e = 0; e < 21; ++e) C[e] = sCf[e * kTeamTracks + lane];
      if (k == 0) {
        // state 0 starts as its own filtered estimate
#pragma unroll
        for (int r = 0; r < 6; ++r)
          if (srow_owner<W>(r) == w) {
            xs[r] = dx[r];  // the offset from the seed
#pragma unroll
            for (int c = 0; c < 6; ++c) {
              S[r][c] = C[sym(r, c)];
              if (c <= r) P0[sy(r, c)] = C[sy(r, c)];
            }
          }
      } else if (states && w == W - 1) {
#pragma unroll
        for (int e = 0; e < 6; ++e) {
          ws.d(k, StateRec::K + 2 * e) = K[e][0];
          ws.d(k, StateRec::K + 2 * e + 1) = K[e][1];
          ws.d(k, StateRec::XF + e) = x[e];
        }
        ws.d(k, StateRec::IR) = ir[0];
        ws.d(k, StateRec::IR + 1) = ir[1];
#pragma unroll
        for (int e = 0; e < 21; ++e) ws.d(k, StateRec::CF + e) = C[e];
      }
      if (REC && k < n - 1) {
        constexpr int kRec = REC == 2 ? AdjRec::kWhole : AdjRec::kFilter;
        auto put = [&](int e, double v) { rec[((size_t)k * kRec + e) * (size_t)p.n_tracks + i] = v; };
        if (w == 0) {
          put(AdjRec::X + 0, x[0]);
          put(AdjRec::X + 1, x[1]);
          put(AdjRec::X + 2, x[4]);
        }
        if (w == turn_owner<W>()) {
          put(AdjRec::X + 3, ang.cp);
          put(AdjRec::X + 4, ang.sp);
          put(AdjRec::X + 5, ang.ct);
          put(AdjRec::X + 6, ang.st);
        }
        if (w == W - 1)
#pragma unroll
          for (int e = 0; e < 21; ++e) put(AdjRec::C + e, C[e]);
        if (REC == 2)
#pragma unroll
          for (int r = 0; r < 6; ++r)
            if (srow_owner<W>(r) == w)
#pragma unroll
              for (int c = 0; c < 6; ++c) put(AdjRec::S + 6 * r + c, S[r][c]);
      }
    }
  }

  // gather the smoothed state 0 (and, with states, the records) in warp 0
  if (status == ST_OK) {
#pragma unroll
    for (int r = 0; r < 6; ++r)
      if (srow_owner<W>(r) == w) {
        sOut[r * kTeamTracks + lane] = xs[r] + p.seed_params[r * TT + t];
#pragma unroll
        for (int c = 0; c <= r; ++c) sOut[(6 + sy(r, c)) * kTeamTracks + lane] = P0[sy(r, c)];
      }
  }
  if (states || REC) __threadfence_block();  // the other warps' records, read by warp 0
  team_sync<W>();
  if (!valid || w != 0) return status;
  double Cs[21];
  if (status == ST_OK && !spd) status = ST_NON_SPD;
  if (status == ST_OK) {
#pragma unroll
    for (int e = 0; e < 6; ++e) xs[e] = sOut[e * kTeamTracks + lane];
#pragma unroll
    for (int e = 0; e < 21; ++e) Cs[e] = sOut[(6 + e) * kTeamTracks + lane];
    if (states) {
      smooth_states(ws, n, p.out_states, p.n_states, o0);
#pragma unroll
      for (int e = 0; e < 6; ++e) p.out_states[e * p.n_states + o0] = xs[e];
    }
    bool fin = isfinite(chi2sum);
#pragma unroll
    for (int e = 0; e < 6; ++e) fin = fin && isfinite(xs[e]);
#pragma unroll
    for (int e = 0; e < 21; ++e) fin = fin && isfinite(Cs[e]);
    if (!fin && !REC) status = ST_NONFINITE;
  }
  if (status != ST_OK) {
    const double nan = qnan();
#pragma unroll
    for (int e = 0; e < 6; ++e) xs[e] = nan;
#pragma unroll
    for (int e = 0; e < 21; ++e) Cs[e] = nan;
    chi2sum = nan;
    nmeas = 0;
    if (p.out_states && n >= 1 && o0 >= 0 && o1 <= p.n_states && n <= p.max_states)
      for (int k = 0; k < n; ++k)
        for (int e = 0; e < 6; ++e) p.out_states[e * p.n_states + o0 + k] = nan;
  }
  // (the adjoint may want fewer outputs)
  if (p.out_params)
#pragma unroll
    for (int e = 0; e < 6; ++e) p.out_params[e * TT + t] = xs[e];
  if (p.out_cov)
#pragma unroll
    for (int e = 0; e < 21; ++e) p.out_cov[e * TT + t] = Cs[e];
  if (p.out_chi2) p.out_chi2[t] = chi2sum;
  if (p.out_ndf) p.out_ndf[t] = 2 * nmeas;
  if (p.out_status) p.out_status[t] = (uint8_t)status;
  return status;
}

}  // namespace dev
}  // namespace kfgb
