// kf_kernels.cu -- the FP64 fit kernel (sm_103a) of the Kalman-filter track
// fit (arXiv 2105.01796): forward filter (Runge-Kutta-Nystrom propagation in
// a constant field, Jacobian transport, multiple-scattering noise, gain-matrix
// update with the Joseph covariance form, chi2) with the smoothed estimate of
// state 0 carried along (the fixed-point form of the smoother, kf_fp64.cuh),
// one launch, one track per thread, every step in double precision; plus the
// small helper kernels (surface packing, the length sort of the sorted
// schedule, a self-check).  The mixed-precision kernel is in kf_mixed.cu, the
// method variants in kf_variants.cu.
// Paper references: Sect. 2 (filter step list, smoother), Sect. 4.1 (RKN
// transport; local<->global Jacobians at both surfaces), Sect. 4.3 (surfaces
// in global memory accessed once; constant field).
//
// The bound is the FP64 pipe (2 DFMA per clock and SM), so the design spends
// as few FP64 instructions as the method allows: about 885 per state with the
// field along z, where the stage-by-stage transport with the backward
// smoother took 2370.  100k tracks of 31 states: 15.28 -> 6.47 ms with the
// closed-form transport and the fixed-point smoother, 6.22 ms with teams for
// the last round, 5.43 ms without the time row (kf_filter.cuh), 5.29 ms with
// cheaper reciprocals and logarithms, 4.88 ms in waves of 7 warps per SM; 20k
// tracks of 24 tilted planes in a general field with every smoothed state 3.56
// -> 1.55 ms.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "kf_device.cuh"
#include "kf_filter.cuh"
#include "kf_fp64.cuh"
#include "kf_internal.h"

namespace kfgb {
namespace {
using namespace dev;


// ---------------------------------------------------------------------------
// the fused fit: forward filter and fixed-point smoother in one pass
// ---------------------------------------------------------------------------
// STATES: the smoothed parameters of every state are wanted.
template <bool BZ, bool STATES>
__device__ __forceinline__ void fit_one_fp64(const FitParams& p, const double* s_surf, int i) {
  const int t = track_of(p, i);
  const size_t TT = (size_t)p.n_tracks_total;
  const WS ws{p.ws64, p.ws32, (size_t)p.n_tracks, kRec64Fp64, 0, i};
  int64_t o0, o1;
  int n;
  int status = track_input(p, t, o0, o1, n);
  Filter f;
  if (status == ST_OK) status = filter_first(p, t, o0, f);
  if (status == ST_OK) {
    if (STATES) {
      status = filter_states<BZ, 6, true, 0>(p, s_surf, ws, o0, n, true, nullptr, f);
    } else if (time_is_settled(f.C)) {
      status = filter_states<BZ, 5, false, 0>(p, s_surf, ws, o0, n, true, nullptr, f);
    } else {
      Filter g = f;
      status = filter_states_with_time<BZ, 0>(p, s_surf, ws, o0, n, true, nullptr, &g);
      f = g;
    }
  }
  if (status == ST_OK) {
    if (!f.spd) status = ST_NON_SPD;
#pragma unroll
    for (int e = 0; e < 6; ++e) f.xs[e] += p.seed_params[e * TT + t];
  }
  if (STATES && status == ST_OK) {
    smooth_states(ws, n, p.out_states, p.n_states, o0);
#pragma unroll
    for (int e = 0; e < 6; ++e) p.out_states[e * p.n_states + o0] = f.xs[e];
  }
  if (status == ST_OK) {
    bool fin = isfinite(f.chi2);
#pragma unroll
    for (int e = 0; e < 6; ++e) fin = fin && isfinite(f.xs[e]);
#pragma unroll
    for (int e = 0; e < 21; ++e) fin = fin && isfinite(f.P0[e]);
    if (!fin) status = ST_NONFINITE;
  }
  if (status != ST_OK) {
    const double nan = qnan();
#pragma unroll
    for (int e = 0; e < 6; ++e) f.xs[e] = nan;
#pragma unroll
    for (int e = 0; e < 21; ++e) f.P0[e] = nan;
    f.chi2 = nan;
    f.nmeas = 0;
    if (STATES && n >= 1 && o0 >= 0 && o1 <= p.n_states && n <= p.max_states)
      for (int k = 0; k < n; ++k)
        for (int e = 0; e < 6; ++e) p.out_states[e * p.n_states + o0 + k] = nan;
  }
#pragma unroll
  for (int e = 0; e < 6; ++e) p.out_params[e * TT + t] = f.xs[e];
#pragma unroll
  for (int e = 0; e < 21; ++e) p.out_cov[e * TT + t] = f.P0[e];
  p.out_chi2[t] = f.chi2;
  if (p.out_ndf) p.out_ndf[t] = 2 * f.nmeas;
  if (p.out_status) p.out_status[t] = (uint8_t)status;
}

// self-check of the full-range Newton helpers against CUDA's double 1/sqrt
// and 1/x over positive and negative values across 1e-300 .. 1e300, and of the
// logarithm against CUDA's; counter: cases beyond 4 ulp
__global__ void selftest_any_kernel(long long n, unsigned long long* counter) {
  const long long i0 = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const long long stride = (long long)gridDim.x * blockDim.x;
  unsigned long long c = 0;
  for (long long i = i0; i < n; i += stride) {
    uint64_t z = (uint64_t)i * 0x9E3779B97F4A7C15ULL;
    z = (z ^ (z >> 31)) * 0xBF58476D1CE4E5B9ULL;
    z ^= z >> 29;
    const double y = exp2((double)((int)(z % 1990) - 995)) * (1.0 + (double)((z >> 20) & 0xfffff) / 1048576.0);
    const double rs_ref = 1.0 / sqrt(y), rc_ref = 1.0 / y;
    if (fabs(rsqrt_any(y) - rs_ref) > 8.9e-16 * rs_ref) ++c;
    if (fabs(rcp_any(y) - rc_ref) > 8.9e-16 * rc_ref) ++c;
    if (fabs(rcp_any(-y) + rc_ref) > 8.9e-16 * rc_ref) ++c;
    // the logarithm over the whole range and close to 1, either side
    const double step = exp2(-(double)(z >> 58) * 0.8125) * (1.0 + (double)((z >> 20) & 0xfffff) / 1048576.0);
    const double args[3] = {y, 1.0 + 0.5 * step, 1.0 - 0.25 * step};
    for (int k = 0; k < 3; ++k) {
      const double l = log(args[k]), a = fabs(l);
      if (!(fabs(log_df(args[k]) - l) <= 8.9e-16 * a)) ++c;
    }
  }
  if (c) atomicAdd(counter, c);
}

__global__ void pack_surfaces_kernel(int n, const double* __restrict__ center, const double* __restrict__ rot,
                                     const double* __restrict__ xx0, double* __restrict__ out) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  double* o = out + (size_t)s * kSurfStride;
  for (int i = 0; i < 3; ++i) o[i] = center[(size_t)i * n + s];
  for (int i = 0; i < 9; ++i) o[3 + i] = rot[(size_t)i * n + s];
  o[12] = xx0[s];
  o[13] = 0.0;
  // the mixed kernel's table: each FP64 value v as hi = (float)v and
  // lo = (float)(v - hi)
  float* m = reinterpret_cast<float*>(out + (size_t)n * kSurfStride + (size_t)s * kSurfStrideM);
  auto split = [](double v, float* hi, float* lo) {
    const float h = (float)v;
    *hi = h;
    *lo = (float)(v - (double)h);
  };
  for (int i = 0; i < 3; ++i) {
    split(o[3 + 3 * i + 2], &m[i], &m[10 + i]);      // n
    split(o[3 + 3 * i + 0], &m[3 + i], &m[13 + i]);  // u
    split(o[3 + 3 * i + 1], &m[6 + i], &m[16 + i]);  // v
    const int j = (i + 2) % 3;  // n.c, u.c, v.c: column j of R is o[3 + 3 k + j], k = 0..2
    split(o[3 + j] * o[0] + o[6 + j] * o[1] + o[9 + j] * o[2], &m[19 + i], &m[22 + i]);
    split(o[i], &m[25 + i], &m[28 + i]);             // c
  }
  m[9] = (float)o[12];
  m[31] = 0.0f;
}

template <bool BZ, bool STATES>
struct Fp64Body {
  static constexpr int kStride = kSurfStride;
  static __device__ __forceinline__ void run(const FitParams& p, const double* s_surf, int i) {
    fit_one_fp64<BZ, STATES>(p, s_surf, i);
  }
};

template <bool BZ>
cudaError_t launch_fp64(const FitParams& p, int block, int min_blocks, cudaStream_t stream, int* launched) {
  (void)min_blocks;  // a register cap below 255 spills this kernel heavily
  if (p.out_states) return launch_body<Fp64Body<BZ, true>, 1>(p, block, stream, launched);
  return launch_body<Fp64Body<BZ, false>, 1>(p, block, stream, launched);
}

// counting sort of tracks by state count (longest first)
__global__ void length_hist_kernel(int n, int max_states, const int32_t* __restrict__ offsets,
                                   int32_t* __restrict__ hist) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  int len = offsets[t + 1] - offsets[t];
  len = len < 0 ? 0 : (len > max_states ? max_states + 1 : len);
  atomicAdd(&hist[max_states + 1 - len], 1);  // bin 0 = longest
}

__global__ void length_scan_kernel(int nbins, int32_t* hist) {
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    int acc = 0;
    for (int b = 0; b < nbins; ++b) {
      const int c = hist[b];
      hist[b] = acc;
      acc += c;
    }
  }
}

__global__ void length_scatter_kernel(int n, int max_states, const int32_t* __restrict__ offsets,
                                      int32_t* __restrict__ hist, int32_t* __restrict__ order) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  int len = offsets[t + 1] - offsets[t];
  len = len < 0 ? 0 : (len > max_states ? max_states + 1 : len);
  const int slot = atomicAdd(&hist[max_states + 1 - len], 1);
  order[slot] = t;
}

}  // namespace

cudaError_t launch_selftest_any(long long n, unsigned long long* counter, cudaStream_t stream) {
  selftest_any_kernel<<<152 * 4, 256, 0, stream>>>(n, counter);
  return cudaGetLastError();
}

cudaError_t launch_pack_surfaces(int n_surfaces, const double* center, const double* rot,
                                 const double* x_over_x0, double* packed, cudaStream_t stream) {
  const int block = 128;
  pack_surfaces_kernel<<<(n_surfaces + block - 1) / block, block, 0, stream>>>(n_surfaces, center, rot,
                                                                              x_over_x0, packed);
  return cudaGetLastError();
}

cudaError_t launch_fit_mixed(const FitParams& p, int block, int min_blocks, cudaStream_t stream, int* launched);

namespace {

// The FP64 fit with the launch shape left to the library.  Equally long tracks
// run in waves of one CTA per SM (plan_waves; 100k tracks of 31 states 5.29 ->
// 4.90 ms).  Else a sub-partition's FP64 pipe is busy with one warp, so a batch
// takes rounds of one warp (32 tracks) per sub-partition, and a last round
// that fills few of them takes as long as a full one.  The tracks of a last
// round go to teams of warps instead (kf_team.cu; the same results bit for
// bit): with U warp units left over
// after the full rounds, teams of 4 while they fit one per SM (U <= SMs:
// 0.60 to 0.64 of a round's time, measured 421-453 against 706 us at 20
// planes), teams of 2 up to two per SM (0.72 to 0.75, 510-531 us), else the
// round as it is (a second round of teams takes 0.9 and more).  On the
// length-sorted schedule the last round holds the shortest tracks; without
// teams its CTAs share SMs with some of the longest (20k tracks of 6 to 25
// states: 2.07-2.41 ms by the luck of the placement, 1.58-1.64 ms with them).
cudaError_t launch_fp64_auto(const FitParams& p, int block, int min_blocks, bool bz, cudaStream_t stream,
                             int* launched) {
  int dev = 0, nsm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const long long units = ((long long)p.n_tracks + 31) / 32, round = 4LL * nsm;
  long long rest = units % round;
  int team = rest == 0 ? 1 : rest <= nsm ? 4 : rest <= 2 * nsm ? 2 : 1;
  FitParams a = p;
  if (p.uniform() && !p.order) {
    const WavePlan plan = plan_waves(units, nsm, true);
    rest = units - plan.main;
    team = plan.last == 1 ? 4 : plan.last == 2 ? 2 : 1;
    a.work_counter = nullptr;
    block = 32 * plan.warps;
    if (team == 1 && rest > 0) {
      a.n_tracks = (int32_t)(plan.main * 32);
      int l = 0;
      if (a.n_tracks > 0) {
        e = bz ? launch_fp64<true>(a, block, min_blocks, stream, &l)
               : launch_fp64<false>(a, block, min_blocks, stream, &l);
        if (e != cudaSuccess) return e;
      }
      if (launched) *launched = l;
      a.track0 = p.track0 + a.n_tracks;
      a.n_tracks = p.n_tracks - a.n_tracks;
      block = 32 * plan.last;
      e = bz ? launch_fp64<true>(a, block, min_blocks, stream, &l)
             : launch_fp64<false>(a, block, min_blocks, stream, &l);
      if (launched) *launched += l;
      return e;
    }
  }
  if (team > 1) a.n_tracks = (int32_t)((units - rest) * 32);
  int l = 0, count = 0;
  if (a.n_tracks > 0) {
    e = bz ? launch_fp64<true>(a, block, min_blocks, stream, &l) : launch_fp64<false>(a, block, min_blocks, stream, &l);
    if (e != cudaSuccess) return e;
    count = l;
  }
  if (team > 1) {
    FitParams b = p;
    b.track0 = p.track0 + a.n_tracks;
    b.n_tracks = p.n_tracks - a.n_tracks;
    b.work_counter = nullptr;
    e = launch_fit_team(b, team, stream, &l);
    if (e != cudaSuccess) return e;
    count += l;
  }
  if (launched) *launched = count;
  return cudaSuccess;
}

}  // namespace

cudaError_t launch_fit(const FitParams& p, int precision, int block, int min_blocks, cudaStream_t stream,
                       int* launched) {
  if (launched) *launched = 0;
  if (p.n_tracks <= 0) return cudaSuccess;
  if (block <= 0) block = 128;
  const bool bz = p.bfield[0] == 0.0 && p.bfield[1] == 0.0;
  if (precision == 0 && p.team_warps > 1) return launch_fit_team(p, p.team_warps, stream, launched);
  if (precision == 0 && p.auto_shape) return launch_fp64_auto(p, block, min_blocks, bz, stream, launched);
  if (precision == 0) return bz ? launch_fp64<true>(p, block, min_blocks, stream, launched)
                                : launch_fp64<false>(p, block, min_blocks, stream, launched);
  return launch_fit_mixed(p, block, min_blocks, stream, launched);
}

cudaError_t launch_length_order(int n_tracks, int max_states, const int32_t* offsets, int32_t* hist,
                                int32_t* order, cudaStream_t stream) {
  if (n_tracks <= 0) return cudaSuccess;
  const int nbins = max_states + 2;
  cudaError_t e = cudaMemsetAsync(hist, 0, sizeof(int32_t) * nbins, stream);
  if (e != cudaSuccess) return e;
  const int block = 256, grid = (n_tracks + block - 1) / block;
  length_hist_kernel<<<grid, block, 0, stream>>>(n_tracks, max_states, offsets, hist);
  length_scan_kernel<<<1, 32, 0, stream>>>(nbins, hist);
  length_scatter_kernel<<<grid, block, 0, stream>>>(n_tracks, max_states, offsets, hist, order);
  return cudaGetLastError();
}

}  // namespace kfgb
