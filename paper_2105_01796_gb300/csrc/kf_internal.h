// Internal interface between the C ABI (kf_api.cu) and the kernels
// (kf_kernels.cu).  Not part of the public header.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace kfgb {

// Packed surface record staged into shared memory: 14 doubles (112 B, a
// whole number of 16-byte units for the bulk copy):
//   [0..2] centre c, [3..11] R row-major (columns u, v, n), [12] x/X0, [13] 0
// The mixed kernel stages a table of its own, 32 floats (128 B) per surface,
// packed after the FP64 table in the same buffer ([n_surfaces][kSurfStride]
// doubles, then [n_surfaces][kSurfStrideM] doubles): every FP64 quantity as
// a double-float pair hi + lo (hi = the nearest float, lo = the nearest
// float to the rest), so it converts nothing per step:
//   [0..2] n hi, [3..5] u hi, [6..8] v hi, [9] x/X0,
//   [10..12] n lo, [13..15] u lo, [16..18] v lo,
//   [19..21] (n.c, u.c, v.c) hi, [22..24] (n.c, u.c, v.c) lo,
//   [25..27] c hi, [28..30] c lo, [31] 0
constexpr int kSurfStride = 14;
constexpr int kSurfStrideM = 16;
constexpr int kSurfPacked = kSurfStride + kSurfStrideM;  // doubles per surface in the packed buffer
constexpr int kMaxSurfaces = 1024;  // 112 KiB of shared memory (FP64 table), 128 KiB (mixed)

// Per-state record of a fit's workspace.
// FP64 path, all in ws64: 90 doubles.  The fit itself writes none (its
//   smoother runs along with the filter); with smoothed states wanted, what
//   their backward pass reads (StateRec, kf_fp64.cuh).  The method variants
//   with the backward filter keep the filtered states there.
// Mixed path, ws64:        xp 6                                   (6 doubles)
//             ws32:        F 25 | q_phi | q_theta | dxf 6 | Cp 21 (54 floats)
//   xp is written for state 0 always and for the others only when smoothed
//   states are output.
//   F_k: rows loc0, loc1, phi, theta over columns 0..4 (20), then the time
//   row over columns 0..4 (5); q = the multiple-scattering variances added to
//   Var(phi) and Var(theta) at state k; dxf = x_f - x_p (the filter's
//   increment, zero on a hole); Cp = the predicted covariance of state k
//   (FP32 products, so exact as floats; states k >= 1).
// Register-cap variants of the fit kernels ("min_blocks"): variant 1 (the
// default) may use 255 registers, 3 caps at 168 and 4 at 128, i.e. the
// registers of 1, 3 or 4 CTAs of 128 threads per SM. Each variant accepts
// CTAs of up to the threads those registers allow.
constexpr int max_threads_of(int min_blocks) { return min_blocks == 4 ? 512 : min_blocks == 3 ? 384 : 256; }
// largest CTA a launch may ask for: only the mixed kernel has the capped
// variants; the FP64 and method-variant kernels are variant 1
inline int max_block(bool mixed, int min_blocks) { return max_threads_of(mixed ? min_blocks : 1); }

constexpr int kRec64Fp64 = 90;
constexpr int kRec64Mixed = 6;
constexpr int kRec32Mixed = 54;

struct FitParams {
  int32_t n_tracks;        // tracks in this launch (chunk)
  int32_t track0;          // global index of the chunk's first track
  int32_t n_tracks_total;  // row stride of [k][n_tracks_total] inputs/outputs
  int32_t max_states;      // states per track the workspace holds
  const int32_t* offsets;
  const double* seed_params;
  const double* seed_cov;
  int32_t n_surfaces;
  const double* surf;      // packed [n_surfaces][kSurfStride]
  int64_t n_states;
  const int32_t* surface_id;
  const double* loc;
  const double* cov;
  const uint8_t* is_hole;
  double bfield[3];
  double mass;
  double h_max;
  int32_t n_iter;
  double* out_params;
  double* out_cov;
  double* out_chi2;
  int32_t* out_ndf;
  uint8_t* out_status;
  double* out_states;
  double* ws64;            // [max_states][rec64][n_tracks]
  float* ws32;             // [max_states][rec32][n_tracks] (mixed only)
  int32_t* error_flag;     // set to 1 when a bounded device wait gives up
  int32_t wait_limit;      // polls of a bounded wait (0 = the default)
  int32_t skip_stage_copy; // diagnostic: announce but skip the surface-table
                           // copy, so that every staging wait runs out
  int32_t* work_counter;   // non-null: persistent launch, warps take 32-track
                           // units from this counter (zeroed before launch)
  const int32_t* order;    // non-null: slot s fits track order[s]
  int32_t resident_warps;  // persistent launch: warps per SM (0 = occupancy)
  int32_t waves;           // grid launch split into full waves + one spread wave (host side)
  int32_t team_warps;      // FP64 path: > 1 shares each track over that many warps (host side)
  int32_t auto_shape;      // FP64 kernels: the launch shape is the library's choice (host side)
  // method variants (the FP64 variant kernel)
  int32_t smoother;        // 0 RTS, 1 backward filter + weighted mean
  int32_t energy_loss;     // 1: mean loss and straggling on q/p
  double bf_scale;         // backward filter start: bf_scale * Cf_{n-1}
  double mat[9];           // z_over_a, i_exc, x0_rho, Sternheimer cbar, x0,
                           // x1, a, k, delta0
  int32_t map_n[3];        // field-map grid points per axis
  double map_origin[3];
  double map_inv_spacing[3];
  double map_off[3];       // -origin / spacing
  const double* map_b;     // null: the constant field bfield
  // every track of the batch has max_states states
  bool uniform() const { return (long long)n_tracks_total * max_states == (long long)n_states; }
};

// Record a failed CUDA call for kf_last_cuda_error() and map it to a
// kf_error code (KF_ENOMEM for allocation failures, else KF_ECUDA).
int cuda_fail(cudaError_t e, const char* what);

// True when the options or the field ask for a method variant.
inline bool wants_variants(int smoother, int energy_loss, const void* map) {
  return smoother != 0 || energy_loss != 0 || map != nullptr;
}

// Pack the SoA surface table into [S][kSurfStride] doubles followed by the
// mixed kernel's [S][kSurfStrideM] (packed must hold S * kSurfPacked doubles).
cudaError_t launch_pack_surfaces(int n_surfaces, const double* center,
                                 const double* rot, const double* x_over_x0,
                                 double* packed, cudaStream_t stream);

// Check the integer-pipe conversions and the Newton 1/sqrt, 1/x helpers on n
// patterns; counters[0..4] receive the mismatch counts.
cudaError_t launch_selftest(long long n, unsigned long long* counters, cudaStream_t stream);
// Check the mixed kernel's double-float arithmetic against FP64 on n
// patterns; counters[0..3] receive the counts beyond 2^-44, counters[4] the
// patterns a plain float sum already misses.
cudaError_t launch_selftest_df(long long n, unsigned long long* counters, cudaStream_t stream);
// The full-range 1/sqrt and 1/x helpers of the FP64 path; counter[0] gets
// the cases beyond 4 ulp.
cudaError_t launch_selftest_any(long long n, unsigned long long* counter, cudaStream_t stream);

// One fused filter + smoother launch over p.n_tracks tracks.  min_blocks
// selects the register-cap variant (__launch_bounds__ minimum CTAs per SM;
// 0 = the default variant).
// *launched (optional) gets the number of kernel launches queued.
cudaError_t launch_fit(const FitParams& p, int precision, int block, int min_blocks,
                       cudaStream_t stream, int* launched = nullptr);

// The FP64 fit with each track's work shared by a team of 2 or 4 warps
// (kf_team.cu): one CTA per 32 tracks, grid schedule.
cudaError_t launch_fit_team(const FitParams& p, int team_warps, cudaStream_t stream, int* launched = nullptr);

// Whether the options leave the FP64 fit's launch shape to the library (every
// launch option but the schedule at its default; the wave-split schedule
// spreads its last round itself).
inline bool shape_is_default(bool waves, int block, int min_blocks, int resident_warps, int team_warps) {
  return !waves && (block == 0 || block == 128) && min_blocks == 0 && resident_warps == 0 &&
         team_warps == 0;
}

// How an FP64 batch of equally long tracks is spread when the launch shape is
// left to the library: full waves of one CTA of `warps` warps per SM (255
// registers leave room for 8), then one last wave of CTAs of `last` warps.
// The FP64 pipe is the bound, yet a wave's time does not step with the warps
// per sub-partition: in units of the time of 1 to 4 warps per SM (one per
// sub-partition, 932 us at 31 states) 5 warps take 1.45, 6 1.53, 7 1.76 and 8
// 2.0.  So a batch of 10.3 warps per SM, which took three rounds of 4 (two
// CTAs per SM), takes a wave of 7 and one of 4: 2.76; 20.6 warps per SM take
// three waves of 7: 5.28 instead of 5 rounds and a team's 0.62.  With teams
// (kf_team.cu) a last wave of one or two warps per SM takes 0.62 or 0.74.
// All tracks equally long is what the host can see (n_states = n_tracks x
// max_states); uneven ones keep the work counter's order of smaller CTAs.
// The costs are the FP64 kernel's with the field along z.  The other kernels
// that follow them (a general field, every state output, the method variants
// with and without a map: ten kinds, 1 to 20.6 warps per SM, 15 planes) take
// 0.64 to 1.00 of the persistent grid's time, 1.02 to 1.03 (0.82 with a map)
// at 12 warps per SM, where three even rounds leave nothing to gain.
struct WavePlan {
  long long main = 0;  // 32-track units of the full waves
  int warps = 0, last = 0;
};
inline WavePlan plan_waves(long long units, int nsm, bool teams) {
  const double cost[9] = {0.0, teams ? 0.62 : 1.0, teams ? 0.74 : 1.0, 1.0, 1.0, 1.45, 1.53, 1.76, 2.0};
  WavePlan best;
  double best_cost = 1e300;
  for (int w = 8; w >= 6; --w) {
    const long long wave = (long long)w * nsm;
    long long k = (units - 8LL * nsm + wave - 1) / wave;  // the last wave takes what is left
    if (k < 0) k = 0;
    for (; ; ++k) {
      const long long rest = units - k * wave;
      const int b = rest > 0 ? (int)((rest + nsm - 1) / nsm) : 0;
      const double c = (double)k * cost[w] + cost[b];
      if (c < best_cost - 1e-9) {
        best_cost = c;
        best.main = rest > 0 ? k * wave : units;
        best.warps = w;
        best.last = b;
      }
      if (rest <= 0) break;
    }
  }
  return best;
}

// The FP64 kernel of the method variants (kf_variants.cu): backward-filter
// smoother, energy loss, field map; same records as the FP64 path.
cudaError_t launch_fit_variants(const FitParams& p, int block, cudaStream_t stream, int* launched = nullptr);

// Inputs and outputs of the adjoint (kf_adjoint.cu): the objective
// L = sum_t [w_t chi2_t + v_t . x_s0,t + W_t . C_s0,t] (x_s0, C_s0 the
// smoothed parameters and packed covariance of state 0) and its gradient
// with respect to the seeds and the per-surface alignment.
struct GradArgs {
  const double* dl_dchi2;    // w [T] or null (ones)
  const double* dl_dparams;  // v [6][T] or null (zero)
  const double* dl_dcov;     // W [21][T] or null (zero)
  double* chi2;              // [T] or null
  double* params;            // [6][T] or null: x_s0
  double* cov;               // [21][T] or null: C_s0
  double* grad_seed;         // [6][T] or null
  double* grad_align;        // [6][S] or null: accumulated (the caller zeroes it)
};

// Doubles of the adjoint's surface tables, and their computation from the
// packed table: the surfaces moved by align ([6][S], null: zero) in the fit
// kernels' layout, then the derivatives of their axes.
size_t grad_table_doubles(int n_surfaces);
cudaError_t launch_align_tables(int n_surfaces, const double* packed, const double* align, double* tables,
                                cudaStream_t stream);

// Scratch doubles per track of one adjoint launch: the filtered states, with
// the smoother's adjoint also their cross-covariances with state 0.
size_t grad_scratch_doubles(int max_states, bool smoother_adjoint);

// One launch over tracks [f.track0, f.track0 + f.n_tracks) of
// f.n_tracks_total; scratch holds grad_scratch_doubles(...) x f.n_tracks.
// team_warps: 1 one thread per track, 2 a team of warps per 32 tracks (block
// and min_blocks do not apply), 0 by the batch's size.
cudaError_t launch_grad(const FitParams& f, const GradArgs& a, const double* tables, double* scratch, int block,
                        int min_blocks, int team_warps, cudaStream_t stream);

// Counting sort of the tracks by state count, longest first:
// order[0..n_tracks) receives track indices.  hist needs max_states + 2 ints.
cudaError_t launch_length_order(int n_tracks, int max_states, const int32_t* offsets,
                                int32_t* hist, int32_t* order, cudaStream_t stream);

}  // namespace kfgb
