// kf_team.cu -- the FP64 fit with each track's work shared by a team of W
// warps (W = 2 or 4), for batches too small to fill the GPU (paper Sect. 4.1:
// parallelism inside one track's fit, for small batches).
//
// On this part an FP64 warp instruction holds its SM sub-partition's FP64
// pipe for the same time whatever the number of active lanes (measured: 79.6
// cycles per DFMA warp instruction with 32, 16, 8, 4, 2 or 1 active lanes),
// and one warp of the one-thread-per-track kernel keeps that pipe busy on its
// own: a batch of fewer tracks than sub-partitions x 32 runs at one warp's
// FP64 instruction count per state (885).  Splitting a track over the
// lanes of one warp cannot shorten that; splitting it over W warps, each on
// its own sub-partition, can.
//
// Lane l of each of a CTA's W warps works on track l of the CTA's 32.  The
// warps all propagate the state (point, direction) and take the same discrete
// decisions; they split
//   * the columns of F (the q/p column's derivatives along the path, the path
//     correction and the free -> bound projection),
//   * F C and F C F^T, the Joseph update (by row of C),
//   * the fixed-point smoother (by row of S = Cov(x_0, x_k): every warp keeps
//     its rows of S and P_0 in registers, they are never exchanged),
// and exchange F, Cp, Cf and a few scalars through shared memory, three
// barriers per state and no second pass.  A team spends 1664 FP64 instructions
// per state where one thread per track spends 885, on pipes that would idle:
// where fits on several streams fill the GPU, one thread per track is the
// better choice (events of 3000 tracks, 11 states: 223 us by teams against 347
// on one stream, 112 against 49 us per event on sixteen).
//
// The 32 tracks of a CTA step through the states in lockstep (a track with
// fewer states, or one that failed, idles at its barriers).  The arithmetic of
// every element is that of the one-thread-per-track FP64 kernel
// (kf_kernels.cu), bit for bit: the shared functions write their fused
// multiply-adds out, and the compiler fuses nothing more.  1000 tracks of 11
// states, 4 warps: 0.535 ms with the backward smoother as a second pass of two
// barriers per state, 0.201 ms now.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "kf_team.cuh"

namespace kfgb {
namespace {
using namespace dev;

// One CTA of W warps per 32 tracks; dynamic shared memory: the surface table,
// then the exchange buffers.
template <bool BZ, int W>
__global__ void __launch_bounds__(32 * W, 1) team_kernel(const FitParams p) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  double* s_surf = reinterpret_cast<double*>(smem_raw);
  double* sh = s_surf + (size_t)p.n_surfaces * kSurfStride;
  __shared__ __align__(8) uint64_t s_mbar;
  const bool ok = stage_surfaces(s_surf, p.surf, (uint32_t)(p.n_surfaces * kSurfStride * 8), &s_mbar,
                                 p.error_flag, p.wait_limit, p.skip_stage_copy != 0);
  const int base = blockIdx.x * kTeamTracks;
  if (!ok) {
    const int i = base + (int)threadIdx.x;
    if (threadIdx.x < kTeamTracks && i < p.n_tracks) write_failed_track(p, i, ST_TIMEOUT);
    return;
  }
  switch (threadIdx.x >> 5) {
    case 0: fit_team<BZ, W, 0>(p, s_surf, sh, base); break;
    case 1: fit_team<BZ, W, 1>(p, s_surf, sh, base); break;
    case 2: fit_team<BZ, W, (W > 2 ? 2 : 0)>(p, s_surf, sh, base); break;
    default: fit_team<BZ, W, (W > 2 ? 3 : 1)>(p, s_surf, sh, base); break;
  }
}

// dynamic shared memory of one of its CTAs
size_t team_smem_bytes(int n_surfaces) {
  static_assert((kMaxSurfaces * kSurfStride + kShFields * kTeamTracks) * 8 + 1024 <= 227 * 1024,
                "fits beside the largest surface table");
  return (size_t)n_surfaces * kSurfStride * sizeof(double) + (size_t)kShFields * kTeamTracks * sizeof(double);
}

template <bool BZ, int W>
cudaError_t launch_team_v(const FitParams& p, cudaStream_t stream) {
  const size_t smem = team_smem_bytes(p.n_surfaces);
  auto kern = team_kernel<BZ, W>;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  const int grid = (p.n_tracks + kTeamTracks - 1) / kTeamTracks;
  kern<<<grid, 32 * W, smem, stream>>>(p);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_fit_team(const FitParams& p, int team_warps, cudaStream_t stream, int* launched) {
  if (launched) *launched = 0;
  if (p.n_tracks <= 0) return cudaSuccess;
  const bool bz = p.bfield[0] == 0.0 && p.bfield[1] == 0.0;
  if (launched) *launched = 1;
  if (team_warps == 4) return bz ? launch_team_v<true, 4>(p, stream) : launch_team_v<false, 4>(p, stream);
  return bz ? launch_team_v<true, 2>(p, stream) : launch_team_v<false, 2>(p, stream);
}

}  // namespace kfgb
