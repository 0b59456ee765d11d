// The single-case particle kernels (see vlb_particle_body.cuh).
#include "vlb_particle_body.cuh"

namespace vlb {

__global__ void particle_range_kernel(const ParticleConst c, const ParticleArrays P, unsigned* err) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= c.np) return;
  const int4 rg = tile_range(c, P.x[p], P.y[p], P.r[p]);
  P.prange[p] = rg;
  write_record(P, p, P.x[p], P.y[p], P.r[p], P.rb[p], P.ux[p], P.uy[p], P.om[p], float(P.lam_s[p]), float(P.T0[p]));
}

// Lists of every particle and band tables of the disks at the initial state,
// one warp per particle.  HELD: of a lattice with held particles.
template <bool HELD>
__global__ void __launch_bounds__(32 * BAND_WARPS) particle_band_kernel(const ParticleConst c, const ParticleArrays P,
                                                                        const TileLists TL, unsigned* err) {
  __shared__ int s_queue[BAND_WARPS][BAND_QUEUE];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int p = blockIdx.x * BAND_WARPS + warp;
  if (p >= c.np) return;  // the whole warp
  band_one<HELD>(c, P, TL, err, p, c.band_stamp, s_queue[warp], lane);
}

// Band tables of the ellipses (their ids: see ParticleArrays::pk), one warp per row.
__global__ void __launch_bounds__(32 * ELL_WARPS)
    particle_ellipse_kernel(const ParticleConst c, const ParticleArrays P, int blocks) {
  __shared__ int s_queue[ELL_WARPS][32];
  begin_chained();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x / blocks, by = (blockIdx.x - i * blocks) * ELL_WARPS + warp;
  if (by >= 2 * c.band_off + 1) return;  // the whole warp
  ellipse_row(c, P, (int)P.pk[8 * (long long)i + 6], c.band_stamp, by, lane, s_queue[warp]);
}

// One particle step (update, then lists and band tables) in one launch: the
// two depend on the particle alone (see step_group).  `group` particles per
// CTA.  Ellipses get their band tables from particle_ellipse_kernel after it.
// HELD: of a lattice with held particles.
template <bool HELD>
__global__ void __launch_bounds__(STEP_THREADS) particle_step_kernel(const __grid_constant__ ParticleConst c,
                                                                     const __grid_constant__ ParticleArrays P,
                                                                     const __grid_constant__ TileLists TL,
                                                                     unsigned* err, int group) {
  __shared__ StepShared sh;
  begin_chained();
  const int p0 = blockIdx.x * group;
  step_group<HELD>(min(group, c.np - p0), [&](int s) { return StepRef{&c, &P, &TL, err, p0 + s, c.band_stamp}; }, sh);
}

static inline dim3 pgrid(int n) { return dim3((unsigned)((n + 127) / 128)); }

cudaError_t launch_particle_range(const ParticleConst& c, const ParticleArrays& P, unsigned* err,
                                  cudaStream_t st) {
  if (c.np == 0) return cudaSuccess;
  particle_range_kernel<<<pgrid(c.np), 128, 0, st>>>(c, P, err);
  return cudaGetLastError();
}
static cudaError_t launch_ellipses(const ParticleConst& c, const ParticleArrays& P, int nell, cudaStream_t st) {
  if (nell > 0) {
    const int blocks = (2 * c.band_off + ELL_WARPS) / ELL_WARPS;  // rows 0 .. 2 band_off
    return launch_chained(particle_ellipse_kernel, true, dim3((unsigned)(blocks * nell)), dim3(32 * ELL_WARPS), st, c, P,
                          blocks);
  }
  return cudaSuccess;
}
cudaError_t launch_particle_band(const ParticleConst& c, const ParticleArrays& P, const TileLists& TL, int nell,
                                 unsigned* err, cudaStream_t st) {
  if (c.np == 0) return cudaSuccess;
  const unsigned grid = (unsigned)((c.np + BAND_WARPS - 1) / BAND_WARPS);
  (c.any_held ? particle_band_kernel<true> : particle_band_kernel<false>)<<<grid, 32 * BAND_WARPS, 0, st>>>(c, P, TL, err);
  if (const cudaError_t e = cudaGetLastError(); e != cudaSuccess) return e;
  return launch_ellipses(c, P, nell, st);
}
cudaError_t launch_particle_step(const ParticleConst& c, const ParticleArrays& P, const TileLists& TL, int nell,
                                 unsigned* err, cudaStream_t st) {
  if (c.np == 0) return cudaSuccess;
  const int group = step_group_size(c.np);
  const cudaError_t e = launch_chained(c.any_held ? particle_step_kernel<true> : particle_step_kernel<false>, true,
                                       dim3((unsigned)((c.np + group - 1) / group)), dim3(STEP_THREADS), st, c, P, TL, err, group);
  if (e != cudaSuccess) return e;
  return launch_ellipses(c, P, nell, st);
}
}  // namespace vlb
