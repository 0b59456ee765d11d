// The single-case lattice kernels: the fused step (see vlb_lattice_body.cuh),
// the ownership dump and the FP64 audits.
#include "vlb_lattice_held.cuh"

namespace vlb {

// One CTA per tile (FP32: TILE_Y warps), or per strip of a tile (FP64: one
// warp per CTA, grid ntx * TILE_Y across).  FP64 arithmetic bounds the FP64
// kernel (a warp's FP64 instruction takes the SM about 16 cycles whether one
// lane needs it or 32), so its warps are spread evenly over the SMs and kept
// full: on a 100 x 400 channel, tiles of four warps put three CTAs on some SMs
// and two on others and gave the fourth tile column 4 live lanes in 32.
// The first `duty` rows of the grid have the once-per-tile work (tile_duties).
//
// What bounds it (GB300, one launch per step, FP32 at 152 B per cell update):
//   FP32, 2048^2 with 2048 disks: memory and the particle tiles' chain of list,
//     record and band table; 111.0 us = 5.75 TB/s (127 us before: a list per
//     CTA behind a barrier, exchange sums over shared memory, f and g in planes
//     of their own, both collisions by the full moment matrices).  Without
//     particles 96 us = 6.6 TB/s.
//   16-bit storage, same case: instruction issue, 539 per warp of 32 cells
//     (880 before); FP16 92.6 us, BF16 92.7 us.
//   FP64, 100 x 400: the FP64 pipe (67 % busy); 37 us (56 before).
//   A lattice of less than a wave of warps (100 x 400 FP32): the latency of one
//     cell, 3.7 us.
template <class S, class C, int MODE, bool HOLD>
__global__ void __launch_bounds__(32 * tile_warps<C>(), sizeof(C) == 4 ? VLB_LATTICE_MIN_BLOCKS : 1)
lattice_kernel(const LatticeConst<C> K, const StepBuffers B, const ParticleArrays P, const TileLists TL, int duty) {
  constexpr int WARPS = tile_warps<C>();
  __shared__ PartTile<C> list[WARPS][TILE_CAP];
  begin_chained();
  const int lane = threadIdx.x, warp = threadIdx.y;
  if (blockIdx.y < duty) {
    const int ntiles = K.ntx * K.nty, span = duty_span(ntiles);
    tile_duties(K, P, TL, span * ((blockIdx.y * gridDim.x + blockIdx.x) * WARPS + warp), span, ntiles, lane, B.err);
    return;
  }
  const int tile_x = blockIdx.x / (TILE_Y / WARPS), tile_y = blockIdx.y - duty;
  const CellAt at = cell_at<S>(tile_x, tile_y, WARPS == 1 ? blockIdx.x % TILE_Y : warp, lane);
  if (WARPS == 1 && tile_x * TILE_X + at.bx >= K.nx) return;  // a strip beyond the lattice
  const ListHead head = list_head(TL, tile_y * K.ntx + tile_x, lane);
  lattice_cell<S, C, MODE, HOLD>(K, B, P, at, head, list[warp], K.band_stamp);
}

// Ownership of every cell at the current level, from the same raster code as
// the lattice kernel (inspection of the integer part of Sec. 2's f_s).
template <class C>
__global__ void __launch_bounds__(TILE_X * TILE_Y)
raster_dump_kernel(const LatticeConst<C> K, const ParticleArrays P, const TileLists TL, unsigned char* count,
                   int* owner, unsigned char* flag, double* fsp, unsigned* err) {
  __shared__ PartTile<C> lists[TILE_Y][TILE_CAP];
  const CellAt at = cell_at<float>(blockIdx.x, blockIdx.y, threadIdx.y, threadIdx.x);
  PartTile<C>* list = lists[threadIdx.y];
  const ListHead head = list_head(TL, at.tile_y * K.ntx + at.tile_x, at.lane);
  const int np = load_block_particles<float, C>(P, head, at, false, list);
  const int x = at.tile_x * TILE_X + at.tx, y = at.tile_y * TILE_Y + at.ty;
  if (x >= K.nx || y >= K.ny) return;
  int nown = 0, own[MAX_OWNERS] = {-1, -1, -1, -1}, cls[MAX_OWNERS] = {};
  C ofs[MAX_OWNERS] = {}, fs = C(0);
  for (int s = 0; s < np; ++s) {
    C f;
    const int c = particle_share(list[s], at.tx, at.ty, x, y, P.band, K.band_off, K.band_stamp, f, err);
    if (c == CELL_FLUID) continue;
    if (nown == MAX_OWNERS) { atomicOr(err, ERR_OWNER_OVERFLOW); break; }
    own[nown] = list[s].id;
    cls[nown] = c;
    ofs[nown++] = f;
    fs += f;
  }
  const C scale = fs > C(1) ? C(1) / fs : C(1);
  const long long c = (long long)y * K.nx + x;
  count[c] = (unsigned char)nown;
  for (int k = 0; k < MAX_OWNERS; ++k) {
    owner[4 * c + k] = own[k];
    flag[4 * c + k] = (unsigned char)cls[k];
    fsp[4 * c + k] = double(ofs[k] * scale);
  }
}
static_assert(MAX_OWNERS == 4, "four owners per cell in the dump");

// FP64 audit of the stored state: per-block sums of f (populations are
// deviations from w_i, so each cell adds 1), eps and g (macro planes 5, 6),
// then one ordered pass over the block sums.
template <class S, class C>
__global__ void audit_blocks_kernel(const LatticeConst<C> K, const typename StoredPair<S>::type* pop, const C* macro,
                                    double* scratch, unsigned* err) {
  __shared__ double red[3][256];
  double sf = 0.0, se = 0.0, sg = 0.0;
  bool bad = false;
  const long long ncell = (long long)K.nx * K.ny;
  for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < ncell;
       c += (long long)gridDim.x * blockDim.x) {
    const long long x = c % K.nx, y = c / K.nx;
    const long long cell = y * K.pitch + x;
    double cf = 1.0;
    for (int i = 0; i < 9; ++i) {
      const typename StoredPair<S>::type fg = pop[(long long)i * K.plane + cell];
      const double v = double(stored_value<C, S>(fg.x));
      const double w = double(stored_value<C, S>(fg.y));
      bad |= !(v == v) || !(w == w);
      cf += v;
    }
    sf += cf;
    se += double(macro[5 * K.plane + cell]);
    sg += double(macro[6 * K.plane + cell]);
  }
  if (bad) atomicOr(err, ERR_NAN);
  red[0][threadIdx.x] = sf;
  red[1][threadIdx.x] = se;
  red[2][threadIdx.x] = sg;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s)
      for (int q = 0; q < 3; ++q) red[q][threadIdx.x] += red[q][threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x < 3) scratch[3 * blockIdx.x + threadIdx.x] = red[threadIdx.x][0];
}

__global__ void audit_final_kernel(const double* scratch, int nblocks, double* out) {
  if (threadIdx.x >= 3) return;
  double s = 0.0;
  for (int b = 0; b < nblocks; ++b) s += scratch[3 * b + threadIdx.x];
  out[threadIdx.x] = s;
}

template <class S, class C>
static cudaError_t launch_mode(int mode, const LatticeConst<C>& K, const StepBuffers& B,
                               const ParticleArrays& P, const TileLists& TL, cudaStream_t st) {
  constexpr int WARPS = tile_warps<C>();
  const int across = K.ntx * (TILE_Y / WARPS);
  // rows of CTAs for the once-per-tile work
  const int ntiles = K.ntx * K.nty, per_cta = duty_span(ntiles) * WARPS;
  const int duty_ctas = (ntiles + per_cta - 1) / per_cta;
  const int duty = mode != MODE_MACROS && K.np > 0 ? (duty_ctas + across - 1) / across : 0;
  const dim3 grid(across, K.nty + duty), block(32, WARPS);
  const bool early = lattice_early(K.np, ntiles);
  auto go = [&](auto kernel) { return launch_chained(kernel, early, grid, block, st, K, B, P, TL, duty); };
  // kernels with the held-temperature path only where some particle is held
  // (FP64 holds nothing at the initial state, which is an equilibrium)
  if (mode == MODE_INIT)
    return sizeof(C) == 4 && K.any_held ? go(lattice_kernel<S, C, MODE_INIT, sizeof(C) == 4>)
                                        : go(lattice_kernel<S, C, MODE_INIT, false>);
  if (mode == MODE_STEP) return K.any_held ? go(lattice_kernel<S, C, MODE_STEP, true>) : go(lattice_kernel<S, C, MODE_STEP, false>);
  return K.any_held ? go(lattice_kernel<S, C, MODE_MACROS, true>) : go(lattice_kernel<S, C, MODE_MACROS, false>);
}

cudaError_t launch_lattice_f32(int mode, const LatticeConst<float>& K, const StepBuffers& B,
                               const ParticleArrays& P, const TileLists& TL, cudaStream_t st, int storage) {
  if (storage == STORE_F16) return launch_mode<__half, float>(mode, K, B, P, TL, st);
  if (storage == STORE_BF16) return launch_mode<__nv_bfloat16, float>(mode, K, B, P, TL, st);
  return launch_mode<float, float>(mode, K, B, P, TL, st);
}
cudaError_t launch_lattice_f64(int mode, const LatticeConst<double>& K, const StepBuffers& B,
                               const ParticleArrays& P, const TileLists& TL, cudaStream_t st) {
  return launch_mode<double, double>(mode, K, B, P, TL, st);
}

}  // namespace vlb

namespace vlb {

cudaError_t launch_raster_dump_f32(const LatticeConst<float>& K, const ParticleArrays& P,
                                   const TileLists& TL, unsigned char* count, int* owner,
                                   unsigned char* flag, double* fsp, unsigned* err, cudaStream_t st) {
  raster_dump_kernel<float><<<dim3(K.ntx, K.nty), dim3(TILE_X, TILE_Y), 0, st>>>(K, P, TL, count, owner, flag,
                                                                                 fsp, err);
  return cudaGetLastError();
}
cudaError_t launch_raster_dump_f64(const LatticeConst<double>& K, const ParticleArrays& P,
                                   const TileLists& TL, unsigned char* count, int* owner,
                                   unsigned char* flag, double* fsp, unsigned* err, cudaStream_t st) {
  raster_dump_kernel<double><<<dim3(K.ntx, K.nty), dim3(TILE_X, TILE_Y), 0, st>>>(K, P, TL, count, owner, flag,
                                                                                  fsp, err);
  return cudaGetLastError();
}

template <class S, class C>
static cudaError_t audit(const LatticeConst<C>& K, const void* pop, const void* macro, double* scratch,
                         int nblocks, double* out, unsigned* err, cudaStream_t st) {
  audit_blocks_kernel<S, C><<<nblocks, 256, 0, st>>>(K, static_cast<const typename StoredPair<S>::type*>(pop),
                                                     static_cast<const C*>(macro), scratch, err);
  audit_final_kernel<<<1, 32, 0, st>>>(scratch, nblocks, out);
  return cudaGetLastError();
}
cudaError_t launch_audit_f32(const LatticeConst<float>& K, const void* pop, const void* macro, double* scratch,
                             int nblocks, double* out, unsigned* err, cudaStream_t st, int storage) {
  if (storage == STORE_F16) return audit<__half, float>(K, pop, macro, scratch, nblocks, out, err, st);
  if (storage == STORE_BF16) return audit<__nv_bfloat16, float>(K, pop, macro, scratch, nblocks, out, err, st);
  return audit<float, float>(K, pop, macro, scratch, nblocks, out, err, st);
}
cudaError_t launch_audit_f64(const LatticeConst<double>& K, const void* pop, const void* macro,
                             double* scratch, int nblocks, double* out, unsigned* err, cudaStream_t st) {
  return audit<double, double>(K, pop, macro, scratch, nblocks, out, err, st);
}

// Planes of (f_i, g_i) pairs to or from as many planes f_i and g_i (the form of a
// state image), n pairs in all; W: an unsigned word of a population's size.
template <class W>
__global__ void split_plane_kernel(W* __restrict__ pairs, W* __restrict__ f, W* __restrict__ g, long long n, int join) {
  for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x) {
    if (join) {
      pairs[2 * c] = f[c];
      pairs[2 * c + 1] = g[c];
    } else {
      f[c] = pairs[2 * c];
      g[c] = pairs[2 * c + 1];
    }
  }
}
template <class W>
static cudaError_t split(void* pairs, void* f, void* g, long long n, bool join, cudaStream_t st) {
  split_plane_kernel<W><<<608, 256, 0, st>>>(static_cast<W*>(pairs), static_cast<W*>(f), static_cast<W*>(g), n, join);
  return cudaGetLastError();
}
cudaError_t launch_split_plane(void* pairs, void* f, void* g, long long n, size_t bytes, bool join, cudaStream_t st) {
  if (bytes == 8) return split<unsigned long long>(pairs, f, g, n, join, st);
  if (bytes == 4) return split<unsigned>(pairs, f, g, n, join, st);
  return split<unsigned short>(pairs, f, g, n, join, st);
}

}  // namespace vlb
