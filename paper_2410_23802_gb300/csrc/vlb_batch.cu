// Batched stepping of many cases (vlb_step_batch), in two forms: per step a
// particle kernel over the particles of every case and a lattice kernel of
// one CTA per tile of any case (form 0); or one persistent launch per step
// that takes the tiles and then the next level's particle steps from a
// device counter, each particle step after a bounded wait for its case's
// tiles (form 1).
#include <atomic>

#include "vlb_lattice_held.cuh"
#include "vlb_particle_body.cuh"

namespace vlb {

// Part `part` of tile t of case d at step k of a batch call.
template <class S, class C, bool HOLD>
__device__ __forceinline__ void batch_tile(const BatchLattice<C>& d, int t, int part, int lane, int k,
                                           PartTile<C>* list) {
  const int par = k & 1;
  const StepBuffers& B = d.B[d.cur ^ par];
  const int tile_y = t / d.K.ntx, tile_x = t - tile_y * d.K.ntx;
  const CellAt at = cell_at<S>(tile_x, tile_y, part, lane);
  if (tile_warps<C>() == 1 && tile_x * TILE_X + at.bx >= d.K.nx) return;  // a strip beyond the lattice
  const ListHead head = list_head(d.TL[1 - (d.tl ^ par)], t, lane);
  lattice_cell<S, C, MODE_STEP, HOLD>(d.K, B, d.P, at, head, list, band_stamp_after(d.stamp, k + 1));
}
// Storage of a launch whose cases do not share one: each tile takes the code
// of its case's.  A round of served cases of both kinds then takes one launch
// where two small ones followed each other (10 cases of 0.94 M cells, 300
// steps: 19.7 -> 18.5 ms; 6 cases of 0.11 M, 200 steps: 5.7 -> 4.8; 40 cases of
// 6.9 M, 100 steps, where either fills the GPU: 70.1 -> 69.8).
struct AnyStorage {};

// Step k of a batch call (vlb_step_batch) over the tiles of many cases, one
// CTA per tile (FP64: per strip of a tile): the tile's case descriptor is
// copied to shared memory, then the single-case code (vlb_lattice_body.cuh)
// runs on it.  The first `duty` CTAs have the once-per-tile work, a lane per
// tile (tile_duties).
template <class S, class C, bool HOLD>
__global__ void __launch_bounds__(32 * tile_warps<C>(), sizeof(C) == 4 ? VLB_LATTICE_MIN_BLOCKS : 1)
lattice_batch_kernel(const BatchLattice<C>* __restrict__ cases, const int* __restrict__ tile_case, int ntiles, int k,
                     int duty) {
  constexpr int WARPS = tile_warps<C>(), PARTS = TILE_Y / WARPS;
  __shared__ PartTile<C> list[WARPS][TILE_CAP];
  __shared__ BatchLattice<C> d;
  static_assert(sizeof(BatchLattice<C>) % 4 == 0, "descriptor copied as words");
  begin_chained();
  const int lane = threadIdx.x, warp = threadIdx.y, par = k & 1;
  if (blockIdx.x < duty) {
    const int span = duty_span(ntiles), first = span * (blockIdx.x * WARPS + warp), t = first + lane;
    int n = 0, c = 0;
    if (lane < span && t < ntiles) {
      c = tile_case[t];
      const BatchLattice<C>& e = cases[c];
      const TileLists& TL = e.TL[1 - (e.tl ^ par)];
      n = min(TL.count[t - e.tile0], TILE_CAP);
      TL.next_count[t - e.tile0] = 0;
    }
    for (unsigned m = __ballot_sync(0xffffffffu, n > 1); m; m &= m - 1) {
      const int l = __ffs(m) - 1;
      const BatchLattice<C>& e = cases[__shfl_sync(0xffffffffu, c, l)];
      contact_pairs(e.K, e.P, e.TL[1 - (e.tl ^ par)].ids, __shfl_sync(0xffffffffu, n, l), first + l - e.tile0, lane,
                    e.B[0].err);
    }
    return;
  }
  const int block = blockIdx.x - duty, tile = block / PARTS, part = WARPS == 1 ? block % PARTS : warp;
  {
    const int* src = reinterpret_cast<const int*>(cases + tile_case[tile]);
    int* dst = reinterpret_cast<int*>(&d);
    for (int w = 32 * warp + lane; w < (int)(sizeof(d) / 4); w += 32 * WARPS) dst[w] = src[w];
  }
  __syncthreads();
  if constexpr (!std::is_same<S, AnyStorage>::value) {
    batch_tile<S, C, HOLD>(d, tile - d.tile0, part, lane, k, list[warp]);
  } else if (d.storage == STORE_F16) {
    batch_tile<__half, C, HOLD>(d, tile - d.tile0, part, lane, k, list[warp]);
  } else if (d.storage == STORE_BF16) {
    batch_tile<__nv_bfloat16, C, HOLD>(d, tile - d.tile0, part, lane, k, list[warp]);
  } else {
    batch_tile<float, C, HOLD>(d, tile - d.tile0, part, lane, k, list[warp]);
  }
}

// The same over the particles of many cases, step k of a batch call; `group`
// (case, particle) items per CTA (see step_group).  HELD: some case of the
// batch has held particles.
template <bool HELD>
__global__ void __launch_bounds__(STEP_THREADS)
    particle_step_batch_kernel(const BatchParticles* __restrict__ cases, const int2* __restrict__ items, int nitems,
                               int k, int group) {
  __shared__ StepShared sh;
  begin_chained();
  const int i0 = blockIdx.x * group;
  step_group<HELD>(min(group, nitems - i0), [&](int s) {
    const int2 it = items[i0 + s];
    const BatchParticles& d = cases[it.x];
    return StepRef{&d.c, &d.P, &d.TL[1 - (d.tl ^ (k & 1))], d.err, it.y, band_stamp_after(d.stamp, k + 1)};
  }, sh);
}
// The ellipses' band tables of step k (of step *kdev when kdev is given).
__global__ void __launch_bounds__(32 * ELL_WARPS)
    particle_ellipse_batch_kernel(const BatchParticles* __restrict__ cases, const int2* __restrict__ items, int blocks,
                                  int k, const int* __restrict__ kdev) {
  __shared__ int s_queue[ELL_WARPS][32];
  begin_chained();
  if (kdev) k = *kdev;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x / blocks, by = (blockIdx.x - i * blocks) * ELL_WARPS + warp;
  const int2 it = items[i];
  const BatchParticles& d = cases[it.x];
  if (by >= 2 * d.c.band_off + 1) return;  // the whole warp
  ellipse_row(d.c, d.P, it.y, band_stamp_after(d.stamp, k + 1), by, lane, s_queue[warp]);
}

template <class S, class C>
static cudaError_t launch_batch(const BatchLattice<C>* cases, const int* tile_case, int ntiles, int k, int particles,
                                bool held, cudaStream_t st) {
  constexpr bool HOLD = !std::is_same<S, AnyStorage>::value;  // (held lattices of one launch share their storage)
  if (ntiles == 0) return cudaSuccess;
  constexpr int WARPS = tile_warps<C>();
  const dim3 block(32, WARPS);
  const int per_cta = duty_span(ntiles) * WARPS, duty = (ntiles + per_cta - 1) / per_cta;
  const unsigned grid = (unsigned)duty + (unsigned)ntiles * (TILE_Y / WARPS);
  return launch_chained(held ? lattice_batch_kernel<S, C, HOLD> : lattice_batch_kernel<S, C, false>,
                        lattice_early(particles, ntiles), dim3(grid), block, st, cases, tile_case, ntiles, k, duty);
}

cudaError_t launch_lattice_batch_f32(const BatchLattice<float>* cases, const int* tile_case, int ntiles, int k,
                                     int storage, int particles, bool held, cudaStream_t st) {
  if (storage == STORE_ANY) return launch_batch<AnyStorage, float>(cases, tile_case, ntiles, k, particles, held, st);
  if (storage == STORE_F16) return launch_batch<__half, float>(cases, tile_case, ntiles, k, particles, held, st);
  if (storage == STORE_BF16) return launch_batch<__nv_bfloat16, float>(cases, tile_case, ntiles, k, particles, held, st);
  return launch_batch<float, float>(cases, tile_case, ntiles, k, particles, held, st);
}
cudaError_t launch_lattice_batch_f64(const BatchLattice<double>* cases, const int* tile_case, int ntiles, int k,
                                     int particles, bool held, cudaStream_t st) {
  return launch_batch<double, double>(cases, tile_case, ntiles, k, particles, held, st);
}

cudaError_t launch_ellipse_batch(const BatchParticles* cases, const BatchEllipses& ell, int k, const int* kdev,
                                 cudaStream_t st) {
  if (ell.n == 0) return cudaSuccess;
  const int blocks = (ell.rows + ELL_WARPS - 1) / ELL_WARPS;
  const dim3 grid((unsigned)(blocks * ell.n)), block(32 * ELL_WARPS);
  if (!kdev) return launch_chained(particle_ellipse_batch_kernel, true, grid, block, st, cases, ell.items, blocks, k, kdev);
  // (behind a persistent launch, captured into a graph: an ordinary launch)
  particle_ellipse_batch_kernel<<<grid, block, 0, st>>>(cases, ell.items, blocks, k, kdev);
  return cudaGetLastError();
}
cudaError_t launch_particle_step_batch(const BatchParticles* cases, const int2* items, int nitems, int k, bool held,
                                       const BatchEllipses& ell, cudaStream_t st) {
  if (nitems == 0) return cudaSuccess;
  const int group = step_group_size(nitems);
  const cudaError_t e = launch_chained(held ? particle_step_batch_kernel<true> : particle_step_batch_kernel<false>, true,
                                       dim3((unsigned)((nitems + group - 1) / group)), dim3(STEP_THREADS), st, cases, items, nitems, k, group);
  return e != cudaSuccess ? e : launch_ellipse_batch(cases, ell, k, nullptr, st);
}

// ---- the persistent form ------------------------------------------------------

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ int load_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// One thread waits until *count >= target: true when it got there, false when
// limit_ns passed first (or, as a backstop should the timer stall, after an
// iteration count that takes longer than that limit at any sleep length).
__device__ bool wait_count(const int* count, int target, long long limit_ns) {
  if (load_acquire(count) >= target) return true;
  const unsigned long long t0 = global_ns();
  const long long max_iter = 4 * (limit_ns / 1024) + 4096;
  unsigned ns = 32;
  for (long long it = 0; it < max_iter; ++it) {
    __nanosleep(ns);
    if (load_acquire(count) >= target) return true;
    if ((long long)(global_ns() - t0) > limit_ns) return false;
    ns = ns < 1024u ? 2u * ns : 1024u;
  }
  return false;
}

// Particle item i of a persistent launch (one warp): the particle step of
// level kn, after the last tile of its case (whose exchange sums, contact
// partners and cleared list buffer it reads).  Inlined: as a call it cost
// the tile path more (spills around the call) than its own FP64 code does.
template <class C, bool HOLD>
__device__ __forceinline__ void persistent_particle(const PersistentBatch<C>& A, int i, int kn, int* queue) {
  const int lane = threadIdx.x & 31;
  if (i >= A.npitems) return;
  const int2 it = A.pitems[i];
  const BatchParticles& pd = A.pcases[A.case_handle[it.x]];
  int ok = 1;
  if (lane == 0) {
    const LatticeConst<C>& K = A.cases[it.x].K;
    ok = wait_count(A.done + it.x, K.ntx * K.nty + (it.x == A.stuck_case ? 1 : 0), A.wait_ns);
    if (!ok) atomicOr(pd.err, ERR_TIMEOUT);
  }
  ok = __shfl_sync(0xffffffffu, ok, 0);
  if (!ok) return;  // the whole warp
  __syncwarp();     // what lane 0 waited for is visible to every lane
  const UpdateLane u = update_position(pd.c, pd.P, it.y, lane, lane < 4, pd.err);
  RasterRec rq;
  record_constants(pd.P, it.y, u.R, u.Rb, rq);
  update_velocity(pd.c, pd.P, it.y, lane, lane < 4, u, rq, pd.err);
  __syncwarp();  // the record and tile range are visible to every lane
  band_one<HOLD>(pd.c, pd.P, pd.TL[1 - (pd.tl ^ (kn & 1))], pd.err, it.y, band_stamp_after(pd.stamp, kn + 1), queue, lane);
}

// Tiles per work chunk of the persistent launch: a CTA takes the next chunk
// from the counter (one atomic round trip, which its first warp waits for)
// only after its last one, so the trip is paid once per chunk.
#ifndef VLB_BATCH_CHUNK
#define VLB_BATCH_CHUNK 4
#endif
constexpr int BATCH_CHUNK = VLB_BATCH_CHUNK;

// The persistent batched step (see PersistentBatch).  Work items: tiles
// 0 .. ntiles - 1, then particle groups ntiles + m (particles 4m .. 4m + 3 of
// the launch, one per warp).  Chunk j of the counter is tiles
// BATCH_CHUNK j .. BATCH_CHUNK (j + 1) - 1 while j < tchunks, else the one
// particle group j - tchunks.  A CTA keeps its case's descriptor in shared
// memory while consecutive tiles share it.  The loop's state lives in shared
// memory.
template <class S, class C, bool HOLD>
__global__ void __launch_bounds__(TILE_X * TILE_Y, sizeof(C) == 4 ? VLB_LATTICE_MIN_BLOCKS : 1)
lattice_persistent_kernel(const __grid_constant__ PersistentBatch<C> A) {
  constexpr int NWARPS = TILE_X * TILE_Y / 32;
  union Shared {
    PartTile<C> list[NWARPS][TILE_CAP];  // the particles of each warp's block
    int queue[NWARPS][BAND_QUEUE];       // the band queues of a particle group
  };
  __shared__ Shared sh;
  __shared__ BatchLattice<C> d;
  __shared__ int s_item, s_end, s_case, s_k, s_pend, s_pend_case;
  static_assert(sizeof(BatchLattice<C>) % 4 == 0, "descriptor copied as words");
  const int tid = threadIdx.y * TILE_X + threadIdx.x;
  const int tchunks = (A.ntiles + BATCH_CHUNK - 1) / BATCH_CHUNK;
  const int nitems = A.ntiles + (A.with_particles ? (A.npitems + NWARPS - 1) / NWARPS : 0);
  // (thread 0) publish the finished tiles of one case: a fence, then one add
  auto publish = [&]() {
    if (s_pend > 0) {
      __threadfence();
      atomicAdd(A.done + s_pend_case, s_pend);
      s_pend = 0;
    }
  };
  auto take_chunk = [&]() {
    const int j = atomicAdd(&A.ctl->next, 1);
    s_item = j < tchunks ? j * BATCH_CHUNK : A.ntiles + (j - tchunks);
    s_end = j < tchunks ? min(A.ntiles, (j + 1) * BATCH_CHUNK) : s_item + 1;
  };
  if (tid == 0) {
    take_chunk();
    s_case = -1;
    s_k = A.ctl->k;
    s_pend = 0;
    s_pend_case = -1;
  }
  __syncthreads();
  int item = s_item, end = s_end;
  for (;;) {
    if (item >= nitems) break;
    if (item < A.ntiles) {
      const int c = A.tile_case[item];
      if (c != s_case) {  // (the barrier ending the previous item keeps d free)
        const int* src = reinterpret_cast<const int*>(A.cases + c);
        int* dst = reinterpret_cast<int*>(&d);
        for (int w = tid; w < (int)(sizeof(d) / 4); w += TILE_X * TILE_Y) dst[w] = src[w];
        __syncthreads();
        if (tid == 0) s_case = c;
      }
      const int par = s_k & 1;
      const StepBuffers& B = d.B[d.cur ^ par];
      const TileLists& TL = d.TL[1 - (d.tl ^ par)];
      const int lt = item - d.tile0;
      const int tile_y = lt / d.K.ntx, tile_x = lt - tile_y * d.K.ntx;
      const int lane = threadIdx.x, warp = threadIdx.y;
      const CellAt at = cell_at<S>(tile_x, tile_y, warp, lane);
      const ListHead head = list_head(TL, lt, lane);
      lattice_cell<S, C, MODE_STEP, HOLD>(d.K, B, d.P, at, head, sh.list[warp], band_stamp_after(d.stamp, s_k + 1));
      if (warp == 0) {
        if (lane == 0) TL.next_count[lt] = 0;  // the next particle step fills the other list buffer
        if (head.count > 1) contact_pairs(d.K, d.P, TL.ids, head.count, lt, lane, B.err);
      }
      __syncthreads();  // every thread's stores and sums of this tile are issued; sh and d are free
      if (tid == 0 && A.with_particles && d.K.np > 0) {
        // counted now, published (fence + add) when the case changes or the
        // chunk ends, so that a chunk of one case pays one fence
        if (s_pend_case != s_case) {
          publish();
          s_pend_case = s_case;
        }
        ++s_pend;
      }
    } else {
      persistent_particle<C, HOLD>(A, (item - A.ntiles) * NWARPS + (tid >> 5), s_k + 1, sh.queue[tid >> 5]);
      __syncthreads();  // the band queues are free
    }
    if (item + 1 < end) {  // the next tile of this chunk (every thread knows it)
      ++item;
      continue;
    }
    if (tid == 0) {
      publish();
      take_chunk();
    }
    __syncthreads();
    item = s_item;
    end = s_end;
  }
  if (tid == 0) {
    __threadfence();
    if (atomicAdd(&A.ctl->exited, 1) == (int)gridDim.x - 1) {
      // the last CTA: every other one has left, so nothing reads these now
      for (int c = 0; c < A.ncases; ++c) A.done[c] = 0;
      A.ctl->next = 0;
      A.ctl->exited = 0;
      A.ctl->k = s_k + 1;
      __threadfence();
    }
  }
}

template <class S, class C, bool HOLD>
static int resident_ctas(int device) {
  // per device, filled by the first call (calls from several host threads
  // may race to fill it; they store the same value)
  static std::atomic<int> cached[64];
  if (device < 0 || device >= 64) return 0;
  const int known = cached[device].load(std::memory_order_relaxed);
  if (known > 0) return known;
  int nb = 0, nsm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, lattice_persistent_kernel<S, C, HOLD>, TILE_X * TILE_Y, 0) !=
          cudaSuccess ||
      cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, device) != cudaSuccess)
    return 0;
  cached[device].store(nb * nsm, std::memory_order_relaxed);
  return nb * nsm;
}

int persistent_grid(int device, bool f64, int storage, bool held) {
  if (f64) return held ? resident_ctas<double, double, true>(device) : resident_ctas<double, double, false>(device);
  if (storage == STORE_F16)
    return held ? resident_ctas<__half, float, true>(device) : resident_ctas<__half, float, false>(device);
  if (storage == STORE_BF16)
    return held ? resident_ctas<__nv_bfloat16, float, true>(device)
                : resident_ctas<__nv_bfloat16, float, false>(device);
  return held ? resident_ctas<float, float, true>(device) : resident_ctas<float, float, false>(device);
}

template <class S, class C>
static cudaError_t launch_persistent(const PersistentBatch<C>& A, int grid, bool held, cudaStream_t st) {
  const int nwarps = TILE_X * TILE_Y / 32;
  const int total = (A.ntiles + BATCH_CHUNK - 1) / BATCH_CHUNK +
                    (A.with_particles ? (A.npitems + nwarps - 1) / nwarps : 0);
  grid = grid < total ? grid : total;
  if (grid <= 0) return cudaSuccess;
  const dim3 block(TILE_X, TILE_Y);
  if (held) lattice_persistent_kernel<S, C, true><<<(unsigned)grid, block, 0, st>>>(A);
  else lattice_persistent_kernel<S, C, false><<<(unsigned)grid, block, 0, st>>>(A);
  return cudaGetLastError();
}

cudaError_t launch_lattice_persistent_f32(const PersistentBatch<float>& A, int grid, int storage, bool held,
                                          cudaStream_t st) {
  if (storage == STORE_F16) return launch_persistent<__half, float>(A, grid, held, st);
  if (storage == STORE_BF16) return launch_persistent<__nv_bfloat16, float>(A, grid, held, st);
  return launch_persistent<float, float>(A, grid, held, st);
}
cudaError_t launch_lattice_persistent_f64(const PersistentBatch<double>& A, int grid, bool held, cudaStream_t st) {
  return launch_persistent<double, double>(A, grid, held, st);
}

}  // namespace vlb
