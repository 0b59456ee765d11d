// Device code of the particle step (Sec. 2.3), shared by the single-case
// kernels (vlb_particles.cu) and the batched ones (vlb_batch.cu).
//
// Particle kernels (Sec. 2.3).
//
//   particle_step (one launch per time step): for each particle
//     update (FP64, one lane per component): F_MES, T_MES of Eq. 28 from the
//       integer accumulators the lattice kernel filled (then cleared); the
//       inside-fluid force and torque of Eq. 29 with backward differences;
//       the short-range contact force; Eqs. 26 and 30 by forward Euler; the
//       raster record and the tile range of the new position;
//     lists: appends the particle to the tile lists of its range (the lattice
//       kernel ranks each list by id and finds the contact partners of the
//       level);
//     band table: classes and areas of the cells near the boundary (FP32 for a
//       disk; an ellipse's table is filled in FP64 by particle_ellipse_kernel).
//   particle_range, particle_band: the same for the initial state.
#pragma once

#include <math.h>

#include "vlb_common.cuh"
#include "vlb_kernels.h"
#include "vlb_raster.cuh"
#include "vlb_raster_held.cuh"

namespace vlb {

// First tile and number of tiles (of T cells) covered along an axis of n cells by
// [X - R - m, X + R + m], none outside the domain; in FP32: the margin m >= 2
// cells absorbs the rounding, and the range is computed once per step and
// stored, so every use of it agrees.
__device__ __forceinline__ int2 tile_span(const ParticleConst& c, double X, double R, int n, int T) {
  const float Xf = float(X), e = add_rn(float(R), float(c.margin));
  const int c0 = max((int)floorf(add_rn(Xf, -e)), 0), c1 = min((int)floorf(add_rn(Xf, e)), n - 1);
  return c1 < c0 ? make_int2(0, 0) : make_int2(c0 / T, c1 / T - c0 / T + 1);
}
// The tiles of a particle along both axes (tx0, ty0, ntx, nty).
__device__ __forceinline__ int4 tile_range(const ParticleConst& c, double X, double Y, double R) {
  const int2 x = tile_span(c, X, R, c.nx, TILE_X), y = tile_span(c, Y, R, c.ny, TILE_Y);
  return x.y == 0 || y.y == 0 ? make_int4(0, 0, 0, 0) : make_int4(x.x, y.x, x.y, y.y);
}

// Raster record of particle p at centre (X, Y) with velocity (ux, uy, om);
// R its radius (an ellipse's semi-major axis), Rb its semi-minor axis: the
// quick test's bounds are the circumscribed and inscribed circles.
__device__ __forceinline__ void write_record(const ParticleArrays& P, int p, double X, double Y, double R, double Rb,
                                             double ux, double uy, double om, float lam_s, float T0) {
  RasterRec q;
  const double Q = double(1 << QBITS);
  q.xi = (int)floor(X);
  q.yi = (int)floor(Y);
  q.qfx = (int)(__double2ll_rn(X * Q) - (long long)q.xi * (1ll << QBITS));
  q.qfy = (int)(__double2ll_rn(Y * Q) - (long long)q.yi * (1ll << QBITS));
  const long long rq = __double2ll_rn(R * Q);
  q.rq2 = rq * rq;
  const double fx = X - double(q.xi), fy = Y - double(q.yi);
  q.xfh = float(fx); q.xfl = float(fx - double(q.xfh));
  q.yfh = float(fy); q.yfl = float(fy - double(q.yfh));
  q.r = float(R);
  q.far2 = float((R + 0.75) * (R + 0.75));
  q.near2 = Rb > 0.75 ? float((Rb - 0.75) * (Rb - 0.75)) : -1.0f;
  q.ux = float(ux); q.uxl = float(ux - double(q.ux));
  q.uy = float(uy); q.uyl = float(uy - double(q.uy));
  q.om = float(om);
  q.lam_s = lam_s;
  q.T0 = T0;
  P.rec[p] = q;
}


// ---- the update, one lane per component --------------------------------------
// Four lanes of a warp hold one particle: lane k = 0, 1 its x and y motion, 2
// its rotation, 3 nothing.  An FP64 instruction costs a warp the same whether
// one lane needs it or all do (the FP64 pipe takes it in about 16 cycles and
// its result returns after about 50), and the three components follow the same
// formulas, so the chain a particle waits for is about a third of the
// instructions of one lane doing all three in turn.  Every operation is
// rounded on its own or an explicit fused one, so that all kernels that
// contain this code give the same bits.
struct UpdateLane {
  int k;
  double at, at1, vel, prev;         // position, new position, velocity, previous velocity (or angle, rates)
  double R, Rb;
  unsigned long long acc0, acc1;     // exchange sums, taken and cleared
  int cell, qf;                      // raster record: cell, 2^-20 offset,
  float fh, fl;                      // fraction as hi + lo
  int t0, nt;                        // first tile and tiles of the range along this axis
};

// New position, its raster coordinates and tile range (lanes k = 0, 1; all 32
// lanes take part).
__device__ __forceinline__ UpdateLane update_position(const ParticleConst& c, const ParticleArrays& P, int p, int lane,
                                                      bool on, unsigned* err) {
  UpdateLane u;
  u.k = lane & 3;
  const int k = u.k;
  u.at = (k == 0 ? P.x : (k == 1 ? P.y : P.theta))[p];
  u.vel = (k == 0 ? P.ux : (k == 1 ? P.uy : P.om))[p];
  u.prev = (k == 0 ? P.ux_prev : (k == 1 ? P.uy_prev : P.om_prev))[p];
  u.R = P.r[p];
  u.Rb = P.rb[p];
  // momentum-exchange force and torque of the current level (Eq. 28) plus the
  // particle-particle contact forces of that level: the lattice kernel's
  // integer accumulators, read and cleared for the next level (at the L2 with
  // atomic exchanges, so that a particle step inside a lattice launch never
  // reads an L1 line this SM loaded before other SMs added to the words)
  u.acc0 = u.acc1 = 0ull;
  if (on && k < 3) {
    unsigned long long* acc = P.mes + 6 * (long long)p + 2 * k;
    u.acc0 = atomicExch(acc, 0ull);
    u.acc1 = atomicExch(acc + 1, 0ull);
  }
  u.at1 = __dadd_rn(u.at, u.vel);
  u.cell = u.qf = u.t0 = u.nt = 0;
  u.fh = u.fl = 0.0f;
  if (k < 2) {
    const int n = k == 0 ? c.nx : c.ny;
    const double X = u.at1;
    bool bad = !(X >= 0.0 && X <= double(n));
    if (k == 0 ? c.per_x : c.per_y)
      bad |= __dadd_rn(__dadd_rn(X, -u.R), -1.0) < 0.0 || __dadd_rn(__dadd_rn(X, u.R), 1.0) > double(n);
    if (on && bad) atomicOr(err, ERR_OUT_OF_DOMAIN);
    u.cell = __double2int_rd(X);
    u.qf = (int)(__double2ll_rn(__dmul_rn(X, double(1 << QBITS))) - (long long)u.cell * (1ll << QBITS));
    const double f = __dadd_rn(X, -double(u.cell));
    u.fh = float(f);
    u.fl = float(__dadd_rn(f, -double(u.fh)));
    const int2 span = tile_span(c, X, u.R, n, k == 0 ? TILE_X : TILE_Y);
    u.t0 = span.x;
    u.nt = span.y;
  }
  // outside along one axis: no tiles at all
  const int other = __shfl_xor_sync(0xffffffffu, u.nt, 1);
  if (other == 0 || u.nt == 0) u.t0 = u.nt = 0;
  return u;
}

// The particle's constants of its raster record.
__device__ __forceinline__ void record_constants(const ParticleArrays& P, int p, double R, double Rb, RasterRec& q) {
  const long long rq = __double2ll_rn(__dmul_rn(R, double(1 << QBITS)));
  q.rq2 = rq * rq;
  const double Ro = __dadd_rn(R, 0.75), Ri = __dadd_rn(Rb, -0.75);
  q.r = float(R);
  q.far2 = float(__dmul_rn(Ro, Ro));
  q.near2 = Rb > 0.75 ? float(__dmul_rn(Ri, Ri)) : -1.0f;
  q.lam_s = float(P.lam_s[p]);
  q.T0 = float(P.T0[p]);
}

// The particle's force, velocity, state arrays and raster record (rq: its
// constants; all 32 lanes take part).
__device__ __forceinline__ void update_velocity(const ParticleConst& c, const ParticleArrays& P, int p, int lane,
                                                bool on, const UpdateLane& u, const RasterRec& rq, unsigned* err) {
  const int k = u.k;
  const double* kp = P.pk + 8 * (long long)p;  // 1/M, 1/I, M_in, I_in, body factor, wall factor
  const double inv_m = kp[k == 2 ? 1 : 0], m_in = kp[k == 2 ? 3 : 2], body = kp[4], wall = kp[5];
  // the total force or torque: word 0 in units of 2^-40, word 1 of 2^-104
  const double Fm = __fma_rn((double)(long long)u.acc0, 1.0 / MES_SCALE_HI,
                             __dmul_rn((double)u.acc1, 1.0 / (MES_SCALE_HI * MES_SCALE_LO)));
  // wall contact forces: walls x-, x+ (lane 0), y-, y+ (lane 1), none on open
  // sides; an ellipse meets a wall with its extent along the wall's normal
  // (reading R13)
  double ext = u.R;
  const double theta = __shfl_sync(0xffffffffu, u.at, lane | 2);
  if (u.Rb != u.R) {
    double sn, cs;
    sincos(theta, &sn, &cs);
    const double a = __dmul_rn(u.R, k == 0 ? cs : sn), b = __dmul_rn(u.Rb, k == 0 ? sn : cs);
    ext = sqrt(__fma_rn(a, a, __dmul_rn(b, b)));
  }
  double Fc = 0.0;
  if (k < 2 && !(k == 0 ? c.per_x : c.per_y)) {
    const double reach = __fma_rn(2.0, ext, c.zeta);
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      if (c.outflow[2 * k + side]) continue;
      const double dist = side == 0 ? u.at : __dadd_rn(double(k == 0 ? c.nx : c.ny), -u.at);
      const double gap = __fma_rn(-2.0, dist, reach);
      if (gap <= 0.0) continue;
      const double gz = __dmul_rn(gap, c.inv_zeta);
      const double mag = __dmul_rn(__dmul_rn(wall, gz), gz);
      Fc = __dadd_rn(Fc, side == 0 ? mag : -mag);
    }
  }
  // Eqs. 26, 29, 30: F_c = F_MES - F_in + (rho_s - rho_f) V g + F_contact
  // (F_MES carries the particle-particle part of F_contact)
  double F = __fma_rn(m_in, __dadd_rn(u.vel, -u.prev), Fm);
  if (k < 2) F = __dadd_rn(__fma_rn(body, k == 0 ? c.gx : c.gy, F), Fc);
  const double vel1 = __fma_rn(F, inv_m, u.vel);
  const double other = __shfl_xor_sync(0xffffffffu, vel1, 1);
  const int cell_y = __shfl_down_sync(0xffffffffu, u.t0, 1), nt_y = __shfl_down_sync(0xffffffffu, u.nt, 1);
  if (!on) return;
  if (k == 0 && !(__fma_rn(vel1, vel1, __dmul_rn(other, other)) <= 0.25)) atomicOr(err, ERR_TOO_FAST);
  RasterRec* rec = P.rec + p;
  if (k < 3) {
    (k == 0 ? P.x : (k == 1 ? P.y : P.theta))[p] = u.at1;
    (k == 0 ? P.ux_prev : (k == 1 ? P.uy_prev : P.om_prev))[p] = u.vel;
    (k == 0 ? P.ux : (k == 1 ? P.uy : P.om))[p] = vel1;
    (k == 0 ? P.fcx : (k == 1 ? P.fcy : P.tc))[p] = F;
    const float vh = float(vel1), vl = float(__dadd_rn(vel1, -double(vh)));
    if (k == 0) {
      rec->xi = u.cell; rec->qfx = u.qf; rec->xfh = u.fh; rec->xfl = u.fl;
      rec->ux = vh; rec->uxl = vl;
      P.prange[p] = make_int4(u.t0, cell_y, u.nt, nt_y);
    } else if (k == 1) {
      rec->yi = u.cell; rec->qfy = u.qf; rec->yfh = u.fh; rec->yfl = u.fl;
      rec->uy = vh; rec->uyl = vl;
    } else {
      rec->om = vh;
    }
  } else {
    rec->rq2 = rq.rq2;
    rec->r = rq.r; rec->far2 = rq.far2; rec->near2 = rq.near2;
    rec->lam_s = rq.lam_s; rec->T0 = rq.T0;
    P.nbr_count[p] = 0;  // the lattice kernel of this step lists the next partners
  }
}

// ---- band tables of disks -------------------------------------------------------
// Exact classes and areas (Sec. 2) of the cells whose centre lies in the band
// |d - R| < 0.75 of a disk, i.e. the cells the lattice kernel's quick test
// leaves open.  Results go to the particle's band table with the level's
// stamp.

// Row by of a particle's box: the cells of the row that can be in the band
// (|x - X| between sqrt((R - 0.75)^2 - dy^2) and sqrt((R + 0.75)^2 - dy^2),
// widened by half a cell on either side, far more than the FP32 error of these
// bounds) as runs [a0, a0 + na), [b0, b0 + nb) of bx.
struct BandRow {
  int a0, na, b0, nb;
};
__device__ __forceinline__ BandRow band_row(const RasterRec& rc, int off, int ny, int by) {
  const int bw = 2 * off + 1;
  const float cx = float(off) + rc.xfh, cy = float(off) + rc.yfh;  // centre in box coordinates
  const float ro = rc.r + 0.75f, ri = rc.near2 > 0.0f ? sqrtf(rc.near2) : 0.0f;
  const int y = rc.yi - off + by;
  int a0 = 0, a1 = -1, b0 = 0, b1 = -1;
  if (y >= 0 && y < ny) {
    const float dy = (float(by) + 0.5f) - cy;
    const float oa = ro * ro - dy * dy;
    if (oa > -1.0f) {  // the row meets the widened outer circle
      const float wa = sqrtf(fmaxf(oa, 0.0f)) + 0.5f;
      const float ib = ri * ri - dy * dy;
      const float wb = (ri > 0.0f && ib > 0.0f) ? sqrtf(ib) - 0.5f : 0.0f;
      // cell bx is a candidate when |bx + 0.5 - cx| lies in [wb, wa]
      a0 = max(0, (int)ceilf(cx - wa - 0.5f));
      b1 = min(bw - 1, (int)floorf(cx + wa - 0.5f));
      if (wb > 0.0f) {
        a1 = (int)floorf(cx - wb - 0.5f);
        b0 = (int)ceilf(cx + wb - 0.5f);
      } else {  // one run through the middle
        a1 = b1;
        b0 = 0;
        b1 = -1;
      }
      a1 = min(a1, bw - 1);
      b0 = max(b0, 0);
    }
  }
  BandRow r;
  r.a0 = a0;
  r.na = max(a1 - a0 + 1, 0);
  r.b0 = b0;
  r.nb = max(b1 - b0 + 1, 0);
  return r;
}
// The lattice kernel's quick test of lattice cell (x, y), in the coordinates
// of the cell's own tile (as that kernel takes it).
__device__ __forceinline__ bool in_band(const RasterRec& rc, int x, int y) {
  const int tx = x % TILE_X, ty = y % TILE_Y;
  float xh, xl, yh, yl;
  tile_coordinate(rc.xi - (x - tx), rc.xfh, rc.xfl, xh, xl);
  tile_coordinate(rc.yi - (y - ty), rc.yfh, rc.yfl, yh, yl);
  return quick_class_at(tx, ty, xh, xl, yh, yl, rc.far2, rc.near2) == CELL_BAND;
}
// Entry (bx, by) of a particle's table.  HELD: compiled with the areas of
// lattices with held particles, taken where `held` says so (in the kernels of
// all other lattices they would cost registers).
template <bool HELD>
__device__ __forceinline__ void band_fill(const RasterRec& rc, int2* table, int off, int stamp, float i2R, int bx,
                                          int by, int held) {
  float f;
  const int cls = HELD && held ? held_band_cell(rc, rc.xi - off + bx, rc.yi - off + by, f)
                               : disk_band_cell(rc, bx - off, by - off, i2R, f);
  table[(long long)by * (2 * off + 1) + bx] = make_int2(cls | (stamp << 2), __float_as_int(f));
}
__device__ __forceinline__ int2* band_table(const ParticleArrays& P, int off, int p) {
  const long long bw = 2 * off + 1;
  return P.band + (long long)p * bw * bw;
}

// A particle's tile lists, one lane of a warp per tile.
__device__ __forceinline__ void append_to_tiles(const TileLists& TL, int ntx, int4 rg, int p, int lane, unsigned* err) {
  const int n = rg.z * rg.w;
  for (int t = lane; t < n; t += 32) {
    const int ty = t / rg.z, tx = t - ty * rg.z;
    const int tile = (rg.y + ty) * ntx + (rg.x + tx);
    const int slot = atomicAdd(&TL.count[tile], 1);
    if (slot < TILE_CAP) TL.ids[(long long)tile * TILE_CAP + slot] = p;
    else atomicOr(err, ERR_TILE_OVERFLOW);
  }
}

// Lists and, for a disk, the band table of one particle by one warp (queue:
// BAND_QUEUE ints of shared memory of this warp): the initial state, and the
// particle steps inside a persistent launch.
constexpr int BAND_WARPS = 4;    // particles per CTA
constexpr int BAND_QUEUE = 256;  // queued band cells per warp before an evaluation pass
template <bool HELD>
__device__ __forceinline__ void band_one(const ParticleConst& c, const ParticleArrays& P, const TileLists& TL,
                                         unsigned* err, int p, int stamp, int* queue, int lane) {
  const RasterRec rc = P.rec[p];
  append_to_tiles(TL, c.ntx, P.prange[p], p, lane, err);
  if (P.rb[p] != P.r[p]) return;  // (the whole warp)
  const int off = c.band_off, bw = 2 * off + 1;
  int2* table = band_table(P, off, p);
  const float i2R = 0.5f / rc.r;
  auto evaluate = [&](int nq) {
    __syncwarp();
    for (int j = lane; j < nq; j += 32) band_fill<HELD>(rc, table, off, stamp, i2R, queue[j] % bw, queue[j] / bw, c.any_held);
    __syncwarp();
  };
  int nq = 0;
  for (int by0 = 0; by0 < bw; by0 += 32) {
    const int by = by0 + lane;
    BandRow r{0, 0, 0, 0};
    if (by < bw) r = band_row(rc, off, c.ny, by);
    int nmax = r.na + r.nb;
    for (int o = 16; o > 0; o >>= 1) nmax = max(nmax, __shfl_xor_sync(0xffffffffu, nmax, o));
    for (int j = 0; j < nmax; ++j) {
      bool band = false;
      int bx = 0;
      if (j < r.na + r.nb) {
        bx = j < r.na ? r.a0 + j : r.b0 + (j - r.na);
        const int x = rc.xi - off + bx;
        band = x >= 0 && x < c.nx && in_band(rc, x, rc.yi - off + by);
      }
      const unsigned m = __ballot_sync(0xffffffffu, band);
      if (band) queue[nq + __popc(m & ((1u << lane) - 1u))] = by * bw + bx;
      nq += __popc(m);
      if (nq > BAND_QUEUE - 32) {  // evaluate what is queued before it can overflow
        evaluate(nq);
        nq = 0;
      }
    }
  }
  evaluate(nq);
}

// ---- the particle step of a CTA ---------------------------------------------------
// A CTA of eight warps takes up to STEP_GROUP particles.  Warp 0 moves them
// (update_position); after a barrier it finishes their update, warp 1 appends
// them to the tile lists, and six warps fill the band tables: the rows of all
// the CTA's boxes are dealt out one per thread, their candidate cells are
// counted and scanned, then the candidates and after them the band cells are
// dealt out one per thread.  A disk of D = 16 has about 125 candidates and 75
// band cells, so a particle alone in a CTA takes one pass of each where one
// warp per particle took 12 and 3, one after the other: the step is a chain of
// latencies, and this cuts the chain (per launch under ncu, one warp per
// particle against this: one disk 14.1 -> 7.9 us, 128 disks 15.8 -> 7.5, 2048
// disks 16.0 -> 12.0, 48 cases of one disk 32.7 -> 10.8; about 5 us of each is
// the launch itself).
constexpr int STEP_THREADS = 256;
constexpr int STEP_GROUP = 8;                   // most particles of a CTA (four lanes of warp 0 each)
constexpr int STEP_BAND = STEP_THREADS - 64;    // threads that fill band tables

struct StepRef {  // a particle of the CTA and where it lives
  const ParticleConst* c;
  const ParticleArrays* P;
  const TileLists* TL;
  unsigned* err;
  int p, stamp;
};
struct StepSlot {
  RasterRec rc;
  int2* table;
  int4 rg;
  float i2R;
  int nx, ny, off, stamp, held, row0;  // row0: rows of the slots before
};
struct StepShared {
  StepSlot slot[STEP_GROUP];
  int4 run[STEP_BAND];  // a row: slot << 20 | by, a0, na, b0
  int pre[STEP_BAND];   // candidates of the rows before
  int2 queue[2 * STEP_BAND];
  int warp_total[STEP_BAND / 32];
  int queued[2];
  int rows;
};

__device__ __forceinline__ void band_barrier() { asm volatile("bar.sync 1, %0;" ::"n"(STEP_BAND) : "memory"); }

// The band tables of the CTA's slots (t: 0 .. STEP_BAND - 1).
template <bool HELD>
__device__ __forceinline__ void band_group(StepShared& sh, int n, int t) {
  const int lane = t & 31, warp = t >> 5;
  const int rows = sh.rows;
  int left = 0, pass = 0;  // queued cells not yet evaluated; passes so far (the same in every thread)
  for (int r0 = 0; r0 < rows; r0 += STEP_BAND) {
    const int r = r0 + t;
    int cnt = 0;
    if (r < rows) {
      int s = 0;
      for (int q = 1; q < n; ++q) s += r >= sh.slot[q].row0;
      const StepSlot& S = sh.slot[s];
      const int by = r - S.row0;
      const BandRow b = band_row(S.rc, S.off, S.ny, by);
      sh.run[t] = make_int4(s << 20 | by, b.a0, b.na, b.b0);
      cnt = b.na + b.nb;
    }
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    if (lane == 31) sh.warp_total[warp] = incl;
    band_barrier();
    int total = 0, before = 0;
#pragma unroll
    for (int w = 0; w < STEP_BAND / 32; ++w) {
      const int v = sh.warp_total[w];
      before += w < warp ? v : 0;
      total += v;
    }
    sh.pre[t] = before + incl - cnt;
    band_barrier();
    for (int c0 = 0; c0 < total; c0 += STEP_BAND, ++pass) {
      const int j = c0 + t;
      bool band = false;
      int2 cell = make_int2(0, 0);
      if (j < total) {
        int i = 0;  // the last row that starts at or before candidate j
#pragma unroll
        for (int o = 128; o > 0; o >>= 1)
          if (i + o < STEP_BAND && sh.pre[i + o] <= j) i += o;
        const int4 run = sh.run[i];
        const int s = run.x >> 20, by = run.x & 0xfffff, q = j - sh.pre[i];
        const int bx = q < run.z ? run.y + q : run.w + (q - run.z);
        const StepSlot& S = sh.slot[s];
        const int x = S.rc.xi - S.off + bx;
        band = x >= 0 && x < S.nx && in_band(S.rc, x, S.rc.yi - S.off + by);
        cell = make_int2(s << 20 | bx, by);
      }
      const unsigned m = __ballot_sync(0xffffffffu, band);
      int base = 0;
      if (lane == 0 && m) base = atomicAdd(&sh.queued[pass & 1], __popc(m));
      base = left + __shfl_sync(0xffffffffu, base, 0);
      if (band) sh.queue[base + __popc(m & ((1u << lane) - 1u))] = cell;
      if (t == 0) sh.queued[(pass + 1) & 1] = 0;  // (last read before the barrier that ended the last pass)
      band_barrier();
      left += sh.queued[pass & 1];
      const bool last = c0 + STEP_BAND >= total;
      // at most 2 STEP_BAND - 1 cells are queued; what stays behind is fewer
      // than STEP_BAND, or nothing after the last pass
      int2 e[2];
      bool mine[2];
#pragma unroll
      for (int g = 0; g < 2; ++g) {
        const int take = left >= STEP_BAND || last ? min(left, STEP_BAND) : 0;
        left -= take;
        mine[g] = t < take;
        if (mine[g]) e[g] = sh.queue[left + t];
      }
      band_barrier();  // every thread has its cells: the queue may change
#pragma unroll
      for (int g = 0; g < 2; ++g) {
        if (!mine[g]) continue;
        const int s = e[g].x >> 20, bx = e[g].x & 0xfffff, by = e[g].y;
        const StepSlot& S = sh.slot[s];
        band_fill<HELD>(S.rc, S.table, S.off, S.stamp, S.i2R, bx, by, S.held);
      }
    }
  }
}

// The particle step of the n <= STEP_GROUP particles ref(0) .. ref(n - 1).
template <bool HELD, class Ref>
__device__ __forceinline__ void step_group(int n, const Ref& ref, StepShared& sh) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  UpdateLane u;
  if (warp == 0) {
    const StepRef r = ref(min(lane >> 2, n - 1));
    u = update_position(*r.c, *r.P, r.p, lane, (lane >> 2) < n, r.err);
    const int t0y = __shfl_down_sync(0xffffffffu, u.t0, 1), nty = __shfl_down_sync(0xffffffffu, u.nt, 1);
    if ((lane >> 2) < n) {
      StepSlot& S = sh.slot[lane >> 2];
      if (u.k == 0) {
        S.rc.xi = u.cell; S.rc.qfx = u.qf; S.rc.xfh = u.fh; S.rc.xfl = u.fl;
        S.rg = make_int4(u.t0, t0y, u.nt, nty);
      } else if (u.k == 1) {
        S.rc.yi = u.cell; S.rc.qfy = u.qf; S.rc.yfh = u.fh; S.rc.yfl = u.fl;
      }
    }
  } else if (warp == 1) {
    int rows = 0;
    if (lane < n) {
      const StepRef r = ref(lane);
      StepSlot& S = sh.slot[lane];
      const double R = r.P->r[r.p], Rb = r.P->rb[r.p];
      record_constants(*r.P, r.p, R, Rb, S.rc);
      S.nx = r.c->nx; S.ny = r.c->ny; S.off = r.c->band_off; S.stamp = r.stamp;
      if (HELD) S.held = r.c->any_held;
      S.table = band_table(*r.P, S.off, r.p);
      S.i2R = 0.5f / S.rc.r;
      rows = R == Rb ? 2 * S.off + 1 : 0;  // an ellipse has a kernel of its own
    }
    int incl = rows;
#pragma unroll
    for (int o = 1; o < STEP_GROUP; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    if (lane < n) sh.slot[lane].row0 = incl - rows;
    if (lane == n - 1) sh.rows = incl;
    if (lane < 2) sh.queued[lane] = 0;
  }
  __syncthreads();
  if (warp == 0) {
    const StepRef r = ref(min(lane >> 2, n - 1));
    update_velocity(*r.c, *r.P, r.p, lane, (lane >> 2) < n, u, sh.slot[min(lane >> 2, n - 1)].rc, r.err);
  } else if (warp == 1) {
    for (int s = 0; s < n; ++s) {
      const StepRef r = ref(s);
      append_to_tiles(*r.TL, r.c->ntx, sh.slot[s].rg, r.p, lane, r.err);
    }
  } else {
    band_group<HELD>(sh, n, threadIdx.x - 64);
  }
}

// Particles per CTA of the particle step: one while every particle can have a
// CTA to itself (four of them are resident per SM, 608 on 152 SMs), then as
// many as keep the grid at that size, up to STEP_GROUP (2048 disks, us per
// step of the 2048^2 cavity: at most 304 CTAs 117.4, 456 115.7, 608 114.7,
// 1216 117.2).
inline int step_group_size(int n) {
  const int g = (n + 607) / 608;
  return g < 1 ? 1 : (g > STEP_GROUP ? STEP_GROUP : g);
}

// ---- band tables of ellipses (reading R13) ------------------------------------------
// One warp per row of an ellipse's box.  Most cells of the row are decided in
// FP32: the quadratic form is convex, so over a cell it is at least its tangent
// plane at the cell's centre and at most the value at a corner; both bounds are
// kept ELL_SLACK (relative) away from 1, over 25 times the FP32 error of the
// form.  The rest (about four to twelve cells a row) get the FP64 class and
// area, four lanes per cell: FP64 runs at 1/64 of the FP32 rate here and a
// dependent FP64 operation takes about 50 cycles, so the corners, edges and
// arcs of a cell go to one lane each, and the rows of one ellipse to as many
// SMs as it has rows (a = 13, b = 6.5: one warp per ellipse took 328 us, this
// 12.4).
constexpr float ELL_SLACK = 1e-5f;

// Class and area of cell (x, y), one lane per corner, edge and arc (lane & 3);
// the class takes the decisions of ellipse_cell_class, operation for operation.
__device__ __forceinline__ int ellipse_cell_by_four(int x, int y, double X, double Y, double a, double b, double c,
                                                    double s, int lane, unsigned mask, double& area) {
  const int k = lane & 3, next = (lane & ~3) | ((k + 1) & 3);
  const EllFrame f = ellipse_frame(double(x + (k == 1 || k == 2)), double(y + (k >> 1)), X, Y, a, b, c, s);
  const double u1 = __shfl_sync(mask, f.u, next), v1 = __shfl_sync(mask, f.v, next);
  const double q = quad_uv(f.u, f.v);
  double qmax = fmax(q, __shfl_xor_sync(mask, q, 1)), qmin = fmin(q, __shfl_xor_sync(mask, q, 1));
  qmax = fmax(qmax, __shfl_xor_sync(mask, qmax, 2));
  // edge k, from corner k to the next: its convex quadratic at its clamped vertex
  const double du = add_rn(u1, -f.u), dv = add_rn(v1, -f.v);
  const double A = quad_uv(du, dv);
  const double B = add_rn(mul_rn(f.u, du), mul_rn(f.v, dv));
  double t = __ddiv_rn(-B, A);
  t = t < 0.0 ? 0.0 : (t > 1.0 ? 1.0 : t);
  const double qe = quad_uv(add_rn(f.u, mul_rn(t, du)), add_rn(f.v, mul_rn(t, dv)));
  qmin = fmin(qmin, qe);
  qmin = fmin(qmin, __shfl_xor_sync(mask, qmin, 1));
  qmin = fmin(qmin, __shfl_xor_sync(mask, qmin, 2));
  const bool holds = double(x) <= X && X <= double(x + 1) && double(y) <= Y && Y <= double(y + 1);
  const int cls = qmax <= 1.0 ? CELL_SOLID : (holds || qmin < 1.0 ? CELL_INTERFACE : CELL_FLUID);
  // the area of an interface cell (quad_unit_disk_area): edge k's part inside
  // the disk is [t0, t1]; after it an arc leads to the next edge that has one
  const double C = f.u * f.u + f.v * f.v - 1.0, disc = B * B - A * C;
  bool on = disc > 0.0 && A != 0.0;
  const double r = sqrt(on ? disc : 1.0);
  const double iA = 1.0 / (on ? A : 1.0);
  const double t0 = fmax((-B - r) * iA, 0.0), t1 = fmin((-B + r) * iA, 1.0);
  on = on && t1 > t0;
  const double pu = f.u + t0 * du, pv = f.v + t0 * dv, eu = f.u + t1 * du, ev = f.v + t1 * dv;
  const unsigned edges = (__ballot_sync(mask, on) >> (lane & ~3)) & 15u;
  int step = 4;  // edges to the next one that meets the disk (4: itself)
#pragma unroll
  for (int o = 3; o > 0; --o)
    if (edges >> ((k + o) & 3) & 1u) step = o;
  const int to = (lane & ~3) | ((k + step) & 3);
  const double nu = __shfl_sync(mask, pu, to), nv = __shfl_sync(mask, pv, to);
  double part = 0.0;
  if (on && cls == CELL_INTERFACE) {
    part = 0.5 * (pu * ev - eu * pv);
    const double gu = nu - eu, gv = nv - ev;
    if (!(step == 1 && gu * gu + gv * gv < 1e-24)) {
      double ang = atan2(eu * nv - ev * nu, eu * nu + ev * nv);
      if (ang < 0.0) ang += 2.0 * 3.14159265358979323846;
      part += 0.5 * ang;
    }
  }
  part += __shfl_xor_sync(mask, part, 1);
  part += __shfl_xor_sync(mask, part, 2);
  // (an ellipse of semi_b >= 1 does not fit into a cell: without a crossing
  // edge an interface cell is only grazed)
  area = a * b * part;
  return cls;
}

// Row by of the band table of ellipse p (one warp; queue: 32 ints of shared memory).
__device__ __forceinline__ void ellipse_row(const ParticleConst& c, const ParticleArrays& P, int p, int stamp, int by,
                                            int lane, int* queue) {
  const RasterRec rc = P.rec[p];
  const int off = c.band_off, bw = 2 * off + 1;
  const int y = rc.yi - off + by;
  if (y < 0 || y >= c.ny) return;  // (the whole warp)
  const double ea = P.r[p], eb = P.rb[p], ex = P.x[p], ey = P.y[p];
  double ec, es;
  sincos(P.theta[p], &es, &ec);
  // the form q = A dx^2 + 2 B dx dy + C dy^2 in FP32, from the unit-disk frame
  const float cf = float(ec), sf = float(es), ia = 1.0f / float(ea), ib = 1.0f / float(eb);
  const float ua = cf * ia, ub = sf * ia, va = -sf * ib, vb = cf * ib;  // u = ua dx + ub dy, v = va dx + vb dy
  const float corner = 0.25f * (ua * ua + ub * ub + va * va + vb * vb) + 0.5f * fabsf(ua * ub + va * vb);
  int2* row = band_table(P, off, p) + (long long)by * bw;
  for (int bx0 = 0; bx0 < bw; bx0 += 32) {
    const int bx = bx0 + lane, x = rc.xi - off + bx;
    int cls = CELL_BAND + 1;  // outside the table's duty
    if (bx < bw && x >= 0 && x < c.nx && in_band(rc, x, y)) {
      const float dx = (float(bx - off) + 0.5f - rc.xfh) - rc.xfl, dy = (float(by - off) + 0.5f - rc.yfh) - rc.yfl;
      const float u = ua * dx + ub * dy, v = va * dx + vb * dy;
      const float q = u * u + v * v;
      // half the gradient's largest change over the cell: |q_x| / 2 + |q_y| / 2
      const float g = fabsf(u * ua + v * va) + fabsf(u * ub + v * vb);
      const float slack = ELL_SLACK * (1.0f + (dx * dx + dy * dy + 1.0f) * ib * ib);
      cls = q + g + corner <= 1.0f - slack ? CELL_SOLID : (q - g >= 1.0f + slack ? CELL_FLUID : CELL_BAND);
    }
    if (cls == CELL_SOLID || cls == CELL_FLUID)
      row[bx] = make_int2(cls | (stamp << 2), __float_as_int(cls == CELL_SOLID ? 1.0f : 0.0f));
    const unsigned m = __ballot_sync(0xffffffffu, cls == CELL_BAND);
    const int nq = __popc(m);
    if (cls == CELL_BAND) queue[__popc(m & ((1u << lane) - 1u))] = bx;
    __syncwarp();
    for (int j0 = 0; j0 < nq; j0 += 8) {
      const int j = j0 + (lane >> 2);
      const int ebx = queue[min(j, nq - 1)];
      double ar;
      const int ecls = ellipse_cell_by_four(rc.xi - off + ebx, y, ex, ey, ea, eb, ec, es, lane, 0xffffffffu, ar);
      ar = ecls == CELL_SOLID ? 1.0 : (ecls == CELL_FLUID ? 0.0 : fmin(fmax(ar, 0.0), 1.0));
      if (j < nq && (lane & 3) == 0) row[ebx] = make_int2(ecls | (stamp << 2), __float_as_int(float(ar)));
    }
    __syncwarp();
  }
}
constexpr int ELL_WARPS = 2;  // rows per CTA of the ellipses' kernels

}  // namespace vlb
