// Solid fraction of a disk in one lattice cell (Sec. 2: f_s is the volume
// fraction of solid in the cell, fixed by the particle position).
//
// Classification (integer, identical on every device): a cell is SOLID when
// its four corners lie in the closed disk and FLUID when its nearest point is
// at distance >= R, tested on centres and radii rounded to a 2^-20 grid.
// INTERFACE cells get the exact area of disk ∩ cell, computed in cell-local
// coordinates as a polygon (the parts of the cell edges inside the disk) plus
// the circular segments between each chord and its arc -- all quantities are
// O(1), so FP32 keeps ~1e-7 absolute error.
#pragma once

#include <math.h>

#include "vlb_common.cuh"

namespace vlb {

__host__ __device__ __forceinline__ float vsqrt(float v) { return sqrtf(v); }
__host__ __device__ __forceinline__ double vsqrt(double v) { return sqrt(v); }

// Products and sums rounded one by one (no contraction into FMA), so that a
// test gives the same answer in every kernel that makes it.
__host__ __device__ __forceinline__ float mul_rn(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fmul_rn(a, b);
#else
  return a * b;
#endif
}
__host__ __device__ __forceinline__ float add_rn(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fadd_rn(a, b);
#else
  return a + b;
#endif
}
__host__ __device__ __forceinline__ double mul_rn(double a, double b) {
#ifdef __CUDA_ARCH__
  return __dmul_rn(a, b);
#else
  return a * b;
#endif
}
__host__ __device__ __forceinline__ double add_rn(double a, double b) {
#ifdef __CUDA_ARCH__
  return __dadd_rn(a, b);
#else
  return a + b;
#endif
}

__host__ __device__ __forceinline__ float fma_rn(float a, float b, float c) {
#ifdef __CUDA_ARCH__
  return __fmaf_rn(a, b, c);
#else
  return fmaf(a, b, c);
#endif
}
__host__ __device__ __forceinline__ double fma_rn(double a, double b, double c) {
#ifdef __CUDA_ARCH__
  return __fma_rn(a, b, c);
#else
  return fma(a, b, c);
#endif
}

enum : int { CELL_FLUID = 0, CELL_INTERFACE = 1, CELL_SOLID = 2 };

// An ellipse as the FP64 lattice kernel sees it (the FP32 kernel reads
// ellipses from their band tables and carries none of this).
template <class C>
struct EllPart {};
template <>
struct EllPart<double> {
  int ell;                        // an ellipse
  double ex, ey, ea, eb, ec, es;  // its centre, semi-axes, cos and sin of its angle
};

// One particle as seen from one tile (shared memory).  Coordinates are
// relative to the tile's lower-left corner.
template <class C>
struct PartTile : EllPart<C> {
  long long xq, yq, rq2;  // fixed-point centre and R^2 (2^-20 grid)
  C xh, xl, yh, yl;       // centre as an unevaluated sum hi + lo
  C r, far2, near2;       // radius, quick-reject bounds on the centre distance^2
  C ux, uy, om;           // rigid-body motion (Eq. 27)
  C uxl, uyl;             // low parts of U (U = ux + uxl to FP64 accuracy)
  C lam_s, T0;
  int id;                 // particle id
  int ci, cj;             // cell of the centre (band table origin)
  int fixed;              // held at T0: 1 covered part (reading R11), 2 whole cells (R11b)
};

// Class of the cell whose lower-left corner lies at (cx0, cy0) from the disk's
// centre (2^-20 grid).  I: long long, or int where every |cx0| + 2^20 fits 31
// bits (each product is then one 32 x 32 -> 64 bit multiply).
template <class I>
__host__ __device__ __forceinline__ int cell_class_at(I cx0, I cy0, long long rq2) {
  const I Q = I(1) << QBITS;
  const I cx1 = cx0 + Q, cy1 = cy0 + Q;
  const I ax0 = cx0 < 0 ? -cx0 : cx0, ax1 = cx1 < 0 ? -cx1 : cx1;
  const I ay0 = cy0 < 0 ? -cy0 : cy0, ay1 = cy1 < 0 ? -cy1 : cy1;
  const I fx = ax0 > ax1 ? ax0 : ax1, fy = ay0 > ay1 ? ay0 : ay1;  // farthest corner
  if ((long long)fx * fx + (long long)fy * fy <= rq2) return CELL_SOLID;
  const I nx = (cx0 <= 0 && cx1 >= 0) ? 0 : (ax0 < ax1 ? ax0 : ax1);  // nearest point
  const I ny = (cy0 <= 0 && cy1 >= 0) ? 0 : (ay0 < ay1 ? ay0 : ay1);
  if ((long long)nx * nx + (long long)ny * ny >= rq2) return CELL_FLUID;
  return CELL_INTERFACE;
}
// Integer classification of cell (il, jl) of the tile against one disk.
template <class C>
__host__ __device__ __forceinline__ int cell_class_exact(int il, int jl, const PartTile<C>& p) {
  const long long Q = 1ll << QBITS;
  return cell_class_at((long long)il * Q - p.xq, (long long)jl * Q - p.yq, p.rq2);
}

// Area of the circular segment on a chord of squared length L2 (<= 4 R^2),
// with i2R = 1 / (2R): R^2 (asin z - z sqrt(1 - z^2)), z = L / (2R).  Its
// Taylor series is R^2 z^3 sum_k 2 b_k / (2k + 3) z^2k with b_k = C(2k, k) / 4^k
// (the derivative is 2 z^2 / sqrt(1 - z^2)); for z below the given bound it is
// cut where its terms pass the type's precision, and needs one square root
// instead of three library calls and a division.
__host__ __device__ __forceinline__ double segment_area(double L2, double R, double i2R) {
  const double z2 = mul_rn(mul_rn(L2, i2R), i2R);
  const double L = vsqrt(L2);
  if (z2 < 1.0 / 64.0) {
    double s = 12155.0 / 688128.0;
    s = fma_rn(s, z2, 6435.0 / 311296.0);
    s = fma_rn(s, z2, 429.0 / 17408.0);
    s = fma_rn(s, z2, 77.0 / 2560.0);
    s = fma_rn(s, z2, 63.0 / 1664.0);
    s = fma_rn(s, z2, 35.0 / 704.0);
    s = fma_rn(s, z2, 5.0 / 72.0);
    s = fma_rn(s, z2, 3.0 / 28.0);
    s = fma_rn(s, z2, 0.2);
    s = fma_rn(s, z2, 2.0 / 3.0);
    return mul_rn(mul_rn(mul_rn(L, L2), mul_rn(0.25, i2R)), s);
  }
  double z = mul_rn(L, i2R);
  z = z < 1.0 ? z : 1.0;
  return mul_rn(mul_rn(R, R), add_rn(asin(z), -mul_rn(z, vsqrt(fma_rn(-z, z, 1.0)))));
}
__host__ __device__ __forceinline__ float segment_area(float L2, float R, float i2R) {
  const float z2 = mul_rn(mul_rn(L2, i2R), i2R);
  const float L = vsqrt(L2);
  if (z2 < 0.0625f) {
    float s = 35.0f / 704.0f;
    s = fma_rn(s, z2, 5.0f / 72.0f);
    s = fma_rn(s, z2, 3.0f / 28.0f);
    s = fma_rn(s, z2, 0.2f);
    s = fma_rn(s, z2, 2.0f / 3.0f);
    return mul_rn(mul_rn(mul_rn(L, L2), mul_rn(0.25f, i2R)), s);
  }
  float z = mul_rn(L, i2R);
  z = z < 1.0f ? z : 1.0f;
  return mul_rn(mul_rn(R, R), add_rn(asinf(z), -mul_rn(z, vsqrt(fma_rn(-z, z, 1.0f)))));
}

// Exact area of disk((cx, cy), R) ∩ [0,1]^2 (cell-local coordinates), R >= 1,
// i2R = 1 / (2R).
//
// Walking the square's boundary counter-clockwise, each edge meets the closed
// disk in one interval (possibly empty), found from that edge's own line.  The
// region's boundary is those intervals joined, between one interval's end and
// the next interval's start, by arcs of the circle; so the area is the polygon
// of the interval end points plus, for every such link, the circular segment
// on its chord.  No entry/exit decision is taken: when rounding puts a circle
// point on one or the other side of a corner, the link's chord is just tiny
// and so is its segment.
//
// The four intervals are computed without branches (four independent square
// roots in flight), the walk keeps the links' squared chords, and the segments
// come last: a cell has one arc as a rule, so a warp evaluates one or two
// segments where evaluating each link at its place in the walk cost it four.
// Every operation is rounded on its own, so that the kernels that compute a
// cell's area agree to the last bit however each was compiled.
template <class C>
__host__ __device__ __forceinline__ C disk_unit_cell_area(C cx, C cy, C R, C i2R) {
  // edge 0: y = 0, x 0 -> 1; edge 1: x = 1, y 0 -> 1; edge 2: y = 1, x 1 -> 0;
  // edge 3: x = 0, y 1 -> 0
  C lo[4], hi[4];
  bool on[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const bool horiz = (k == 0 || k == 2);
    const C d = add_rn((k == 1 || k == 2) ? C(1) : C(0), -(horiz ? cy : cx));
    const C ad = d < C(0) ? -d : d;
    const bool meets = ad < R;
    const C h = mul_rn(add_rn(R, -ad), add_rn(R, ad));
    const C s = vsqrt(meets ? h : C(1));
    const C c_run = horiz ? cx : cy;
    lo[k] = add_rn(c_run, -s);
    hi[k] = add_rn(c_run, s);
    lo[k] = lo[k] < C(0) ? C(0) : lo[k];
    hi[k] = hi[k] > C(1) ? C(1) : hi[k];
    on[k] = meets && hi[k] > lo[k];
  }
  // the walk: interval ends (ax, ay) -> (bx, by) in order, links between them
  C x0 = C(0), y0 = C(0), xp = C(0), yp = C(0);
  C twice = C(0), l2[4];
  bool any = false;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const bool horiz = (k == 0 || k == 2), up = (k == 0 || k == 1);
    const C fixed = (k == 1 || k == 2) ? C(1) : C(0);
    const C a = up ? lo[k] : hi[k], b = up ? hi[k] : lo[k];
    const C ax = horiz ? a : fixed, ay = horiz ? fixed : a;
    const C bx = horiz ? b : fixed, by = horiz ? fixed : b;
    const bool link = on[k] && any;
    const C lx = add_rn(ax, -xp), ly = add_rn(ay, -yp);
    l2[k] = link ? fma_rn(lx, lx, mul_rn(ly, ly)) : C(0);
    C add = link ? fma_rn(xp, ay, -mul_rn(ax, yp)) : C(0);
    // the interval's own term ax by - bx ay: zero on the edges through (0, 0)
    if (k == 1 || k == 2) add = add_rn(add, on[k] ? add_rn(hi[k], -lo[k]) : C(0));
    twice = add_rn(twice, add);
    x0 = (on[k] && !any) ? ax : x0;
    y0 = (on[k] && !any) ? ay : y0;
    xp = on[k] ? bx : xp;
    yp = on[k] ? by : yp;
    any = any || on[k];
  }
  if (!any) return C(0);
  // closing link from the last end back to the first start (l2[0] is free:
  // no link leads to the first edge)
  twice = add_rn(twice, fma_rn(xp, y0, -mul_rn(x0, yp)));
  {
    const C lx = add_rn(x0, -xp), ly = add_rn(y0, -yp);
    l2[0] = fma_rn(lx, lx, mul_rn(ly, ly));
  }
  const C most = mul_rn(mul_rn(C(4), R), R);
  C seg = C(0);
  for (;;) {  // the links of non-zero length, in the order 1, 2, 3, closing
    const bool b1 = l2[1] > C(0), b2 = l2[2] > C(0), b3 = l2[3] > C(0);
    const C L2 = b1 ? l2[1] : (b2 ? l2[2] : (b3 ? l2[3] : l2[0]));
    if (!(L2 > C(0))) break;
    if (b1) l2[1] = C(0);
    else if (b2) l2[2] = C(0);
    else if (b3) l2[3] = C(0);
    else l2[0] = C(0);
    seg = add_rn(seg, segment_area(L2 < most ? L2 : most, R, i2R));
  }
  const C area = fma_rn(C(0.5), twice, seg);
  return area < C(0) ? C(0) : (area > C(1) ? C(1) : area);
}

// Quick class of tile cell (il, jl): CELL_FLUID or CELL_SOLID where the
// centre distance decides it, CELL_BAND where the exact test is needed.  The
// FP32 lattice kernel and the band kernel both take this decision, so it is
// rounded step by step (mul_rn, add_rn) to come out the same in both.
enum : int { CELL_BAND = 3 };
template <class C>
__host__ __device__ __forceinline__ int quick_class_at(int il, int jl, C xh, C xl, C yh, C yl, C far2, C near2) {
  // centre distance from the cell centre (hi/lo sums keep FP32 exact enough)
  const C dx = add_rn(add_rn(add_rn(C(il), C(0.5)), -xh), -xl);
  const C dy = add_rn(add_rn(add_rn(C(jl), C(0.5)), -yh), -yl);
  const C d2 = add_rn(mul_rn(dx, dx), mul_rn(dy, dy));
  if (d2 >= far2) return CELL_FLUID;   // nearest point > R + 0.04
  if (d2 <= near2) return CELL_SOLID;  // farthest corner < R - 0.04
  return CELL_BAND;
}
template <class C>
__host__ __device__ __forceinline__ int quick_class(int il, int jl, const PartTile<C>& p) {
  return quick_class_at(il, jl, p.xh, p.xl, p.yh, p.yl, p.far2, p.near2);
}

// ---------------------------------------------------------------------------
// Ellipses (reading R13), in FP64 with every product, sum and quotient
// rounded one at a time, so that the class decisions are those of any other
// FP64 evaluation in the same order (the oracle's among them).
// ---------------------------------------------------------------------------
struct EllFrame { double u, v; };
// Point (px, py) in the ellipse's unit-disk frame: ((c dx + s dy) / a, (c dy - s dx) / b).
__host__ __device__ __forceinline__ EllFrame ellipse_frame(double px, double py, double X, double Y, double a,
                                                           double b, double c, double s) {
  const double dx = add_rn(px, -X), dy = add_rn(py, -Y);
  EllFrame f;
#ifdef __CUDA_ARCH__
  f.u = __ddiv_rn(add_rn(mul_rn(c, dx), mul_rn(s, dy)), a);
  f.v = __ddiv_rn(add_rn(mul_rn(c, dy), -mul_rn(s, dx)), b);
#else
  f.u = (c * dx + s * dy) / a;
  f.v = (c * dy - s * dx) / b;
#endif
  return f;
}
__host__ __device__ __forceinline__ double quad_uv(double u, double v) { return add_rn(mul_rn(u, u), mul_rn(v, v)); }

// Class of cell [i, i+1] x [j, j+1]: SOLID when its four corners lie in the
// closed ellipse, FLUID when the least value of the quadratic form over the
// cell (each edge's convex quadratic at its clamped vertex) is >= 1.
__host__ __device__ __forceinline__ int ellipse_cell_class(int i, int j, double X, double Y, double a, double b,
                                                           double c, double s) {
  double cu[4], cv[4];
  const double xs[4] = {double(i), double(i + 1), double(i + 1), double(i)};
  const double ys[4] = {double(j), double(j), double(j + 1), double(j + 1)};
  double qmax = 0.0, qmin = 0.0;
  for (int k = 0; k < 4; ++k) {
    const EllFrame f = ellipse_frame(xs[k], ys[k], X, Y, a, b, c, s);
    cu[k] = f.u; cv[k] = f.v;
    const double q = quad_uv(f.u, f.v);
    qmax = k == 0 ? q : (q > qmax ? q : qmax);
    qmin = k == 0 ? q : (q < qmin ? q : qmin);
  }
  if (qmax <= 1.0) return CELL_SOLID;
  if (double(i) <= X && X <= double(i + 1) && double(j) <= Y && Y <= double(j + 1)) return CELL_INTERFACE;
  for (int k = 0; k < 4; ++k) {
    const int k1 = (k + 1) & 3;
    const double du = add_rn(cu[k1], -cu[k]), dv = add_rn(cv[k1], -cv[k]);
    const double A = quad_uv(du, dv);
#ifdef __CUDA_ARCH__
    double t = __ddiv_rn(-add_rn(mul_rn(cu[k], du), mul_rn(cv[k], dv)), A);
#else
    double t = -(cu[k] * du + cv[k] * dv) / A;
#endif
    t = t < 0.0 ? 0.0 : (t > 1.0 ? 1.0 : t);
    const double q = quad_uv(add_rn(cu[k], mul_rn(t, du)), add_rn(cv[k], mul_rn(t, dv)));
    qmin = q < qmin ? q : qmin;
  }
  return qmin >= 1.0 ? CELL_FLUID : CELL_INTERFACE;
}

// Area of the unit disk within the convex quadrilateral (us, vs) (counter-
// clockwise), by Green's theorem on the intersection's boundary: inside
// parts of the edges contribute (u_a v_b - u_b v_a) / 2, the arcs between
// leaving the disk on one edge and entering it on a later one half their
// counter-clockwise angle; a vertex on the circle (exit and entry at the same
// point of consecutive edges) adds no arc.
__host__ __device__ __forceinline__ double quad_unit_disk_area(const double (&us)[4], const double (&vs)[4]) {
  double pa_u[4], pa_v[4], pb_u[4], pb_v[4];
  int edge[4];
  int m = 0;
  for (int k = 0; k < 4; ++k) {
    const int k1 = (k + 1) & 3;
    const double u0 = us[k], v0 = vs[k];
    const double du = us[k1] - u0, dv = vs[k1] - v0;
    const double A = du * du + dv * dv, B = u0 * du + v0 * dv, C = u0 * u0 + v0 * v0 - 1.0;
    const double disc = B * B - A * C;
    if (A == 0.0 || disc <= 0.0) continue;
    const double r = sqrt(disc);
    double t0 = (-B - r) / A, t1 = (-B + r) / A;
    t0 = t0 > 0.0 ? t0 : 0.0;
    t1 = t1 < 1.0 ? t1 : 1.0;
    if (t1 <= t0) continue;
    pa_u[m] = u0 + t0 * du; pa_v[m] = v0 + t0 * dv;
    pb_u[m] = u0 + t1 * du; pb_v[m] = v0 + t1 * dv;
    edge[m] = k;
    ++m;
  }
  if (m == 0) {
    bool inside = true;  // the disk's centre inside the polygon (then the whole disk is)
    for (int k = 0; k < 4; ++k) {
      const int k1 = (k + 1) & 3;
      inside = inside && ((us[k1] - us[k]) * (0.0 - vs[k]) - (vs[k1] - vs[k]) * (0.0 - us[k]) >= 0.0);
    }
    return inside ? 3.14159265358979323846 : 0.0;
  }
  double area = 0.0;
  for (int q = 0; q < m; ++q) {
    area += 0.5 * (pa_u[q] * pb_v[q] - pb_u[q] * pa_v[q]);
    const int n1 = q + 1 < m ? q + 1 : 0;
    const double qu = pa_u[n1], qv = pa_v[n1];
    const double gu = qu - pb_u[q], gv = qv - pb_v[q];
    if (edge[n1] == ((edge[q] + 1) & 3) && gu * gu + gv * gv < 1e-24) continue;
    double ang = atan2(pb_u[q] * qv - pb_v[q] * qu, pb_u[q] * qu + pb_v[q] * qv);
    if (ang < 0.0) ang += 2.0 * 3.14159265358979323846;
    area += 0.5 * ang;
  }
  return area;
}

// Exact area of the ellipse in cell [i, i+1] x [j, j+1] (the cell is a
// parallelogram in the unit-disk frame; areas scale by a b).
__host__ __device__ __forceinline__ double ellipse_cell_area(int i, int j, double X, double Y, double a, double b,
                                                             double c, double s) {
  const double xs[4] = {double(i), double(i + 1), double(i + 1), double(i)};
  const double ys[4] = {double(j), double(j), double(j + 1), double(j + 1)};
  double us[4], vs[4];
  for (int k = 0; k < 4; ++k) {
    const EllFrame f = ellipse_frame(xs[k], ys[k], X, Y, a, b, c, s);
    us[k] = f.u; vs[k] = f.v;
  }
  return a * b * quad_unit_disk_area(us, vs);
}

// Class and fraction of cell (gi, gj) of the lattice for an ellipse; the
// quick test on the circumscribed and inscribed circles first (its SOLID and
// FLUID answers are exact), the FP64 class and area for the band cells.
template <class C>
__host__ __device__ __forceinline__ int ellipse_cell_fraction(int il, int jl, int gi, int gj, const PartTile<C>& p,
                                                              C& fsp) {
  const int qc = quick_class(il, jl, p);
  if (qc == CELL_FLUID) { fsp = C(0); return CELL_FLUID; }
  if (qc == CELL_SOLID) { fsp = C(1); return CELL_SOLID; }
  const int cls = ellipse_cell_class(gi, gj, p.ex, p.ey, p.ea, p.eb, p.ec, p.es);
  if (cls == CELL_SOLID) { fsp = C(1); return cls; }
  if (cls == CELL_FLUID) { fsp = C(0); return cls; }
  const double ar = ellipse_cell_area(gi, gj, p.ex, p.ey, p.ea, p.eb, p.ec, p.es);
  fsp = C(ar < 0.0 ? 0.0 : (ar > 1.0 ? 1.0 : ar));
  return cls;
}

// Class and solid fraction of tile cell (il, jl) for one particle.
template <class C>
__host__ __device__ __forceinline__ int cell_fraction(int il, int jl, const PartTile<C>& p, C& fsp) {
  const int qc = quick_class(il, jl, p);
  if (qc == CELL_FLUID) { fsp = C(0); return CELL_FLUID; }
  if (qc == CELL_SOLID) { fsp = C(1); return CELL_SOLID; }
  const int cls = cell_class_exact(il, jl, p);
  if (cls == CELL_SOLID) { fsp = C(1); return cls; }
  if (cls == CELL_FLUID) { fsp = C(0); return cls; }
  const C cx = (p.xh - C(il)) + p.xl;  // disk centre in cell-local coordinates
  const C cy = (p.yh - C(jl)) + p.yl;
  fsp = disk_unit_cell_area(cx, cy, p.r, C(0.5) / p.r);
  return cls;
}

// A centre coordinate (cell `cells` from the tile's origin, fraction fh + fl)
// relative to the tile, as an unevaluated sum h + l.
__host__ __device__ __forceinline__ void tile_coordinate(int cells, float fh, float fl, float& h, float& l) {
  const float f = float(cells);  // exact small integer
  h = add_rn(f, fh);
  l = add_rn(add_rn(add_rn(f, -h), fh), fl);
}
// The geometry fields of a particle's raster record as seen from the tile with
// origin (x0, y0) (FP32, no FP64 arithmetic): everything cell_fraction reads.
__host__ __device__ __forceinline__ void tile_geometry(const RasterRec& rc, int x0, int y0, PartTile<float>& q) {
  const long long Q = 1ll << QBITS;
  q.xq = (long long)(rc.xi - x0) * Q + rc.qfx;
  q.yq = (long long)(rc.yi - y0) * Q + rc.qfy;
  q.rq2 = rc.rq2;
  tile_coordinate(rc.xi - x0, rc.xfh, rc.xfl, q.xh, q.xl);
  tile_coordinate(rc.yi - y0, rc.yfh, rc.yfl, q.yh, q.yl);
  q.r = rc.r; q.far2 = rc.far2; q.near2 = rc.near2;
  q.ci = rc.xi; q.cj = rc.yi;
}

// Class and area of the cell at offset (dx, dy) from the record's own cell
// against its disk (a band-table entry).  i2R = 1 / (2 R).
__host__ __device__ __forceinline__ int disk_band_cell(const RasterRec& rc, int dx, int dy, float i2R, float& f) {
  int cls;
  if (rc.rq2 < (1ll << 61)) {  // R < 1448 cells: every corner within 2^31 grid units of the centre
    cls = cell_class_at(dx * (1 << QBITS) - rc.qfx, dy * (1 << QBITS) - rc.qfy, rc.rq2);
  } else {
    cls = cell_class_at((long long)dx * (1ll << QBITS) - rc.qfx, (long long)dy * (1ll << QBITS) - rc.qfy, rc.rq2);
  }
  if (cls != CELL_INTERFACE) {
    f = cls == CELL_SOLID ? 1.0f : 0.0f;
    return cls;
  }
  const float cx = add_rn(add_rn(float(-dx), rc.xfh), rc.xfl), cy = add_rn(add_rn(float(-dy), rc.yfh), rc.yfl);
  f = disk_unit_cell_area(cx, cy, rc.r, i2R);
  return cls;
}

}  // namespace vlb
