// FP32 areas of band cells in lattices with held particles: the same geometry
// as disk_unit_cell_area (vlb_raster.cuh) in the one order of operations those
// lattices keep (see vlb_lattice_held.cuh for the reason): the centre relative
// to the cell comes from its tile's coordinates, each segment is added where
// the walk meets its link, and sums of products may contract.
#pragma once

#include "vlb_raster.cuh"

namespace vlb {

// Area of the circular segment cut off by a chord of length L (L <= 2R):
// R^2 (asin z - z sqrt(1 - z^2)), z = L / (2R); below z = 1/4 its series
// 2/3 z^3 + 1/5 z^5 + 3/28 z^7 + 5/72 z^9 + 35/704 z^11 + O(z^13).
__device__ __forceinline__ float held_segment_area(float L, float R) {
  const float z = L / (2.0f * R);
  if (z < 0.25f) {
    const float z2 = z * z;
    float s = 35.0f / 704.0f;
    s = s * z2 + 5.0f / 72.0f;
    s = s * z2 + 3.0f / 28.0f;
    s = s * z2 + 0.2f;
    s = s * z2 + 2.0f / 3.0f;
    return R * R * s * z2 * z;
  }
  return R * R * (asinf(z) - z * sqrtf(fmaxf(1.0f - z * z, 0.0f)));
}

// Area of disk((cx, cy), R) in [0,1]^2 (cell-local coordinates), R >= 1: the
// walk of disk_unit_cell_area, shoelace terms and link segments summed on the
// fly in walking order.
__device__ __forceinline__ float held_unit_cell_area(float cx, float cy, float R) {
  float x0 = 0.0f, y0 = 0.0f;  // first point (a_0)
  float xp = 0.0f, yp = 0.0f;  // last point so far
  bool any = false;
  float twice = 0.0f, seg = 0.0f;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    // edge 0: y = 0, x 0 -> 1; edge 1: x = 1, y 0 -> 1; edge 2: y = 1, x 1 -> 0;
    // edge 3: x = 0, y 1 -> 0
    const bool horiz = (k == 0 || k == 2);
    const float fixed = (k == 1 || k == 2) ? 1.0f : 0.0f;
    const float d = fixed - (horiz ? cy : cx);
    const float ad = d < 0.0f ? -d : d;
    if (ad >= R) continue;
    const float s = vsqrt((R - ad) * (R + ad));
    const float c_run = horiz ? cx : cy;
    float lo = c_run - s, hi = c_run + s;
    lo = lo < 0.0f ? 0.0f : lo;
    hi = hi > 1.0f ? 1.0f : hi;
    if (!(hi > lo)) continue;
    const bool up = (k == 0 || k == 1);
    const float a = up ? lo : hi, b = up ? hi : lo;  // start and end in walking order
    const float ax = horiz ? a : fixed, ay = horiz ? fixed : a;
    const float bx = horiz ? b : fixed, by = horiz ? fixed : b;
    if (any) {
      // link from the previous interval's end to this start: a chord and its arc
      twice += xp * ay - ax * yp;
      const float lx = ax - xp, ly = ay - yp;
      const float L = vsqrt(lx * lx + ly * ly);
      if (L > 0.0f) seg += held_segment_area(L < 2.0f * R ? L : 2.0f * R, R);
    } else {
      x0 = ax; y0 = ay;
      any = true;
    }
    twice += ax * by - bx * ay;
    xp = bx; yp = by;
  }
  if (!any) return 0.0f;
  // closing link from the last end back to the first start
  twice += xp * y0 - x0 * yp;
  {
    const float lx = x0 - xp, ly = y0 - yp;
    const float L = vsqrt(lx * lx + ly * ly);
    if (L > 0.0f) seg += held_segment_area(L < 2.0f * R ? L : 2.0f * R, R);
  }
  const float area = 0.5f * twice + seg;
  return area < 0.0f ? 0.0f : (area > 1.0f ? 1.0f : area);
}

// As disk_band_cell: class and area of lattice cell (x, y), a band cell of the
// record's disk.
__device__ __forceinline__ int held_band_cell(const RasterRec& rc, int x, int y, float& f) {
  const int tx = x % TILE_X, ty = y % TILE_Y;
  PartTile<float> q;
  tile_geometry(rc, x - tx, y - ty, q);
  const int cls = cell_class_exact(tx, ty, q);
  if (cls != CELL_INTERFACE) {
    f = cls == CELL_SOLID ? 1.0f : 0.0f;
    return cls;
  }
  const float cx = (q.xh - float(tx)) + q.xl;  // disk centre in cell-local coordinates
  const float cy = (q.yh - float(ty)) + q.yl;
  f = held_unit_cell_area(cx, cy, q.r);
  return cls;
}

}  // namespace vlb
