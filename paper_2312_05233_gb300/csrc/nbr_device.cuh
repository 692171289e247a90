// Device helpers of the candidate scans (nbr.cu, wide.cu).
#pragma once

#include "tnep_internal.cuh"

namespace tnep {

// Stencil cells along one axis.  Periodic axes with at least 2k + 1 cells wrap
// and carry the image shift that the minimum-image rule would pick for any
// pair within the cutoff (in units of the box edge, as the float32 product
// L * k); shorter periodic axes list every cell once and leave the shift to
// rint; open axes list the cells that exist.
__device__ __forceinline__ bool axis_short(int nc, float L, int k) { return L > 0.0f && nc < 2 * k + 1; }
__device__ __forceinline__ int axis_count(int c, int nc, float L, int k) {
  if (L > 0.0f) return nc >= 2 * k + 1 ? 2 * k + 1 : nc;
  return min(nc - 1, c + k) - max(0, c - k) + 1;
}
// Entry `idx` of the stencil: its cell, image shift, offset from the centre
// cell before wrapping, and distance in whole cells, max(|offset| - 1, 0), from
// the centre cell (0 where it is not known).
struct AxisCell {
  int cell, off, unit;
  float shift;
};
__device__ __forceinline__ AxisCell axis_cell(int c, int nc, float L, int k, int idx) {
  AxisCell a;
  if (axis_short(nc, L, k)) {
    a.cell = idx; a.off = idx - c; a.unit = 0; a.shift = 0.0f;
    return a;
  }
  const int o = L > 0.0f ? idx - k : max(0, c - k) + idx - c;
  a.cell = c + o;
  a.off = o;
  a.unit = max(abs(o) - 1, 0);
  a.shift = 0.0f;
  if (L > 0.0f) {
    if (a.cell < 0) { a.cell += nc; a.shift = L; }
    else if (a.cell >= nc) { a.cell -= nc; a.shift = -L; }
  }
  return a;
}

// Lower bound on the distance between points of two cells `u` whole cells
// apart along an axis of edge e, less a margin for positions binned across
// a face by rounding.
__device__ __forceinline__ float cell_gap(int u, float e) { return fmaxf((float)u * e - 1e-3f, 0.0f); }

// Margin (Angstrom) for float32 rounding of cell bounds, of binning and of
// the pair rule in the window scan below.
constexpr float kWindowMargin = 1e-3f;

// Lower bound on the distance along one axis between a point at x (relative
// to the grid origin) in cell c and the points of cell c + o, edge e.
__device__ __forceinline__ float point_cell_gap(float x, int c, int o, float e) {
  float g = 0.0f;
  if (o > 0) g = (float)(c + o) * e - x;
  else if (o < 0) g = x - (float)(c + o + 1) * e;
  return fmaxf(g - kWindowMargin, 0.0f);
}

// Minimum-image difference with every operation rounded separately.
__device__ __forceinline__ float mi_diff(float xj, float xi, float L, float invL) {
  float d = __fsub_rn(xj, xi);
  d = __fsub_rn(d, __fmul_rn(L, rintf(__fmul_rn(d, invL))));
  return d;
}

// The candidates of an atom at pi in cell lc of its structure: contiguous
// ranges of cell-ordered atoms, row by row of the (y, z) stencil.
struct Stencil {
  int cx, cy, cz, k, kx, nx, ny, nz;
  float ex, ey, ez, rc2R;
  bool use_rint, window;
  float xr, yr, zr, rcm2;
  __device__ __forceinline__ Stencil(const NbrArgs& a, int s, const StructGrid& G, int lc, float4 pi, float rc2R_)
      : rc2R(rc2R_) {
    cx = lc % G.nc[0];
    cy = (lc / G.nc[0]) % G.nc[1];
    cz = lc / (G.nc[0] * G.nc[1]);
    k = a.cell_div;
    kx = k == 1 ? a.x_div : k;  // x_div subdivides x only, and only with cell_div = 1
    nx = axis_count(cx, G.nc[0], G.L[0], kx);
    ny = axis_count(cy, G.nc[1], G.L[1], k);
    nz = axis_count(cz, G.nc[2], G.L[2], k);
    // stencil cells farther than the cutoff from the centre cell are skipped
    ex = 1.0f / G.cinv[0]; ey = 1.0f / G.cinv[1]; ez = 1.0f / G.cinv[2];
    // The shift of a stencil cell equals L * rint((p_j - p_i) / L) for every pair
    // the cutoff can accept when all coordinates lie in [0, L); otherwise (or
    // when an axis has too few cells to carry shifts) use rint per pair.  Both
    // give the float32 rule of the header bit for bit.
    use_rint = axis_short(G.nc[0], G.L[0], kx) || axis_short(G.nc[1], G.L[1], k) || axis_short(G.nc[2], G.L[2], k) ||
               (a.struct_flags[s] & 1);
    window = kx > 1 && k == 1 && !use_rint;
    xr = pi.x - G.origin[0]; yr = pi.y - G.origin[1]; zr = pi.z - G.origin[2];
    const float rcm = a.rc_R + kWindowMargin;
    rcm2 = rcm * rcm;
  }
  __device__ __forceinline__ int rows() const { return ny * nz; }
  // Calls emit(j0, j1, sx, sy, sz, rint_pairs) for the ranges of row iz * ny + iy, in
  // a fixed order, at most three.  The shift applies to the whole range unless
  // rint_pairs asks for the minimum image per pair.
  template <class Emit>
  __device__ __forceinline__ void row(const NbrArgs& a, const StructGrid& G, int iy, int iz, Emit&& emit) const {
    const AxisCell z = axis_cell(cz, G.nc[2], G.L[2], k, iz), y = axis_cell(cy, G.nc[1], G.L[1], k, iy);
    const int ncx = G.nc[0];
    const int row = G.cell_offset + (z.cell * G.nc[1] + y.cell) * ncx;
    if (window) {
      // Window scan: cells are thin along x.  In each (y, z) row of the stencil
      // only the x-cells meeting [x_i - h, x_i + h] can hold pairs, where
      // h^2 = rc_R^2 - (distance from atom i to the row)^2; on a periodic axis
      // the window splits at the box faces into ranges with shifts +L, 0, -L.
      // A window longer than the row falls back to the whole row with rint.
      const float gz = point_cell_gap(zr, cz, z.off, ez);
      if (gz * gz >= rcm2) return;
      const float gy = point_cell_gap(yr, cy, y.off, ey);
      const float h2 = rcm2 - gy * gy - gz * gz;
      if (h2 <= 0.0f) return;
      const float h = sqrtf(h2) + kWindowMargin;
      int clo = (int)floorf((xr - h) * G.cinv[0]);
      int chi = (int)floorf((xr + h) * G.cinv[0]);
      if (G.L[0] > 0.0f) {
        if (chi - clo + 1 > ncx) {
          emit(a.cell_start[row], a.cell_start[row + ncx], 0.0f, y.shift, z.shift, true);
          return;
        }
        if (clo < 0) emit(a.cell_start[row + clo + ncx], a.cell_start[row + ncx], G.L[0], y.shift, z.shift, false);
        const int b0 = max(clo, 0), b1 = min(chi, ncx - 1);
        if (b0 <= b1) emit(a.cell_start[row + b0], a.cell_start[row + b1 + 1], 0.0f, y.shift, z.shift, false);
        if (chi >= ncx) emit(a.cell_start[row], a.cell_start[row + chi - ncx + 1], -G.L[0], y.shift, z.shift, false);
      } else {
        clo = max(clo, 0);
        chi = min(chi, ncx - 1);
        if (clo <= chi) emit(a.cell_start[row + clo], a.cell_start[row + chi + 1], 0.0f, y.shift, z.shift, false);
      }
      return;
    }
    const float gz = cell_gap(z.unit, ez);
    if (gz * gz >= rc2R) return;
    const float gy = cell_gap(y.unit, ey);
    const float gyz = gy * gy + gz * gz;
    if (gyz >= rc2R) return;
    int ix = 0;
    while (ix < nx) {
      const AxisCell x = axis_cell(cx, ncx, G.L[0], kx, ix);
      const float gx = cell_gap(x.unit, ex);
      if (gx * gx + gyz >= rc2R) { ++ix; continue; }
      // merge x-cells that are contiguous, within reach and share a shift into one range
      int ie = ix + 1, last = x.cell;
      while (ie < nx) {
        const AxisCell e = axis_cell(cx, ncx, G.L[0], kx, ie);
        if (e.cell != last + 1 || e.shift != x.shift) break;
        const float ge = cell_gap(e.unit, ex);
        if (ge * ge + gyz >= rc2R) break;
        last = e.cell;
        ++ie;
      }
      ix = ie;
      emit(a.cell_start[row + x.cell], a.cell_start[row + last + 1], x.shift, y.shift, z.shift, use_rint);
    }
  }
};

}  // namespace tnep
