// grid_walk.cuh -- layout of the cell grid over an obstacle cloud and the walk
// of its rows near a footprint (cloud_grid.cuh builds the grid and says what
// it is for).
#pragma once

#include "common.cuh"

namespace exact {

constexpr int kCells = 8192;          // cell-start table size (nx * ny <= kCells)
constexpr float kCellTarget = 7600.f; // nx * ny aimed at: (a + 1)(b + 1) <= kCells for a b <= 7600, a, b < 256
constexpr int kGridDim = 256;         // most cells along one axis

// Most that a safety distance counts for: beyond, squares would overflow.
constexpr float kCapMax = 1e15f;

struct __align__(16) GridHead {
    float lx, ly, inv, cell;   // lower corner, 1 / cell size, cell size
    float vmax;                // largest point speed (predicted clouds)
    int open;                  // points outside lie in the border cells
    int nx, ny;
};
struct CloudGrid {
    GridHead head;
    int start[kCells + 8];     // first point of each cell; kCells + 1 used, padded to whole 32-byte sectors
};
constexpr size_t kGridBytes = (sizeof(CloudGrid) + 255) / 256 * 256;
// A predicted cloud gets one grid per horizon step over its points' positions
// at that step, while those fit kStepGridBytes (8 bytes per point and step: the
// most try_work gives); else one grid whose cells are searched as far as the
// fastest point can have moved.  (Measured with K = 1,024, T = 20, 2,048 points
// on boxes and discs at 0.5 m/s: the cycle takes 27 to 29 us with a grid per step,
// 45 to 52 us with one; K = 256, T = 100, 100,000 points at 0.3 m/s 0.29 ms against
// 9.2, at 30 m/s 0.19 against 17.3.)
constexpr size_t kStepGridBytes = (size_t)1 << 30;
// The grid of step h and the first of its points: grid + h * grids, point
// h * points (both 0 for a static cloud).
struct GridStride {
    int grids, points;
};
inline size_t step_points(int N) { return ((size_t)N + 31) / 32 * 32; }   // points of one step, padded to 256 bytes
inline size_t step_grid_bytes(int N, int T) {
    return ((size_t)T * sizeof(CloudGrid) + 255) / 256 * 256 + (size_t)T * step_points(N) * sizeof(float2);
}
// Runs of points are counted in 32-bit integers over 32 steps at a time.
constexpr int kGridMaxPoints = 1 << 25;
// Bytes of a grid and the ordered copy of N points (and velocities).
inline size_t grid_copy_bytes(int N, bool moving) {
    return kGridBytes + ((size_t)N * sizeof(float2) + 255) / 256 * 256 * (moving ? 2 : 1);
}
// The grid and the ordered copy are read with __ldca (cached, ordered loads):
// a kernel launched early may not take them through the read-only path, whose
// loads the compiler may move above griddepcontrol.wait.
__device__ __forceinline__ GridHead load_head(const CloudGrid *g) {
    const float4 a = __ldca(reinterpret_cast<const float4 *>(&g->head));
    const float4 b = __ldca(reinterpret_cast<const float4 *>(&g->head) + 1);
    return GridHead{a.x, a.y, a.z, a.w, b.x, __float_as_int(b.y), __float_as_int(b.z), __float_as_int(b.w)};
}

// Cell index along one axis: monotone in x, so the cells of an interval's
// ends bound the cells of every point inside it.
__device__ __forceinline__ int cell_axis(float x, float lo, float inv, int n) {
    return min(n - 1, max(0, (int)((x - lo) * inv)));
}

// The rows of the grid that the footprint's bounding box at one step crosses
// and, per row, the run of points in the cells that the box can touch.
// pose = (x, y, cos, sin) of the body frame; fb = box (centre, half extents)
// in the body frame.  The box is grown by lim at each row, which may shrink
// from row to row (and below 0) but not exceed the lim of the start.
struct RowWalk {
    float cwx, cwy;              // box centre (world)
    float hx, hy;                // half extents in the body frame, with the slack for rounding
    float ac, as;                // |cos|, |sin|
    float k1, k2, i1, i2;        // slabs |c dx + s dy| <= ex, |-s dx + c dy| <= ey as x = k dy +- i e
    float y0, dy;                // lower edge of row 0 relative to the centre, row height, both with a tolerance
    int jc, j0, j1;              // centre row, first and last row (none: j1 < j0)
};
__device__ __forceinline__ RowWalk row_walk(const GridHead &g, float4 pose, float4 fb, float lim) {
    RowWalk r;
    const float c = pose.z, s = pose.w;
    r.cwx = fmaf(c, fb.x, fmaf(-s, fb.y, pose.x));
    r.cwy = fmaf(s, fb.x, fmaf(c, fb.y, pose.y));
    // Above every rounding below and in the evaluation, each taken relative to
    // what it rounds (u = 2^-24): the centre's two fmas, 2 u of its coordinates;
    // cell indices, 6 u of the grid's extent; the body frame's transform, the
    // slabs' products and the replaced c or s (1e-6), of the box and of lim.
    // Map coordinates of 1e5 m thus widen the box by 0.1 m (with one slack for
    // all, 1e-5 of every term, by 4 m: K = 1,024, T = 30, 4,000 points at
    // (5e5, -5e5) m 37 us instead of 535).
    const float slack = 5e-7f * (fabsf(r.cwx) + fabsf(r.cwy)) + 1e-6f * g.cell * (float)(g.nx + g.ny) +
                        1e-5f * (fabsf(fb.x) + fabsf(fb.y) + fb.z + fb.w) + 2e-6f * fmaxf(lim, 0.f);
    r.hx = fb.z + slack;
    r.hy = fb.w + slack;
    r.ac = fabsf(c);
    r.as = fabsf(s);
    // a vanishing c or s is replaced by 1e-6 (an error of 1e-6 |dx|, inside the slack)
    const float ic = copysignf(1.f / fmaxf(r.ac, 1e-6f), c), is = copysignf(1.f / fmaxf(r.as, 1e-6f), s);
    r.k1 = -s * ic;
    r.k2 = c * is;
    r.i1 = fabsf(ic);
    r.i2 = fabsf(is);
    const float tol = 1e-6f * g.cell * (float)(g.nx + g.ny) + 1e-6f;
    r.y0 = g.ly - r.cwy - tol;
    r.dy = g.cell + 2.f * tol;
    const float ex = r.hx + lim, ey = r.hy + lim;
    const float rx = fmaf(r.ac, ex, r.as * ey), ry = fmaf(r.as, ex, r.ac * ey);
    const float a = (r.cwy - ry - g.ly) * g.inv, b = (r.cwy + ry - g.ly) * g.inv;
    const float u = (r.cwx - rx - g.lx) * g.inv, v = (r.cwx + rx - g.lx) * g.inv;
    // points lie in [0, ny] x [0, nx] of these coordinates: a box beyond holds
    // none, unless the border cells hold the points beyond
    const bool meets = g.open || !(a > (float)g.ny || b < 0.f || u > (float)g.nx || v < 0.f);
    r.j0 = max(0, min(g.ny - 1, (int)a));
    r.j1 = meets ? min(g.ny - 1, max(0, (int)b)) : -1;
    r.jc = max(r.j0, min(r.j1, (int)((r.cwy - g.ly) * g.inv)));
    if (g.open && (r.j0 == 0 || r.j1 == g.ny - 1)) {   // a border row has no outer edge: the whole width of the box
        r.k1 = r.k2 = 0.f;
        r.i1 = r.i2 = 1e6f;
        r.y0 = -finf();
        r.dy = finf();
    }
    return r;
}
// Rows from the centre outwards: the k-th (k = 0, 1, ...) is jc, jc + 1,
// jc - 1, ..., and may lie outside [j0, j1]; walk_rows of them reach all.
__device__ __forceinline__ int walk_row(const RowWalk &r, int k) { return r.jc + ((k & 1) ? (k + 1) >> 1 : -(k >> 1)); }
__device__ __forceinline__ int walk_rows(const RowWalk &r) {
    return r.j1 < r.j0 ? 0 : 2 * max(r.j1 - r.jc, r.jc - r.j0) + 1;
}
// Points [p0, p1) of row j that can lie in the box grown by lim.
__device__ __forceinline__ void row_run(const GridHead &g, const int *start, const RowWalk &r, int j, float lim,
                                        int &p0, int &p1) {
    p0 = p1 = 0;
    if (j < r.j0 || j > r.j1) return;
    const float ex = r.hx + lim, ey = r.hy + lim;
    const float rx = fmaf(r.ac, ex, r.as * ey), ry = fmaf(r.as, ex, r.ac * ey);
    const float lo_y = fmaf((float)j, g.cell, r.y0);
    const float a = fmaxf(lo_y, -ry), b = fminf(lo_y + r.dy, ry);
    const float u1 = r.k1 * a, v1 = r.k1 * b, w1 = ex * r.i1, u2 = r.k2 * a, v2 = r.k2 * b, w2 = ey * r.i2;
    const float lo = fmaxf(-rx, fmaxf(fminf(u1, v1) - w1, fminf(u2, v2) - w2));
    const float hi = fminf(rx, fminf(fmaxf(u1, v1) + w1, fmaxf(u2, v2) + w2));
    // a box shrunk to nothing, a row beyond it, or a non-finite pose
    if (!(ex >= 0.f && ey >= 0.f && a <= b && lo <= hi)) return;
    const float fa = (r.cwx + lo - g.lx) * g.inv, fb = (r.cwx + hi - g.lx) * g.inv;
    const int i0 = max(0, min(g.nx - 1, (int)fa)), i1 = min(g.nx - 1, max(0, (int)fb));
    p0 = __ldca(start + j * g.nx + i0);
    p1 = __ldca(start + j * g.nx + i1 + 1);
}

}  // namespace exact
