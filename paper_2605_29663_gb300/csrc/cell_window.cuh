// cell_window.cuh -- where most of a cloud lies, from the counts of its first
// sort into cells: a few points far from all others would stretch the cells until
// most of the cloud shares one.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

namespace exact {

// A sort is repeated over the window at most kZooms times (a point at 1e6 m
// beside a room takes four).
constexpr int kZooms = 6;

template <int NA, int NB>
struct WindowSmem {
    int a[NA], b[NB];   // points per row and column of cells
    int lo[2], hi[2];   // the window
};

// Counts cnt[i * nb + j] (rows with odd i run backwards when SERPENTINE), i < na
// <= NA, j < nb <= NB.  Along each axis the cells [lo, hi] beyond which about 1/64
// of the points lie on either side.  Every thread of the block calls; ends with a
// block barrier.
template <bool SERPENTINE, int NA, int NB>
__device__ __noinline__ void cell_window(const int *cnt, int na, int nb, WindowSmem<NA, NB> &w) {
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
    for (int c = tid; c < nb; c += nt) w.b[c] = 0;
    __syncthreads();
    for (int j0 = 0; j0 < nb; j0 += 32) {
        const int j = j0 + lane;
        int col = 0;
        for (int i = warp; i < na; i += nw) {
            const int n = j < nb ? cnt[i * nb + (SERPENTINE && (i & 1) ? nb - 1 - j : j)] : 0;
            col += n;
            const int row = __reduce_add_sync(0xffffffffu, n);
            if (lane == 0) w.a[i] = j0 ? w.a[i] + row : row;   // row i is this warp's
        }
        if (j < nb && col) atomicAdd(&w.b[j], col);
    }
    __syncthreads();
    if (warp < 2) {
        const int *h = warp ? w.b : w.a, n = warp ? nb : na, seg = (n + 31) / 32;
        const int e0 = lane * seg, e1 = min(n, e0 + seg);
        int sum = 0;
        for (int e = e0; e < e1; ++e) sum += h[e];
        int run = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, run, o);
            if (lane >= o) run += t;
        }
        const int all = __shfl_sync(0xffffffffu, run, 31), cut = all / 64;
        run -= sum;
        int lo = n - 1, hi = 0;
        for (int e = e0; e < e1; ++e) {
            const int before = run;
            run += h[e];
            if (before <= cut && run > cut) lo = e;
            if (before < all - cut && run >= all - cut) hi = e;
        }
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        if (lane == 0) { w.lo[warp] = lo; w.hi[warp] = hi; }
    }
    __syncthreads();
}

// Whether an axis of n cells of size step over [l, h] is worth cutting to the
// window: then [l, h] become its ends, a cell farther out.
__device__ __forceinline__ bool cut_axis(int n, float step, int lo, int hi, float &l, float &h) {
    if ((hi - lo + 3) * 4 > n || !(h - l > 1e-5f)) return false;
    const float l0 = l;
    if (lo > 0) l = l0 + (float)(lo - 1) * step;
    if (hi < n - 1) h = l0 + (float)(hi + 2) * step;
    return true;
}

}  // namespace exact
