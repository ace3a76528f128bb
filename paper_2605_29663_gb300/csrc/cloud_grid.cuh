// cloud_grid.cuh -- the cell grid over an obstacle cloud and the sample phase
// that walks it.
//
// A cycle without a d_min output needs, per (sample, step), only the points
// within d_safe of the footprint: every cost term and the validation test
// are the same for any d >= d_safe.  So one block per cloud sorts the points
// into the cells of a uniform grid (row-major, so consecutive cells of a row
// hold consecutive points), and the sample phase walks, per (sample, step),
// the grid rows that the footprint's bounding box (grown by d_safe and a
// slack far above rounding) crosses: each row contributes one contiguous run
// of points, found with two reads of the cell-start table.  A distance field
// of the footprint bounds each of those points' distances from both sides
// (fill_field), and only the points that can be a step's minimum are evaluated.
// No output changes by a bit: a point in no walked cell is farther than
// d_safe, and a point not evaluated is farther than one that is.
//
// What bounds it: instruction issue (49 to 71 % of the cycles issue) where
// many points lie inside the footprints, else the latency of one sample's
// rollout, walk and evaluation.  Measured against sub-chunk circles over a
// Morton-ordered copy (cycle times, the nominal driven to where the samples
// touch obstacles): forklift K = 2,048, T = 40, N = 4,096 120 to 135 -> 82 to 94 us; hybrid
// 3 x K = 1,024, N = 2,048 73 -> 41 us; 64 scenes of up to 20,000 points 6.47 ->
// 1.28 ms; predicted K = 1,024, N = 2,048 57 -> 27 us.  One warp per sample was
// slower than a block's warps sharing its samples (the forklift's near points
// range from 0 to 4,700 per sample).  Clouds below 1,024 points stay with
// the point-level pruning of steps_min_keys, which needs no launch before the
// samples (512 points, K = 256: 18 against 22 us; 100 points, K = 1,000: 24
// against 34 us).
#pragma once

#include "cell_window.cuh"
#include "mppi_cycle.cuh"

namespace exact {

constexpr int kGridThreads = 1024;
constexpr int kGridRegs = 4;          // points per thread kept in registers (clouds of up to 4,096)

struct GridSmem {
    int cnt[kCells + 1];
    float red[5][kGridThreads / 32];
    int part[kGridThreads / 32];
    WindowSmem<kGridDim, kGridDim> window;
};

// One block sorts the cloud's valid points (unmasked, finite position and
// velocity) into cells: opts / ovel in cell order, grid header and cell
// starts.  The order inside a cell follows the scatter's atomics; nothing
// computed from the cloud depends on it (minima are exact in any order).
// Where a cell holds more than 1/64 of the points and most of them lie in a small
// window, the cells are laid over that window again, and what lies outside goes
// to its border cells (GridHead::open): a cloud of 8,000 points on 12 m x 12 m and
// one point 10 km away, K = 2,048, T = 30, 80 us against 1,835 with cells over all of
// it.
// PREDICT: the points are taken where they are at time th.
template <bool MOVING, bool PREDICT = false>
__device__ __forceinline__ void build_grid(const float2 *__restrict__ pts, const float2 *__restrict__ vel,
                                           const uint8_t *__restrict__ mask, int N, float2 *__restrict__ opts,
                                           float2 *__restrict__ ovel, CloudGrid *__restrict__ grid, GridSmem &sm,
                                           float th = 0.f) {
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
    grid_dep_release();   // the sample kernel may start its rollouts meanwhile
    auto fetch = [&](int i, float2 &p, float2 &v) {
        p = pts[i];
        v = MOVING || PREDICT ? vel[i] : make_float2(0.f, 0.f);
        if (PREDICT) p = make_float2(fmaf(th, v.x, p.x), fmaf(th, v.y, p.y));
        return (!mask || mask[i]) && isfinite(p.x) && isfinite(p.y) && (!MOVING || (isfinite(v.x) && isfinite(v.y)));
    };
    // clouds of up to kGridRegs points per thread are read once and kept in
    // registers (point tid + k nt in slot k); larger ones are re-read per pass
    const bool inreg = N <= kGridRegs * nt;
    float2 rp[kGridRegs], rv[kGridRegs];
    bool ok[kGridRegs];
    if (inreg) {
#pragma unroll
        for (int k = 0; k < kGridRegs; ++k) {
            const int i = tid + k * nt;
            ok[k] = i < N && fetch(i, rp[k], rv[k]);
        }
    }
    float lx, ly, hx, hy, vm = 0.f;
    float wx0 = 0.f, wy0 = 0.f, wx1 = 0.f, wy1 = 0.f;   // the window
    float cell, inv;
    int nx, ny, ncell, rc[kGridRegs], rank[kGridRegs];   // cell, place among its points
    auto cell_of = [&](float2 p) { return cell_axis(p.y, ly, inv, ny) * nx + cell_axis(p.x, lx, inv, nx); };
    int c0, c1, s, inc;   // this thread's cells, their points, the warp's prefix
    // cells over the points (those in the window), the counts of all and the start
    // of their prefix; whether some cell holds more than 1/64 of them (from the
    // counts: a look at what the atomics return would wait for them)
    auto lay = [&](auto windowed) {
        constexpr bool W = decltype(windowed)::value;
        lx = ly = finf();
        hx = hy = -finf();
        auto grow = [&](float2 p, float2 v) {
            if (W && (p.x < wx0 || p.x > wx1 || p.y < wy0 || p.y > wy1)) return;
            lx = fminf(lx, p.x); hx = fmaxf(hx, p.x); ly = fminf(ly, p.y); hy = fmaxf(hy, p.y);
            if (MOVING && !W) vm = fmaxf(vm, fabsf(v.x) + fabsf(v.y));
        };
        if (inreg) {
#pragma unroll
            for (int k = 0; k < kGridRegs; ++k)
                if (ok[k]) grow(rp[k], rv[k]);
        } else {
#pragma unroll 4
            for (int i = tid; i < N; i += nt) {
                float2 p, v;
                if (fetch(i, p, v)) grow(p, v);
            }
        }
        for (int c = tid; c <= kCells; c += nt) sm.cnt[c] = 0;
        lx = warp_min_f(lx); ly = warp_min_f(ly); hx = -warp_min_f(-hx); hy = -warp_min_f(-hy);
        if (MOVING && !W) vm = -warp_min_f(-vm);
        if (lane == 0) {
            sm.red[0][warp] = lx; sm.red[1][warp] = ly; sm.red[2][warp] = hx; sm.red[3][warp] = hy;
            if (!W) sm.red[4][warp] = vm;
        }
        __syncthreads();
        {   // every warp reduces the warps' boxes itself: one barrier less
            const bool w = lane < nw;
            lx = warp_min_f(w ? sm.red[0][lane] : finf());
            ly = warp_min_f(w ? sm.red[1][lane] : finf());
            hx = -warp_min_f(w ? -sm.red[2][lane] : finf());
            hy = -warp_min_f(w ? -sm.red[3][lane] : finf());
            if (MOVING && !W) vm = -warp_min_f(w ? -sm.red[4][lane] : 0.f);
        }
        // square cells over the box; a cloud without a valid point gets one cell
        const bool any = lx <= hx;
        if (!any) lx = ly = hx = hy = 0.f;
        const float w = hx - lx, h = hy - ly, wide = fmaxf(w, h);
        const float target = fminf(kCellTarget, fmaxf(1000.f, 2.f * (float)N));
        cell = fmaxf(fmaxf(sqrtf(w * (h / target)), wide / (float)(kGridDim - 1)), 1e-6f);
        inv = 1.f / cell;
        nx = min(kGridDim, (int)(w * inv) + 1);
        ny = min(kGridDim, (int)(h * inv) + 1);
        ncell = min(kCells, nx * ny);
        if (inreg) {
#pragma unroll
            for (int k = 0; k < kGridRegs; ++k)
                if (ok[k]) {
                    rc[k] = min(ncell - 1, cell_of(rp[k]));
                    rank[k] = atomicAdd(&sm.cnt[rc[k]], 1);
                }
        } else {
#pragma unroll 4
            for (int i = tid; i < N; i += nt) {
                float2 p, v;
                if (fetch(i, p, v)) atomicAdd(&sm.cnt[min(ncell - 1, cell_of(p))], 1);
            }
        }
        __syncthreads();
        // exclusive prefix over the counts: contiguous segments per thread
        const int per = ((ncell + nt) / nt) | 1;   // odd: no bank conflicts
        c0 = tid * per;
        c1 = min(ncell + 1, c0 + per);
        bool crowded = false;
        s = 0;
        for (int c = c0; c < c1; ++c) {
            const int n = sm.cnt[c];
            s += n;
            crowded |= n > N / 64;
        }
        inc = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        if (lane == 31) sm.part[warp] = inc;
        return __syncthreads_or(crowded) != 0;
    };
    int open = 0;
    if (lay(std::false_type{}))
        for (int zoom = 0; zoom < kZooms; ++zoom) {
            cell_window<false>(sm.cnt, ny, nx, sm.window);
            wx0 = lx; wx1 = hx; wy0 = ly; wy1 = hy;
            const bool cx = cut_axis(nx, cell, sm.window.lo[1], sm.window.hi[1], wx0, wx1);
            const bool cy = cut_axis(ny, cell, sm.window.lo[0], sm.window.hi[0], wy0, wy1);
            if (!cx && !cy) break;
            open = 1;
            if (!lay(std::true_type{})) break;
        }
    {   // the totals of the warps below, again by every warp itself
        int v = lane < warp ? sm.part[lane] : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        int run = v + inc - s;
        for (int c = c0; c < c1; ++c) {
            const int n = sm.cnt[c];
            sm.cnt[c] = run;   // cell ncell holds no point: the number of valid points
            run += n;
        }
    }
    if (tid == 0) {
        grid->head = GridHead{lx, ly, inv, cell, MOVING ? vm * 1.0001f : 0.f, open, nx, ny};
    }
    __syncthreads();
    for (int c = tid; c <= ncell; c += nt) grid->start[c] = sm.cnt[c];
    if (inreg) {
#pragma unroll
        for (int k = 0; k < kGridRegs; ++k)
            if (ok[k]) {
                const int pos = sm.cnt[rc[k]] + rank[k];
                opts[pos] = rp[k];
                if (MOVING) ovel[pos] = rv[k];
            }
    } else {
        __syncthreads();   // the starts are written: the counts may move
#pragma unroll 4
        for (int i = tid; i < N; i += nt) {
            float2 p, v;
            if (fetch(i, p, v)) {
                const int pos = atomicAdd(&sm.cnt[min(ncell - 1, cell_of(p))], 1);
                opts[pos] = p;
                if (MOVING) ovel[pos] = v;
            }
        }
    }
}

// ---------------------------------------------------------------- sample phase
// One block takes up to kGroup samples of a scene at a time: one warp each
// rolls them out, then all warps share out the (sample, step) slots, a few
// steps at a time from a shared counter (a sample that drives through a wall
// has thousands of near points, its neighbour none), then one warp each forms
// the J~.
constexpr int kGroup = 16;
constexpr int kRuns = 64;     // a warp's queued runs: 32 are handled at a time, at most 31 stay
constexpr int kEvals = 128;   // a warp's queued points: 64 are evaluated at a time, at most 63 stay
constexpr int kField = 32;    // cells of the footprint's distance field along one axis
__host__ __device__ constexpr int grid_T_pad(int T) { return (T + 3) / 4 * 4; }
__host__ __device__ constexpr size_t grid_smem_bytes(int T, int samples, int warps) {
    return kField * kField * 4 + (size_t)grid_T_pad(T) * 32 * samples + kGroup * 4 + (size_t)warps * (kRuns * 12 + kEvals * 8);
}
// grid_group keeps a block of 256 threads to kGridSmem; the largest block has
// 512.  The kernels' limit is always set to kGridSmemMax, whatever a call or a
// plan needs itself: the limit belongs to the kernel, and a smaller one would
// be another plan's or thread's too.
constexpr size_t kGridSmem = 70 * 1024, kGridSmemMax = kGridSmem + (512 - kBlock) / 32 * (kRuns * 12 + kEvals * 8);
static_assert(grid_smem_bytes(EXACT_MAX_HORIZON, 1, kBlock / 32) <= kGridSmem, "one sample of the longest horizon fits");

// Samples per block: as few as keep the blocks to three per SM, so that a small
// sample count still spreads over the GPU, and up to 16 beyond, which is where
// a block's three phases and their barriers cost least (64 scenes with 114,688
// samples: groups of 4, 8, 16, 24 take 1.94, 1.55, 1.35, 1.41 ms; the forklift's
// 2,048 samples: groups of 3, 5, 7 take 94, 87, 93 us).
// A long horizon lowers it to what leaves three blocks their shared memory.
inline int grid_group(long long samples, int T, int warps, int sms) {
    const long long slots = 3LL * (sms > 0 ? sms : 148), want = (samples + slots - 1) / slots;
    int g = (int)(want < 1 ? 1 : want > kGroup ? kGroup : want);
    while (g > 1 && grid_smem_bytes(T, g, warps) > kGridSmem) --g;
    return g;
}

// Minimum of floats of either sign (not NaN): their bits order as signed
// integers when positive, the other way round when negative.
__device__ __forceinline__ void atomic_min(float *a, float v) {
    if (v >= 0.f)
        atomicMin(reinterpret_cast<int *>(a), __float_as_int(v));
    else
        atomicMax(reinterpret_cast<unsigned *>(a), __float_as_uint(v));
}

// The footprint's signed distance at the centres of kField x kField cells over
// its bounding box grown by d_safe (and the slack): for a point in a cell the
// distance is within rd (half the cell's diagonal, and a slack far above
// rounding) of the centre's, because every signed distance is 1-Lipschitz.
// So one shared-memory read bounds a point's distance from both sides: the
// smallest upper bound of a step's points replaces d_safe as what still
// matters, and only the points whose lower bound is below it are evaluated
// (a few per step, whatever the number of points inside the footprint).
// A safety distance far beyond the footprint's size would leave the cells too
// coarse to tell its points apart: the field then ends at twice the box's half
// extent, and beyond it the box bounds the distance (its own, and that of its
// farthest corner).  (K = 1,024, T = 30, 4,000 points all within d_safe = 50 m:
// 207 us against 923 with the field over all of it, forklift 142 against 654.)
struct Field {
    float x0, y0, ix, iy, rd;
};
// Whether the field ends before d_safe (the kernels' FAR: as a branch at run time
// it cost every cycle 1 to 2 %).
__host__ __device__ inline bool field_ends(float d_safe, float hx, float hy) { return d_safe > 2.f * fmaxf(hx, hy); }
template <class EV>
__device__ __forceinline__ Field make_field(const EV &ev, float cap) {
    const float4 fb = ev.box();
    const float m = fminf(cap, 2.f * fmaxf(fb.z, fb.w));
    const float hx = fb.z + m + 2.f * kPruneSlack, hy = fb.w + m + 2.f * kPruneSlack;
    const float cx = 2.f * hx / kField, cy = 2.f * hy / kField;
    return Field{fb.x - hx, fb.y - hy, 1.f / cx, 1.f / cy, fmaf(0.50001f, sqrtf(fmaf(cx, cx, cy * cy)), 0.1f * kPruneSlack)};
}
template <class EV>
__device__ __forceinline__ void fill_field(const EV &ev, const Field &f, float *field) {
    const float cx = 1.f / f.ix, cy = 1.f / f.iy;
    for (int i = 2 * threadIdx.x; i < kField * kField; i += 2 * blockDim.x) {
        const float x = fmaf((float)(i % kField) + 0.5f, cx, f.x0), y = fmaf((float)(i / kField) + 0.5f, cy, f.y0);
        float k0, k1;
        ev.eval2(x, y, x + cx, y, k0, k1);
        *reinterpret_cast<float2 *>(field + i) = make_float2(ev.dist(k0), ev.dist(k1));
    }
}

// Samples [r0, r0 + ns) of a scene, ns <= kGroup; every thread of the block
// calls.  mem holds grid_smem_bytes(V.P.T, ns, warps) bytes, first the
// footprint's distance field (filled here when fill is set), and next is a
// shared counter.  The keys are the same bits whatever warp takes a slot.
// FAR: field_ends for the scene (and right, but slower, where it does not).
template <bool MOVING, bool FAR, class EV>
__device__ __forceinline__ void grid_samples(const SceneView &V, const CloudGrid *grid, GridStride gst, const EV &ev,
                                             int r0, int ns, char *mem, bool fill, int *next) {
    const MppiP &P = V.P;
    const int T = P.T, nu = P.nu, Tp = grid_T_pad(T), lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nwarps = blockDim.x >> 5;
    const unsigned full = 0xffffffffu;
    // per slot (sample s, step h) = s Tp + h
    float *field = reinterpret_cast<float *>(mem);
    float4 *pose = reinterpret_cast<float4 *>(field + kField * kField);
    unsigned *key = reinterpret_cast<unsigned *>(pose + ns * Tp);   // minimum order key
    float *lim = reinterpret_cast<float *>(key + ns * Tp);          // distance that still matters
    float *stage = lim + ns * Tp;                                   // stage cost without the obstacle term
    float *time = stage + ns * Tp;                                  // time of the scored state
    float *term = time + ns * Tp;                                   // per sample: terminal cost
    // this warp's queues: points to evaluate (slot, point); runs of points (slot, first, count)
    char *own = reinterpret_cast<char *>(term + kGroup) + warp * (kRuns * 12 + kEvals * 8);
    int2 *eval = reinterpret_cast<int2 *>(own);
    int *run_p = reinterpret_cast<int *>(eval + kEvals), *run_n = run_p + kRuns, *run_s = run_n + kRuns;
    const float cap = fminf(fmaxf(P.d_safe, 0.f), kCapMax);
    const Field fd = make_field(ev, cap);
    if (fill) fill_field(ev, fd, field);
    for (int s = warp; s < ns; s += nwarps) {
        const int r = r0 + s, off = s * Tp;
        if (r == 0 && lane == 0 && !(isfinite(V.state[0]) && isfinite(V.state[1]) && isfinite(V.state[2])))
            report_error(V.err, EXACT_EINVAL);   // a start state the host could not see is not finite
        const float *U = V.U;
        const float *eps = V.noise + (size_t)r * T * nu;
        LaneRollout R;
        warp_rollout(P, V.state[0], V.state[1], V.state[2],
                     [&](int h, int j) { return clamp_u(P, j, U[h * nu + j] + eps[h * nu + j]); }, R);
#pragma unroll
        for (int e = 0; e < kMaxPerLane; ++e) {
            const int h = lane * R.per + e;
            if (e < R.per && h < T) {
                float sn, cs;
                sincosf(R.th[e], &sn, &cs);
                pose[off + h] = make_float4(R.x[e], R.y[e], cs, sn);
                key[off + h] = f2ord(finf());
                lim[off + h] = cap;
                time[off + h] = (float)(h + P.state_offset) * P.dt;
                const float u2 = fmaf(R.u[e][0], R.u[e][0], fmaf(R.u[e][1], R.u[e][1], R.u[e][2] * R.u[e][2]));
                stage[off + h] = fmaf(P.w_goal, guidance_dist(R.x[e], R.y[e], V.wp, V.W), P.w_ctrl * u2);
            }
        }
        if (lane == 0) term[s] = P.w_term * guidance_dist(R.qTx, R.qTy, V.wp, V.W);
    }
    if (threadIdx.x == 0) *next = 0;
    grid_dep_wait();   // launched early behind the kernel that builds the grid
    __syncthreads();
    {
        const float4 fb = ev.box();
        int nruns = 0, nev = 0;   // queued runs and points (warp-uniform)

        auto point_at = [&](int i, int slot) -> float2 {
            float2 o = __ldca(V.pts + i);
            if constexpr (MOVING) {
                const float th = time[slot];
                const float2 v = __ldca(V.vel + i);
                o = make_float2(fmaf(th, v.x, o.x), fmaf(th, v.y, o.y));
            }
            return o;
        };
        auto evaluate = [&](int cnt) {   // queued points [0, cnt), cnt <= 64: two per lane
            __syncwarp();
            const int a = 2 * lane;
            if (a < cnt) {
                const bool two = a + 1 < cnt;
                const int2 ea = eval[a], eb = two ? eval[a + 1] : ea;
                const float2 oa = point_at(ea.y, ea.x), ob = point_at(eb.y, eb.x);
                const float4 pa = pose[ea.x], pb = pose[eb.x];
                float pxa, pya, pxb, pyb;
                body_frame(oa.x, oa.y, pa.x, pa.y, pa.z, pa.w, pxa, pya);
                body_frame(ob.x, ob.y, pb.x, pb.y, pb.z, pb.w, pxb, pyb);
                float ka, kb;
                ev.eval2(pxa, pya, pxb, pyb, ka, kb);
                const unsigned oa2 = f2ord(ka), ob2 = f2ord(kb);
                if (oa2 < key[ea.x]) atomicMin(key + ea.x, oa2);
                if (ob2 < key[eb.x]) atomicMin(key + eb.x, ob2);
            }
            __syncwarp();
        };
        // the points of queued runs [0, n), n <= 32, dealt 64 at a time: those
        // whose lower bound is below their slot's limit go to the evaluation
        // queue.  The run of a dealt point is found by counting the runs that
        // start at or before it: a bit per start in the window's mask
        auto walk_runs = [&](int n) {
            __syncwarp();
            const int cnt = lane < n ? run_n[lane] : 0, rs = lane < n ? run_s[lane] : 0;
            int incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(full, incl, o);
                if (lane >= o) incl += t;
            }
            const int excl = incl - cnt, off = (lane < n ? run_p[lane] : 0) - excl;   // first point, from the dealt index
            const int total = __shfl_sync(full, incl, 31);
            const unsigned upto = (2u << lane) - 1u;
            for (int b = 0; b < total; b += 64) {
                float lb[2], ub[2], now[2];   // bounds of the distance; the slot's limit
                int i[2], sl[2];
                bool lower = false;
                const int rel = excl - b;
                const unsigned lo = __reduce_or_sync(full, (unsigned)rel < 32u ? 1u << rel : 0u);
                const unsigned hi = __reduce_or_sync(full, (unsigned)(rel - 32) < 32u ? 1u << (rel - 32) : 0u);
                const int before = __popc(__ballot_sync(full, rel < 0)) - 1;
                const int k[2] = {before + __popc(lo & upto), before + __popc(lo) + __popc(hi & upto)};
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int t = b + 32 * q + lane;
                    i[q] = t + __shfl_sync(full, off, k[q] & 31);
                    sl[q] = __shfl_sync(full, rs, k[q] & 31);
                    lb[q] = ub[q] = finf();
                    now[q] = lim[sl[q]];
                    if (t < total) {
                        const float4 p = pose[sl[q]];
                        const float2 o = point_at(i[q], sl[q]);
                        float px, py;
                        body_frame(o.x, o.y, p.x, p.y, p.z, p.w, px, py);
                        // cell of the field; a point outside one that reaches as far is farther than d_safe
                        const float u = (px - fd.x0) * fd.ix, v = (py - fd.y0) * fd.iy;
                        if (u >= 0.f && u < (float)kField && v >= 0.f && v < (float)kField) {
                            const float f = field[(int)v * kField + (int)u];
                            lb[q] = f - fd.rd;
                            ub[q] = f + fd.rd;
                        } else if constexpr (FAR) {
                            const float ax = fabsf(px - fb.x), ay = fabsf(py - fb.y);
                            const float e = fmaf(1e-5f, ax + ay, 0.1f * kPruneSlack);
                            lb[q] = fmaxf(ax - fb.z, ay - fb.w) - e;
                            ub[q] = (ax + fb.z) + (ay + fb.w) + e;
                        }
                    }
                    lower |= ub[q] < now[q];
                }
                if (__any_sync(full, lower)) {   // some point's distance is below the limit: it falls
#pragma unroll
                    for (int q = 0; q < 2; ++q)
                        if (ub[q] < now[q]) atomic_min(lim + sl[q], ub[q]);
                    __syncwarp();
#pragma unroll
                    for (int q = 0; q < 2; ++q) now[q] = *(volatile float *)(lim + sl[q]);
                }
                const bool keep[2] = {lb[0] <= now[0], lb[1] <= now[1]};
                const unsigned b0 = __ballot_sync(full, keep[0]), b1 = __ballot_sync(full, keep[1]);
                if (b0 | b1) {
                    const unsigned below = (1u << lane) - 1u;
                    if (keep[0]) eval[nev + __popc(b0 & below)] = make_int2(sl[0], i[0]);
                    nev += __popc(b0);
                    if (keep[1]) eval[nev + __popc(b1 & below)] = make_int2(sl[1], i[1]);
                    nev += __popc(b1);
                    if (nev >= 64) {
                        evaluate(64);
                        int2 m0 = make_int2(0, 0), m1 = m0;
                        if (lane < nev - 64) m0 = eval[64 + lane];
                        if (lane + 32 < nev - 64) m1 = eval[96 + lane];
                        __syncwarp();
                        if (lane < nev - 64) eval[lane] = m0;
                        if (lane + 32 < nev - 64) eval[32 + lane] = m1;
                        nev -= 64;
                    }
                }
            }
        };

        // slots in groups of `per` steps of one sample from the shared counter:
        // about three groups per warp, 4 to 8 steps; 32 / per' lanes share a
        // step's rows (per' = per rounded up to a power of two)
        const int per = max(4, min(8, ns * T / (3 * nwarps)));
        const int groups = (T + per - 1) / per, items = ns * groups;
        int lg = 5;
        while ((32 >> lg) < per) --lg;
        const int lanes = 1 << lg, phase = lane & (lanes - 1);
        for (;;) {
            int item = 0;
            if (lane == 0) item = atomicAdd(next, 1);
            item = __shfl_sync(full, item, 0);
            if (item >= items) break;
            const int sm = item / groups, q = lane >> lg, h = (item - sm * groups) * per + q, slot = sm * Tp + h;
            RowWalk w;
            GridHead g;
            const CloudGrid *gh = grid + h * gst.grids;
            const int base = h * gst.points;
            int rows = 0;
            float reach = kPruneSlack;   // a predicted point may have moved by t_h vmax
            if (q < per && h < T) {
                g = load_head(gh);
                if (MOVING) reach = fmaf(time[slot], g.vmax, reach);
                w = row_walk(g, pose[slot], fb, cap + reach);
                rows = walk_rows(w);
            }
            for (int k = phase; __any_sync(full, k < rows); k += lanes) {
                int p0 = 0, p1 = 0;
                if (k < rows) row_run(g, gh->start, w, walk_row(w, k), lim[slot] + reach, p0, p1);
                const bool some = p1 > p0;
                const unsigned b = __ballot_sync(full, some);
                if (b) {
                    if (some) {
                        const int at = nruns + __popc(b & ((1u << lane) - 1u));
                        run_p[at] = base + p0;
                        run_n[at] = p1 - p0;
                        run_s[at] = slot;
                    }
                    nruns += __popc(b);
                    if (nruns >= 32) {
                        walk_runs(32);
                        int a = 0, n = 0, c = 0;
                        if (lane < nruns - 32) { a = run_p[32 + lane]; n = run_n[32 + lane]; c = run_s[32 + lane]; }
                        __syncwarp();
                        if (lane < nruns - 32) { run_p[lane] = a; run_n[lane] = n; run_s[lane] = c; }
                        nruns -= 32;
                    }
                }
            }
        }
        if (nruns > 0) walk_runs(nruns);
        if (nev > 0) evaluate(nev);
    }
    __syncthreads();
    for (int s = warp; s < ns; s += nwarps) {
        const int off = s * Tp;
        ff acc{0.f, 0.f};
        bool unsafe = false;
        for (int h = lane; h < T; h += 32) {
            const float kh = ord2f(key[off + h]);
            const float d = kh == finf() ? finf() : ev.dist(kh);
            acc = add_phi_obs(P, d, ff_add(acc, stage[off + h]));
            unsafe |= d < P.d_safe;
        }
        acc = warp_sum_ff(acc);
        const bool chi = __any_sync(full, unsafe);
        if (lane == 0) finish_cost(V, r0 + s, acc, term[s], chi);
    }
}

}  // namespace exact
