// sdf_near.cu -- exact_sdf_batch for many poses against one cloud: the same
// distances, minima and argmins as sdf_batch.cu, with the work that cannot
// matter left out.
//
// A block first sorts every chunk of kChunk points into spatial order (strips
// about as wide as a patch of 64 points is, each walked up and down by turns:
// compact patches, 0.73 m against 1.22 m mean radius in Morton order for 8,192
// points on 12 m x 12 m) and takes the bounding circle of every patch of 64
// consecutive points.  The matrix kernel and the minimum
// kernel below then decide per (pose, patch), for 64 points at once, what
// each point would otherwise pay for.  Measured (calls of exact_sdf_batch):
// 16,384 poses x 8,192 points x 32 edges 1,227 -> 710 to 728 us; the minimum of
// 3,000 poses x 20,001 points x 12 edges 240 -> 40 to 47 us.
#include "cell_window.cuh"
#include "mppi_cycle.cuh"
#include "sdf_near.h"

namespace exact {

constexpr int kChunk = kSdfChunk;        // points sorted together; their copy fits a block's shared memory
constexpr int kPatch = 64;               // points of a patch: two per lane
constexpr int kPatches = kChunk / kPatch;
constexpr int kSortThreads = 1024;
constexpr int kNearThreads = 1024;       // matrix kernel: one block per SM
constexpr int kRows = 4;                 // row buffers of a block
constexpr int kMinThreads = 128;

// Points of each chunk of a cloud: as equal as whole patches allow.
inline int chunk_points(int N) {
    const int n = (N + kChunk - 1) / kChunk, per = (N + n - 1) / n;
    return (per + kPatch - 1) / kPatch * kPatch;
}

// One sorted chunk: points (invalid ones last, as NaN, which every evaluation
// turns into +inf), their indices in the chunk, and the patches' circles
// (centre, radius or -1 for a patch without a valid point).
struct __align__(256) SortedChunk {
    float2 pts[kChunk];
    unsigned short idx[kChunk];
    float4 circ[kPatches];
};

size_t sdf_near_bytes(int n_points) { return sizeof(SortedChunk) * (((size_t)n_points + kChunk - 1) / kChunk); }

// Latency-bound (one block per chunk): the chunk is read once into registers,
// eight points per thread, and counting-sorted through shared memory.
__global__ void __launch_bounds__(kSortThreads)
sdf_sort_kernel(const float2 *__restrict__ pts, const uint8_t *__restrict__ mask, int N, int csize,
                SortedChunk *__restrict__ out) {
    constexpr int kCellsS = 64 * 64, kPer = kChunk / kSortThreads, kSeg = kCellsS / kSortThreads;
    __shared__ int cnt[kCellsS + 1];
    __shared__ float red[4][32];
    __shared__ int part[32];
    extern __shared__ __align__(16) char s_sort[];   // the sorted chunk
    float2 *s_pts = reinterpret_cast<float2 *>(s_sort);
    unsigned short *s_idx = reinterpret_cast<unsigned short *>(s_pts + kChunk);
    using Window = WindowSmem<64, kCellsS>;   // in the same place, before the points are sorted
    static_assert(sizeof(Window) <= kChunk * sizeof(float2), "the window's counts fit");
    Window &window = *reinterpret_cast<Window *>(s_sort);
    SortedChunk &C = out[blockIdx.x];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int base = blockIdx.x * csize, n = min(csize, N - base);
    float2 p[kPer];
    bool ok[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const int i = tid + k * kSortThreads;
        ok[k] = false;
        if (i < n) {
            p[k] = pts[base + i];
            ok[k] = (!mask || mask[base + i]) && isfinite(p[k].x) && isfinite(p[k].y);
        }
    }
    // strips across x, bins along y within each, over all points or, where most
    // of them share a few cells, over the window these lie in (cell_window): what
    // lies outside goes to its border (4,096 poses x 8,192 points x 32 edges, one
    // point 10 km away: 217 us against 732)
    float wx0 = 0.f, wy0 = 0.f, wx1 = 0.f, wy1 = 0.f;
    float lx, ly, hx, hy, w, h;
    int cell[kPer], strips, bins;
    int s, inc, c[kSeg];
    // counts, and the start of their prefix; whether some cell holds more than
    // 1/64 of the points
    auto lay = [&](auto windowed) {
        constexpr bool W = decltype(windowed)::value;
        lx = ly = finf();
        hx = hy = -finf();
#pragma unroll
        for (int k = 0; k < kPer; ++k)
            if (ok[k] && !(W && (p[k].x < wx0 || p[k].x > wx1 || p[k].y < wy0 || p[k].y > wy1))) {
                lx = fminf(lx, p[k].x); hx = fmaxf(hx, p[k].x); ly = fminf(ly, p[k].y); hy = fmaxf(hy, p[k].y);
            }
        for (int q = tid; q <= kCellsS; q += kSortThreads) cnt[q] = 0;
        lx = warp_min_f(lx); ly = warp_min_f(ly); hx = -warp_min_f(-hx); hy = -warp_min_f(-hy);
        if (lane == 0) { red[0][warp] = lx; red[1][warp] = ly; red[2][warp] = hx; red[3][warp] = hy; }
        __syncthreads();
        lx = warp_min_f(red[0][lane]); ly = warp_min_f(red[1][lane]);
        hx = -warp_min_f(-red[2][lane]); hy = -warp_min_f(-red[3][lane]);
        w = fmaxf(hx - lx, 1e-6f);
        h = fmaxf(hy - ly, 1e-6f);
        const float side = sqrtf(w * (h * ((float)kPatch / (float)n)));
        strips = min(64, max(1, (int)(w / side + 0.5f)));
        bins = kCellsS / strips;
        const float sx = (float)strips / w, sy = (float)bins / h;
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            cell[k] = kCellsS;   // invalid (and absent) points last
            if (ok[k]) {
                const int a = min(strips - 1, max(0, (int)((p[k].x - lx) * sx)));
                const int b = min(bins - 1, max(0, (int)((p[k].y - ly) * sy)));
                cell[k] = a * bins + ((a & 1) ? bins - 1 - b : b);
            }
            if (tid + k * kSortThreads < n) atomicAdd(&cnt[cell[k]], 1);
        }
        __syncthreads();
        bool crowded = false;
        s = 0;   // the last count (invalid points) needs no prefix of its own
#pragma unroll
        for (int k = 0; k < kSeg; ++k) {
            s += c[k] = cnt[tid * kSeg + k];
            crowded |= c[k] > n / 64;
        }
        inc = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        if (lane == 31) part[warp] = inc;
        return __syncthreads_or(crowded) != 0;
    };
    if (lay(std::false_type{}))
        for (int zoom = 0; zoom < kZooms; ++zoom) {
            cell_window<true>(cnt, strips, bins, window);
            wx0 = lx; wx1 = hx; wy0 = ly; wy1 = hy;
            const bool cx = cut_axis(strips, w / (float)strips, window.lo[0], window.hi[0], wx0, wx1);
            const bool cy = cut_axis(bins, h / (float)bins, window.lo[1], window.hi[1], wy0, wy1);
            if ((!cx && !cy) || !lay(std::true_type{})) break;
        }
    int run = lane < warp ? part[lane] : 0, all = part[lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        run += __shfl_xor_sync(0xffffffffu, run, o);
        all += __shfl_xor_sync(0xffffffffu, all, o);
    }
    run += inc - s;
#pragma unroll
    for (int k = 0; k < kSeg; ++k) {
        cnt[tid * kSeg + k] = run;
        run += c[k];
    }
    if (tid == 0) cnt[kCellsS] = all;
    __syncthreads();
    const float qnan = __int_as_float(0x7fffffff);
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const int i = tid + k * kSortThreads;
        // absent points fill the end of the chunk (their results are not stored)
        const int at = i < n ? atomicAdd(&cnt[cell[k]], 1) : i;
        s_pts[at] = ok[k] ? p[k] : make_float2(qnan, qnan);
        s_idx[at] = (unsigned short)i;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kPer / 2; ++k)
        reinterpret_cast<float4 *>(C.pts)[tid + k * kSortThreads] = reinterpret_cast<const float4 *>(s_pts)[tid + k * kSortThreads];
    static_assert(kChunk / 8 == kSortThreads, "one 16-byte piece of indices per thread");
    reinterpret_cast<uint4 *>(C.idx)[tid] = reinterpret_cast<const uint4 *>(s_idx)[tid];
    for (int q = warp; q < kPatches; q += kSortThreads / 32) {
        const float2 a = s_pts[q * kPatch + lane], b = s_pts[q * kPatch + 32 + lane];
        const float x0 = warp_min_f(fminf(a.x, b.x)), y0 = warp_min_f(fminf(a.y, b.y));   // NaN ignored
        const float x1 = -warp_min_f(-fmaxf(a.x, b.x)), y1 = -warp_min_f(-fmaxf(a.y, b.y));
        const float cx = 0.5f * (x0 + x1), cy = 0.5f * (y0 + y1);
        float r2 = 0.f;
        if (a.x == a.x) r2 = fmaxf(r2, fmaf(a.x - cx, a.x - cx, (a.y - cy) * (a.y - cy)));
        if (b.x == b.x) r2 = fmaxf(r2, fmaf(b.x - cx, b.x - cx, (b.y - cy) * (b.y - cy)));
        r2 = -warp_min_f(-r2);
        const float r = sqrtf(r2) * 1.000001f;
        if (lane == 0) C.circ[q] = x0 <= x1 ? make_float4(cx, cy, r, 0.f) : make_float4(0.f, 0.f, -1.f, 0.f);
    }
}

// ---------------------------------------------------------------- matrix
// Polygons: which edges can be the nearest of some point of a patch.  With
// the patch's circle (c, r) in the body frame, f the edge nearest to c and a
// its nearest point, every p in the circle has d_f(p) <= |p - a|, and for any
// b on edge e
//   |p - b|^2 - |p - a|^2 = |c - b|^2 - |c - a|^2 + 2 (p - c) . (a - b)
//                        >= d_e(c)^2 - d_f(c)^2 - 2 r |a - b|,
// so edge e is not needed where d_e(c)^2 > d_f(c)^2 + 2 r max_b |a - b| (b an
// end of e).  A margin of 1e-5 of the squared coordinates in the body frame,
// far above the rounding of the squared distances (that of o - t is relative to
// the difference, wherever both lie on the map), keeps every edge whose computed
// distance could be the minimum: the minimum over the kept edges is the same
// bits.  One
// lane per edge, two ballots per patch; far from a 32-gon about 4 edges stay.
struct EdgeLane {
    float vx, vy, ex, ey, exn, eyn;
    bool on;
};
__device__ __forceinline__ EdgeLane edge_lane(const float4 *C, int E, int n, int e) {
    EdgeLane l = {};
    l.on = e < n;
    if (l.on) {
        const float4 v = C[3 * e], k = C[3 * e + 1], d = C[3 * e + 2];
        l.vx = -v.x; l.vy = -v.z; l.ex = -d.x; l.ey = -d.z;
        l.exn = k.x;
        l.eyn = reinterpret_cast<const float *>(C + 3 * E + 1)[e];
    }
    return l;
}
struct EdgeNear {
    float d2, qx, qy, dx, dy;   // squared distance of the centre, centre - nearest point, centre - v
};
__device__ __forceinline__ EdgeNear edge_near(const EdgeLane &l, float cx, float cy) {
    const float dx = cx - l.vx, dy = cy - l.vy;
    const float t = __saturatef(fmaf(dy, l.eyn, dx * l.exn));
    const float qx = fmaf(-t, l.ex, dx), qy = fmaf(-t, l.ey, dy);
    return EdgeNear{l.on ? fmaf(qy, qy, qx * qx) : finf(), qx, qy, dx, dy};
}

// Block b takes its equal share of the (chunk, pose) rows.  A chunk's sorted
// points stay in shared memory over all its poses; a row is gathered in
// shared memory in the caller's order and leaves as one bulk copy (or, when
// its address or length is not a multiple of 16 bytes, by coalesced stores).
// All warps but the last take the (pose, patch) items round-robin over all the
// block's poses, a near patch costing three far ones, and run up to kRows rows
// ahead; the last warp waits for a row's warps (mbarrier full), stores it,
// reduces its minimum and hands the buffer back (mbarrier empty).  Bound by
// instruction issue.  (With a block barrier after each pair of poses instead,
// the warps waited for the slowest: 777 against 704 us for 16,384 poses x 8,192
// points x 32 edges.)
template <bool WIDE>   // more than 32 edges
__global__ void __launch_bounds__(kNearThreads)
sdf_matrix_kernel(const SortedChunk *__restrict__ chunks, int N, int csize, int nch, const float *__restrict__ poses, int P,
                  const __grid_constant__ FpTable fp, int n_edges, float *__restrict__ dist, int bulk,
                  float *__restrict__ dmin, int *__restrict__ argmin, unsigned long long *__restrict__ keys, int *err) {
    extern __shared__ __align__(128) char s_mem[];
    float2 *pts = reinterpret_cast<float2 *>(s_mem);
    float *rows = reinterpret_cast<float *>(pts + kChunk);                     // kRows of kChunk
    float4 *circ = reinterpret_cast<float4 *>(rows + kRows * kChunk);
    unsigned short *idx = reinterpret_cast<unsigned short *>(circ + kPatches);
    __shared__ float4 s_fp[kFpSlots];
    __shared__ float4 s_edge[3 * EXACT_MAX_POLY_VERTICES];   // (-v, -v), (e/|e|^2: x, x, y), (-e, -e) per edge
    constexpr int nwarps = kNearThreads / 32 - 1;            // computing warps
    __shared__ unsigned long long red[kRows][nwarps + 1];
    __shared__ unsigned long long full[kRows], empty[kRows];
    __shared__ int gone;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int E = fp.n;
    if (tid == 0) gone = 0;
    if (tid == 0)
        for (int k = 0; k < kRows; ++k) {
            mbar_init(full + k, nwarps);
            mbar_init(empty + k, 1);
            red[k][nwarps] = kNoKey;
        }
    // Bounded, as every wait here: when the phase has not come the error is
    // recorded and the thread leaves the kernel, its copies in flight completed;
    // the storing warp then stores no further row, and the others' waits end the
    // same way.  Two limits in a row: the first may have passed while the GPU ran
    // another program.  (An exit that the compiler does not see: a return or a
    // vote here cost registers, and the loop over the patches 5 % on clouds
    // dense on the footprint.)
    auto leave = []() { asm volatile("cp.async.bulk.wait_group 0;\n\texit;" ::: "memory"); };
    auto wait = [&](unsigned long long *bar, unsigned parity) {
        if (!mbar_wait(bar, parity) && !mbar_wait(bar, parity)) {
            report_error(err, EXACT_ETIMEOUT);
            *(volatile int *)&gone = 1;
            __threadfence_block();
            leave();
        }
    };
    auto arrive = [&](unsigned long long *bar) {
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
    };
    load_table(s_fp, fp);
    __syncthreads();
    for (int e = tid; e < E; e += kNearThreads) {
        const float4 k = s_fp[3 * e + 1];
        s_edge[3 * e] = s_fp[3 * e];
        s_edge[3 * e + 1] = make_float4(k.x, k.y, reinterpret_cast<const float *>(s_fp + 3 * E + 1)[e], 0.f);
        s_edge[3 * e + 2] = s_fp[3 * e + 2];
    }
    // padding edges repeat vertex 0: one of them counts, the rest are the same
    const int ne = min(E, n_edges + 1);
    const EdgeLane e0 = edge_lane(s_fp, E, ne, lane), e1 = WIDE ? edge_lane(s_fp, E, ne, 32 + lane) : EdgeLane{};
    const float lim = fmaf(fp.bc.z, 1e-5f, fp.bc.z) + 1e-5f, lim2 = lim * lim;   // as in poly_rows
    // 1e-5 (|cx| + |cy| + r + span)^2, span bounding the footprint's coordinates,
    // is at most 6e-5 of the centre's squared distance + 1.8e-4 span^2 + 3e-5 r^2
    const float span = fabsf(fp.bc.x) + fabsf(fp.bc.y) + fp.bc.z, k0 = 1.8e-4f * span * span;
    const ulonglong2 *T = reinterpret_cast<const ulonglong2 *>(s_edge);
    const ulonglong2 *S = reinterpret_cast<const ulonglong2 *>(s_fp);
    __syncthreads();

    // this block's share of the (chunk, pose) rows, chunk by chunk; i counts its rows
    const long long w1 = (long long)nch * P * (blockIdx.x + 1) / gridDim.x;
    int i = 0;
    for (long long w = (long long)nch * P * blockIdx.x / gridDim.x; w < w1;) {
        const int chunk = (int)(w / P), pose0 = (int)(w - (long long)chunk * P), npose = (int)min((long long)(P - pose0), w1 - w);
        const int base = chunk * csize, n = min(csize, N - base), npatch = (n + kPatch - 1) / kPatch, iend = i + npose;
        w += npose;
        __syncthreads();   // nobody reads the previous chunk
        {
            const SortedChunk &C = chunks[chunk];
            const float4 *src = reinterpret_cast<const float4 *>(C.pts);
            for (int j = tid; j < kChunk / 2; j += kNearThreads) reinterpret_cast<float4 *>(pts)[j] = src[j];
            const uint4 *si = reinterpret_cast<const uint4 *>(C.idx);
            for (int j = tid; j < kChunk / 8; j += kNearThreads) reinterpret_cast<uint4 *>(idx)[j] = si[j];
            for (int j = tid; j < kPatches; j += kNearThreads) {
                float4 c = C.circ[j];
                const float rz = fmaxf(c.z, 0.f);
                c.w = fmaf(1e-5f, rz + span, rz);   // the radius, with the slack that does not depend on the pose
                circ[j] = c;
            }
        }
        __syncthreads();
        if (warp == nwarps) {   // the storing warp
            for (int pose = pose0; i < iend; ++i, ++pose) {
                const int k = i % kRows;
                if (chunk == 0 && lane == 0 && !(isfinite(poses[3 * (size_t)pose]) && isfinite(poses[3 * (size_t)pose + 1]) &&
                                                 isfinite(poses[3 * (size_t)pose + 2])))
                    report_error(err, EXACT_EINVAL);
                wait(full + k, (i / kRows) & 1);
                if (*(volatile int *)&gone) leave();   // a row may lack the part of a thread that left
                const float *row = rows + k * kChunk;
                float *out = dist + (size_t)pose * N + base;
                if (bulk && lane == 0)
                    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n\tcp.async.bulk.commit_group;" ::"l"(
                                     out),
                                 "r"(smem_addr(row)), "r"(n * 4)
                                 : "memory");
                if (dmin || argmin) {
                    const unsigned long long b = warp_min_u64(red[k][lane]);
                    if (lane == 0 && keys) {
                        if (b != kNoKey) atomicMin(keys + pose, b);
                    } else if (lane == 0) {
                        if (dmin) dmin[pose] = b == kNoKey ? finf() : table_eval(fp, s_fp).dist(ord2f((unsigned)(b >> 32)));
                        if (argmin) argmin[pose] = b == kNoKey ? -1 : (int)(unsigned)(b & 0xffffffffu);
                    }
                }
                if (!bulk) {
#pragma unroll 8
                    for (int j = lane; j < n; j += 32) __stcs(out + j, row[j]);
                    __syncwarp();
                    if (lane == 0) arrive(empty + k);
                } else if (lane == 0) {
                    // the copy issued just before this one has read its row
                    asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                    if (i > 0) arrive(empty + (i - 1) % kRows);
                }
            }
            continue;
        }
        // a computing warp: items warp, warp + nwarps, ... of the (pose, patch) pairs
        int q = warp;
        for (size_t pose = pose0; i < iend; ++i, ++pose) {
            const int k = i % kRows;
            const float tx = poses[3 * pose], ty = poses[3 * pose + 1], th = poses[3 * pose + 2];
            float sn, cs;
            sincosf(th, &sn, &cs);
            float *row = rows + k * kChunk;
            if (i >= kRows) wait(empty + k, ((i / kRows) & 1) ^ 1);   // the last row in this buffer has left it
            float bk = finf();
            int bi = -1;
            for (; q < npatch; q += nwarps) {
                const float4 cc = circ[q];
                float cx, cy;
                body_frame(cc.x, cc.y, tx, ty, cs, sn, cx, cy);
                const float r = fmaf(1e-5f, fabsf(cx) + fabsf(cy), cc.w);
                // edges that can be nearest
                const EdgeNear n0 = edge_near(e0, cx, cy), n1 = WIDE ? edge_near(e1, cx, cy) : EdgeNear{finf(), 0.f, 0.f, 0.f, 0.f};
                const float own = WIDE ? fminf(n0.d2, n1.d2) : n0.d2;
                const float best = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(own)));
                const int who = __ffs(__ballot_sync(0xffffffffu, own == best)) - 1;   // -1: not finite, every edge is kept
                const bool second = WIDE && n0.d2 != best;
                const float ax = __shfl_sync(0xffffffffu, second ? n1.qx : n0.qx, who & 31);
                const float ay = __shfl_sync(0xffffffffu, second ? n1.qy : n0.qy, who & 31);
                const float r4 = 4.0001f * r * r, thr = fmaf(7.5e-6f, r4, fmaf(best, 1.00006f, k0));
                auto needed = [&](const EdgeLane &l, const EdgeNear &m) {
                    const float ux = ax - m.dx, uy = ay - m.dy, wx = ux + l.ex, wy = uy + l.ey;   // the ends - a
                    const float s2 = fmaxf(fmaf(ux, ux, uy * uy), fmaf(wx, wx, wy * wy));
                    const float g = m.d2 - thr;   // dropped iff g > 2 r s, s = sqrt(s2)
                    return l.on && (who < 0 || !(g > 0.f && g * g > r4 * s2));
                };
                unsigned m0 = __ballot_sync(0xffffffffu, needed(e0, n0));
                unsigned m1 = WIDE ? __ballot_sync(0xffffffffu, needed(e1, n1)) : 0u;

                const float4 o = reinterpret_cast<const float4 *>(pts)[q * 32 + lane];   // points 2 lane, 2 lane + 1
                const unsigned ii = reinterpret_cast<const unsigned *>(idx)[q * 32 + lane];
                float px0, py0, px1, py1;
                body_frame(o.x, o.y, tx, ty, cs, sn, px0, py0);
                body_frame(o.z, o.w, tx, ty, cs, sn, px1, py1);
                const f2x PX = pack2(px0, px1), PY = pack2(py0, py1);
                float k0 = finf(), k1 = finf();
                auto edge = [&](int b) {   // the distance part of poly_edge
                    const ulonglong2 v = T[3 * b], c = T[3 * b + 1], d = T[3 * b + 2];
                    const f2x dx = add2(PX, v.x), dy = add2(PY, v.y);
                    float u0, u1, d0, d1, eyn, pad, q0, q1;
                    unpack2(mul2(dx, c.x), u0, u1);
                    unpack2(dy, d0, d1);
                    unpack2(c.y, eyn, pad);
                    const f2x t = pack2(__saturatef(fmaf(d0, eyn, u0)), __saturatef(fmaf(d1, eyn, u1)));
                    const f2x qx = fma2(t, d.x, dx), qy = fma2(t, d.y, dy);
                    unpack2(fma2(qy, qy, mul2(qx, qx)), q0, q1);
                    k0 = fminf(k0, q0);
                    k1 = fminf(k1, q1);
                };
                for (; m0; m0 &= m0 - 1u) edge(__ffs(m0) - 1);
                if (WIDE)
                    for (; m1; m1 &= m1 - 1u) edge(31 + __ffs(m1));
                // only a point within the bounding circle can be inside
                const float fx = cx - fp.bc.x, fy = cy - fp.bc.y, far = r + lim;
                if (!(fmaf(fx, fx, fy * fy) > far * far)) {
                    const float bx0 = px0 - fp.bc.x, by0 = py0 - fp.bc.y, bx1 = px1 - fp.bc.x, by1 = py1 - fp.bc.y;
                    const bool f0 = fmaf(bx0, bx0, by0 * by0) <= lim2, f1 = fmaf(bx1, bx1, by1 * by1) <= lim2;
                    if (__any_sync(0xffffffffu, f0 || f1)) {
                        unsigned s0 = 0u, s1 = 0u;
                        f2x dxa = add2(PX, S[0].x), dya = add2(PY, S[0].y);
#pragma unroll 4
                        for (int b = 0; b < E; ++b) {   // the parity part of poly_edge
                            const ulonglong2 vn = S[3 * b + 3];
                            const f2x nkx = S[3 * b + 1].y, dxb = add2(PX, vn.x), dyb = add2(PY, vn.y);
                            float h0, h1, x0, x1;
                            unpack2(fma2(dya, nkx, dxa), h0, h1);
                            unpack2(mul2(dya, dyb), x0, x1);
                            s0 ^= __float_as_uint(x0) & __float_as_uint(h0);
                            s1 ^= __float_as_uint(x1) & __float_as_uint(h1);
                            dxa = dxb;
                            dya = dyb;
                        }
                        if (f0) k0 = __uint_as_float(__float_as_uint(k0) | (s0 & 0x80000000u));
                        if (f1) k1 = __uint_as_float(__float_as_uint(k1) | (s1 & 0x80000000u));
                    }
                }
                const int i0 = (int)(ii & 0xffffu), i1 = (int)(ii >> 16);
                auto to_dist = [](float key) {
                    const unsigned b = __float_as_uint(key);
                    return __uint_as_float(__float_as_uint(sqrtf(__uint_as_float(b & 0x7fffffffu))) | (b & 0x80000000u));
                };
                const int at = q * kPatch + 2 * lane;
                if (at < n) row[i0] = to_dist(k0);   // absent points come last
                if (at + 1 < n) row[i1] = to_dist(k1);
                if (fminf(k0, k1) <= bk) {   // lowest index among equal keys; +inf never wins
                    if (k0 < bk || (k0 == bk && i0 < bi)) { bk = k0; bi = i0; }
                    if (k1 < bk || (k1 == bk && i1 < bi)) { bk = k1; bi = i1; }
                }
            }
            q -= npatch;
            if (dmin || argmin) {
                const unsigned u = bi < 0 ? ~0u : f2ord(bk), m = __reduce_min_sync(0xffffffffu, u);
                const unsigned at = __reduce_min_sync(0xffffffffu, u == m ? (unsigned)(base + bi) : ~0u);
                if (lane == 0) red[k][warp] = m == ~0u ? kNoKey : ((unsigned long long)m << 32) | at;
            }
            fence_proxy_async_smem();   // this warp's part of the row comes before its bulk copy
            __syncwarp();
            if (lane == 0) arrive(full + k);
        }
    }
    if (warp == nwarps && bulk && lane == 0)
        asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");   // the last rows are written
}

// ---------------------------------------------------------------- minimum
// Minimum and argmin only, W warps per pose (one when the poses alone fill the
// GPU: no barrier): the patch whose centre is nearest to the footprint's
// bounding box is evaluated first, then only the patches whose lower bound (the
// centre's box distance less the radius) is below the minimum so far; a
// dropped patch holds no point at the minimum, so ties keep their lowest
// index.
__device__ __forceinline__ float sqrt_approx(float x) {
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
template <int W>
__global__ void __launch_bounds__(kMinThreads)
sdf_min_kernel(const SortedChunk *__restrict__ chunks, int N, int csize, const float *__restrict__ poses, int P,
               const __grid_constant__ FpTable fp, float *__restrict__ dmin, int *__restrict__ argmin, int *err) {
    constexpr int kGroups = kMinThreads / 32 / W;   // poses per block
    static_assert(W == 1 || kGroups == 1, "several warps per pose meet at the block's barrier");
    __shared__ float4 s_fp[kFpSlots];
    __shared__ unsigned long long s_best[kGroups], s_first[kGroups];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, group = warp / W, sub = warp % W;
    const int pose = blockIdx.x * kGroups + group;
    auto meet = [&]() {
        if (W == 1) __syncwarp();
        else __syncthreads();
    };
    load_table(s_fp, fp);
    unsigned long long *best = s_best + group;
    if (sub == 0 && lane == 0) *best = s_first[group] = kNoKey;
    __syncthreads();
    if (pose >= P) return;   // W == 1 only: no later barrier
    const float tx = poses[3 * (size_t)pose], ty = poses[3 * (size_t)pose + 1], th = poses[3 * (size_t)pose + 2];
    if (sub == 0 && lane == 0 && !(isfinite(tx) && isfinite(ty) && isfinite(th))) report_error(err, EXACT_EINVAL);
    float sn, cs;
    sincosf(th, &sn, &cs);
    const SmemEval ev = table_eval(fp, s_fp);
    const float4 box = ev.box();
    const float span = fabsf(box.x) + fabsf(box.y) + box.z + box.w;
    const int npatch = (N + kPatch - 1) / kPatch, per = csize / kPatch;   // chunks are whole patches
    // box distance of patch q's centre, and its radius with a slack far above
    // every rounding (the square root's too)
    auto centre = [&](int q, float &r) {
        const float4 cc = __ldg(&chunks[q / per].circ[q % per]);
        float cx, cy;
        body_frame(cc.x, cc.y, tx, ty, cs, sn, cx, cy);
        r = cc.z < 0.f ? -1.f : fmaf(1e-5f, fabsf(cx) + fabsf(cy) + cc.z + span, cc.z) + 1e-5f;
        const float ax = fabsf(cx - box.x) - box.z, ay = fabsf(cy - box.y) - box.w;
        const float mx = fmaxf(ax, 0.f), my = fmaxf(ay, 0.f);
        return sqrt_approx(fmaf(mx, mx, my * my)) + fminf(fmaxf(ax, ay), 0.f);
    };
    auto evaluate = [&](int q) {   // the whole warp: the patch's points against every edge or box
        const SortedChunk &C = chunks[q / per];
        const int at = (q % per) * 32 + lane;
        const float4 o = __ldg(reinterpret_cast<const float4 *>(C.pts) + at);
        const unsigned ii = __ldg(reinterpret_cast<const unsigned *>(C.idx) + at);
        float px0, py0, px1, py1, k0, k1;
        body_frame(o.x, o.y, tx, ty, cs, sn, px0, py0);
        body_frame(o.z, o.w, tx, ty, cs, sn, px1, py1);
        ev.eval2(px0, py0, px1, py1, k0, k1);
        const unsigned base = (unsigned)(q / per) * (unsigned)csize;
        // +inf and NaN are no minimum; then the lowest index among equal keys
        const unsigned u0 = k0 < finf() ? f2ord(k0) : ~0u, u1 = k1 < finf() ? f2ord(k1) : ~0u;
        const unsigned m = __reduce_min_sync(0xffffffffu, min(u0, u1));
        if (m == ~0u) return;
        const unsigned i0 = u0 == m ? base + (ii & 0xffffu) : ~0u, i1 = u1 == m ? base + (ii >> 16) : ~0u;
        const unsigned long long b = ((unsigned long long)m << 32) | __reduce_min_sync(0xffffffffu, min(i0, i1));
        if (lane == 0 && b < *(volatile unsigned long long *)best) atomicMin(best, b);
    };
    unsigned long long near = kNoKey;
    for (int q = sub * 32 + lane; q < npatch; q += W * 32) {
        float r;
        const float d = centre(q, r);
        if (r >= 0.f) {
            const unsigned long long k = pack_key(d, (unsigned)q);
            near = k < near ? k : near;
        }
    }
    near = warp_min_u64(near);
    if (W > 1) {
        if (lane == 0) atomicMin(&s_first[group], near);
        meet();
        near = s_first[group];
    }
    const int first = near == kNoKey ? -1 : (int)(unsigned)(near & 0xffffffffu);
    if (sub == 0 && first >= 0) evaluate(first);
    meet();
    for (int q0 = sub * 32; q0 < npatch; q0 += W * 32) {
        const int q = q0 + lane;
        float r = -1.f, d = 0.f;
        if (q < npatch) d = centre(q, r);
        for (unsigned todo = __ballot_sync(0xffffffffu, r >= 0.f && q != first); todo;) {
            const unsigned long long b = *(volatile unsigned long long *)best;
            const float now = b == kNoKey ? finf() : ev.dist(ord2f((unsigned)(b >> 32)));
            // a non-finite pose keeps everything
            todo &= __ballot_sync(0xffffffffu, !(d - r > now));
            if (!todo) break;
            evaluate(q0 + __ffs(todo) - 1);
            todo &= todo - 1u;
            __syncwarp();
        }
    }
    meet();
    if (sub == 0 && lane == 0) {
        const unsigned long long b = *best;
        if (dmin) dmin[pose] = b == kNoKey ? finf() : ev.dist(ord2f((unsigned)(b >> 32)));
        if (argmin) argmin[pose] = b == kNoKey ? -1 : (int)(unsigned)(b & 0xffffffffu);
    }
}

// ---------------------------------------------------------------- launches
// Where the sort (a launch of about 12 us) pays.  Matrix: a patch costs the
// pruned kernel a search, the transform, the root and the store whatever the
// number of edges, about what 14 edges cost the general one, and patches of few
// points are too wide to leave edges out: from 16 edges and 8,192 points, or 32
// and 4,096, on (4,096 poses x 8,192 points: 12 edges 166 us against 157 with the
// general kernel, 16 edges 171 against 178, 24 edges 187 against 252, 64 edges 288
// against 568; 16 edges x 4,096 points 112 against 94).  A cloud dense on the
// footprint keeps most edges and still gains (within 0.3 m of the origin: 16
// edges 279 against 284, 32 edges 392 against 478).  Minimum: general calls from
// about 45 us on, of 1,024 points (200,000 poses x 128 points lost up to 17 %); a
// cover's general evaluation is so cheap that it takes 768 poses (256 poses x
// 300,000 points, 3 boxes: 179 against 125 us).  It loses where nearly every patch
// can hold the minimum: points all at one place 2.3x, on a circle about every
// pose 1.5x, all inside the footprint 1.2x.
constexpr int kMinPoses = 256, kMinPoints = 1024, kMatrixPoses = 64, kMatrixPoints = 4096;
bool sdf_near_fits(const exact_footprint *fp, int n_points, int n_poses, bool dist) {
    const bool polygon = fp->kind == EXACT_FP_POLYGON;
    const long long pairs = (long long)n_points * n_poses, work = pairs * (polygon ? fp->n_pad : 2 * fp->n_pad);
    if (!dist) return n_poses >= (polygon ? kMinPoses : 3 * kMinPoses) && n_points >= kMinPoints && work >= (1ll << 27);
    return polygon && fp->n_pad >= 16 && n_points >= kMatrixPoints && (long long)n_points * fp->n_pad >= 16 * 8192 &&
           n_poses >= kMatrixPoses && work >= (1ll << 28);
}
bool sdf_near_possible(int n_points, int n_poses) {
    if ((long long)n_points * n_poses < (1ll << 27) / EXACT_MAX_POLY_VERTICES) return false;
    return (n_poses >= kMinPoses && n_points >= kMinPoints) || (n_poses >= kMatrixPoses && n_points >= kMatrixPoints);
}

int sdf_near_launch(const float2 *pts, const uint8_t *mask, int N, const float *poses, int P, const exact_footprint *fp,
                    float *dist, float *dmin, int *argmin, unsigned long long *keys, void *scratch, int sms, int *err,
                    cudaStream_t st) {
    SortedChunk *chunks = static_cast<SortedChunk *>(scratch);
    const int csize = chunk_points(N), nch = (N + csize - 1) / csize;
    const FpTable t = make_table(fp);
    constexpr int sort_smem = kChunk * 10;
    if (cudaFuncSetAttribute(sdf_sort_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, sort_smem) != cudaSuccess)
        return EXACT_ECUDA;
    sdf_sort_kernel<<<nch, kSortThreads, sort_smem, st>>>(pts, mask, N, csize, chunks);
    if (cudaGetLastError() != cudaSuccess) return EXACT_ECUDA;
    if (!dist) {
        if (P >= 8 * sms)
            sdf_min_kernel<1><<<(P + kMinThreads / 32 - 1) / (kMinThreads / 32), kMinThreads, 0, st>>>(chunks, N, csize, poses, P, t,
                                                                                                      dmin, argmin, err);
        else
            sdf_min_kernel<kMinThreads / 32><<<P, kMinThreads, 0, st>>>(chunks, N, csize, poses, P, t, dmin, argmin, err);
        return cuda_status(cudaGetLastError());
    }
    const size_t smem = (size_t)kChunk * (8 + kRows * 4 + 2) + kPatches * sizeof(float4);
    const int bulk = ((uintptr_t)dist & 15u) == 0 && N % 4 == 0;
    auto k = fp->n_pad > 32 ? sdf_matrix_kernel<true> : sdf_matrix_kernel<false>;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return EXACT_ECUDA;
    const long long rows = (long long)nch * P;
    k<<<(unsigned)(rows < sms ? rows : sms), kNearThreads, smem, st>>>(chunks, N, csize, nch, poses, P, t, fp->n, dist, bulk,
                                                                      dmin, argmin, keys, err);
    return cuda_status(cudaGetLastError());
}

}  // namespace exact
