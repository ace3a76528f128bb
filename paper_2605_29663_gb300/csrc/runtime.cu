// runtime.cu -- footprint objects, contexts, scratch and status strings of
// the EXACT-MPPI C ABI.
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <mutex>
#include <new>

#include "internal.h"

namespace {

// Orientation of (a, b, c): sign of the cross product (b - a) x (c - a).
int orient(double ax, double ay, double bx, double by, double cx, double cy) {
    const double v = (bx - ax) * (cy - ay) - (by - ay) * (cx - ax);
    return (v > 0.0) - (v < 0.0);
}

// c collinear with segment ab: does it lie within the segment's box?
bool on_segment(double ax, double ay, double bx, double by, double cx, double cy) {
    return fmin(ax, bx) <= cx && cx <= fmax(ax, bx) && fmin(ay, by) <= cy && cy <= fmax(ay, by);
}

bool segments_touch(const double *p, const double *q, const double *r, const double *s) {
    const int o1 = orient(p[0], p[1], q[0], q[1], r[0], r[1]);
    const int o2 = orient(p[0], p[1], q[0], q[1], s[0], s[1]);
    const int o3 = orient(r[0], r[1], s[0], s[1], p[0], p[1]);
    const int o4 = orient(r[0], r[1], s[0], s[1], q[0], q[1]);
    if (o1 != o2 && o3 != o4) return true;
    if (o1 == 0 && on_segment(p[0], p[1], q[0], q[1], r[0], r[1])) return true;
    if (o2 == 0 && on_segment(p[0], p[1], q[0], q[1], s[0], s[1])) return true;
    if (o3 == 0 && on_segment(r[0], r[1], s[0], s[1], p[0], p[1])) return true;
    if (o4 == 0 && on_segment(r[0], r[1], s[0], s[1], q[0], q[1])) return true;
    return false;
}

// Simple-polygon check (O(n^2)): no repeated vertex, non-adjacent edges do
// not meet, adjacent edges do not fold back onto each other, non-zero area.
int check_simple(const double *v, int n) {
    for (int i = 0; i < n; ++i)
        for (int j = i + 1; j < n; ++j)
            if (v[2 * i] == v[2 * j] && v[2 * i + 1] == v[2 * j + 1]) return EXACT_ENOTSIMPLE;
    for (int i = 0; i < n; ++i) {
        const double *a = v + 2 * i, *b = v + 2 * ((i + 1) % n);
        for (int j = i + 1; j < n; ++j) {
            const double *c = v + 2 * j, *d = v + 2 * ((j + 1) % n);
            const bool adjacent = (j == i + 1) || (i == 0 && j == n - 1);
            if (adjacent) {
                // shared vertex: the far end of one edge must not lie on the other
                const double *far_i = (j == i + 1) ? a : b;
                const double *far_j = (j == i + 1) ? d : c;
                if (orient(a[0], a[1], b[0], b[1], far_j[0], far_j[1]) == 0 &&
                    on_segment(a[0], a[1], b[0], b[1], far_j[0], far_j[1]))
                    return EXACT_ENOTSIMPLE;
                if (orient(c[0], c[1], d[0], d[1], far_i[0], far_i[1]) == 0 &&
                    on_segment(c[0], c[1], d[0], d[1], far_i[0], far_i[1]))
                    return EXACT_ENOTSIMPLE;
            } else if (segments_touch(a, b, c, d)) {
                return EXACT_ENOTSIMPLE;
            }
        }
    }
    double area2 = 0.0;
    for (int i = 0; i < n; ++i) {
        const double *a = v + 2 * i, *b = v + 2 * ((i + 1) % n);
        area2 += a[0] * b[1] - a[1] * b[0];
    }
    if (!(fabs(area2) > 1e-12)) return EXACT_ENOTSIMPLE;
    return EXACT_OK;
}

int poly_bucket(int n) {
    static const int sizes[] = {4, 6, 8, 10, 12, 14, 16, 24, 32, 40, 48, 56, 64};
    for (int s : sizes)
        if (n <= s) return s;
    return -1;
}

int rect_bucket(int n) {
    static const int sizes[] = {1, 2, 3, 4, 5, 6, 7, 8};
    for (int s : sizes)
        if (n <= s) return s;
    return -1;
}

}  // namespace

extern "C" const char *exact_status_string(int status) {
    switch (status) {
    case EXACT_OK: return "ok";
    case EXACT_EINVAL: return "invalid argument";
    case EXACT_ENOTSIMPLE: return "polygon is not simple";
    case EXACT_ECAPACITY: return "size beyond the supported maximum";
    case EXACT_ECUDA: return "CUDA runtime error";
    case EXACT_ETIMEOUT: return "device-side wait timed out";
    default: return "unknown status";
    }
}

extern "C" int exact_footprint_create(int kind, const float *host_data, int n, exact_footprint **out) {
    if (!out || !host_data) return EXACT_EINVAL;
    *out = nullptr;
    const int per = kind == EXACT_FP_POLYGON ? 2 : kind == EXACT_FP_RECTS ? 4 : 0;
    if (per == 0 || n <= 0) return EXACT_EINVAL;
    for (int i = 0; i < n * per; ++i)
        if (!isfinite(host_data[i])) return EXACT_EINVAL;
    exact_footprint *fp = new (std::nothrow) exact_footprint();
    if (!fp) return EXACT_EINVAL;
    memset(fp, 0, sizeof(*fp));
    fp->kind = kind;
    fp->n = n;
    if (kind == EXACT_FP_POLYGON) {
        if (n < 3) { delete fp; return EXACT_EINVAL; }
        if (n > EXACT_MAX_POLY_VERTICES) { delete fp; return EXACT_ECAPACITY; }
        double v[2 * EXACT_MAX_POLY_VERTICES];
        for (int i = 0; i < 2 * n; ++i) v[i] = (double)host_data[i] + 0.0;  // -0 -> +0
        const int rc = check_simple(v, n);
        if (rc != EXACT_OK) { delete fp; return rc; }
        const int E = poly_bucket(n);
        fp->n_pad = E;
        for (int b = 0; b < E; ++b) {
            const int ib = b < n ? b : 0;
            const int nb = (b + 1) < n ? b + 1 : 0;   // padded vertices repeat vertex 0
            const double vx = v[2 * ib], vy = v[2 * ib + 1];
            const double wx = v[2 * nb], wy = v[2 * nb + 1];
            const double ex = (b < n) ? wx - vx : 0.0, ey = (b < n) ? wy - vy : 0.0;
            const double len2 = ex * ex + ey * ey;
            fp->vx[b] = (float)vx;
            fp->vy[b] = (float)vy;
            fp->ex[b] = (float)ex;
            fp->ey[b] = (float)ey;
            fp->exn[b] = len2 > 0.0 ? (float)(ex / len2) : 0.f;
            fp->eyn[b] = len2 > 0.0 ? (float)(ey / len2) : 0.f;
            fp->kx[b] = ey != 0.0 ? (float)(ex / ey) : 0.f;
        }
    } else {
        if (n > EXACT_MAX_RECTS) { delete fp; return EXACT_ECAPACITY; }
        for (int j = 0; j < n; ++j)
            if (!(host_data[4 * j + 2] > 0.f) || !(host_data[4 * j + 3] > 0.f)) { delete fp; return EXACT_EINVAL; }
        const int R = rect_bucket(n);
        fp->n_pad = R;
        for (int j = 0; j < R; ++j) {
            const int s = j < n ? j : 0;   // padded boxes repeat box 0
            fp->cx[j] = host_data[4 * s] + 0.f;
            fp->cy[j] = host_data[4 * s + 1] + 0.f;
            fp->sx[j] = host_data[4 * s + 2];
            fp->sy[j] = host_data[4 * s + 3];
        }
    }
    // bounding circle of the footprint (centre of the bounding box, largest
    // vertex / box-corner distance) and the bounding box itself (half
    // extents about that centre), both rounded outwards so that the float
    // circle and box contain the footprint, for the bounds that let the
    // MPPI kernels skip far point chunks and far points
    double lo[2] = {1e300, 1e300}, hi[2] = {-1e300, -1e300};
    auto corners = [&](auto &&visit) {
        if (kind == EXACT_FP_POLYGON) {
            for (int b = 0; b < n; ++b) visit((double)host_data[2 * b], (double)host_data[2 * b + 1]);
        } else {
            for (int j = 0; j < n; ++j)
                for (int sx = -1; sx <= 1; sx += 2)
                    for (int sy = -1; sy <= 1; sy += 2)
                        visit((double)host_data[4 * j] + sx * (double)host_data[4 * j + 2],
                              (double)host_data[4 * j + 1] + sy * (double)host_data[4 * j + 3]);
        }
    };
    corners([&](double x, double y) {
        lo[0] = fmin(lo[0], x); lo[1] = fmin(lo[1], y);
        hi[0] = fmax(hi[0], x); hi[1] = fmax(hi[1], y);
    });
    const double bcx = 0.5 * (lo[0] + hi[0]), bcy = 0.5 * (lo[1] + hi[1]);
    double r2 = 0.0;
    corners([&](double x, double y) { r2 = fmax(r2, (x - bcx) * (x - bcx) + (y - bcy) * (y - bcy)); });
    fp->bcx = (float)bcx;
    fp->bcy = (float)bcy;
    fp->brad = (float)(sqrt(r2) * (1.0 + 1e-6) + 1e-6 + fabs((double)fp->bcx - bcx) + fabs((double)fp->bcy - bcy));
    const double shift = fabs((double)fp->bcx - bcx) + fabs((double)fp->bcy - bcy);
    fp->bhx = (float)(0.5 * (hi[0] - lo[0]) * (1.0 + 1e-6) + 1e-6 + shift);
    fp->bhy = (float)(0.5 * (hi[1] - lo[1]) * (1.0 + 1e-6) + 1e-6 + shift);
    *out = fp;
    return EXACT_OK;
}

extern "C" void exact_footprint_destroy(exact_footprint *fp) { delete fp; }

extern "C" int exact_footprint_info(const exact_footprint *fp, int *kind, int *n) {
    if (!fp) return EXACT_EINVAL;
    if (kind) *kind = fp->kind;
    if (n) *n = fp->n;
    return EXACT_OK;
}

namespace exact {

int current_sm_count() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    return sms;
}

static void free_retired(exact_ctx *ctx) {
    while (ctx->n_retired > 0) cudaFree(ctx->retired[--ctx->n_retired]);
}
static void retire(exact_ctx *ctx, void *p) {
    if (p) ctx->retired[ctx->n_retired++] = p;   // growth looks for room first
}

// Outgrown arenas stay allocated until the context goes: a captured graph may
// still replay with their addresses, whichever later call grew the scratch.
// Doubling keeps them below the current arena's size in sum.  Where there is no
// memory for twice the size, the size asked for is tried; only where that does
// not fit beside them are they given back (before that the call would have
// been refused).
int ensure_scratch(exact_ctx *ctx, size_t bytes) {
    if (!ctx) return EXACT_EINVAL;
    if (bytes <= ctx->scratch_bytes) return EXACT_OK;
    bytes = align_up(bytes, (size_t)1 << 20);
    const size_t twice = std::max(bytes, 2 * ctx->scratch_bytes);
    size_t got = 0;
    void *p = nullptr;
    for (size_t want : {twice, bytes})
        if (!p && ctx->n_retired < kRetired) {
            if (cudaMalloc(&p, want) == cudaSuccess) got = want;
            else { cudaGetLastError(); p = nullptr; }
        }
    if (!p) {
        if (cudaDeviceSynchronize() != cudaSuccess) return EXACT_ECUDA;
        if (ctx->scratch_alloc) cudaFree(ctx->scratch_alloc);
        free_retired(ctx);
        ctx->scratch = ctx->scratch_alloc = nullptr;
        ctx->scratch_bytes = 0;
        got = bytes;
        if (cudaMalloc(&p, got) != cudaSuccess) return EXACT_ECUDA;
    }
    // counters and flags in the arena must start at zero; the clear runs on the
    // legacy stream, which a caller's non-blocking stream does not wait for: end
    // it here, before the call's kernels write the arena
    if (cudaMemset(p, 0, got) != cudaSuccess || cudaStreamSynchronize(cudaStreamLegacy) != cudaSuccess) {
        cudaFree(p);
        return EXACT_ECUDA;
    }
    retire(ctx, ctx->scratch_alloc);
    ctx->scratch = ctx->scratch_alloc = p;
    ctx->scratch_bytes = got;
    return EXACT_OK;
}

bool try_work(exact_ctx *ctx, size_t bytes, cudaStream_t st) {
    if (bytes <= ctx->work_bytes) return true;
    if (bytes > ((size_t)1 << 30)) return false;
    bytes = align_up(bytes, (size_t)1 << 20);
    size_t got = std::max(bytes, 2 * ctx->work_bytes);
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    void *p = nullptr;
    if (cudaStreamIsCapturing(st, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone ||
        ctx->n_retired >= kRetired ||
        (cudaMalloc(&p, got) != cudaSuccess && cudaMalloc(&p, got = bytes) != cudaSuccess)) {
        cudaGetLastError();   // not this call's error: it has another path
        return false;
    }
    cudaGetLastError();
    retire(ctx, ctx->work_alloc);
    ctx->work = ctx->work_alloc = p;
    ctx->work_bytes = got;
    return true;
}

// One pool per device, shared by the contexts that use it and destroyed with
// the last of them: making a pool and mapping its first memory takes some 130
// us, which a second context need not pay again.
constexpr int kMaxDevices = 64;
static struct SharedPool {
    std::mutex lock;
    cudaMemPool_t pool = nullptr;
    int users = 0;
} g_pools[kMaxDevices];

cudaMemPool_t sdf_pool(exact_ctx *ctx, unsigned long long keep) {
    cudaMemPool_t pool = ctx->pool.load();
    if (pool && keep <= kPoolKeep) return pool;
    if (ctx->device < 0 || ctx->device >= kMaxDevices) return nullptr;
    SharedPool &shared = g_pools[ctx->device];
    std::lock_guard<std::mutex> guard(shared.lock);
    if (!shared.pool) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = ctx->device;
        if (cudaMemPoolCreate(&shared.pool, &props) != cudaSuccess) {
            cudaGetLastError();
            shared.pool = nullptr;
            return nullptr;
        }
        unsigned long long least = kPoolKeep;
        int no = 0;   // a stream does not wait for another's call to end to take its memory
        cudaMemPoolSetAttribute(shared.pool, cudaMemPoolAttrReleaseThreshold, &least);
        cudaMemPoolSetAttribute(shared.pool, cudaMemPoolReuseAllowInternalDependencies, &no);
    }
    pool = shared.pool;
    if (!ctx->pool.load()) {
        ++shared.users;
        ctx->pool = pool;
    }
    unsigned long long now = 0;
    if (cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &now) == cudaSuccess && now < keep)
        cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
    return pool;
}

static void release_pool(exact_ctx *ctx) {
    if (!ctx->pool.load()) return;
    SharedPool &shared = g_pools[ctx->device];
    std::lock_guard<std::mutex> guard(shared.lock);
    if (--shared.users == 0) {
        cudaMemPoolDestroy(shared.pool);
        shared.pool = nullptr;
    }
}

}  // namespace exact

extern "C" int exact_ctx_create(exact_ctx **out) {
    if (!out) return EXACT_EINVAL;
    *out = nullptr;
    exact_ctx *ctx = new (std::nothrow) exact_ctx();
    if (!ctx) return EXACT_EINVAL;
    if (cudaGetDevice(&ctx->device) != cudaSuccess) { delete ctx; return EXACT_ECUDA; }
    ctx->sm_count = exact::current_sm_count();
    // one allocation: split keys, error word, statistics, part tickets, the
    // arena's first 1 MB (all zeroed), then the second arena's, so that a cycle of
    // ordinary size can be captured without any call before it
    const size_t key_bytes = exact::align_up(sizeof(SdfKey) * (size_t)exact::sdf_split_poses(ctx->sm_count), 256);
    const size_t stats_bytes = exact::align_up(sizeof(exact_cycle_stats), 256);
    const size_t first = key_bytes + 256 + stats_bytes +
                         exact::align_up(sizeof(unsigned) * (size_t)exact::ticket_count(ctx->sm_count), 256);
    ctx->scratch_bytes = ctx->work_bytes = (size_t)1 << 20;
    const size_t head = first + ctx->scratch_bytes;
    if (cudaMalloc(&ctx->sdf_keys, head + ctx->work_bytes) != cudaSuccess) { delete ctx; return EXACT_ECUDA; }
    char *base = reinterpret_cast<char *>(ctx->sdf_keys);
    ctx->d_err = reinterpret_cast<int *>(base + key_bytes);
    ctx->d_stats = reinterpret_cast<decltype(ctx->d_stats)>(base + key_bytes + 256);
    ctx->part_tickets = reinterpret_cast<unsigned *>(base + key_bytes + 256 + stats_bytes);
    ctx->scratch = base + first;
    ctx->work = base + head;
    if (cudaMemset(base, 0, head) != cudaSuccess || cudaStreamSynchronize(cudaStreamLegacy) != cudaSuccess) {   // as in ensure_scratch
        cudaFree(base);
        delete ctx;
        return EXACT_ECUDA;
    }
    *out = ctx;
    return EXACT_OK;
}

extern "C" void exact_ctx_destroy(exact_ctx *ctx) {
    if (!ctx) return;
    cudaDeviceSynchronize();
    if (ctx->scratch_alloc) cudaFree(ctx->scratch_alloc);
    if (ctx->work_alloc) cudaFree(ctx->work_alloc);
    exact::release_pool(ctx);
    exact::free_retired(ctx);
    if (ctx->sdf_keys) cudaFree(ctx->sdf_keys);
    delete ctx;
}

extern "C" int exact_ctx_enable_stats(exact_ctx *ctx, int enable) {
    if (!ctx) return EXACT_EINVAL;
    ctx->stats = enable != 0;
    return EXACT_OK;
}

extern "C" int exact_ctx_get_stats(exact_ctx *ctx, exact_cycle_stats *out, void *stream) {
    if (!ctx || !out) return EXACT_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    // read, then zero the two counters (the first 16 bytes), in stream order
    if (cudaMemcpyAsync(out, ctx->d_stats, sizeof(exact_cycle_stats), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaMemsetAsync(ctx->d_stats, 0, 2 * sizeof(long long), st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return EXACT_ECUDA;
    return EXACT_OK;
}

extern "C" int exact_ctx_get_error(exact_ctx *ctx, void *stream) {
    if (!ctx) return EXACT_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    int err = 0;
    // read and clear in stream order, then wait for this stream only
    if (cudaMemcpyAsync(&err, ctx->d_err, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaMemsetAsync(ctx->d_err, 0, sizeof(int), st) != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess)
        return EXACT_ECUDA;
    return err;
}
