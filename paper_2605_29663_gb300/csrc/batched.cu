// batched.cu -- many independent scenes advanced by one EXACT-MPPI control
// cycle each (Algorithm 1 per scene) in one persistent launch.
//
// Plan (exact_batch_create, host, once): a device scene table (parameters,
// pointers, footprint constants, scratch addresses), the work-item list of
// the sample phase -- per scene that walks a cell grid (GridRule) one item per
// group of samples (cloud_grid.cuh); per other scene one per (scene, sample), or per
// (scene, two consecutive samples) when the batch holds at least four samples
// per SM and the scene's horizon fits two in a block's step slots; scenes ordered by
// per-sample cost T * N * edges, heaviest first (longest-processing-time
// order) -- and the block tables of the update and validation phases.
//
// Step (mppi_step_batched, capturable): a memset of the per-scene control
// words and the queue heads, then
//   batched_cloud_grid_kernel, batched_grid_sample_kernel
//                           one block per cloud sorts it into a cell grid;
//                           persistent blocks take groups of samples
//   batched_sample_kernel   persistent: SMs x resident blocks; each block
//                           pulls items from an atomic queue and runs (the
//                           other scenes) sample_body with the scene's footprint constants
//                           in shared memory (reloaded only when the scene
//                           changes; so are the staged points when the cloud
//                           fits the stage);
//   batched_update_kernel   one block per (scene, sample chunk): weights and
//                           weighted noise into the scene's partial slots;
//   batched_validate_kernel one block per (scene, step, point chunk): U_upd
//                           from the partial slots, the nominal rollout, the
//                           clearance check and the scene's shift / reset.
// The per-scene arithmetic is that of mppi_step (same device bodies, same
// operation order), so a scene of a batch gives the same bits as mppi_step.
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <string>
#include <new>
#include <vector>

#include "batched_internal.cuh"

namespace exact {

__global__ void __launch_bounds__(512)
batched_sample_kernel(const SceneDev *__restrict__ scenes, const int2 *__restrict__ items, int n_items,
                      unsigned *queue, int pairs_per_lane) {
    extern __shared__ float4 dyn[];
    float4 *s_fp = dyn;
    float2 *s_pts = reinterpret_cast<float2 *>(dyn + kFpSlots);
    __shared__ SampleSmem sm;
    __shared__ int s_item;
    sample_smem_init(sm);
    int fp_scene = -1, pts_scene = -1;   // block-uniform
    for (;;) {
        if (threadIdx.x == 0) s_item = (int)atomicAdd(queue, 1u);
        __syncthreads();
        const int item = s_item;
        if (item >= n_items) break;
        const int2 it = items[item];
        const SceneDev &D = scenes[it.x];
        if (it.x != fp_scene) {
            load_table(s_fp, D.fp);
            __syncthreads();
            fp_scene = it.x;
        }
        const SmemEval ev = table_eval(D.fp, s_fp);
        sample_body(D.V, ev, item_sample(it), 0, sm, s_pts, it.x == pts_scene, pairs_per_lane, item_second(it));
        pts_scene = D.V.N <= kStage ? it.x : -1;
    }
}

// The scenes that walk a grid: persistent blocks take grid items from
// the queue, a scene's footprint terms and distance field in shared memory.
// FAR: some scene's field ends before its d_safe.
template <bool FAR>
__global__ void __launch_bounds__(1024)   // at most 512 are launched: 64 registers, four blocks of 256 per SM
batched_grid_sample_kernel(const SceneDev *__restrict__ scenes, const int2 *__restrict__ items, int n_items,
                           int group, unsigned *queue) {
    extern __shared__ float4 dyn[];
    __shared__ float4 s_fp[kFpSlots];
    __shared__ int s_item, s_next;
    int fp_scene = -1;   // block-uniform
    for (;;) {
        if (threadIdx.x == 0) s_item = (int)atomicAdd(queue, 1u);
        __syncthreads();   // also: the previous item's costs are formed
        const int item = s_item;
        if (item >= n_items) break;
        const int2 it = items[item];
        const SceneDev &D = scenes[it.x];
        const bool fresh = it.x != fp_scene;
        if (fresh) {
            load_table(s_fp, D.fp);
            __syncthreads();
            fp_scene = it.x;
        }
        grid_samples<false, FAR>(D.V, D.grid, GridStride{0, 0}, table_eval(D.fp, s_fp), it.y, min(group, D.V.P.K - it.y),
                            reinterpret_cast<char *>(dyn), fresh, &s_next);
    }
}

// The cell grids (one block each).
__global__ void __launch_bounds__(kGridThreads)
batched_cloud_grid_kernel(const SceneDev *__restrict__ scenes, const int *__restrict__ list) {
    __shared__ GridSmem sm;
    const SceneDev &D = scenes[list[blockIdx.x]];
    build_grid<false>(D.src_pts, nullptr, D.src_mask, D.V.N, const_cast<float2 *>(D.V.pts), nullptr, D.grid, sm);
}

__global__ void __launch_bounds__(kUpdBlock)
batched_update_kernel(const SceneDev *__restrict__ scenes, const int2 *__restrict__ table) {
    __shared__ UpdateSmem sm;
    __shared__ SceneView V;
    const int2 t = table[blockIdx.x];
    stage_view(V, scenes[t.x].V);
    update_body(V, t.y, sm);
}

__global__ void __launch_bounds__(kBlock)
batched_validate_kernel(const SceneDev *__restrict__ scenes, const int2 *__restrict__ table) {
    __shared__ float4 s_fp[kFpSlots];
    __shared__ ValidateSmem sm;
    const int2 t = table[blockIdx.x];
    __shared__ SceneView V;
    const SceneDev &D = scenes[t.x];
    load_table(s_fp, D.fp);
    const CloudGrid *grid = D.grid;
    const SmemEval ev = table_eval(D.fp, s_fp);
    stage_view(V, D.V);
    validate_body(V, ev, t.y / V.val_chunks, t.y % V.val_chunks, sm, grid);
}

// The tuning views write their d_min to buf instead of the scenes' outputs.
// They share it: nothing reads it.
__global__ void tune_dmin_kernel(SceneDev *tune, const SceneDev *scenes, int n, float *buf) {
    for (int s = threadIdx.x; s < n; s += blockDim.x) tune[s].V.dmin = scenes[s].V.dmin ? buf : nullptr;
}

int check_params(const exact_mppi_params *p);
MppiP to_device_params(const exact_mppi_params *p);

}  // namespace exact

using namespace exact;


static int batch_grid(exact_batch *b) {
    int per_sm = 0;
    // the staged points and footprint slots (dynamic) plus the sample state
    // (static) exceed the default 48 KB per block
    if (cudaFuncSetAttribute(batched_sample_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSampleSmemMax) !=
        cudaSuccess)
        return EXACT_ECUDA;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batched_sample_kernel, sample_threads(b), b->smem) !=
        cudaSuccess)
        return EXACT_ECUDA;
    if (per_sm < 1) return EXACT_EINVAL;
    b->grid = b->sms * per_sm;
    if (b->n_gitems == 0) return EXACT_OK;
    const auto grid_kernel = b->far ? batched_grid_sample_kernel<true> : batched_grid_sample_kernel<false>;
    if (cudaFuncSetAttribute(grid_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kGridSmemMax) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, grid_kernel, b->threads, grid_smem(b)) !=
            cudaSuccess)
        return EXACT_ECUDA;
    if (per_sm < 1) return EXACT_EINVAL;
    b->ggrid = b->sms * per_sm;
    return EXACT_OK;
}

// Which scenes walk a cell grid (cloud_grid.cuh): those without a d_min output
// and with 1,024 points or more, and the smaller ones where grids are built
// anyway or pay.  Else these are items of the other sample kernel, which prunes
// them point by point and is launched for scenes with a d_min output anyway.
// Grids pay from about 2,048 samples on, up to T = 32, and beyond for ten points
// a step (us, items against grids, one footprint: 4 scenes of 256 samples, T = 20,
// 300 points 22.7, 26.4; 16 such scenes 41.8, 37.8, with T = 60 61.9, 68.5, with
// T = 60 and 1,000 points 73.4, 72.5; four footprints: 61.8, 47.7; 84.4, 86.6; 118,
// 94).
struct GridRule {
    bool small = false;   // scenes below kPruneMin points too
    GridRule(const exact_scene *scenes, int n) {
        bool grids = false, items = false;   // launched for other scenes anyway
        long long samples = 0, paying = 0;
        for (int s = 0; s < n; ++s) {
            const exact_scene &S = scenes[s];
            if (S.dmin || S.n_points > kGridMaxPoints) items = true;
            else if (S.n_points >= kPruneMin) grids = true;
            else {
                samples += S.params.K;
                if (S.params.T <= 32 || S.n_points >= 10 * S.params.T) paying += S.params.K;
            }
        }
        const bool pays = paying >= 2048 && 2 * paying >= samples;
        small = items ? grids && pays : grids || pays;
    }
    bool operator()(const exact_scene &S) const {
        return !S.dmin && S.n_points <= kGridMaxPoints && (small || S.n_points >= kPruneMin);
    }
};

extern "C" int exact_batch_create(int n_scenes, const exact_scene *scenes, exact_batch **out) {
    if (!out || !scenes || n_scenes < 1) return EXACT_EINVAL;
    *out = nullptr;
    if (n_scenes > 4096) return EXACT_ECAPACITY;
    const GridRule uses_grid(scenes, n_scenes);
    std::vector<SceneDev> host(n_scenes);
    std::vector<size_t> scratch_off(n_scenes);
    size_t scratch_total = 0;
    int max_stage = 0;
    size_t dmin_len = 0;
    bool pairs_matter = false;
    for (int s = 0; s < n_scenes; ++s) {
        const exact_scene &S = scenes[s];
        int rc = check_params(&S.params);
        if (rc != EXACT_OK) return rc;
        if (!S.fp || !S.state || !S.U || !S.noise || !S.waypoints || S.n_wp < 1 || S.n_points < 0 || !S.u_star)
            return EXACT_EINVAL;
        if (S.n_points > 0 && (!S.cloud || ((uintptr_t)S.cloud & 7u) != 0)) return EXACT_EINVAL;
        scratch_off[s] = scratch_total;
        scratch_total += align_up(scene_scratch_bytes(S.params.K, S.params.T, 1), 256);
        // a grid and a copy of the cloud in cell order
        if (uses_grid(S))
            scratch_total += grid_copy_bytes(S.n_points, false);
        else
            max_stage = std::max(max_stage, std::min(S.n_points, kStage));
        if (S.dmin) dmin_len = std::max(dmin_len, (size_t)S.params.K * S.params.T);
        pairs_matter |= !S.dmin && S.n_points >= kPruneMin && !uses_grid(S);
    }
    std::vector<int> sort_list;
    for (int s = 0; s < n_scenes; ++s)
        if (uses_grid(scenes[s])) sort_list.push_back(s);
    const size_t table_bytes = align_up(sizeof(SceneDev) * n_scenes, 256);
    // items and block tables
    std::vector<int> order(n_scenes);
    for (int s = 0; s < n_scenes; ++s) order[s] = s;
    auto cost = [&](int s) {
        const exact_scene &S = scenes[s];
        return (double)S.params.T * std::max(S.n_points, 1) * (double)S.fp->n_pad;
    };
    std::stable_sort(order.begin(), order.end(), [&](int a, int c) { return cost(a) > cost(c); });
    std::vector<int2> items, gitems, upd, val;
    long long total_k = 0, grid_k = 0;
    int grid_T = 1;
    for (int s = 0; s < n_scenes; ++s) {
        total_k += scenes[s].params.K;
        if (uses_grid(scenes[s])) {
            grid_k += scenes[s].params.K;
            grid_T = std::max(grid_T, scenes[s].params.T);
        }
    }
    const int sms_now = current_sm_count();
    const int group = grid_group(grid_k, grid_T, kBlock / 32, sms_now);
    for (int s : order) {
        const exact_mppi_params &p = scenes[s].params;
        if (uses_grid(scenes[s])) {
            for (int r = 0; r < p.K; r += group) gitems.push_back(make_int2(s, r));
            continue;
        }
        // pairs of samples per item when the whole batch has enough samples
        // to fill the GPU at half the items (and this scene's horizon fits)
        const bool two = pair_samples((int)std::min<long long>(total_k, 1 << 29), p.T, 1, sms_now);
        for (int r = 0; r < p.K; r += two ? 2 : 1)
            items.push_back(make_int2(s, r | (two && r + 1 < p.K ? kItemPair : 0)));
    }
    for (int s = 0; s < n_scenes; ++s) {
        const exact_mppi_params &p = scenes[s].params;
        for (int q = 0; q < upd_blocks_for(p.K, p.T, p.n_u); ++q) upd.push_back(make_int2(s, q));
        for (int q = 0; q < p.T * val_chunks_for(scenes[s].n_points, uses_grid(scenes[s])); ++q) val.push_back(make_int2(s, q));
    }
    const size_t items_bytes = align_up(items.size() * sizeof(int2) + 1, 256);
    const size_t gitems_bytes = align_up(gitems.size() * sizeof(int2) + 1, 256);
    const size_t upd_bytes = align_up(upd.size() * sizeof(int2), 256);
    const size_t val_bytes = align_up(val.size() * sizeof(int2), 256);
    const size_t ctrl_bytes = align_up(kHdrStride * n_scenes + 2 * sizeof(unsigned), 256);
    const size_t sort_bytes = align_up(sort_list.size() * sizeof(int) + 1, 256);
    const size_t err_bytes = 256;
    const size_t total =
        2 * table_bytes + items_bytes + gitems_bytes + upd_bytes + val_bytes + ctrl_bytes + sort_bytes + err_bytes + scratch_total;

    exact_batch *b = new (std::nothrow) exact_batch();
    if (!b) return EXACT_EINVAL;
    if (cudaMalloc(&b->dev, total) != cudaSuccess) { delete b; return EXACT_ECUDA; }
    char *p = static_cast<char *>(b->dev);
    b->d_scenes = reinterpret_cast<SceneDev *>(p); p += table_bytes;
    b->d_tune = reinterpret_cast<SceneDev *>(p); p += table_bytes;
    b->d_items = reinterpret_cast<int2 *>(p); p += items_bytes;
    b->d_gitems = reinterpret_cast<int2 *>(p); p += gitems_bytes;
    b->d_upd = reinterpret_cast<int2 *>(p); p += upd_bytes;
    b->d_val = reinterpret_cast<int2 *>(p); p += val_bytes;
    b->d_ctrl = p; p += ctrl_bytes;
    b->d_sort = reinterpret_cast<int *>(p); p += sort_bytes;
    b->n_sort = (int)sort_list.size();
    b->d_err = reinterpret_cast<int *>(p); p += err_bytes;
    char *scratch = p;
    b->ctrl_bytes = ctrl_bytes;
    b->d_queue = reinterpret_cast<unsigned *>(b->d_ctrl + kHdrStride * n_scenes);
    b->n = n_scenes;
    b->n_items = (int)items.size();
    b->paired = std::any_of(items.begin(), items.end(), [](int2 it) { return (it.y & kItemPair) != 0; });
    b->n_gitems = (int)gitems.size();
    b->grid_group = group;
    b->grid_T = grid_T;
    b->dmin_len = dmin_len;
    b->pairs_matter = pairs_matter;
    for (int s : sort_list) b->far |= field_ends(scenes[s].params.d_safe, scenes[s].fp->bhx, scenes[s].fp->bhy);
    b->n_upd = (int)upd.size();
    b->n_val = (int)val.size();
    b->smem = kFpSlots * sizeof(float4) + (size_t)max_stage * sizeof(float2);
    b->sms = current_sm_count();
    b->uniform = true;
    for (int s = 1; s < n_scenes && b->uniform; ++s)
        b->uniform = memcmp(scenes[s].fp, scenes[0].fp, sizeof(exact_footprint)) == 0;
    if (b->uniform) b->fp = *scenes[0].fp;

    for (int s = 0; s < n_scenes; ++s) {
        const exact_scene &S = scenes[s];
        SceneDev &D = host[s];
        memset(&D, 0, sizeof(D));
        SceneView &V = D.V;
        V.P = to_device_params(&S.params);
        V.state = S.state;
        V.pts = reinterpret_cast<const float2 *>(S.cloud);
        V.mask = S.mask;
        V.N = S.n_points;
        V.wp = S.waypoints;
        V.W = S.n_wp;
        V.U = S.U;
        V.noise = S.noise;
        V.u_star = S.u_star; V.costs = S.costs; V.weights = S.weights; V.U_upd_out = S.U_upd;
        V.dmin = S.dmin; V.valid = S.valid; V.nom_cost = S.nom_cost;
        V.err = b->d_err;
        V.hdr = reinterpret_cast<ArenaHeader *>(b->d_ctrl + kHdrStride * s);
        carve_scene(V, scratch + scratch_off[s], S.params.K, S.params.T, 1);
        D.src_pts = V.pts;
        D.src_mask = V.mask;
        if (uses_grid(S)) {   // filled before each step's sample phase
            char *q = scratch + scratch_off[s] + align_up(scene_scratch_bytes(S.params.K, S.params.T, 1), 256);
            D.grid = reinterpret_cast<CloudGrid *>(q);
            V.pts = reinterpret_cast<const float2 *>(q + kGridBytes);
            V.mask = nullptr;
        }
        V.upd_chunk = upd_chunk_for(S.params.K, S.params.T, S.params.n_u);
        V.upd_blocks = upd_blocks_for(S.params.K, S.params.T, S.params.n_u);
        V.val_chunks = val_chunks_for(S.n_points, uses_grid(S));
        const exact_footprint *fp = S.fp;
        D.fp = make_table(fp);
    }
    int rc = EXACT_OK;
    if (cudaMemcpy(b->d_scenes, host.data(), sizeof(SceneDev) * n_scenes, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(b->d_tune, host.data(), sizeof(SceneDev) * n_scenes, cudaMemcpyHostToDevice) != cudaSuccess ||
        (b->n_items &&
         cudaMemcpy(b->d_items, items.data(), items.size() * sizeof(int2), cudaMemcpyHostToDevice) != cudaSuccess) ||
        (b->n_gitems && cudaMemcpy(b->d_gitems, gitems.data(), gitems.size() * sizeof(int2), cudaMemcpyHostToDevice) !=
                            cudaSuccess) ||
        cudaMemcpy(b->d_upd, upd.data(), upd.size() * sizeof(int2), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(b->d_val, val.data(), val.size() * sizeof(int2), cudaMemcpyHostToDevice) != cudaSuccess ||
        (b->n_sort && cudaMemcpy(b->d_sort, sort_list.data(), sort_list.size() * sizeof(int), cudaMemcpyHostToDevice) !=
                          cudaSuccess) ||
        cudaMemset(b->d_ctrl, 0, ctrl_bytes) != cudaSuccess || cudaMemset(b->d_err, 0, err_bytes) != cudaSuccess ||
        (scratch_total && cudaMemset(scratch, 0, scratch_total) != cudaSuccess))
        rc = EXACT_ECUDA;
    if (rc == EXACT_OK) rc = batch_grid(b);
    if (rc != EXACT_OK) {
        cudaFree(b->dev);
        delete b;
        return rc;
    }
    *out = b;
    return EXACT_OK;
}

extern "C" void exact_batch_destroy(exact_batch *b) {
    if (!b) return;
    cudaDeviceSynchronize();
    cudaFree(b->dev);
    delete b;
}

static int launch_uniform(exact_batch *b, const SceneDev *table, cudaStream_t st, BatchPhase phase) {
    return b->fp.kind == EXACT_FP_POLYGON && b->fp.n_pad > 16 ? launch_uniform_large(b, table, st, phase)
                                                               : launch_uniform_small(b, table, st, phase);
}

static int launch_sample(exact_batch *b, const SceneDev *table, cudaStream_t st) {
    if (cudaMemsetAsync(b->d_ctrl, 0, b->ctrl_bytes, st) != cudaSuccess) return EXACT_ECUDA;
    if (b->n_items > 0) {   // scenes that walk no grid
        if (!b->uniform) {
            batched_sample_kernel<<<b->grid, sample_threads(b), b->smem, st>>>(table, b->d_items, b->n_items, b->d_queue,
                                                                         b->pairs);
            if (cudaGetLastError() != cudaSuccess) return EXACT_ECUDA;
        } else {
            const int rc = launch_uniform(b, table, st, kPhaseSample);
            if (rc != EXACT_OK) return rc;
        }
    }
    if (b->n_gitems == 0) return EXACT_OK;
    batched_cloud_grid_kernel<<<b->n_sort, kGridThreads, 0, st>>>(table, b->d_sort);
    if (cudaGetLastError() != cudaSuccess) return EXACT_ECUDA;
    // the persistent warps start early (rollouts first; grid_sample waits
    // before it reads a grid)
    // no more blocks than items: idle ones would crowd the busy ones on an SM
    return cuda_status(launch_dependent(b->far ? batched_grid_sample_kernel<true> : batched_grid_sample_kernel<false>, (unsigned)std::min(b->ggrid, b->n_gitems), (unsigned)b->threads,
                                        grid_smem(b), st, table, (const int2 *)b->d_gitems, b->n_gitems, b->grid_group,
                                        b->d_queue + 1));
}

extern "C" int mppi_step_batched(exact_batch *b, void *stream) {
    if (!b) return EXACT_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    int rc = launch_sample(b, b->d_scenes, st);
    if (rc != EXACT_OK) return rc;
    // update and validation start while their predecessor drains
    // (programmatic dependent launch; the bodies wait where they read its
    // results, as in the single-scene cycle)
    if (launch_dependent(batched_update_kernel, (unsigned)b->n_upd, (unsigned)kUpdBlock, 0, st,
                         (const SceneDev *)b->d_scenes, (const int2 *)b->d_upd) != cudaSuccess)
        return EXACT_ECUDA;
    if (!b->uniform)
        return cuda_status(launch_dependent(batched_validate_kernel, (unsigned)b->n_val, (unsigned)kBlock, 0, st,
                                            (const SceneDev *)b->d_scenes, (const int2 *)b->d_val));
    return launch_uniform(b, b->d_scenes, st, kPhaseValidate);
}

extern "C" int exact_batch_get_error(exact_batch *b, void *stream) {
    if (!b) return EXACT_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    int err = 0;
    if (cudaMemcpyAsync(&err, b->d_err, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaMemsetAsync(b->d_err, 0, sizeof(int), st) != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess)
        return EXACT_ECUDA;
    return err;
}

extern "C" int exact_batch_get_tiles(const exact_batch *b, int *threads, int *pairs_per_lane) {
    if (!b) return EXACT_EINVAL;
    if (threads) *threads = b->threads;
    if (pairs_per_lane) *pairs_per_lane = b->pairs;
    return EXACT_OK;
}

extern "C" int exact_batch_set_tiles(exact_batch *b, int threads, int pairs_per_lane) {
    if (!b) return EXACT_EINVAL;
    if (!(threads == 64 || threads == 128 || threads == 256 || threads == 512)) return EXACT_EINVAL;
    if (pairs_per_lane < 1 || pairs_per_lane > 8) return EXACT_EINVAL;
    const int ot = b->threads, op = b->pairs;
    b->threads = threads;
    b->pairs = pairs_per_lane;
    b->grid_c = 0;
    const int rc = batch_grid(b);
    if (rc != EXACT_OK) {
        b->threads = ot;
        b->pairs = op;
        batch_grid(b);
    }
    return rc;
}

extern "C" int exact_batch_autotune(exact_batch *b, int iters, char *json_out, int json_cap, void *stream) {
    if (!b || iters < 1) return EXACT_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    static const int kThreads[] = {128, 256, 512};
    static const int kPairs[] = {1, 2, 4, 8};
    const int now[] = {b->pairs, b->pairs};
    // point pairs per lane only shape the sub-chunks of a cloud pruned without
    // a grid; elsewhere each block size is timed twice instead
    const int *pairs = b->pairs_matter ? kPairs : now;
    const int n_pairs = b->pairs_matter ? 4 : 2;
    float *dmin = nullptr;
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess ||
        (b->dmin_len && cudaMalloc(&dmin, b->dmin_len * sizeof(float)) != cudaSuccess))
        return EXACT_ECUDA;
    tune_dmin_kernel<<<1, 256, 0, st>>>(b->d_tune, b->d_scenes, b->n, dmin);
    float best_ms = 3.0e38f;
    int best_t = b->threads, best_p = b->pairs;
    std::string json = "{\"candidates\": [";
    bool first = true;
    int rc = cuda_status(cudaGetLastError());
    for (int c = 0; c < 3 * n_pairs && rc == EXACT_OK; ++c) {
        const int t = kThreads[c % 3], pl = pairs[c / 3];
        if (exact_batch_set_tiles(b, t, pl) != EXACT_OK) continue;
        if ((rc = launch_sample(b, b->d_tune, st)) != EXACT_OK) break;   // warm-up
        cudaEventRecord(e0, st);
        for (int i = 0; i < iters && rc == EXACT_OK; ++i) rc = launch_sample(b, b->d_tune, st);
        cudaEventRecord(e1, st);
        if (rc != EXACT_OK || cudaEventSynchronize(e1) != cudaSuccess) { rc = EXACT_ECUDA; break; }
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        ms /= iters;
        char buf[128];
        snprintf(buf, sizeof(buf), "%s{\"threads\": %d, \"pairs_per_lane\": %d, \"ms\": %.6f}", first ? "" : ", ", t, pl, ms);
        json += buf;
        first = false;
        if (ms < best_ms) { best_ms = ms; best_t = t; best_p = pl; }
    }
    cudaStreamSynchronize(st);
    if (dmin) cudaFree(dmin);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    const int src = exact_batch_set_tiles(b, best_t, best_p);
    if (rc == EXACT_OK) rc = src;
    char buf[160];
    snprintf(buf, sizeof(buf), "], \"best\": {\"threads\": %d, \"pairs_per_lane\": %d, \"ms\": %.6f}}", best_t, best_p,
             best_ms);
    json += buf;
    if (json_out && json_cap > 0) {
        strncpy(json_out, json.c_str(), (size_t)json_cap - 1);
        json_out[json_cap - 1] = '\0';
    }
    return rc;
}
