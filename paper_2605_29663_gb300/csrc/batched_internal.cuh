// batched_internal.cuh -- what batched.cu (plan, generic kernels) and
// batched_uniform.cuh (constant-footprint kernels) share: the device scene
// table entry and the batch plan.
#pragma once

#include "cloud_grid.cuh"

namespace exact {

constexpr size_t kHdrStride = 64;                            // bytes between scene headers
// Most dynamic shared memory of the sample kernels: footprint slots and staged
// points.  Every plan sets this limit (see kGridSmemMax).
constexpr size_t kSampleSmemMax = kFpSlots * sizeof(float4) + kStage * sizeof(float2);

struct SceneDev {
    SceneView V;
    const float2 *src_pts;      // the caller's cloud (V.pts may be its copy in cell order)
    const uint8_t *src_mask;
    CloudGrid *grid;            // cell grid of the ordered copy, or NULL
    FpTable fp;
};

// The scene's view in shared memory, read before the block waits for its
// predecessor: its fields are otherwise fetched from the table one dependent
// load after the other behind the wait.  Ends with a block barrier.
__device__ __forceinline__ void stage_view(SceneView &dst, const SceneView &src) {
    static_assert(sizeof(SceneView) % 4 == 0, "copied in words");
    for (int i = threadIdx.x; i < (int)(sizeof(SceneView) / 4); i += blockDim.x)
        reinterpret_cast<int *>(&dst)[i] = reinterpret_cast<const int *>(&src)[i];
    __syncthreads();
}

// A sample item of a scene that walks no grid is (scene, r); bit 30 of r
// marks an item that also takes sample r + 1 of the same scene (see
// sample_body).  A grid item is (scene, r): grid_group consecutive samples
// from r on (see grid_samples).
constexpr int kItemPair = 1 << 30;
__device__ __forceinline__ int item_sample(int2 it) { return it.y & (kItemPair - 1); }
__device__ __forceinline__ int item_second(int2 it) { return (it.y & kItemPair) ? (it.y & (kItemPair - 1)) + 1 : -1; }

}  // namespace exact

struct exact_batch {
    int n = 0;
    void *dev = nullptr;
    exact::SceneDev *d_scenes = nullptr;      // for steps
    exact::SceneDev *d_tune = nullptr;        // same, with another d_min output (autotuning)
    int2 *d_items = nullptr, *d_gitems = nullptr, *d_upd = nullptr, *d_val = nullptr;
    int n_items = 0, n_gitems = 0, n_upd = 0, n_val = 0;
    int grid_group = 1, grid_T = 1;      // samples per grid item, longest horizon of a grid scene
    size_t dmin_len = 0;                 // most d_min values of a scene that outputs them
    bool far = false;                    // some grid scene's field ends before its d_safe
    bool paired = false;                 // some items take two samples
    bool pairs_matter = false;           // some scene is pruned without a grid
    char *d_ctrl = nullptr;            // n headers (kHdrStride apart) + queue head
    size_t ctrl_bytes = 0;
    unsigned *d_queue = nullptr;       // queue heads: items, grid items
    int *d_sort = nullptr;             // scenes whose cloud gets a grid
    int n_sort = 0;
    size_t smem = 0;
    int threads = exact::kBlock, pairs = 1, sms = 0, grid = 0;
    int ggrid = 0;                     // persistent grid of the grid kernel
    bool uniform = false;              // every scene has the same footprint constants
    exact_footprint fp;                // their copy (uniform batches)
    int grid_c = 0;                    // persistent grid of the constant-footprint kernel (0 = not yet known)
    int *d_err = nullptr;              // device error word of the batch (not cleared by steps)
};

namespace exact {
// Sample or validation launch of a batch whose scenes share one footprint,
// footprint constants as kernel parameters (batched_uniform.cuh): rectangle
// covers and polygons of up to 16 edges, and larger polygons.
enum BatchPhase { kPhaseSample, kPhaseValidate };
int launch_uniform_small(exact_batch *b, const SceneDev *table, cudaStream_t st, BatchPhase phase);
int launch_uniform_large(exact_batch *b, const SceneDev *table, cudaStream_t st, BatchPhase phase);

// Threads of the sample kernel: the tile's, and a third warp where items take
// two samples, for the first two roll these out while the others stage the points.
inline int sample_threads(const exact_batch *b) { return b->paired && b->threads < 96 ? 96 : b->threads; }
inline size_t grid_smem(const exact_batch *b) { return grid_smem_bytes(b->grid_T, b->grid_group, b->threads / 32); }
}  // namespace exact
