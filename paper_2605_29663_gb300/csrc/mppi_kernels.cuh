// mppi_kernels.cuh -- the three kernels of one single-scene control cycle
// and their stream-ordered launch, templated on static / predicted
// (time-indexed) obstacle points and on the sample kernel's minimum resident
// blocks per SM (MINB).  MINB = 4 caps the sample kernel at 64 registers:
// four blocks per SM, which pays when the grid spans several waves and the
// footprint is small; otherwise MINB = 0 leaves the register count to the
// compiler (about 120 for these bodies; an explicit minimum of one or two
// blocks changed its choices and measured slower, and so did 512-thread
// blocks for small grids).  mppi.cu instantiates the static uncapped cycle,
// mppi_dense.cu the static capped one, mppi_predicted.cu the predicted
// (capped) one and mppi_grid.cu the cycle on a cell grid, so that they compile
// in parallel.
#pragma once
#include "cloud_grid.cuh"

namespace exact {

// The validation kernel that follows on the stream counts its finished
// blocks on this ticket: it starts from zero.
__device__ __forceinline__ void reset_validation(const SceneView &V) {
    V.hdr->ticket[1] = 0u;
    V.hdr->vticket = 0ull;
    V.hdr->bad = 0;
}

template <class FPC, bool MOVING, int MINB, int PATH>
__global__ void __launch_bounds__(kBlock, MINB)
mppi_sample_kernel(const SceneView V, const ConstEval<FPC> ev, int pair) {
    extern __shared__ float2 s_pts[];   // min(N, stage) staged points (float4 each when MOVING)
    __shared__ SampleSmem sm;
    sample_smem_init(sm);
    if (blockIdx.x == 0 && threadIdx.x == 0) reset_validation(V);
    // pair: block b takes samples 2b and 2b + 1; else sample b / parts,
    // horizon part b % parts.  Only the register-capped static instantiations
    // carry the two-sample path: in the uncapped ones (large polygons) it cost
    // the compiler spills, and predicted clouds measured slower with it.
    const bool two = MINB != 0 && !MOVING && pair;
    const int r = two ? 2 * (int)blockIdx.x : (int)blockIdx.x / V.parts;
    const int p = two ? 0 : (int)blockIdx.x % V.parts;
    sample_body<MOVING, PATH>(V, ev, r, p, sm, s_pts, false, 1, two && r + 1 < V.P.K ? r + 1 : -1);
}

template <bool MOVING>
__global__ void __launch_bounds__(kUpdBlock) mppi_update_kernel(const SceneView V) {
    __shared__ UpdateSmem sm;
    update_body(V, blockIdx.x, sm);
}

template <class FPC, bool MOVING>
__global__ void __launch_bounds__(kBlock) mppi_validate_kernel(const SceneView V, const ConstEval<FPC> ev) {
    __shared__ ValidateSmem sm;
    validate_body<MOVING>(V, ev, blockIdx.x / V.val_chunks, blockIdx.x % V.val_chunks, sm);
}

// The cycle of a cloud with a grid evaluates few points (cloud_grid.cuh), so
// its kernels take the footprint as a slot table in the kernel parameters,
// copied to shared memory: one kernel for every footprint, small enough to be
// fetched quickly.  Sample phase: block b takes samples b group ...
template <bool MOVING, bool FAR>
__global__ void __launch_bounds__(kBlock, 3)
mppi_grid_sample_kernel(const SceneView V, const __grid_constant__ FpTable fp, const CloudGrid *grid, GridStride gst,
                        int group) {
    extern __shared__ float4 s_mem[];
    __shared__ float4 s_fp[kFpSlots];
    __shared__ int s_next;
    if (blockIdx.x == 0 && threadIdx.x == 0) reset_validation(V);
    grid_dep_release();   // the update blocks may stage their noise meanwhile
    load_table(s_fp, fp);
    __syncthreads();
    const int r0 = (int)blockIdx.x * group;
    grid_samples<MOVING, FAR>(V, grid, gst, table_eval(fp, s_fp), r0, min(group, V.P.K - r0), reinterpret_cast<char *>(s_mem),
                         true, &s_next);
}
template <bool MOVING>
__global__ void __launch_bounds__(kBlock)
mppi_grid_validate_kernel(const SceneView V, const __grid_constant__ FpTable fp, const CloudGrid *grid, GridStride gst) {
    __shared__ ValidateSmem sm;
    __shared__ float4 s_fp[kFpSlots];
    load_table(s_fp, fp);   // validate_body synchronises before it evaluates
    const int h = blockIdx.x;
    validate_body<MOVING>(V, table_eval(fp, s_fp), h, 0, sm, grid + h * gst.grids, h * gst.points);
}

// The three launches of one cycle for a scene whose scratch is carved.
// PATH = kPathPoints: only for footprints whose evaluator prunes point by
// point (ConstEval::kQueueOk), cycles without a d_min output and clouds below
// kPruneMin points.
template <bool MOVING, int MINB, int PATH = kPathAny>
int launch_cycle_t(const SceneView &V, const exact_footprint *fp, cudaStream_t st, int sms) {
    const size_t smem = (size_t)min(V.N, stage_points_of<MOVING>()) * (MOVING ? sizeof(float4) : sizeof(float2));
    const int pair = MINB != 0 && !MOVING ? pair_samples(V.P.K, V.P.T, V.parts, sms) : 0;
    const int grid = pair ? (V.P.K + 1) / 2 : V.P.K * V.parts;
    auto launch = [&](auto fpc) -> int {
        using FPC = decltype(fpc);
        const ConstEval<FPC> ev{fpc};
        mppi_sample_kernel<FPC, MOVING, MINB, PATH><<<grid, kBlock, smem, st>>>(V, ev, pair);
        if (cudaGetLastError() != cudaSuccess) return EXACT_ECUDA;
        if (launch_dependent(mppi_update_kernel<MOVING>, V.upd_blocks, kUpdBlock, 0, st, V) != cudaSuccess)
            return EXACT_ECUDA;
        return cuda_status(
            launch_dependent(mppi_validate_kernel<FPC, MOVING>, V.P.T * V.val_chunks, kBlock, 0, st, V, ev));
    };
    if constexpr (PATH == kPathPoints)
        return with_small_footprint(fp, launch);
    else
        return with_footprint(fp, launch);
}

// The launches of one cycle behind the kernel that builds the cloud's grid:
// the sample kernel may start early too (its rollouts do not read the cloud).
template <bool MOVING>
int launch_grid_cycle_t(const SceneView &V, const exact_footprint *fp, cudaStream_t st, const CloudGrid *grid,
                        GridStride gst, int sms) {
    const int group = grid_group(V.P.K, V.P.T, kBlock / 32, sms);
    const size_t smem = grid_smem_bytes(V.P.T, group, kBlock / 32);
    auto sample = field_ends(V.P.d_safe, fp->bhx, fp->bhy) ? mppi_grid_sample_kernel<MOVING, true>
                                                            : mppi_grid_sample_kernel<MOVING, false>;
    // beyond the default 48 KB with the footprint's slots
    if (smem > 40u * 1024u &&
        cudaFuncSetAttribute(sample, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGridSmemMax) != cudaSuccess)
        return EXACT_ECUDA;
    const FpTable t = make_table(fp);
    if (launch_dependent(sample, (V.P.K + group - 1) / group, kBlock, smem, st, V, t, grid,
                         gst, group) != cudaSuccess ||
        launch_dependent(mppi_update_kernel<MOVING>, V.upd_blocks, kUpdBlock, 0, st, V) != cudaSuccess)
        return EXACT_ECUDA;
    return cuda_status(launch_dependent(mppi_grid_validate_kernel<MOVING>, V.P.T, kBlock, 0, st, V, t, grid, gst));
}

// Any cycle without a grid (mppi.cu: picks one of the four below), the static
// capped cycle (mppi_dense.cu), the predicted cycle (mppi_predicted.cu), and
// the cycles with a grid (mppi_grid.cu).  sms is the
// SM count of the device the cycle runs on (it sizes the grids).
int launch_cycle(const SceneView &V, const exact_footprint *fp, cudaStream_t st, int sms);
int launch_cycle_dense(const SceneView &V, const exact_footprint *fp, cudaStream_t st, int sms);
int launch_cycle_moving(const SceneView &V, const exact_footprint *fp, cudaStream_t st, int sms);
int launch_cycle_grid(const SceneView &V, const exact_footprint *fp, cudaStream_t st, const CloudGrid *grid,
                      GridStride gst, int sms);
// The static capped cycle whose sample kernel holds only the point-level
// pruning (mppi_points.cu): small footprints, no d_min output, N < kPruneMin.
int launch_cycle_points(const SceneView &V, const exact_footprint *fp, cudaStream_t st, int sms);

// mppi_step with optional point velocities (NULL: static cloud).
int mppi_step_impl(exact_ctx *ctx, const float *state, const float *cloud, const float *velocity,
                   const uint8_t *mask, int n_points, const float *waypoints, int n_wp, float *U,
                   const float *noise, const exact_footprint *fp, const exact_mppi_params *params, float *u_star,
                   float *costs, float *weights, int *valid, float *U_upd, float *dmin, void *stream);

}  // namespace exact
