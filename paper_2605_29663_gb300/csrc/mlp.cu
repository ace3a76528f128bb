// mlp.cu -- the learned sampling proposal's network on the tensor cores.
//
// y = W3 g(W2 g(W1 x + b1) + b2) + b3 with the exact GELU g(z) = z Phi(z).
// Every product is a BF16 x BF16 -> FP32 tensor-core GEMM (mma.sync
// m16n8k16).  FP32 master weights and Adam moments; BF16 copies of the
// weights and of every GEMM operand (activations, output and hidden
// gradients); FP32 pre-activations for the GELU derivative; FP32 gradients.
//
// What bounds it: latency.  A training step of the 111-256-256-40 network on
// a batch of 1,024 is 0.6 GFLOP over a few MB that stay in L2, so what counts
// is the number of dependent launches and the depth of each.  A step is seven:
// three forward layers (the last one forms the output gradient and the loss
// too), two input gradients, all weight and bias gradients together, and one
// that adds their partial sums, steps Adam and refreshes the BF16 weights.
// Each starts while its predecessor drains (programmatic dependent launch) and
// fetches its weights before it waits.  The GEMMs stage 16-byte cp.async
// copies of whole 64-wide k tiles, four in flight (K = 256 is in flight
// entirely), in XOR-swizzled rows read with ldmatrix; 32 x 64 output tiles
// spread a batch of 1,024 over 128 blocks.  Operand rows are padded to whole
// 16-byte chunks, zero-filled.  Every sum runs in a fixed order: k ascending in
// the products, gradients over the batch in kchunk slices added in order, the
// loss over the output tiles' double sums.
// Measured, host calls included: 8 steps and one loss_grad on a batch of 1,024
// in 376 us (2,627 us with one strided-load GEMM kernel and 27 launches per
// step), the proposal's inference for 256 robots in 39 to 49 us (123 us).
#include <cuda_bf16.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <vector>

#include "mppi_cycle.cuh"

namespace exact {

typedef __nv_bfloat16 bf16;

constexpr int kMlpInPad = 128;   // inputs are zero-padded to this width
constexpr int kBN = 64, kBK = 64, kStages = 4;

__device__ __forceinline__ float gelu_f(float z) { return 0.5f * z * (1.f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad_f(float z) {
    return 0.5f * (1.f + erff(z * 0.70710678118654752f)) + z * expf(-0.5f * z * z) * 0.39894228040143268f;
}

__device__ __forceinline__ void mma_bf16(float *d, const uint32_t *a, const uint32_t *b) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// ---------------------------------------------------------------- tiles
// A tile is R rows of 64 bf16 (128 bytes) in shared memory, the 16-byte chunks
// of a row XORed with the row's low bits, so that the eight rows an ldmatrix
// reads fall into different banks.
__device__ __forceinline__ unsigned tile_addr(const bf16 *tile, int row, int chunk) {
    return smem_addr(tile) + row * 128 + ((chunk ^ (row & 7)) << 4);
}
// Rows [r0, r0 + R) x columns [c0, c0 + 64) of a row-major matrix (ld a
// multiple of 8, 16-byte aligned); rows from rmax and chunks from cmax (a
// multiple of 8) on are zero.  128 threads, no wait.
template <int R>
__device__ __forceinline__ void tile_load(bf16 *tile, const bf16 *__restrict__ g, int ld, int r0, int rmax, int c0,
                                          int cmax) {
#pragma unroll
    for (int k = 0; k < R * 8 / 128; ++k) {
        const int e = k * 128 + threadIdx.x, row = e >> 3, chunk = e & 7;
        const bool ok = r0 + row < rmax && c0 + chunk * 8 < cmax;
        const bf16 *src = ok ? g + (size_t)(r0 + row) * ld + c0 + chunk * 8 : g;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(tile_addr(tile, row, chunk)), "l"(src),
                     "r"(ok ? 16 : 0)
                     : "memory");
    }
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
template <bool TRANS>
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], unsigned addr) {
    if constexpr (TRANS)
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                     : "r"(addr)
                     : "memory");
    else
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                     : "r"(addr)
                     : "memory");
}
// A fragment (16 x 16 at m0, k0) of a tile stored [m][k], or [k][m] (TRANS).
template <bool TRANS>
__device__ __forceinline__ void frag_a(uint32_t (&a)[4], const bf16 *tile, int m0, int k0) {
    const int lane = threadIdx.x & 31, r = lane & 7, mi = lane >> 3;
    if constexpr (TRANS)
        ldsm4<true>(a, tile_addr(tile, k0 + r + (mi >> 1) * 8, (m0 >> 3) + (mi & 1)));
    else
        ldsm4<false>(a, tile_addr(tile, m0 + r + (mi & 1) * 8, (k0 >> 3) + (mi >> 1)));
}
// B fragments of two neighbouring 8-column tiles (b[0..1] at n0, b[2..3] at
// n0 + 8) of a tile stored [n][k], or [k][n] (TRANS).
template <bool TRANS>
__device__ __forceinline__ void frag_b2(uint32_t (&b)[4], const bf16 *tile, int n0, int k0) {
    const int lane = threadIdx.x & 31, r = lane & 7, mi = lane >> 3;
    if constexpr (TRANS)
        ldsm4<true>(b, tile_addr(tile, k0 + r + (mi & 1) * 8, (n0 >> 3) + (mi >> 1)));
    else
        ldsm4<false>(b, tile_addr(tile, n0 + r + (mi >> 1) * 8, (k0 >> 3) + (mi & 1)));
}
// One 64-wide k tile: four warps in a 2 x 2 grid, each MT x 4 mma tiles.
template <int MT, bool TA, bool TB>
__device__ __forceinline__ void tile_mma(float (&acc)[MT][4][4], const bf16 *As, const bf16 *Bs) {
    const int warp = threadIdx.x >> 5, wm = (warp >> 1) * MT * 16, wn = (warp & 1) * 32;
#pragma unroll
    for (int kk = 0; kk < kBK; kk += 16) {
        uint32_t a[MT][4], b[2][4];
#pragma unroll
        for (int mi = 0; mi < MT; ++mi) frag_a<TA>(a[mi], As, wm + mi * 16, kk);
#pragma unroll
        for (int p = 0; p < 2; ++p) frag_b2<TB>(b[p], Bs, wn + p * 16, kk);
#pragma unroll
        for (int mi = 0; mi < MT; ++mi)
#pragma unroll
            for (int ni = 0; ni < 4; ++ni) mma_bf16(acc[mi][ni], a[mi], &b[ni >> 1][(ni & 1) * 2]);
    }
}

// ---------------------------------------------------------------- layers
enum { LAYER_IN, LAYER_HIDDEN, LAYER_OUT, LAYER_GRAD };

struct LayerArgs {
    int M, N, K;          // batch rows, output columns, inner size
    const float *x;       // LAYER_IN: the FP32 input, M x K
    bf16 *Xb;             // LAYER_IN: its BF16 copy (kMlpInPad columns), written for the weight gradient
    const bf16 *A;        // else: M x K activations (row stride lda)
    int lda;
    const bf16 *W;        // N x K weights; LAYER_GRAD: K x N
    int ldw;
    const float *bias;    // N
    float *C;             // M x N FP32: pre-activations, outputs or gradients (row stride N)
    bf16 *Cb;             // BF16 activations or gradients (row stride ldcb)
    int ldcb;
    const float *gz;      // LAYER_GRAD: pre-activations (row stride N)
    const float *target;  // LAYER_OUT: M x N, or NULL
    float *dY;            // LAYER_OUT with a target: 2 (y - target) / (M N)
    float scale;
    double *lossp;        // LAYER_OUT with a target: per block, sum of squares
};

// 32 rows x 64 columns of one layer.  Only the weights are read before the
// wait: they were written at least two launches ago.
template <int MODE>
__global__ void __launch_bounds__(128) layer_kernel(const LayerArgs g) {
    constexpr int BM = 32;
    constexpr bool NN = MODE == LAYER_GRAD;   // weights stored [k][n]
    __shared__ __align__(128) bf16 As[kStages][BM * kBK];
    __shared__ __align__(128) bf16 Bs[kStages][kBN * kBK];
    const int i0 = blockIdx.y * BM, j0 = blockIdx.x * kBN;
    const int kt_n = (g.K + kBK - 1) / kBK;
    const int kpad = (g.K + 7) & ~7, npad = (g.N + 7) & ~7;
    auto load_b = [&](int kt) {
        bf16 *t = Bs[kt % kStages];
        if constexpr (NN) tile_load<kBK>(t, g.W, g.ldw, kt * kBK, g.K, j0, npad);
        else tile_load<kBN>(t, g.W, g.ldw, j0, g.N, kt * kBK, MODE == LAYER_IN ? kMlpInPad : kpad);
    };
    auto load_a = [&](int kt) {
        bf16 *t = As[kt % kStages];
        if constexpr (MODE == LAYER_IN) {
            float v[BM * kBK / 128];   // every load in flight before the first store
#pragma unroll
            for (int p = 0; p < BM * kBK / 128; ++p) {
                const int e = p * 128 + threadIdx.x, i = i0 + e / kBK, k = kt * kBK + e % kBK;
                v[p] = i < g.M && k < g.K ? __ldca(g.x + (size_t)i * g.K + k) : 0.f;
            }
#pragma unroll
            for (int p = 0; p < BM * kBK / 128; ++p) {
                const int e = p * 128 + threadIdx.x, row = e / kBK, c = e % kBK, i = i0 + row;
                const bf16 h = __float2bfloat16_rn(v[p]);
                t[row * kBK + (((c >> 3) ^ (row & 7)) << 3) + (c & 7)] = h;
                if (blockIdx.x == 0 && g.Xb && i < g.M) g.Xb[(size_t)i * kMlpInPad + kt * kBK + c] = h;
            }
        } else {
            tile_load<BM>(t, g.A, g.lda, i0, g.M, kt * kBK, kpad);
        }
    };
    if constexpr (MODE == LAYER_IN) grid_dep_wait();   // the weights may come from the launch before this one
    for (int kt = 0; kt < kt_n && kt < kStages; ++kt) load_b(kt);
    if constexpr (MODE != LAYER_IN) grid_dep_wait();
    grid_dep_release();   // after the wait: a launch that starts now finds everything before this one complete
    for (int kt = 0; kt < kStages; ++kt) {
        if (kt < kt_n) load_a(kt);
        cp_commit();
    }
    float acc[1][4][4] = {};
    for (int kt = 0; kt < kt_n; ++kt) {
        cp_wait<kStages - 1>();
        __syncthreads();
        tile_mma<1, false, NN>(acc, As[kt % kStages], Bs[kt % kStages]);
        if (kt + kStages < kt_n) {
            __syncthreads();
            load_a(kt + kStages);
            load_b(kt + kStages);
        }
        cp_commit();
    }

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gid = lane >> 2, t4 = lane & 3;
    double sq = 0.0;
#pragma unroll
    for (int ni = 0; ni < 4; ++ni)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = i0 + (warp >> 1) * 16 + gid + 8 * (q >> 1), j = j0 + (warp & 1) * 32 + ni * 8 + 2 * t4 + (q & 1);
            if (i >= g.M || j >= g.N) continue;
            float v = acc[0][ni][q];
            const size_t c = (size_t)i * g.N + j;
            if constexpr (MODE == LAYER_GRAD) {
                v = v * gelu_grad_f(g.gz[c]);
                g.C[c] = v;
                g.Cb[(size_t)i * g.ldcb + j] = __float2bfloat16_rn(v);
            } else {
                v += g.bias[j];
                g.C[c] = v;
                if constexpr (MODE == LAYER_OUT) {
                    if (g.target) {
                        const float d = v - g.target[c], gv = d * g.scale;
                        sq += (double)d * (double)d;
                        g.dY[c] = gv;
                        g.Cb[(size_t)i * g.ldcb + j] = __float2bfloat16_rn(gv);
                    }
                } else {
                    g.Cb[(size_t)i * g.ldcb + j] = __float2bfloat16_rn(gelu_f(v));
                }
            }
        }
    if constexpr (MODE == LAYER_OUT) {
        if (!g.target) return;
        __syncthreads();
        double *s_sq = reinterpret_cast<double *>(As[0]);   // the tiles are consumed
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
        if (lane == 0) s_sq[warp] = sq;
        __syncthreads();
        if (threadIdx.x == 0) g.lossp[blockIdx.y * gridDim.x + blockIdx.x] = ((s_sq[0] + s_sq[1]) + s_sq[2]) + s_sq[3];
    }
}

// ---------------------------------------------------------------- parameter gradients
// Weight gradients G[i][j] = sum_b D[b][i] H[b][j] (M x N, K = the batch) in
// S slices of kchunk rows each: block (tile, slice) leaves its partial tile in
// P[slice]; bias gradients sum_b F[b][j] in kColSlices slices (slice s adds rows
// s, s + kColSlices, ...).  All layers' blocks run in one launch.
constexpr int kColSlices = 32;
struct GradArgs {
    const bf16 *D, *H;   // B x M (row stride ldd), B x N (row stride ldh)
    int ldd, ldh, M, N, S, kchunk;
    float *P;            // S x M x N
    const float *F;      // B x M: FP32 gradient of the layer's output
    float *Q;            // kColSlices x M
    int gemm_blocks, blocks;   // blocks of this layer: GEMM blocks first
};
struct GradSet {
    GradArgs l[3];
    int B;
};

__global__ void __launch_bounds__(128) grad_kernel(const GradSet gs) {
    constexpr int BM = 64;
    __shared__ __align__(128) bf16 As[2][BM * kBK];
    __shared__ __align__(128) bf16 Bs[2][kBN * kBK];
    int b = blockIdx.x, li = 0;
    while (li < 2 && b >= gs.l[li].blocks) b -= gs.l[li++].blocks;
    const GradArgs &g = gs.l[li];
    grid_dep_wait();
    grid_dep_release();
    if (b >= g.gemm_blocks) {   // bias: one thread per column
        b -= g.gemm_blocks;
        const int tiles = (g.M + 127) / 128, sl = b / tiles, j = (b - sl * tiles) * 128 + threadIdx.x;
        if (j >= g.M) return;
        float a = 0.f;
#pragma unroll 8
        for (int r = sl; r < gs.B; r += kColSlices) a += g.F[(size_t)r * g.M + j];
        g.Q[(size_t)sl * g.M + j] = a;
        return;
    }
    const int nt = (g.N + kBN - 1) / kBN, mt = (g.M + BM - 1) / BM;
    const int z = b / (nt * mt), t = b - z * nt * mt, i0 = (t / nt) * BM, j0 = (t % nt) * kBN;
    const int kb = z * g.kchunk, ke = min(gs.B, kb + g.kchunk);
    const int kt_n = ke > kb ? (ke - kb + kBK - 1) / kBK : 0;
    auto load = [&](int kt) {   // rows of the batch are k
        tile_load<kBK>(As[kt & 1], g.D, g.ldd, kb + kt * kBK, ke, i0, (g.M + 7) & ~7);
        tile_load<kBK>(Bs[kt & 1], g.H, g.ldh, kb + kt * kBK, ke, j0, (g.N + 7) & ~7);
    };
    for (int kt = 0; kt < 2; ++kt) {
        if (kt < kt_n) load(kt);
        cp_commit();
    }
    float acc[2][4][4] = {};
    for (int kt = 0; kt < kt_n; ++kt) {
        cp_wait<1>();
        __syncthreads();
        tile_mma<2, true, true>(acc, As[kt & 1], Bs[kt & 1]);
        if (kt + 2 < kt_n) {
            __syncthreads();
            load(kt + 2);
        }
        cp_commit();
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gid = lane >> 2, t4 = lane & 3;
    float *P = g.P + (size_t)z * g.M * g.N;
#pragma unroll
    for (int mi = 0; mi < 2; ++mi)
#pragma unroll
        for (int ni = 0; ni < 4; ++ni)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int i = i0 + (warp >> 1) * 32 + mi * 16 + gid + 8 * (q >> 1);
                const int j = j0 + (warp & 1) * 32 + ni * 8 + 2 * t4 + (q & 1);
                if (i < g.M && j < g.N) P[(size_t)i * g.N + j] = acc[mi][ni][q];
            }
}

// ---------------------------------------------------------------- finish
struct FinishArgs {
    const float *P[3], *Q[3];   // partial weight and bias gradients per layer
    int M[3], N[3], S[3];
    bf16 *Wb[3];                // BF16 weight copies (row stride ldw)
    int ldw[3];
    float *grads;               // packed gradients out, or NULL
    float *w, *m, *v;           // packed parameters and moments (stepped when adam)
    int adam;
    float lr, b1, b2, eps, c1, c2;
    const double *lossp;
    int n_lossp;
    double inv_n;
    float *loss;                // or NULL
    long long n;
};

// The packed gradient (slices added in order), Adam (Kingma & Ba) on the FP32
// parameters (c1 = 1 - beta1^t, c2 = 1 - beta2^t), the BF16 copy of every
// stepped weight, and the mean squared error.
__global__ void __launch_bounds__(256) finish_kernel(const FinishArgs g) {
    grid_dep_wait();
    grid_dep_release();
    const long long e = blockIdx.x * 256ll + threadIdx.x;
    if (e < g.n) {
        long long r = e;
        int li = 0;
        while (li < 2 && r >= (long long)g.M[li] * g.N[li] + g.M[li]) {
            r -= (long long)g.M[li] * g.N[li] + g.M[li];
            ++li;
        }
        const long long nw = (long long)g.M[li] * g.N[li];
        float gk = 0.f;
        if (r < nw) {
#pragma unroll 8
            for (int z = 0; z < g.S[li]; ++z) gk += g.P[li][z * nw + r];
        } else {
#pragma unroll 8
            for (int sl = 0; sl < kColSlices; ++sl) gk += g.Q[li][(long long)sl * g.M[li] + (r - nw)];
        }
        if (g.grads) g.grads[e] = gk;
        if (g.adam) {
            const float mk = fmaf(1.f - g.b1, gk, g.b1 * g.m[e]);   // one rounding order, whatever the compiler fuses
            const float vk = fmaf((1.f - g.b2) * gk, gk, g.b2 * g.v[e]);
            g.m[e] = mk;
            g.v[e] = vk;
            const float w = g.w[e] - g.lr * (mk / g.c1) / (sqrtf(vk / g.c2) + g.eps);
            g.w[e] = w;
            if (r < nw) {
                const int row = (int)(r / g.N[li]), col = (int)(r - (long long)row * g.N[li]);
                g.Wb[li][(size_t)row * g.ldw[li] + col] = __float2bfloat16_rn(w);
            }
        }
    }
    if (blockIdx.x == 0 && g.loss) {
        __shared__ double s[8];
        double a = 0.0;
        for (int k = threadIdx.x; k < g.n_lossp; k += 256) a += g.lossp[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = a;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int k = 0; k < 8; ++k) t += s[k];
            *g.loss = (float)(t * g.inv_n);
        }
    }
}

// BF16 copy of a row-major FP32 matrix (rows x cols) into a row stride `ld`
// (columns cols..ld-1 are zero).
__global__ void to_bf16_kernel(const float *__restrict__ W, int rows, int cols, int ld, bf16 *__restrict__ Wb) {
    const long long n = (long long)rows * ld;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const int r = (int)(e / ld), c = (int)(e - (long long)r * ld);
        Wb[e] = __float2bfloat16_rn(c < cols ? W[(long long)r * cols + c] : 0.f);
    }
}

}  // namespace exact

using namespace exact;

struct exact_mlp {
    int din = 0, H = 0, O = 0, maxB = 0, Hp = 0, Op = 0;   // Hp, Op: BF16 row strides (multiples of 8)
    long long nparam = 0;
    long long oW1, ob1, oW2, ob2, oW3, ob3;   // offsets into the packed parameter vector
    void *dev = nullptr;
    float *w, *m, *v;                         // packed FP32 parameters and moments
    bf16 *W1b, *W2b, *W3b;                    // BF16 weights (W1b rows padded to 128)
    bf16 *Xb, *H1b, *H2b, *dYb, *dZ1b, *dZ2b; // BF16 operands (padding columns stay zero)
    float *Z1, *Z2, *Y, *dY, *dZ1, *dZ2;      // FP32 activations / gradients
    float *P[3], *Q[3];                       // partial weight and bias gradients
    double *lossp;                            // partial losses
    int t = 0;                                // Adam step
};

// Slices of a weight gradient over the batch: enough that its 64 x 64 tiles
// fill the GPU, at least 64 rows each.  (Part of the result: the slices are
// summed in order.)
constexpr int kSplitMax = 16;
static int splits_for(int M, int N, long long K) {
    const int tiles = ((M + 63) / 64) * ((N + 63) / 64);
    int s = 1;
    while (s < kSplitMax && tiles * s * 2 <= 152 && K / (s * 2) >= 64) s *= 2;
    return s;
}
static int chunk_for(int S, int K) { return S > 1 ? ((K + S - 1) / S + 31) / 32 * 32 : K; }

static int grid_for(long long n, int block) {
    long long g = (n + block - 1) / block;
    return (int)(g < 1 ? 1 : (g > 65535 ? 65535 : g));
}

static int refresh_bf16(exact_mlp *m, cudaStream_t st) {
    to_bf16_kernel<<<grid_for((long long)m->H * kMlpInPad, 256), 256, 0, st>>>(m->w + m->oW1, m->H, m->din, kMlpInPad, m->W1b);
    to_bf16_kernel<<<grid_for((long long)m->H * m->Hp, 256), 256, 0, st>>>(m->w + m->oW2, m->H, m->H, m->Hp, m->W2b);
    to_bf16_kernel<<<grid_for((long long)m->O * m->Hp, 256), 256, 0, st>>>(m->w + m->oW3, m->O, m->H, m->Hp, m->W3b);
    return cuda_status(cudaGetLastError());
}

template <int MODE>
static cudaError_t layer(const LayerArgs &g, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((g.N + kBN - 1) / kBN, (g.M + 31) / 32);
    cfg.blockDim = dim3(128);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, layer_kernel<MODE>, g);
}

// forward: x -> Z1, H1b -> Z2, H2b -> y; with a target also dY, dYb and the
// partial losses
static int forward(exact_mlp *m, const float *x, int B, float *y, const float *target, cudaStream_t st) {
    const int H = m->H, O = m->O;
    LayerArgs a;
    memset(&a, 0, sizeof a);
    a.M = B; a.N = H; a.K = m->din; a.x = x; a.Xb = target ? m->Xb : nullptr; a.W = m->W1b; a.ldw = kMlpInPad;
    a.bias = m->w + m->ob1; a.C = m->Z1; a.Cb = m->H1b; a.ldcb = m->Hp;
    LayerArgs b;
    memset(&b, 0, sizeof b);
    b.M = B; b.N = H; b.K = H; b.A = m->H1b; b.lda = m->Hp; b.W = m->W2b; b.ldw = m->Hp;
    b.bias = m->w + m->ob2; b.C = m->Z2; b.Cb = m->H2b; b.ldcb = m->Hp;
    LayerArgs c;
    memset(&c, 0, sizeof c);
    c.M = B; c.N = O; c.K = H; c.A = m->H2b; c.lda = m->Hp; c.W = m->W3b; c.ldw = m->Hp;
    c.bias = m->w + m->ob3; c.C = y; c.Cb = m->dYb; c.ldcb = m->Op;
    c.target = target; c.dY = m->dY; c.scale = 2.f / (float)((long long)B * O); c.lossp = m->lossp;
    if (layer<LAYER_IN>(a, st) != cudaSuccess || layer<LAYER_HIDDEN>(b, st) != cudaSuccess ||
        layer<LAYER_OUT>(c, st) != cudaSuccess)
        return EXACT_ECUDA;
    return EXACT_OK;
}

// Loss and gradients of one batch; grads / loss may be NULL; adam: step the
// parameters with learning rate lr (step m->t).
static int backward(exact_mlp *m, const float *x, const float *target, int B, float *grads, float *loss, bool adam,
                    float lr, cudaStream_t st) {
    int rc = forward(m, x, B, m->Y, target, st);
    if (rc != EXACT_OK) return rc;
    const int H = m->H, O = m->O, D = m->din;
    // dZ2 = (dY W3) g'(Z2), dZ1 = (dZ2 W2) g'(Z1)
    LayerArgs a;
    memset(&a, 0, sizeof a);
    a.M = B; a.N = H; a.K = O; a.A = m->dYb; a.lda = m->Op; a.W = m->W3b; a.ldw = m->Hp;
    a.C = m->dZ2; a.Cb = m->dZ2b; a.ldcb = m->Hp; a.gz = m->Z2;
    LayerArgs b = a;
    b.K = H; b.A = m->dZ2b; b.lda = m->Hp; b.W = m->W2b; b.C = m->dZ1; b.Cb = m->dZ1b; b.gz = m->Z1;
    if (layer<LAYER_GRAD>(a, st) != cudaSuccess || layer<LAYER_GRAD>(b, st) != cudaSuccess) return EXACT_ECUDA;
    GradSet gs;
    memset(&gs, 0, sizeof gs);
    gs.B = B;
    const bf16 *Ds[3] = {m->dZ1b, m->dZ2b, m->dYb}, *Hs[3] = {m->Xb, m->H1b, m->H2b};
    const float *Fs[3] = {m->dZ1, m->dZ2, m->dY};
    const int ldd[3] = {m->Hp, m->Hp, m->Op}, ldh[3] = {kMlpInPad, m->Hp, m->Hp}, Ms[3] = {H, H, O}, Ns[3] = {D, H, H};
    FinishArgs f;
    memset(&f, 0, sizeof f);
    bf16 *Wb[3] = {m->W1b, m->W2b, m->W3b};
    int blocks = 0;
    for (int k = 0; k < 3; ++k) {
        GradArgs &g = gs.l[k];
        g.D = Ds[k]; g.H = Hs[k]; g.ldd = ldd[k]; g.ldh = ldh[k]; g.M = Ms[k]; g.N = Ns[k];
        g.S = splits_for(g.M, g.N, B);
        g.kchunk = chunk_for(g.S, B);
        g.P = m->P[k]; g.F = Fs[k]; g.Q = m->Q[k];
        g.gemm_blocks = ((g.M + 63) / 64) * ((g.N + kBN - 1) / kBN) * g.S;
        g.blocks = g.gemm_blocks + ((g.M + 127) / 128) * kColSlices;
        blocks += g.blocks;
        f.P[k] = g.P; f.Q[k] = g.Q; f.M[k] = g.M; f.N[k] = g.N; f.S[k] = g.S;
        f.Wb[k] = Wb[k]; f.ldw[k] = ldh[k];
    }
    f.grads = grads; f.w = m->w; f.m = m->m; f.v = m->v; f.adam = adam ? 1 : 0;
    const double b1 = 0.9, b2 = 0.999;
    f.lr = lr; f.b1 = (float)b1; f.b2 = (float)b2; f.eps = 1e-8f;
    f.c1 = (float)(1.0 - pow(b1, m->t)); f.c2 = (float)(1.0 - pow(b2, m->t));
    f.lossp = m->lossp; f.n_lossp = ((O + kBN - 1) / kBN) * ((B + 31) / 32);
    f.inv_n = 1.0 / (double)((long long)B * O);
    f.loss = loss;
    f.n = m->nparam;
    if (launch_dependent(grad_kernel, (unsigned)blocks, 128u, 0, st, gs) != cudaSuccess ||
        launch_dependent(finish_kernel, (unsigned)((m->nparam + 255) / 256), 256u, 0, st, f) != cudaSuccess)
        return EXACT_ECUDA;
    return EXACT_OK;
}

extern "C" int exact_mlp_create(int d_in, int hidden, int d_out, int max_batch, exact_mlp **out) {
    if (!out) return EXACT_EINVAL;
    *out = nullptr;
    if (d_in < 1 || hidden < 1 || d_out < 1 || max_batch < 1) return EXACT_EINVAL;
    if (d_in > kMlpInPad || hidden > 1024 || d_out > 256 || max_batch > (1 << 20)) return EXACT_ECAPACITY;
    exact_mlp *m = new (std::nothrow) exact_mlp();
    if (!m) return EXACT_EINVAL;
    m->din = d_in; m->H = hidden; m->O = d_out; m->maxB = max_batch;
    const long long H = hidden, D = d_in, O = d_out, B = max_batch;
    m->oW1 = 0; m->ob1 = H * D; m->oW2 = m->ob1 + H; m->ob2 = m->oW2 + H * H; m->oW3 = m->ob2 + H;
    m->ob3 = m->oW3 + O * H;
    m->nparam = m->ob3 + O;
    m->Hp = (hidden + 7) & ~7;
    m->Op = (d_out + 7) & ~7;
    const long long Hp = m->Hp, Op = m->Op, most = 1ll << 40;
    std::vector<size_t> sz = {
        (size_t)m->nparam * 4, (size_t)m->nparam * 4, (size_t)m->nparam * 4,                            // w m v
        (size_t)(H * kMlpInPad) * 2, (size_t)(H * Hp) * 2, (size_t)(O * Hp) * 2,                        // W1b W2b W3b
        (size_t)(B * kMlpInPad) * 2, (size_t)(B * Hp) * 2, (size_t)(B * Hp) * 2, (size_t)(B * Op) * 2,   // Xb H1b H2b dYb
        (size_t)(B * Hp) * 2, (size_t)(B * Hp) * 2,                                                     // dZ1b dZ2b
        (size_t)(B * H) * 4, (size_t)(B * H) * 4, (size_t)(B * O) * 4, (size_t)(B * O) * 4,             // Z1 Z2 Y dY
        (size_t)(B * H) * 4, (size_t)(B * H) * 4,                                                       // dZ1 dZ2
        (size_t)splits_for(hidden, d_in, most) * H * D * 4, (size_t)splits_for(hidden, hidden, most) * H * H * 4,
        (size_t)splits_for(d_out, hidden, most) * O * H * 4,                                            // P
        (size_t)kColSlices * H * 4, (size_t)kColSlices * H * 4, (size_t)kColSlices * O * 4,             // Q
        (size_t)((O + kBN - 1) / kBN) * ((B + 31) / 32) * 8};                                           // lossp
    size_t total = 0;
    for (auto s : sz) total += align_up(s, 256);
    if (cudaMalloc(&m->dev, total) != cudaSuccess) { delete m; return EXACT_ECUDA; }
    if (cudaMemset(m->dev, 0, total) != cudaSuccess) { cudaFree(m->dev); delete m; return EXACT_ECUDA; }
    char *p = static_cast<char *>(m->dev);
    void **slots[] = {(void **)&m->w, (void **)&m->m, (void **)&m->v, (void **)&m->W1b, (void **)&m->W2b,
                      (void **)&m->W3b, (void **)&m->Xb, (void **)&m->H1b, (void **)&m->H2b, (void **)&m->dYb,
                      (void **)&m->dZ1b, (void **)&m->dZ2b, (void **)&m->Z1, (void **)&m->Z2, (void **)&m->Y,
                      (void **)&m->dY, (void **)&m->dZ1, (void **)&m->dZ2, (void **)&m->P[0], (void **)&m->P[1],
                      (void **)&m->P[2], (void **)&m->Q[0], (void **)&m->Q[1], (void **)&m->Q[2], (void **)&m->lossp};
    for (size_t i = 0; i < sz.size(); ++i) {
        *slots[i] = p;
        p += align_up(sz[i], 256);
    }
    *out = m;
    return EXACT_OK;
}

extern "C" void exact_mlp_destroy(exact_mlp *m) {
    if (!m) return;
    cudaDeviceSynchronize();
    cudaFree(m->dev);
    delete m;
}

extern "C" long long exact_mlp_num_params(const exact_mlp *m) { return m ? m->nparam : -1; }

extern "C" int exact_mlp_set_params(exact_mlp *m, const float *host_params) {
    if (!m || !host_params) return EXACT_EINVAL;
    for (long long k = 0; k < m->nparam; ++k)
        if (!isfinite(host_params[k])) return EXACT_EINVAL;
    if (cudaMemcpy(m->w, host_params, (size_t)m->nparam * 4, cudaMemcpyHostToDevice) != cudaSuccess) return EXACT_ECUDA;
    if (cudaMemset(m->m, 0, (size_t)m->nparam * 4) != cudaSuccess ||
        cudaMemset(m->v, 0, (size_t)m->nparam * 4) != cudaSuccess)
        return EXACT_ECUDA;
    m->t = 0;
    const int rc = refresh_bf16(m, 0);
    if (rc != EXACT_OK) return rc;
    return cuda_status(cudaDeviceSynchronize());
}

extern "C" int exact_mlp_get_params(const exact_mlp *m, float *host_params) {
    if (!m || !host_params) return EXACT_EINVAL;
    if (cudaDeviceSynchronize() != cudaSuccess) return EXACT_ECUDA;
    return cuda_status(cudaMemcpy(host_params, m->w, (size_t)m->nparam * 4, cudaMemcpyDeviceToHost));
}

extern "C" int exact_mlp_get_state(const exact_mlp *m, float *host_params, float *host_m, float *host_v,
                                   long long *step) {
    if (!m || !host_params || !host_m || !host_v || !step) return EXACT_EINVAL;
    if (cudaDeviceSynchronize() != cudaSuccess) return EXACT_ECUDA;
    const size_t bytes = (size_t)m->nparam * 4;
    if (cudaMemcpy(host_params, m->w, bytes, cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(host_m, m->m, bytes, cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(host_v, m->v, bytes, cudaMemcpyDeviceToHost) != cudaSuccess)
        return EXACT_ECUDA;
    *step = m->t;
    return EXACT_OK;
}

extern "C" int exact_mlp_set_state(exact_mlp *m, const float *host_params, const float *host_m, const float *host_v,
                                   long long step) {
    if (!m || !host_params || !host_m || !host_v || step < 0 || step > (1ll << 30)) return EXACT_EINVAL;
    for (long long k = 0; k < m->nparam; ++k)
        if (!isfinite(host_params[k]) || !isfinite(host_m[k]) || !(host_v[k] >= 0.f) || !isfinite(host_v[k]))
            return EXACT_EINVAL;
    const size_t bytes = (size_t)m->nparam * 4;
    if (cudaDeviceSynchronize() != cudaSuccess ||
        cudaMemcpy(m->w, host_params, bytes, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(m->m, host_m, bytes, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(m->v, host_v, bytes, cudaMemcpyHostToDevice) != cudaSuccess)
        return EXACT_ECUDA;
    m->t = (int)step;
    const int rc = refresh_bf16(m, 0);
    if (rc != EXACT_OK) return rc;
    return cuda_status(cudaDeviceSynchronize());
}

extern "C" int exact_mlp_forward(exact_mlp *m, const float *x, int B, float *y, void *stream) {
    if (!m || !x || !y || B < 0) return EXACT_EINVAL;
    if (B == 0) return EXACT_OK;
    if (B > m->maxB) return EXACT_ECAPACITY;
    return forward(m, x, B, y, nullptr, (cudaStream_t)stream);
}

extern "C" int exact_mlp_loss_grad(exact_mlp *m, const float *x, const float *target, int B, float *loss,
                                   float *grads, void *stream) {
    if (!m || !x || !target || B < 1) return EXACT_EINVAL;
    if (B > m->maxB) return EXACT_ECAPACITY;
    return backward(m, x, target, B, grads, loss, false, 0.f, (cudaStream_t)stream);
}

extern "C" int exact_mlp_train_step(exact_mlp *m, const float *x, const float *target, int B, float lr, float *loss,
                                    void *stream) {
    if (!m || !x || !target || B < 1 || !(lr > 0.f)) return EXACT_EINVAL;
    if (B > m->maxB) return EXACT_ECAPACITY;
    m->t += 1;
    const int rc = backward(m, x, target, B, nullptr, loss, true, lr, (cudaStream_t)stream);
    if (rc != EXACT_OK) m->t -= 1;
    return rc;
}
