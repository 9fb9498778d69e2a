// Learned parametric embedder (a project addition; the paper embeds each data
// set by plain optimisation): an MLP d -> 256 -> 256 -> 2 with exact-erf GELU,
// BF16 weights and activations, FP32 accumulation and FP32 master weights,
// trained with Adam on the UMAP cross-entropy over edges of the method's own
// fuzzy graph, then used to embed new points.
//
// Every dense product runs on the tcgen05 tensor cores with BF16 operands (TMA,
// 128-byte swizzle) and FP32 accumulation in TMEM: mlp_layer_kernel with a fused
// epilogue (bias + GELU forward, the GELU derivative backward), mlp_gemm_kernel
// for the weight gradients (plain FP32, split over K).  The weight gradients sum over the batch's rows: they take the
// activations as they lie, MN-major (with transposed copies for K-major
// operands, written by two GEMM epilogues, the layer 3 kernel and the gather, a
// step of 4096 edges took 136 us against 125).  The 256 -> 2 layer, the loss,
// the reductions and Adam are small SIMT kernels.
//
// One training step (batch of B edges, each with `neg` negatives, R = 2 + neg
// rows per edge, M = B R rows):
//   sample     edges proportional to w (integer rejection on q) + negatives
//   gather     X rows -> Xb (M x 64), BF16
//              (both for the next step, beside this step's backward pass)
//   F1, F2     pre_l = H_{l-1} W_l^T + b_l ; H_l = GELU(pre_l)  (BF16) ;
//              GELU'(pre_l) (FP32, blocked)
//   head       z = H2 W3^T + b3, loss and dL/dz per edge
//   L3 back    dpre2 = (dz W3) . GELU'(pre2) ; db2 partial sums
//   dW3, dW2   dW3, db3 partial sums ; dpre2^T H1 (split-K, FP32 partials), on a
//              branch of their own
//   dH1        dpre1 = (dpre2 W2) . GELU'(pre1)
//   dW1        dpre1^T Xb     (split-K) ; db1 partial sums
//   update     gradient (fixed summation order), Adam, BF16 copies
//
// Sums over the batch run in a fixed order: over the rows of chunks of 512 in
// order, then over the chunks (or K splits) in order.
#include <cuda_bf16.h>

#include <cmath>
#include <cstring>
#include <functional>
#include <vector>

#include "common.cuh"
#include "gemm.cuh"
#include "tc_ptx.cuh"

namespace drgb {

// ------------------------------------------------------------------ layout
static constexpr int MLP_IN = 64;   // padded input width (d <= 64)
static constexpr int MLP_H = 256;
static constexpr int MLP_OUT = 2;
static constexpr int64_t OFF_W1 = 0;
static constexpr int64_t OFF_B1 = OFF_W1 + MLP_H * MLP_IN;
static constexpr int64_t OFF_W2 = OFF_B1 + MLP_H;
static constexpr int64_t OFF_B2 = OFF_W2 + MLP_H * MLP_H;
static constexpr int64_t OFF_W3 = OFF_B2 + MLP_H;
static constexpr int64_t OFF_B3 = OFF_W3 + MLP_OUT * MLP_H;
static constexpr int64_t MLP_P = OFF_B3 + MLP_OUT;

typedef __nv_bfloat16 bf16;

// ------------------------------------------------------------------ GELU
__device__ __forceinline__ float gelu(float x) { return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float x) {
    return 0.5f * (1.0f + erff(x * 0.70710678118654752f)) + x * 0.39894228040143268f * expf(-0.5f * x * x);
}

// ------------------------------------------------------------------ tensor-core GEMM
static constexpr int G_BM = 128;
// 128 x 128 (or 64) tiles of C, split over K, two CTAs per SM.
static constexpr int G_EPI_WARPS = 8;  // two per TMEM lane quarter, one per column half
static constexpr int G_THREADS = 64 + G_EPI_WARPS * 32;  // warp 0 TMA, warp 1 MMA

// Blocked FP32 layout of an M x N matrix that only epilogues (and kernels of
// the same tiling) exchange: 128 x 32 blocks, within a block float4 columns of
// 128 rows, so that a warp's accesses are 512 contiguous bytes.
__host__ __device__ __forceinline__ int64_t blocked_at(int64_t row, int col, int N) {
    return ((row >> 7) * (N >> 5) + (col >> 5)) * 4096 + (int64_t((col & 31) >> 2) * 128 + (row & 127)) * 4 + (col & 3);
}

struct GemmArgs {
    int M, N, K;          // M, N multiples of 128 / BN; K multiple of 64
    int kb_per_split;     // 64-wide K blocks per split (grid z)
    float* out_f32;       // [splits][M][N]
    int f16;              // FP16 operands, else BF16
    int* status;
};

template <int BN>
struct GemmSmem {
    static constexpr int STAGES = BN == 128 ? 3 : 4;
    static constexpr int A_BYTES = G_BM * 64 * 2;
    static constexpr int B_BYTES = BN * 64 * 2;
    static constexpr size_t TOTAL = 1024 + size_t(STAGES) * (A_BYTES + B_BYTES) + 256;
};
static constexpr int G_PITCH = 36;  // floats per row of a warp's 32 x 32 transposing tile (16-byte rows)

// With KROWS the operands are stored K rows x M (N) columns, as activations of a
// batch are for a product over its rows, and staged as boxes of 64 x 64.
template <int BN, bool KROWS>
__global__ void __launch_bounds__(G_THREADS, 2)
mlp_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, GemmArgs G) {
    using SM = GemmSmem<BN>;
    constexpr int STAGES = SM::STAGES;
    constexpr int BOX = 64 * 64 * 2;
    static_assert(STAGES * (SM::A_BYTES + SM::B_BYTES) >= G_EPI_WARPS * 32 * G_PITCH * 4, "epilogue tiles fit the ring");
    extern __shared__ uint8_t smem_raw[];
    // 1024-byte aligned (swizzled operand tiles); an offset from the shared
    // array, so that every pointer below stays a known shared-memory address
    uint8_t* base = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    uint8_t* sA = base;
    uint8_t* sB = base + STAGES * SM::A_BYTES;
    uint64_t* bars = reinterpret_cast<uint64_t*>(sB + STAGES * SM::B_BYTES);
    uint64_t* full = bars;
    uint64_t* empty = bars + STAGES;
    uint64_t* acc_full = bars + 2 * STAGES;
    uint64_t* mma_done = acc_full + 1;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mma_done + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = blockIdx.x * G_BM, n0 = blockIdx.y * BN;
    const int kb0 = blockIdx.z * G.kb_per_split;
    int nkb = G.K / 64 - kb0;
    if (nkb > G.kb_per_split) nkb = G.kb_per_split;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(acc_full, 1);
        mbar_init(mma_done, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_slot)), "r"(BN) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    dep_enter();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            int kb = 0;
            for (; kb < nkb; ++kb) {
                const int s = kb % STAGES;
                if (kb >= STAGES && !mbar_wait(&empty[s], ((kb / STAGES) & 1) ^ 1, abort_flag, G.status)) break;
                mbar_expect_tx(&full[s], SM::A_BYTES + SM::B_BYTES);
                if (KROWS) {
#pragma unroll
                    for (int j = 0; j < G_BM / 64; ++j)
                        tma_load_2d(sA + s * SM::A_BYTES + j * BOX, &tmA, m0 + 64 * j, (kb0 + kb) * 64, &full[s]);
#pragma unroll
                    for (int j = 0; j < BN / 64; ++j)
                        tma_load_2d(sB + s * SM::B_BYTES + j * BOX, &tmB, n0 + 64 * j, (kb0 + kb) * 64, &full[s]);
                } else {
                    tma_load_2d(sA + s * SM::A_BYTES, &tmA, (kb0 + kb) * 64, m0, &full[s]);
                    tma_load_2d(sB + s * SM::B_BYTES, &tmB, (kb0 + kb) * 64, n0, &full[s]);
                }
            }
            if (kb < nkb) {  // aborted: let issued loads land before exit
                for (int u = (kb > STAGES ? kb - STAGES : 0); u < kb; ++u) {
                    const unsigned long long t0 = global_timer();
                    while (!mbar_try(&full[u % STAGES], (u / STAGES) & 1) && global_timer() - t0 < 100000000ull) {
                    }
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc = idesc_f16kind(G_BM, BN, G.f16 != 0) | (KROWS ? IDESC_MN_MAJOR : 0u);
            constexpr int KSTEP = KROWS ? 2048 / 16 : 32 / 16;  // 16 of K, in descriptor units
            for (int kb = 0; kb < nkb; ++kb) {
                const int s = kb % STAGES;
                if (!mbar_wait(&full[s], (kb / STAGES) & 1, abort_flag, G.status)) break;
                tc_fence_after();
                const uint32_t pa = smem_u32(sA + s * SM::A_BYTES), pb = smem_u32(sB + s * SM::B_BYTES);
                const uint64_t ad = KROWS ? sdesc_sw128_mn(pa, BOX) : sdesc_sw128(pa);
                const uint64_t bd = KROWS ? sdesc_sw128_mn(pb, BOX) : sdesc_sw128(pb);
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    mma_f16kind(tmem, ad + KSTEP * k, bd + KSTEP * k, idesc, (kb > 0 || k > 0) ? 1u : 0u);
                mma_commit(&empty[s]);
            }
            mma_commit(acc_full);
            mma_commit(mma_done);
            const unsigned long long t0 = global_timer();
            while (!mbar_try(mma_done, 0) && global_timer() - t0 < 100000000ull) {
            }
        }
    } else {
        const int quarter = warp & 3, half = (warp - 2) >> 2;
        // once the accumulator is complete the operand ring is free: each warp
        // transposes its 32 x 32 pieces through its own part of it
        float* tile = reinterpret_cast<float*>(base) + (warp - 2) * 32 * G_PITCH;
        const bool ok = mbar_wait(acc_full, 0, abort_flag, G.status) && nkb > 0;
        tc_fence_after();
        if (ok) {
#pragma unroll 1
            for (int c = half * (BN / 64); c < (half + 1) * (BN / 64); ++c) {
                float v[32];
                __syncwarp();
                tmem_ld32(tmem + (uint32_t(quarter * 32) << 16) + uint32_t(c * 32), v);
                const int gc0 = n0 + c * 32;
#pragma unroll
                for (int i = 0; i < 32; i += 4)
                    *reinterpret_cast<float4*>(tile + lane * G_PITCH + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
                __syncwarp();
                float* o = G.out_f32 + (int64_t(blockIdx.z) * G.M + m0 + quarter * 32) * G.N + gc0;
#pragma unroll
                for (int it = 0; it < 8; ++it) {  // four rows of 128 bytes an instruction
                    const int r = it * 4 + (lane >> 3), i = 4 * (lane & 7);
                    *reinterpret_cast<float4*>(o + int64_t(r) * G.N + i) =
                        *reinterpret_cast<const float4*>(tile + r * G_PITCH + i);
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(BN) : "memory");
    }
}

struct Gemm {
    CUtensorMap a, b;
    GemmArgs g;
    dim3 grid;
    int bn;
    bool krows;
};

// C[M x N] = A[M x K] B[N x K]^T with A, B row-major BF16 (K contiguous), or
// with `krows` A[K x M]^T B[K x N].
static int gemm_setup(Ctx* c, Gemm& G, const bf16* A, const bf16* B, int M, int N, int K, int bn,
                      int splits, bool krows, bool f16 = false) {
    if (M % G_BM || N % bn || K % 64 || splits < 1)
        return set_error(c, DRGB_ERR_INVALID, "mlp gemm: bad shape %d x %d x %d", M, N, K);
    int rc;
    if (krows) {
        if ((rc = make_map_k64(c, &G.a, A, K, M, 64, false)) || (rc = make_map_k64(c, &G.b, B, K, N, 64, false))) return rc;
    } else {
        if ((rc = make_map_k64(c, &G.a, A, M, K, G_BM, f16)) || (rc = make_map_k64(c, &G.b, B, N, K, bn, f16))) return rc;
    }
    std::memset(&G.g, 0, sizeof(G.g));
    G.g.M = M;
    G.g.N = N;
    G.g.K = K;
    G.g.f16 = f16;
    const int kbs = K / 64;
    G.g.kb_per_split = (kbs + splits - 1) / splits;
    G.g.status = c->d_status;
    G.grid = dim3(M / G_BM, N / bn, (kbs + G.g.kb_per_split - 1) / G.g.kb_per_split);
    G.bn = bn;
    G.krows = krows;
    return DRGB_OK;
}

template <int BN, bool KROWS>
static int gemm_attr(Ctx* c) {
    DRGB_CUDA(c, cudaFuncSetAttribute(mlp_gemm_kernel<BN, KROWS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      int(GemmSmem<BN>::TOTAL)));
    return DRGB_OK;
}

static int gemm_launch(Ctx* c, const Gemm& G, bool dep, cudaStream_t st) {
    auto go = [&](auto kernel, size_t smem) { return launch_dep(c, kernel, G.grid, G_THREADS, smem, dep, st, G.a, G.b, G.g); };
    if (G.bn == 128) return go(G.krows ? mlp_gemm_kernel<128, true> : mlp_gemm_kernel<128, false>, GemmSmem<128>::TOTAL);
    if (G.bn == 64 && G.krows) return go(mlp_gemm_kernel<64, true>, GemmSmem<64>::TOTAL);
    return set_error(c, DRGB_ERR_INVALID, "mlp gemm: unsupported tile");
}

// The plain product for other users of the library (the PCA covariance):
// partials[z][M][N] = A[M x K] B[N x K]^T over the z-th share of K.
int tc_gemm_nt_f32(Ctx* c, const void* A, const void* B, int M, int N, int K, int splits, float* partials,
                   int* splits_used, cudaStream_t st, bool f16) {
    Gemm G;
    int rc = gemm_setup(c, G, static_cast<const bf16*>(A), static_cast<const bf16*>(B), M, N, K, 128, splits, false, f16);
    if (rc) return rc;
    G.g.out_f32 = partials;
    if ((rc = gemm_attr<128, false>(c))) return rc;
    if (splits_used) *splits_used = int(G.grid.z);
    return gemm_launch(c, G, false, st);
}

// ------------------------------------------------------------------ layers of a batch
// One layer of the training step over M rows, N = MLP_H: forward
// (pre = A B^T + bias; out = GELU(pre), dgelu = GELU'(pre)) or backward
// (d = (A B^T) . dgelu; out, out_f32 = d).  128 x 64 tiles in persistent CTAs, two
// per SM: the producer and MMA warps run up to two tiles ahead (the accumulator
// has two buffers) of eight epilogue warps, each on 32 x 32 of a tile.
//
// Bound: the epilogue (forward about 60 instructions an element for GELU and
// its derivative; backward the latency of its reads), so the split evens that
// out: 28,672 rows are 896 tiles on 304 CTAs, 2.95 rounds of them.  As 448 CTAs of
// 128 x 128 (1.47 rounds, each load, MMA and epilogue in turn) F1 took 27.1, F2
// 28.5 and dH1 21.3 us; a step went from 125 to 109 us.
static constexpr int LY_BN = 64, LY_STAGES = 3;
static constexpr int LY_A = G_BM * 64 * 2, LY_B = LY_BN * 64 * 2;
static constexpr int LY_TILE = 32 * G_PITCH * 4;  // a warp's transposing tile
static constexpr size_t LY_SMEM = 1024 + size_t(LY_STAGES) * (LY_A + LY_B) + G_EPI_WARPS * LY_TILE + MLP_H * 4 + 128;

struct LayerArgs {
    int M, K;             // multiples of 128 and 64
    const float* bias;    // forward: [MLP_H]
    float* dgelu;         // blocked: forward out, backward in
    bf16* out;            // [M][MLP_H]
    float* out_f32;       // backward: blocked
    int* status;
};

template <bool BACK>
__global__ void __launch_bounds__(G_THREADS, 2)
mlp_layer_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, LayerArgs G) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    uint8_t* sA = base;
    uint8_t* sB = base + LY_STAGES * LY_A;
    uint8_t* s_tile = sB + LY_STAGES * LY_B;
    float* s_bias = reinterpret_cast<float*>(s_tile + G_EPI_WARPS * LY_TILE);
    uint64_t* full = reinterpret_cast<uint64_t*>(s_bias + MLP_H);
    uint64_t* empty = full + LY_STAGES;
    uint64_t* acc_full = empty + LY_STAGES;  // [2]
    uint64_t* acc_free = acc_full + 2;       // [2]
    uint64_t* mma_done = acc_free + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mma_done + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    constexpr int NT = MLP_H / LY_BN;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int tiles = G.M / G_BM * NT, nkb = G.K / 64;
    const int mine = (tiles - int(blockIdx.x) + int(gridDim.x) - 1) / int(gridDim.x);  // tiles blockIdx.x, + gridDim.x, ...

    if (tid == 0) {
        for (int s = 0; s < LY_STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int u = 0; u < 2; ++u) {
            mbar_init(&acc_full[u], 1);
            mbar_init(&acc_free[u], G_EPI_WARPS);
        }
        mbar_init(mma_done, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_slot)), "r"(2 * LY_BN) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    dep_enter();
    if (!BACK)
        for (int t = tid; t < MLP_H; t += G_THREADS) s_bias[t] = G.bias[t];
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            int it = 0;
            bool ok = true;
            for (int i = 0; i < mine && ok; ++i) {
                const int t = int(blockIdx.x) + i * int(gridDim.x), m0 = t / NT * G_BM, n0 = t % NT * LY_BN;
                for (int kb = 0; kb < nkb; ++kb, ++it) {
                    const int s = it % LY_STAGES;
                    if (it >= LY_STAGES && !(ok = mbar_wait(&empty[s], ((it / LY_STAGES) & 1) ^ 1, abort_flag, G.status))) break;
                    mbar_expect_tx(&full[s], LY_A + LY_B);
                    tma_load_2d(sA + s * LY_A, &tmA, kb * 64, m0, &full[s]);
                    tma_load_2d(sB + s * LY_B, &tmB, kb * 64, n0, &full[s]);
                }
            }
            if (!ok) {  // aborted: let issued loads land before exit
                for (int u = (it > LY_STAGES ? it - LY_STAGES : 0); u < it; ++u) {
                    const unsigned long long t0 = global_timer();
                    while (!mbar_try(&full[u % LY_STAGES], (u / LY_STAGES) & 1) && global_timer() - t0 < 100000000ull) {
                    }
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc = idesc_f16kind(G_BM, LY_BN, false);
            int it = 0;
            bool ok = true;
            for (int i = 0; i < mine && ok; ++i) {
                const int u = i & 1;
                if (i >= 2 && !(ok = mbar_wait(&acc_free[u], ((i >> 1) & 1) ^ 1, abort_flag, G.status))) break;
                for (int kb = 0; kb < nkb; ++kb, ++it) {
                    const int s = it % LY_STAGES;
                    if (!(ok = mbar_wait(&full[s], (it / LY_STAGES) & 1, abort_flag, G.status))) break;
                    tc_fence_after();
                    const uint64_t ad = sdesc_sw128(smem_u32(sA + s * LY_A)), bd = sdesc_sw128(smem_u32(sB + s * LY_B));
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        mma_f16kind(tmem + u * LY_BN, ad + 2 * k, bd + 2 * k, idesc, (kb > 0 || k > 0) ? 1u : 0u);
                    mma_commit(&empty[s]);
                }
                if (ok) mma_commit(&acc_full[u]);
            }
            mma_commit(mma_done);  // every MMA issued above has completed once this fires
            const unsigned long long t0 = global_timer();
            while (!mbar_try(mma_done, 0) && global_timer() - t0 < 100000000ull) {
            }
        }
    } else {
        const int quarter = warp & 3, half = (warp - 2) >> 2;
        float* tile = reinterpret_cast<float*>(s_tile + (warp - 2) * LY_TILE);
        auto at = [&](int i, int& m0, int& c0) {
            const int t = int(blockIdx.x) + i * int(gridDim.x);
            m0 = t / NT * G_BM + quarter * 32;
            c0 = t % NT * LY_BN + half * 32;
        };
        float x[32];  // backward: GELU' of the tile to come
        auto load_x = [&](int i) {
            if (!BACK || i >= mine) return;
            int m0, c0;
            at(i, m0, c0);
            const float* p = G.dgelu + blocked_at(m0 + lane, c0, MLP_H);
#pragma unroll
            for (int j = 0; j < 32; j += 4) {
                const float4 f = *reinterpret_cast<const float4*>(p + j * 128);
                x[j] = f.x;
                x[j + 1] = f.y;
                x[j + 2] = f.z;
                x[j + 3] = f.w;
            }
        };
        load_x(0);
        for (int i = 0; i < mine; ++i) {
            const int u = i & 1;
            int m0, c0;
            at(i, m0, c0);
            if (!mbar_wait(&acc_full[u], (i >> 1) & 1, abort_flag, G.status)) break;
            tc_fence_after();
            float v[32];
            __syncwarp();
            tmem_ld32(tmem + (uint32_t(quarter * 32) << 16) + uint32_t(u * LY_BN + half * 32), v);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_free[u]);
            const int64_t bo = blocked_at(m0 + lane, c0, MLP_H);  // this lane's float4 column of the blocked matrices
            if (!BACK) {
                float* bl = G.dgelu + bo;
#pragma unroll
                for (int j = 0; j < 32; j += 4) {
                    const float4 b4 = *reinterpret_cast<const float4*>(s_bias + c0 + j);
                    v[j] += b4.x;
                    v[j + 1] += b4.y;
                    v[j + 2] += b4.z;
                    v[j + 3] += b4.w;
                    *reinterpret_cast<float4*>(bl + j * 128) =
                        make_float4(gelu_grad(v[j]), gelu_grad(v[j + 1]), gelu_grad(v[j + 2]), gelu_grad(v[j + 3]));
                    v[j] = gelu(v[j]);
                    v[j + 1] = gelu(v[j + 1]);
                    v[j + 2] = gelu(v[j + 2]);
                    v[j + 3] = gelu(v[j + 3]);
                }
            } else {
#pragma unroll
                for (int j = 0; j < 32; ++j) v[j] *= x[j];
                load_x(i + 1);
                float* bl = G.out_f32 + bo;
#pragma unroll
                for (int j = 0; j < 32; j += 4)
                    *reinterpret_cast<float4*>(bl + j * 128) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
            }
            uint32_t* wt = reinterpret_cast<uint32_t*>(tile);  // rows of 20 words: 16-byte reads and writes
            __syncwarp();
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                uint32_t packed[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const __nv_bfloat162 h2 = __floats2bfloat162_rn(v[8 * j + 2 * k], v[8 * j + 2 * k + 1]);
                    packed[k] = *reinterpret_cast<const uint32_t*>(&h2);
                }
                *reinterpret_cast<uint4*>(wt + lane * 20 + 4 * j) = make_uint4(packed[0], packed[1], packed[2], packed[3]);
            }
            __syncwarp();
            bf16* o = G.out + int64_t(m0) * MLP_H + c0;
#pragma unroll
            for (int j = 0; j < 4; ++j) {  // eight rows of 64 bytes an instruction
                const int r = j * 8 + (lane >> 2), k = lane & 3;
                *reinterpret_cast<uint4*>(o + int64_t(r) * MLP_H + 8 * k) = *reinterpret_cast<const uint4*>(wt + r * 20 + 4 * k);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * LY_BN) : "memory");
    }
}

struct Layer {
    CUtensorMap a, b;
    LayerArgs g;
};

static int layer_setup(Ctx* c, Layer& L, const bf16* A, const bf16* B, int M, int K) {
    int rc;
    if ((rc = make_map_k64(c, &L.a, A, M, K, G_BM, false)) || (rc = make_map_k64(c, &L.b, B, MLP_H, K, LY_BN, false))) return rc;
    std::memset(&L.g, 0, sizeof(L.g));
    L.g.M = M;
    L.g.K = K;
    L.g.status = c->d_status;
    return DRGB_OK;
}

template <bool BACK>
static int layer_launch(Ctx* c, const Layer& L, bool dep, cudaStream_t st) {
    const dim3 grid(grid_for(int64_t(L.g.M / G_BM) * (MLP_H / LY_BN), 1, 2 * c->num_sms));
    return launch_dep(c, mlp_layer_kernel<BACK>, grid, G_THREADS, LY_SMEM, dep, st, L.a, L.b, L.g);
}

// Opt the training kernels into their shared-memory sizes (before any capture).
static int gemm_prepare(Ctx* c) {
    int rc;
    if ((rc = gemm_attr<128, true>(c)) || (rc = gemm_attr<64, true>(c))) return rc;
    DRGB_CUDA(c, cudaFuncSetAttribute(mlp_layer_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(LY_SMEM)));
    DRGB_CUDA(c, cudaFuncSetAttribute(mlp_layer_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(LY_SMEM)));
    return DRGB_OK;
}

// ------------------------------------------------------------------ SIMT kernels
struct MlpWeights {          // BF16 working copies of the master weights
    bf16* W1b;               // [256][64]
    bf16* W2b;               // [256][256]  (out, in)
    bf16* W2tb;              // [256][256]  (in, out)
    float* W3f;              // [2][256]    BF16-rounded values in FP32
};

// Working copies of master weight p.
__device__ __forceinline__ void mlp_cast_one(float w, int64_t p, const MlpWeights& W) {
    if (p < OFF_B1) {
        W.W1b[p] = __float2bfloat16_rn(w);
    } else if (p >= OFF_W2 && p < OFF_B2) {
        const int t = int(p - OFF_W2), o = t / MLP_H, i = t % MLP_H;
        const bf16 v = __float2bfloat16_rn(w);
        W.W2b[t] = v;
        W.W2tb[i * MLP_H + o] = v;
    } else if (p >= OFF_W3 && p < OFF_B3) {
        W.W3f[p - OFF_W3] = __bfloat162float(__float2bfloat16_rn(w));
    }
}

__global__ void mlp_cast_kernel(const float* __restrict__ P, MlpWeights W) {
    for (int64_t p = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; p < MLP_P; p += int64_t(gridDim.x) * blockDim.x)
        mlp_cast_one(P[p], p, W);
}

// Edge sampling proportional to w: try uniform entries e, accept when the
// next 24 random bits fall below q_e = round(2^24 w_e); 64 tries at most.
// Draws the batch of step *step_dev + 1.
__global__ void mlp_sample_kernel(const int32_t* __restrict__ rp, const int32_t* __restrict__ col,
                                  const uint32_t* __restrict__ q, int64_t n, int64_t nnz, int B, int neg,
                                  const uint32_t* __restrict__ step_dev, uint32_t k0, uint32_t k1,
                                  const int32_t* __restrict__ row_of, int32_t* __restrict__ rows) {
    const int R = 2 + neg;
    const uint32_t step = *step_dev + 1;
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < B; s += gridDim.x * blockDim.x) {
        uint32_t e = 0;
        for (uint32_t r = 0; r < 64; ++r) {
            const U4 u = philox4x32_10(U4{step, uint32_t(s), r, TAG_MLP}, k0, k1);
            e = __umulhi(u.x, uint32_t(nnz));
            if ((u.y >> 8) < q[e]) break;
        }
        // head row: from the table when there is one (a search is 17 dependent
        // loads at 70,000 rows), else the last i with rp[i] <= e
        int64_t lo = row_of ? row_of[e] : -1, hi = lo;
        if (lo < 0) {
            lo = 0;
            hi = n - 1;
        }
        while (lo < hi) {
            const int64_t mid = (lo + hi + 1) >> 1;
            if (rp[mid] <= int32_t(e)) lo = mid; else hi = mid - 1;
        }
        rows[int64_t(s) * R] = int32_t(lo);
        rows[int64_t(s) * R + 1] = col[e];
        for (int t = 0; t < neg; ++t) {
            const U4 u = philox4x32_10(U4{step, uint32_t(s), 64u + uint32_t(t / 4), TAG_MLP}, k0, k1);
            const uint32_t w4[4] = {u.x, u.y, u.z, u.w};
            rows[int64_t(s) * R + 2 + t] = int32_t(__umulhi(w4[t & 3], uint32_t(n)));
        }
    }
}

// Head row of every CSR entry (entries that no row covers keep -1).
__global__ void mlp_heads_kernel(const int32_t* __restrict__ rp, int64_t n, int64_t nnz, int32_t* __restrict__ row_of) {
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
        const int32_t b = rp[i], e = rp[i + 1];
        if (b < 0 || e > nnz) continue;
        for (int32_t t = b; t < e; ++t) row_of[t] = int32_t(i);
    }
}

// Gather BF16 rows (zero-padded to 64 columns), a warp per row; with `kept` the
// row numbers are copied there.
__global__ void mlp_gather_kernel(const float* __restrict__ X, int d, const int32_t* __restrict__ rows, int M,
                                  int M_valid, bf16* __restrict__ Xb, int32_t* __restrict__ kept) {
    const int lane = threadIdx.x & 31;
    for (int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < M; r += (gridDim.x * blockDim.x) >> 5) {
        float v[2] = {0.f, 0.f};
        if (r < M_valid) {
            const int32_t src = rows[r];
            if (kept && lane == 0) kept[r] = src;
            const float* x = X + int64_t(src) * d + 2 * lane;
#pragma unroll
            for (int j = 0; j < 2; ++j)
                if (2 * lane + j < d) v[j] = x[j];
        }
        reinterpret_cast<__nv_bfloat162*>(Xb)[int64_t(r) * (MLP_IN / 2) + lane] = __floats2bfloat162_rn(v[0], v[1]);
    }
}

// z = H2 W3^T + b3 of an edge's rows (head, tail, negatives) and its UMAP
// cross-entropy, with Phi = 1 / (1 + a d^b) clamped to [1e-4, 1 - 1e-4] (zero
// gradient where clamped); loss and dL/dz are divided by the batch size.
// Advances the step counter, which is at the step before until here.
//
// One warp per edge: the rows' products with lanes on columns lane + 32 i, four
// rows' loads in flight together, then one lane per row for the loss (powf and
// logf of all rows at once), whose terms are added in row order.  Latency-bound:
// as two kernels, with a thread per edge for the losses, 8 + 7 us.  (This and
// the split of the layer 3 backward below took a step of 4096 edges from 109 to
// 101 us.)
static constexpr int HEAD_ROWS = 4;

__global__ void __launch_bounds__(256) mlp_head_loss_kernel(const bf16* H2, const float* __restrict__ W3f,
                                                            const float* __restrict__ P, const int32_t* __restrict__ rows,
                                                            int B, int neg, float a, float b, float* __restrict__ dz,
                                                            float* __restrict__ loss_part, uint32_t* __restrict__ step_dev) {
    const int lane = threadIdx.x & 31;
    // (the weights and the rows are older than the kernel before, so they are read
    // before the wait, and qualified)
    float w0[MLP_H / 32], w1[MLP_H / 32];
#pragma unroll
    for (int i = 0; i < MLP_H / 32; ++i) {
        w0[i] = W3f[lane + 32 * i];
        w1[i] = W3f[MLP_H + lane + 32 * i];
    }
    const float b0 = P[OFF_B3], b1 = P[OFF_B3 + 1];
    dep_enter();
    if (blockIdx.x == 0 && threadIdx.x == 0) *step_dev += 1;
    const int R = 2 + neg;
    const float lo = 1e-4f, hi = 1.0f - 1e-4f, invB = 1.0f / float(B);
    const int warps = int((gridDim.x * blockDim.x) >> 5);
    for (int s = int((blockIdx.x * blockDim.x + threadIdx.x) >> 5); s < B; s += warps) {
        const int64_t r0 = int64_t(s) * R;
        const int32_t row = lane < R ? rows[r0 + lane] : 0;
        float z0 = 0.f, z1 = 0.f;  // of row r0 + lane
        for (int q = 0; q < R; q += HEAD_ROWS) {
            bf16 h[HEAD_ROWS][MLP_H / 32];
#pragma unroll
            for (int u = 0; u < HEAD_ROWS; ++u) {
                const int64_t r = r0 + (q + u < R ? q + u : R - 1);
#pragma unroll
                for (int i = 0; i < MLP_H / 32; ++i) h[u][i] = H2[r * MLP_H + lane + 32 * i];
            }
#pragma unroll
            for (int u = 0; u < HEAD_ROWS; ++u) {
                float s0 = 0.f, s1 = 0.f;
#pragma unroll
                for (int i = 0; i < MLP_H / 32; ++i) {
                    const float x = __bfloat162float(h[u][i]);
                    s0 = fmaf(x, w0[i], s0);
                    s1 = fmaf(x, w1[i], s1);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    s0 += __shfl_xor_sync(0xffffffffu, s0, o);
                    s1 += __shfl_xor_sync(0xffffffffu, s1, o);
                }
                if (lane == q + u) {
                    z0 = s0 + b0;
                    z1 = s1 + b1;
                }
            }
        }
        const float d0 = __shfl_sync(0xffffffffu, z0, 0) - z0, d1 = __shfl_sync(0xffffffffu, z1, 0) - z1;
        const int32_t head = __shfl_sync(0xffffffffu, row, 0);
        float g0 = 0.f, g1 = 0.f, l = 0.f;
        if (lane >= 1 && lane < R && !(lane >= 2 && row == head)) {  // (a negative that is the head itself adds nothing)
            const float d = d0 * d0 + d1 * d1;
            const float adb = d > 0.f ? a * powf(d, b) : 0.f;
            const float phi = 1.0f / (1.0f + adb);
            const bool inside = phi > lo && phi < hi;
            const float pc = fminf(fmaxf(phi, lo), hi);
            float dLdd = 0.f;
            if (lane == 1) {
                l = -logf(pc);
                if (inside) dLdd = b * adb / (d * (1.0f + adb));  // a b d^(b-1) / (1 + a d^b)
            } else {
                l = -logf(1.0f - pc);
                if (inside) dLdd = -b / (d * (1.0f + adb));
            }
            g0 = dLdd * 2.0f * d0 * invB;
            g1 = dLdd * 2.0f * d1 * invB;
        }
        float gi0 = 0.f, gi1 = 0.f, L = 0.f;
        for (int t = 1; t < R; ++t) {
            gi0 += __shfl_sync(0xffffffffu, g0, t);
            gi1 += __shfl_sync(0xffffffffu, g1, t);
            L += __shfl_sync(0xffffffffu, l, t);
        }
        if (lane < R)
            *reinterpret_cast<float2*>(dz + 2 * (r0 + lane)) = lane == 0 ? make_float2(gi0, gi1) : make_float2(-g0, -g1);
        if (lane == 0) loss_part[s] = L * invB;
    }
}

// One CTA takes a chunk of MLP_CHUNK rows and 32 columns.  The sums over a
// chunk's rows run in row order, one column a lane, from shared memory: their
// chains of 512 additions take about 2 us when no load sits inside them (56
// CTAs of 256 columns reading each row from L2 took 140 us for dW3, 40 us for
// a bias gradient).
static constexpr int MLP_CHUNK = 512;
static constexpr int MC_THREADS = 256;
static constexpr int MC_PITCH = MLP_CHUNK * 4 + 4;  // floats per float4 column: lanes of a row hit distinct banks

// dpre2 = (dz W3) . GELU'(pre2) (BF16) and, over the chunk, db2 = sum dpre2.
// Loads 64 KB a CTA, a warp per float4 column; one warp then adds while the
// others write dpre2 from shared memory.  (With dW3's sums and H2's tile in the
// same CTA, two CTAs an SM and 1.47 rounds of them, 26 us; mlp_w3grad_kernel now
// runs beside it.)
static constexpr size_t L3_SMEM = size_t(8) * MC_PITCH * 4 + MLP_CHUNK * 8;

__global__ void __launch_bounds__(MC_THREADS, 3)
mlp_l3back_kernel(const float* dz, const float* __restrict__ W3f, const float* __restrict__ dgelu2, int M,
                  bf16* __restrict__ D, float* __restrict__ pb2) {
    extern __shared__ __align__(16) float s_v[];  // [8][MC_PITCH]: dpre2, float4 columns
    float2* s_z = reinterpret_cast<float2*>(s_v + 8 * MC_PITCH);  // [MLP_CHUNK]: dz
    const int r0 = blockIdx.x * MLP_CHUNK, c0 = blockIdx.y * 32, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rows = M - r0 < MLP_CHUNK ? M - r0 : MLP_CHUNK;  // a multiple of 128
    float wx[4], wy[4];
#pragma unroll
    // (the weights and GELU' are older than the kernel before: qualified, so that their
    // first loads may be issued before the wait; unqualified, a step of 4096 edges took 6 us
    // more where the process had used 8 streams)
    for (int j = 0; j < 4; ++j) {
        wx[j] = W3f[c0 + 4 * warp + j];
        wy[j] = W3f[MLP_H + c0 + 4 * warp + j];
    }
    dep_enter();
    for (int r = tid; r < rows; r += MC_THREADS) s_z[r] = *reinterpret_cast<const float2*>(dz + 2 * int64_t(r0 + r));
    __syncthreads();
    for (int q = 0; q < rows; q += 128) {
        const float* p = dgelu2 + blocked_at(r0 + q + lane, c0 + 4 * warp, MLP_H);
        float4 x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = *reinterpret_cast<const float4*>(p + u * 128);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int r = q + 32 * u + lane;
            const float2 dz2 = s_z[r];
            float v[4] = {x[u].x, x[u].y, x[u].z, x[u].w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float g = dz2.x * wx[j] + dz2.y * wy[j];
                v[j] = g * v[j];
            }
            *reinterpret_cast<float4*>(s_v + warp * MC_PITCH + 4 * r) = make_float4(v[0], v[1], v[2], v[3]);
        }
    }
    __syncthreads();
    if (warp == 0) {
        const float* col = s_v + (lane >> 2) * MC_PITCH + (lane & 3);
        float s = 0.f;
#pragma unroll 16
        for (int r = 0; r < rows; ++r) s += col[4 * r];
        pb2[int64_t(blockIdx.x) * MLP_H + c0 + lane] = s;
    } else {
        for (int t = tid - 32; t < rows * 4; t += MC_THREADS - 32) {  // 16 bytes a lane, four lanes a row
            const int r = t >> 2, i = t & 3;
            const float4 f = *reinterpret_cast<const float4*>(s_v + 2 * i * MC_PITCH + 4 * r);
            const float4 g = *reinterpret_cast<const float4*>(s_v + (2 * i + 1) * MC_PITCH + 4 * r);
            const __nv_bfloat162 h[4] = {__floats2bfloat162_rn(f.x, f.y), __floats2bfloat162_rn(f.z, f.w),
                                         __floats2bfloat162_rn(g.x, g.y), __floats2bfloat162_rn(g.z, g.w)};
            *reinterpret_cast<uint4*>(D + int64_t(r0 + r) * MLP_H + c0 + 8 * i) = *reinterpret_cast<const uint4*>(h);
        }
    }
}

// Over the chunk: dW3[o] = sum dz[.][o] H2 and db3[o] = sum dz[.][o].
__global__ void __launch_bounds__(MC_THREADS)
mlp_w3grad_kernel(const float* __restrict__ dz, const bf16* __restrict__ H2, int M, float* __restrict__ pw3) {
    __shared__ __align__(16) bf16 s_h[MLP_CHUNK * 32];  // H2
    __shared__ float2 s_z[MLP_CHUNK];                   // dz
    const int r0 = blockIdx.x * MLP_CHUNK, c0 = blockIdx.y * 32, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rows = M - r0 < MLP_CHUNK ? M - r0 : MLP_CHUNK;
    for (int t = tid; t < rows * 4; t += MC_THREADS) {
        const int r = t >> 2, i = t & 3;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(s_h + r * 32 + 8 * i)),
                     "l"(H2 + int64_t(r0 + r) * MLP_H + c0 + 8 * i) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    for (int r = tid; r < rows; r += MC_THREADS) s_z[r] = *reinterpret_cast<const float2*>(dz + 2 * int64_t(r0 + r));
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    if (warp < 2) {
        const float* zo = reinterpret_cast<const float*>(s_z) + warp;
        float s = 0.f;
#pragma unroll 16
        for (int r = 0; r < rows; ++r) s += zo[2 * r] * __bfloat162float(s_h[r * 32 + lane]);
        pw3[int64_t(blockIdx.x) * (2 * MLP_H + 2) + warp * MLP_H + c0 + lane] = s;
    } else if (warp == 2 && c0 == 0 && lane < 2) {
        const float* zo = reinterpret_cast<const float*>(s_z) + lane;
        float s = 0.f;
#pragma unroll 16
        for (int r = 0; r < rows; ++r) s += zo[2 * r];
        pw3[int64_t(blockIdx.x) * (2 * MLP_H + 2) + 2 * MLP_H + lane] = s;
    }
}

// Column sums of a blocked FP32 M x MLP_H matrix over the chunk's rows.
static constexpr size_t CS_SMEM = size_t(8) * MC_PITCH * 4;

__global__ void __launch_bounds__(MC_THREADS, 3)
mlp_colsum_kernel(const float* __restrict__ A, int M, float* __restrict__ part) {
    extern __shared__ __align__(16) float s_v[];  // [8][MC_PITCH]
    const int r0 = blockIdx.x * MLP_CHUNK, c0 = blockIdx.y * 32, tid = threadIdx.x;
    const int rows = M - r0 < MLP_CHUNK ? M - r0 : MLP_CHUNK;
    dep_enter();
    for (int r = tid; r < rows; r += MC_THREADS) {
        const float* p = A + blocked_at(r0 + r, c0, MLP_H);
#pragma unroll
        for (int i = 0; i < 8; ++i)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(s_v + i * MC_PITCH + 4 * r)),
                         "l"(p + i * 512) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    if (tid < 32) {
        const float* col = s_v + (tid >> 2) * MC_PITCH + (tid & 3);
        float s = 0.f;
#pragma unroll 16
        for (int r = 0; r < rows; ++r) s += col[4 * r];
        part[int64_t(blockIdx.x) * MLP_H + c0 + tid] = s;
    }
}

struct GradParts {
    const float* dW1;   // [s1][256][64]
    int s1;
    const float* dW2;   // [s2][256][256]
    int s2;
    const float* db1;   // [n1][256]
    int n1;
    const float* db2;   // [n2][256]
    int n2;
    const float* w3;    // [n3][514]
    int n3;
    const float* loss;  // [B]
    int B;
};

template <class F>
__device__ __forceinline__ float sum_splits(int count, F&& at) {
    float s = 0.f;
    for (int z0 = 0; z0 < count; z0 += 32) {  // 32 loads in flight, added in order
        float v[32];
#pragma unroll
        for (int u = 0; u < 32; ++u) v[u] = z0 + u < count ? at(z0 + u) : 0.f;
#pragma unroll
        for (int u = 0; u < 32; ++u)
            if (z0 + u < count) s += v[u];
    }
    return s;
}

// Adam's state and step (adam_m null: the gradient alone).
struct AdamArgs {
    float* P;
    float* m;
    float* v;
    float lr, b1, b2, eps;
    MlpWeights W;
};

// Gradient vector from the partial sums (each summed in a fixed order), the
// batch loss, and with `ADAM` the update of the FP32 master weights
// (bias-corrected step t = *step + 1) and their BF16 copies.
template <bool ADAM>
__global__ void __launch_bounds__(256) mlp_update_kernel(GradParts g, AdamArgs A, float* __restrict__ grad,
                                                         float* __restrict__ loss_out,
                                                         const uint32_t* __restrict__ step_dev) {
    const uint32_t step = *step_dev;
    float c1 = 1.f, c2 = 1.f;
    if (ADAM) {
        const float t = float(step + 1);
        c1 = 1.0f - powf(A.b1, t);
        c2 = 1.0f - powf(A.b2, t);
    }
    for (int64_t p = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; p < MLP_P; p += int64_t(gridDim.x) * blockDim.x) {
        float s;
        if (p < OFF_B1) s = sum_splits(g.s1, [&](int z) { return g.dW1[int64_t(z) * MLP_H * MLP_IN + p]; });
        else if (p < OFF_W2) s = sum_splits(g.n1, [&](int z) { return g.db1[int64_t(z) * MLP_H + (p - OFF_B1)]; });
        else if (p < OFF_B2) s = sum_splits(g.s2, [&](int z) { return g.dW2[int64_t(z) * MLP_H * MLP_H + (p - OFF_W2)]; });
        else if (p < OFF_W3) s = sum_splits(g.n2, [&](int z) { return g.db2[int64_t(z) * MLP_H + (p - OFF_B2)]; });
        else s = sum_splits(g.n3, [&](int z) { return g.w3[int64_t(z) * (2 * MLP_H + 2) + (p - OFF_W3)]; });
        if (!ADAM) {
            grad[p] = s;
        } else {
            const float mm = A.b1 * A.m[p] + (1.0f - A.b1) * s;
            const float vv = A.b2 * A.v[p] + (1.0f - A.b2) * s * s;
            A.m[p] = mm;
            A.v[p] = vv;
            float w = A.P[p];
            w -= A.lr * (mm / c1) / (sqrtf(vv / c2) + A.eps);
            A.P[p] = w;
            mlp_cast_one(w, p, A.W);
        }
    }
    if (blockIdx.x == gridDim.x - 1 && loss_out) {  // (a block without parameters)
        __shared__ float red[256];
        float s = 0.f;
#pragma unroll 16
        for (int t = threadIdx.x; t < g.B; t += 256) s += g.loss[t];
        red[threadIdx.x] = s;
        __syncthreads();
        for (int o = blockDim.x / 2; o > 0; o >>= 1) {
            if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
            __syncthreads();
        }
        if (threadIdx.x == 0) loss_out[step] = red[0];
    }
}

// Initial weights: U(-1/sqrt(fan_in), 1/sqrt(fan_in)) from Philox, biases 0,
// columns of W1 beyond d exactly 0.
__global__ void mlp_init_kernel(float* __restrict__ P, int d, uint32_t k0, uint32_t k1) {
    for (int64_t p = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; p < MLP_P; p += int64_t(gridDim.x) * blockDim.x) {
        const U4 u = philox4x32_10(U4{uint32_t(p), 0u, 0u, TAG_MLP | 0x100u}, k0, k1);
        const float r = float(u.x >> 8) * 5.9604644775390625e-08f * 2.0f - 1.0f;  // [-1, 1)
        float val = 0.f;
        if (p < OFF_B1) val = (int(p % MLP_IN) < d) ? r / sqrtf(float(d)) : 0.f;
        else if (p >= OFF_W2 && p < OFF_B2) val = r / 16.0f;     // fan_in 256
        else if (p >= OFF_W3 && p < OFF_B3) val = r / 16.0f;
        P[p] = val;
    }
}

// ------------------------------------------------------------------ fused forward pass
// Y = head(GELU(GELU(X W1^T + b1) W2^T + b2)) for whole 128-row tiles, one
// persistent CTA per SM: both weight matrices stay in shared memory (160 KB),
// X is cast into a swizzled operand tile, H1 goes through shared memory in two
// halves of 128 columns, each multiplied into the second accumulator as soon as
// it is written, and H2 never leaves the registers that form the head's sums.
//
// Bound: the two GELUs' erf (about 40 instructions an element on the FP32 pipe,
// 18,000 cycles a tile against 3,200 of MMA), which the earlier form, two GEMMs
// and a head over chunks of 65,536 rows, joined with three passes over the
// activations.
//
// The sums are those of the training kernels: column pairs of the head in the
// order of mlp_head_loss_kernel (partial sums over columns u + 32 i, i ascending, for
// u = 0..31, joined as its shuffles join lanes).
static constexpr int FE_EPI_WARPS = 16;  // four per TMEM lane quarter
static constexpr int FE_EPI = FE_EPI_WARPS * 32;
static constexpr int FE_THREADS = FE_EPI + 32;  // the last warp loads the weights and issues the MMAs
static constexpr int FE_W1 = MLP_H * MLP_IN * 2, FE_W2 = MLP_H * MLP_H * 2, FE_X = G_BM * MLP_IN * 2, FE_H = G_BM * 128 * 2;
static constexpr size_t FE_SMEM = 1024 + FE_W1 + FE_W2 + FE_X + FE_H + 128 + (4 * MLP_H + 2) * 4;

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float* v) {
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr) : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

__global__ void __launch_bounds__(FE_THREADS, 1)
mlp_embed_kernel(const __grid_constant__ CUtensorMap tmW1, const __grid_constant__ CUtensorMap tmW2,
                 const float* __restrict__ X, int64_t n, int d, const float* __restrict__ P,
                 const float* __restrict__ W3f, float* __restrict__ Y, int* status) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    uint8_t* sW1 = base;
    uint8_t* sW2 = sW1 + FE_W1;  // four K blocks of 64 columns x 256 rows
    uint8_t* sX = sW2 + FE_W2;
    uint8_t* sH = sX + FE_X;     // two K blocks of 64 columns x 128 rows; also the head's partial sums
    uint64_t* bars = reinterpret_cast<uint64_t*>(sH + FE_H);
    uint64_t *w_full = bars, *x_full = bars + 1, *h_full = bars + 2, *d1_full = bars + 3, *h_free = bars + 4,
             *d2_full = bars + 5, *mma_done = bars + 6;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 7);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    float* s_b1 = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(bars) + 128);
    float* s_b2 = s_b1 + MLP_H;
    float* s_w3 = s_b2 + MLP_H;  // [2][256], then the two biases
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t tiles = (n + G_BM - 1) / G_BM;
    const int mine = int((tiles - blockIdx.x + gridDim.x - 1) / gridDim.x);  // tiles blockIdx.x, + gridDim.x, ...

    if (tid == 0) {
        mbar_init(w_full, 1);
        mbar_init(x_full, FE_EPI_WARPS);
        mbar_init(h_full, FE_EPI_WARPS);
        mbar_init(d1_full, 1);
        mbar_init(h_free, 1);
        mbar_init(d2_full, 1);
        mbar_init(mma_done, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == FE_EPI_WARPS) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_slot)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (int t = tid; t < MLP_H; t += FE_THREADS) {
        s_b1[t] = P[OFF_B1 + t];
        s_b2[t] = P[OFF_B2 + t];
        s_w3[t] = W3f[t];
        s_w3[MLP_H + t] = W3f[MLP_H + t];
        if (t < 2) s_w3[2 * MLP_H + t] = P[OFF_B3 + t];
    }
    for (int t = tid; t < FE_X / 16; t += FE_THREADS) reinterpret_cast<uint4*>(sX)[t] = make_uint4(0u, 0u, 0u, 0u);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == FE_EPI_WARPS) {
        if (lane == 0) {
            mbar_expect_tx(w_full, FE_W1 + FE_W2);
            tma_load_2d(sW1, &tmW1, 0, 0, w_full);
            for (int kb = 0; kb < 4; ++kb) tma_load_2d(sW2 + kb * (FE_W2 / 4), &tmW2, kb * 64, 0, w_full);
            const uint32_t idesc = idesc_f16kind(G_BM, MLP_H, false);
            const uint32_t D1 = tmem, D2 = tmem + MLP_H;
            bool ok = mbar_wait(w_full, 0, abort_flag, status);
            for (int t = 0; t < mine && ok; ++t) {
                if (!mbar_wait(x_full, t & 1, abort_flag, status)) break;
                tc_fence_after();
                const uint64_t xd = sdesc_sw128(smem_u32(sX)), w1d = sdesc_sw128(smem_u32(sW1));
#pragma unroll
                for (int k = 0; k < 4; ++k) mma_f16kind(D1, xd + 2 * k, w1d + 2 * k, idesc, k > 0);
                mma_commit(d1_full);
                for (int half = 0; half < 2 && ok; ++half) {
                    if (!(ok = mbar_wait(h_full, half, abort_flag, status))) break;
                    tc_fence_after();
                    for (int kb = 0; kb < 2; ++kb) {
                        const uint64_t hd = sdesc_sw128(smem_u32(sH + kb * (FE_H / 2)));
                        const uint64_t w2d = sdesc_sw128(smem_u32(sW2 + (2 * half + kb) * (FE_W2 / 4)));
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            mma_f16kind(D2, hd + 2 * k, w2d + 2 * k, idesc, (half > 0 || kb > 0 || k > 0) ? 1u : 0u);
                    }
                    mma_commit(half == 0 ? h_free : d2_full);
                }
            }
            // every MMA issued above has completed once this barrier fires
            mma_commit(mma_done);
            const unsigned long long t0 = global_timer();
            while (!mbar_try(mma_done, 0) && global_timer() - t0 < 100000000ull) {
            }
        }
    } else {
        // A failed wait (reported in the status word) does not leave the loop:
        // every later one then returns at once, and the warps still meet at
        // their barriers.
        const int quarter = warp & 3, g = warp >> 2;
        const int row = quarter * 32 + lane;
        const uint32_t tq = tmem + (uint32_t(quarter * 32) << 16);
        // this thread's elements of an X tile (128 d consecutive floats) and
        // their places in the operand tile
        constexpr int NX = G_BM * MLP_IN / FE_EPI;
        uint32_t xo[NX];
#pragma unroll
        for (int u = 0; u < NX; ++u) {
            const int e = tid + u * FE_EPI, r = e / d, c = e - r * d;
            xo[u] = r < G_BM ? uint32_t(r * 128 + ((((c >> 3) ^ r) & 7) << 4) + (c & 7) * 2) : 0xffffffffu;
        }
        float xv[NX];
        auto load_x = [&](int t) {
            const int64_t e0 = (blockIdx.x + int64_t(t) * gridDim.x) * G_BM * d;
#pragma unroll
            for (int u = 0; u < NX; ++u) {
                const int64_t e = e0 + tid + u * FE_EPI;
                xv[u] = t < mine && xo[u] != 0xffffffffu && e < n * d ? X[e] : 0.f;
            }
        };
        auto stage_x = [&]() {
#pragma unroll
            for (int u = 0; u < NX; ++u)
                if (xo[u] != 0xffffffffu) *reinterpret_cast<bf16*>(sX + xo[u]) = __float2bfloat16_rn(xv[u]);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            tc_fence_before();  // (the reads of the first accumulator)
            __syncwarp();
            if (lane == 0) mbar_arrive(x_full);
        };
        load_x(0);
        if (mine > 0) stage_x();
        load_x(1);
        for (int t = 0; t < mine; ++t) {
            mbar_wait(d1_full, t & 1, abort_flag, status);
            tc_fence_after();
#pragma unroll 1
            for (int half = 0; half < 2; ++half) {
                const int c0 = half * 128 + g * 32;
                float v[32];
                __syncwarp();
                tmem_ld32(tq + uint32_t(c0), v);
                uint32_t packed[16];
#pragma unroll
                for (int i = 0; i < 32; i += 4) {
                    const float4 b4 = *reinterpret_cast<const float4*>(s_b1 + c0 + i);
                    v[i] = gelu(v[i] + b4.x);
                    v[i + 1] = gelu(v[i + 1] + b4.y);
                    v[i + 2] = gelu(v[i + 2] + b4.z);
                    v[i + 3] = gelu(v[i + 3] + b4.w);
                    const __nv_bfloat162 h0 = __floats2bfloat162_rn(v[i], v[i + 1]), h1 = __floats2bfloat162_rn(v[i + 2], v[i + 3]);
                    packed[i / 2] = *reinterpret_cast<const uint32_t*>(&h0);
                    packed[i / 2 + 1] = *reinterpret_cast<const uint32_t*>(&h1);
                }
                // the first half's products with H are done (the second's, of the
                // tile before, were when its D2 was read)
                if (half == 1) mbar_wait(h_free, t & 1, abort_flag, status);
                uint8_t* hr = sH + (g >> 1) * (FE_H / 2) + row * 128;
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    *reinterpret_cast<uint4*>(hr + ((((g & 1) * 4 + j) ^ (row & 7)) << 4)) =
                        make_uint4(packed[4 * j], packed[4 * j + 1], packed[4 * j + 2], packed[4 * j + 3]);
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(h_full);
            }
            if (t + 1 < mine) stage_x();
            load_x(t + 2);
            mbar_wait(d2_full, t & 1, abort_flag, status);
            tc_fence_after();
            // residues u = 8 g .. 8 g + 7 of the columns modulo 32
            float p0[8], p1[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) p0[u] = p1[u] = 0.f;
#pragma unroll 1
            for (int i = 0; i < 8; ++i) {
                const int c0 = 32 * i + 8 * g;
                float v[8];
                __syncwarp();
                tmem_ld8(tq + uint32_t(MLP_H + c0), v);
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const float h = __bfloat162float(__float2bfloat16_rn(gelu(v[u] + s_b2[c0 + u])));
                    p0[u] = fmaf(h, s_w3[c0 + u], p0[u]);
                    p1[u] = fmaf(h, s_w3[MLP_H + c0 + u], p1[u]);
                }
            }
            tc_fence_before();
            float* hs = reinterpret_cast<float*>(sH);  // [2][32][128]
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                hs[(8 * g + u) * 128 + row] = p0[u];
                hs[(32 + 8 * g + u) * 128 + row] = p1[u];
            }
            asm volatile("bar.sync 1, %0;" ::"r"(FE_EPI) : "memory");
            if (tid < 2 * G_BM) {
                const int o = tid >> 7, r = tid & 127;
                float q[16];
#pragma unroll
                for (int u = 0; u < 16; ++u) q[u] = hs[(32 * o + u) * 128 + r] + hs[(32 * o + u + 16) * 128 + r];
#pragma unroll
                for (int w = 8; w > 0; w >>= 1)
#pragma unroll
                    for (int u = 0; u < w; ++u) q[u] += q[u + w];
                const int64_t gr = (blockIdx.x + int64_t(t) * gridDim.x) * G_BM + r;
                if (gr < n) Y[2 * gr + o] = q[0] + s_w3[2 * MLP_H + o];
            }
            asm volatile("bar.sync 1, %0;" ::"r"(FE_EPI) : "memory");
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == FE_EPI_WARPS) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

// ------------------------------------------------------------------ host: one forward/backward
// Opt the chunk kernels into their shared-memory sizes (before any capture).
static int chunk_prepare(Ctx* c) {
    DRGB_CUDA(c, cudaFuncSetAttribute(mlp_l3back_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(L3_SMEM)));
    DRGB_CUDA(c, cudaFuncSetAttribute(mlp_colsum_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(CS_SMEM)));
    return DRGB_OK;
}

struct MlpBuffers {
    int M;                       // rows of the batch (padded to 128)
    int32_t* rows;
    bf16 *Xb, *H1b, *H2b, *D2b, *D1b;
    int32_t* next_rows;
    float *dg1, *dg2, *dz, *D1f, *loss_part;
    float *pW2, *pW1, *pb1, *pb2, *pw3;
    float* grad;
    MlpWeights W;
    uint32_t* step;
    int n_chunks;
};

static constexpr int MLP_SPLITS = 32;
static size_t mlp_batch_bytes(int M) {
    const size_t m = size_t(M);
    const int nch = int((m + MLP_CHUNK - 1) / MLP_CHUNK);
    size_t b = Carve::round(m * 4);                                   // rows
    b += Carve::round(m * MLP_IN * 2);                                // Xb
    b += 4 * Carve::round(m * MLP_H * 2);                             // H1b, H2b, D2b, D1b
    b += 3 * Carve::round(m * MLP_H * 4);                             // dg1, dg2, D1f
    b += Carve::round(m * 2 * 4) + 2 * Carve::round(m * 4);           // dz, next_rows, loss_part
    b += Carve::round(size_t(MLP_SPLITS) * MLP_H * MLP_H * 4);        // pW2
    b += Carve::round(size_t(MLP_SPLITS) * MLP_H * MLP_IN * 4);       // pW1
    b += 2 * Carve::round(size_t(nch) * MLP_H * 4);                   // pb1, pb2
    b += Carve::round(size_t(nch) * (2 * MLP_H + 2) * 4);             // pw3
    b += Carve::round(MLP_P * 4);                                     // grad
    b += 2 * Carve::round(MLP_H * MLP_H * 2) + Carve::round(MLP_H * MLP_IN * 2) + Carve::round(2 * MLP_H * 4);
    b += Carve::round(64);
    return b + 8192;
}

static MlpBuffers mlp_carve(void* base, int M) {
    Carve cv(base);
    MlpBuffers b;
    const size_t m = size_t(M);
    b.M = M;
    b.n_chunks = int((m + MLP_CHUNK - 1) / MLP_CHUNK);
    b.rows = cv.take<int32_t>(m);
    b.Xb = cv.take<bf16>(m * MLP_IN);
    b.H1b = cv.take<bf16>(m * MLP_H);
    b.H2b = cv.take<bf16>(m * MLP_H);
    b.D2b = cv.take<bf16>(m * MLP_H);
    b.D1b = cv.take<bf16>(m * MLP_H);
    b.dg1 = cv.take<float>(m * MLP_H);
    b.dg2 = cv.take<float>(m * MLP_H);
    b.D1f = cv.take<float>(m * MLP_H);
    b.next_rows = cv.take<int32_t>(m);
    b.dz = cv.take<float>(m * 2);
    b.loss_part = cv.take<float>(m);
    b.pW2 = cv.take<float>(size_t(MLP_SPLITS) * MLP_H * MLP_H);
    b.pW1 = cv.take<float>(size_t(MLP_SPLITS) * MLP_H * MLP_IN);
    b.pb1 = cv.take<float>(size_t(b.n_chunks) * MLP_H);
    b.pb2 = cv.take<float>(size_t(b.n_chunks) * MLP_H);
    b.pw3 = cv.take<float>(size_t(b.n_chunks) * (2 * MLP_H + 2));
    b.grad = cv.take<float>(MLP_P);
    b.W.W2b = cv.take<bf16>(MLP_H * MLP_H);
    b.W.W2tb = cv.take<bf16>(MLP_H * MLP_H);
    b.W.W1b = cv.take<bf16>(MLP_H * MLP_IN);
    b.W.W3f = cv.take<float>(2 * MLP_H);
    b.step = cv.take<uint32_t>(16);
    return b;
}

// Further branches of a training step: dW2 beside dH1 and what follows from
// it, and the next step's batch.  The batch does not depend on the weights: its
// rows are drawn beside the backward pass and gathered beside the update, when
// dW1 has read this step's Xb.  In line the two took 27 us of a step (dependent loads from memory, under
// one warp an SM): a step of 4096 edges went from 160 to 144 us, one of 512
// from 74 to 58.
// Without the streams everything runs in line and no batch is prepared.
struct MlpFork {
    cudaStream_t side = nullptr, ahead = nullptr;
    cudaEvent_t ev[7] = {};
    std::function<int(cudaStream_t)> draw, gather;
};

// `to` continues after what `from` holds so far.
static int mlp_order(Ctx* c, cudaEvent_t ev, cudaStream_t from, cudaStream_t to) {
    DRGB_CUDA(c, cudaEventRecord(ev, from));
    DRGB_CUDA(c, cudaStreamWaitEvent(to, ev, 0));
    return DRGB_OK;
}

// Padding rows carry no gradient (their part of dz is written by nothing else).
static int mlp_zero_padding(Ctx* c, const MlpBuffers& b, int rows, cudaStream_t st) {
    if (b.M > rows) DRGB_CUDA(c, cudaMemsetAsync(b.dz + 2 * int64_t(rows), 0, size_t(b.M - rows) * 2 * 4, st));
    return DRGB_OK;
}

// The kernels follow each other with programmatic dependencies (launch_dep): 144
// to 136 us a step of 4096 edges.
//
// Forward + backward of the batch whose rows are already gathered (Xb)
// with B edges of R rows; leaves the gradient in b.grad and the loss in
// loss_out[*step] (if given), and with `adam` updates the weights.
static int mlp_fwd_bwd(Ctx* c, MlpBuffers& b, const float* P, int B, int neg, float a, float bb,
                       float* loss_out, const AdamArgs* adam, const MlpFork& fork, cudaStream_t st) {
    const int M = b.M;
    int rc;
    Layer F1, F2, DH1;
    Gemm DW2, DW1;
    if ((rc = layer_setup(c, F1, b.Xb, b.W.W1b, M, MLP_IN))) return rc;
    F1.g.bias = P + OFF_B1;
    F1.g.dgelu = b.dg1;
    F1.g.out = b.H1b;
    if ((rc = layer_setup(c, F2, b.H1b, b.W.W2b, M, MLP_H))) return rc;
    F2.g.bias = P + OFF_B2;
    F2.g.dgelu = b.dg2;
    F2.g.out = b.H2b;
    if ((rc = layer_launch<false>(c, F1, false, st)) || (rc = layer_launch<false>(c, F2, true, st)) ||
        (rc = launch_dep(c, mlp_head_loss_kernel, dim3(grid_for(B, 8, c->num_sms * 8)), 256, 0, true, st, b.H2b, b.W.W3f,
                          P, b.rows, B, neg, a, bb, b.dz, b.loss_part, b.step)))
        return rc;
    if (fork.ahead && ((rc = mlp_order(c, fork.ev[0], st, fork.ahead)) || (rc = fork.draw(fork.ahead)))) return rc;
    // dW3, dW2 = dpre2^T H1 (K = M, split) and later db1 on a branch of their own
    const dim3 cgrid(b.n_chunks, MLP_H / 32);
    const cudaStream_t side = fork.side ? fork.side : st;
    if (fork.side && (rc = mlp_order(c, fork.ev[1], st, side))) return rc;
    if ((rc = launch_dep(c, mlp_l3back_kernel, cgrid, MC_THREADS, L3_SMEM, fork.side != nullptr, st, b.dz, b.W.W3f, b.dg2,
                          M, b.D2b, b.pb2)) ||
        (rc = launch_dep(c, mlp_w3grad_kernel, cgrid, MC_THREADS, 0, false, side, b.dz, b.H2b, M, b.pw3)))
        return rc;
    if (fork.side && (rc = mlp_order(c, fork.ev[5], st, side))) return rc;
    if ((rc = gemm_setup(c, DW2, b.D2b, b.H1b, MLP_H, MLP_H, M, 128, MLP_SPLITS, true))) return rc;
    DW2.g.out_f32 = b.pW2;
    if ((rc = gemm_launch(c, DW2, false, side))) return rc;
    // dpre1 = (dpre2 W2) . GELU'(pre1): A = dpre2 [M x 256(out)], B = W2^T [256(in) x 256(out)]
    if ((rc = layer_setup(c, DH1, b.D2b, b.W.W2tb, M, MLP_H))) return rc;
    DH1.g.dgelu = b.dg1;
    DH1.g.out = b.D1b;
    DH1.g.out_f32 = b.D1f;
    if ((rc = layer_launch<true>(c, DH1, fork.side != nullptr, st))) return rc;
    if (fork.side && (rc = mlp_order(c, fork.ev[2], st, side))) return rc;
    // dW1 = dpre1^T Xb
    if ((rc = gemm_setup(c, DW1, b.D1b, b.Xb, MLP_H, MLP_IN, M, 64, MLP_SPLITS, true))) return rc;
    DW1.g.out_f32 = b.pW1;
    if ((rc = gemm_launch(c, DW1, fork.side != nullptr, st)) ||
        (rc = launch_dep(c, mlp_colsum_kernel, cgrid, MC_THREADS, CS_SMEM, false, side, b.D1f, M, b.pb1)))
        return rc;
    if (fork.ahead && ((rc = mlp_order(c, fork.ev[6], st, fork.ahead)) || (rc = fork.gather(fork.ahead)))) return rc;
    if (fork.side && (rc = mlp_order(c, fork.ev[3], fork.side, st))) return rc;
    GradParts gp;
    gp.dW1 = b.pW1;
    gp.s1 = int(DW1.grid.z);
    gp.dW2 = b.pW2;
    gp.s2 = int(DW2.grid.z);
    gp.db1 = b.pb1;
    gp.n1 = b.n_chunks;
    gp.db2 = b.pb2;
    gp.n2 = b.n_chunks;
    gp.w3 = b.pw3;
    gp.n3 = b.n_chunks;
    gp.loss = b.loss_part;
    gp.B = B;
    const int ugrid = int((MLP_P + 255) / 256) + 1;  // the last block adds the losses
    if (adam) mlp_update_kernel<true><<<ugrid, 256, 0, st>>>(gp, *adam, b.grad, loss_out, b.step);
    else mlp_update_kernel<false><<<ugrid, 256, 0, st>>>(gp, AdamArgs{}, b.grad, loss_out, b.step);
    DRGB_CHECK_LAUNCH(c);
    if (fork.ahead && (rc = mlp_order(c, fork.ev[4], fork.ahead, st))) return rc;
    return DRGB_OK;
}

static int mlp_check(Ctx* c, int d) {
    if (!c) return DRGB_ERR_INVALID;
    if (d < 1 || d > MLP_IN) return set_error(c, DRGB_ERR_INVALID, "mlp: d must be in 1..%d", MLP_IN);
    return DRGB_OK;
}

static int round_up(int64_t x, int64_t m) { return int((x + m - 1) / m * m); }

}  // namespace drgb

using namespace drgb;

extern "C" {

int64_t drgb_mlp_param_count(void) { return MLP_P; }

int drgb_mlp_init(drgb_ctx* c, float* params, int32_t d, uint64_t seed, void* stream) {
    int rc = mlp_check(c, d);
    if (rc) return rc;
    if (!params) return set_error(c, DRGB_ERR_INVALID, "mlp_init: NULL params");
    mlp_init_kernel<<<grid_for(MLP_P, 256, c->num_sms * 4), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        params, d, uint32_t(seed), uint32_t(seed >> 32));
    DRGB_CHECK_LAUNCH(c);
    return DRGB_OK;
}

int drgb_mlp_grad(drgb_ctx* c, const float* params, const float* X, int64_t n, int32_t d, const int32_t* rows,
                  int32_t n_edges, int32_t neg, float a, float b, float* grad_out, float* loss_out, void* stream) {
    int rc = mlp_check(c, d);
    if (rc) return rc;
    if (!params || !X || !rows || !grad_out || n_edges < 1 || neg < 0 || neg > 8 || n < 2)
        return set_error(c, DRGB_ERR_INVALID, "mlp_grad: bad arguments");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if ((rc = gemm_prepare(c)) || (rc = chunk_prepare(c))) return rc;
    const int Mv = n_edges * (2 + neg);
    const int M = round_up(Mv, 128);
    if ((rc = ensure_scratch(c, mlp_batch_bytes(M), st))) return rc;
    MlpBuffers bu = mlp_carve(c->scratch, M);
    DRGB_CUDA(c, cudaMemsetAsync(bu.rows, 0, size_t(M) * 4, st));
    DRGB_CUDA(c, cudaMemcpyAsync(bu.rows, rows, size_t(Mv) * 4, cudaMemcpyDeviceToDevice, st));
    DRGB_CUDA(c, cudaMemsetAsync(bu.step, 0xFF, 64, st));  // (the step before the first)
    if ((rc = mlp_zero_padding(c, bu, Mv, st))) return rc;
    mlp_cast_kernel<<<grid_for(MLP_P, 256, c->num_sms * 4), 256, 0, st>>>(params, bu.W);
    DRGB_CHECK_LAUNCH(c);
    mlp_gather_kernel<<<grid_for(M, 8, c->num_sms * 8), 256, 0, st>>>(X, d, bu.rows, M, Mv, bu.Xb, nullptr);
    DRGB_CHECK_LAUNCH(c);
    if ((rc = mlp_fwd_bwd(c, bu, params, n_edges, neg, a, b, loss_out, nullptr, MlpFork{}, st))) return rc;
    DRGB_CUDA(c, cudaMemcpyAsync(grad_out, bu.grad, MLP_P * 4, cudaMemcpyDeviceToDevice, st));
    return drgb_sync(c, stream);
}

int drgb_mlp_train(drgb_ctx* c, const float* X, int64_t n, int32_t d, const int32_t* row_ptr, const int32_t* col,
                   const uint32_t* q, int64_t nnz, float a, float b, const drgb_mlp_params* mp, float* params,
                   float* adam_m, float* adam_v, float* losses, void* stream) {
    int rc = mlp_check(c, d);
    if (rc) return rc;
    if (!X || !row_ptr || !col || !q || !mp || !params || !adam_m || !adam_v || nnz < 1 || n < 2 ||
        mp->batch_edges < 1 || mp->neg < 0 || mp->neg > 8 || mp->steps < 0)
        return set_error(c, DRGB_ERR_INVALID, "mlp_train: bad arguments");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if ((rc = gemm_prepare(c)) || (rc = chunk_prepare(c))) return rc;
    const int B = mp->batch_edges, neg = mp->neg, R = 2 + neg;
    const int Mv = B * R;
    const int M = round_up(Mv, 128);
    // the heads of the CSR entries, if there is room for them beside the batch
    const size_t least = mlp_batch_bytes(M);
    size_t bytes = Carve::round(least) + size_t(nnz) * 4;
    if ((rc = ensure_scratch_within(c, &bytes, least, st))) return rc;
    MlpBuffers bu = mlp_carve(c->scratch, M);
    int32_t* row_of = bytes > least ? reinterpret_cast<int32_t*>(static_cast<char*>(c->scratch) + Carve::round(least)) : nullptr;
    DRGB_CUDA(c, cudaMemsetAsync(bu.rows, 0, size_t(M) * 4, st));
    DRGB_CUDA(c, cudaMemsetAsync(bu.step, 0xFF, 64, st));  // (the step before the first)
    if ((rc = mlp_zero_padding(c, bu, Mv, st))) return rc;
    if (row_of) {
        DRGB_CUDA(c, cudaMemsetAsync(row_of, 0xFF, size_t(nnz) * 4, st));
        mlp_heads_kernel<<<grid_for(n, 256, c->num_sms * 8), 256, 0, st>>>(row_ptr, n, nnz, row_of);
        DRGB_CHECK_LAUNCH(c);
    }
    mlp_cast_kernel<<<grid_for(MLP_P, 256, c->num_sms * 4), 256, 0, st>>>(params, bu.W);
    DRGB_CHECK_LAUNCH(c);
    const uint32_t k0 = uint32_t(mp->seed), k1 = uint32_t(mp->seed >> 32);

    MlpFork fork;
    int32_t* const next_rows = bu.next_rows;
    fork.draw = [&](cudaStream_t s) -> int {
        mlp_sample_kernel<<<grid_for(B, 32, c->num_sms * 8), 32, 0, s>>>(row_ptr, col, q, n, nnz, B, neg, bu.step, k0,
                                                                        k1, row_of, next_rows);
        DRGB_CHECK_LAUNCH(c);
        return DRGB_OK;
    };
    fork.gather = [&](cudaStream_t s) -> int {
        mlp_gather_kernel<<<grid_for(M, 8, c->num_sms * 8), 256, 0, s>>>(X, d, next_rows, M, Mv, bu.Xb, bu.rows);
        DRGB_CHECK_LAUNCH(c);
        return DRGB_OK;
    };
    if (mp->steps > 0 && ((rc = fork.draw(st)) || (rc = fork.gather(st)))) return rc;

    // capture one step, replay it mp->steps times (the step counter lives on
    // the device, so every replay draws a fresh batch)
    cudaStream_t cap = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    auto release = [&]() {
        if (exec) cudaGraphExecDestroy(exec);
        if (graph) cudaGraphDestroy(graph);
        for (cudaEvent_t ev : fork.ev)
            if (ev) cudaEventDestroy(ev);
        if (fork.side) cudaStreamDestroy(fork.side);
        if (fork.ahead) cudaStreamDestroy(fork.ahead);
        if (cap) cudaStreamDestroy(cap);
    };
    cudaError_t e = cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&fork.side, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&fork.ahead, cudaStreamNonBlocking);
    for (cudaEvent_t& ev : fork.ev)
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) {
        release();
        return set_error(c, DRGB_ERR_CUDA, "mlp_train: begin capture: %s", cudaGetErrorString(e));
    }
    const AdamArgs adam{params, adam_m, adam_v, mp->lr, mp->beta1, mp->beta2, mp->eps, bu.W};
    const int64_t before = c->launches;
    rc = mlp_fwd_bwd(c, bu, params, B, neg, a, b, losses, &adam, fork, cap);
    const int64_t step_launches = c->launches - before;
    c->launches = before;  // counted as they are replayed
    e = cudaStreamEndCapture(cap, &graph);
    if (rc == DRGB_OK && e != cudaSuccess) rc = set_error(c, DRGB_ERR_CUDA, "mlp_train: end capture: %s", cudaGetErrorString(e));
    if (rc == DRGB_OK && (e = cudaGraphInstantiate(&exec, graph, 0)) != cudaSuccess)
        rc = set_error(c, DRGB_ERR_CUDA, "mlp_train: instantiate: %s", cudaGetErrorString(e));
    for (int s = 0; rc == DRGB_OK && s < mp->steps; ++s) {
        e = cudaGraphLaunch(exec, st);
        if (e != cudaSuccess) rc = set_error(c, DRGB_ERR_CUDA, "mlp_train: launch: %s", cudaGetErrorString(e));
        else c->launches += step_launches;
    }
    release();
    if (rc) return rc;
    return drgb_sync(c, stream);
}

int drgb_mlp_sample(drgb_ctx* c, const int32_t* row_ptr, const int32_t* col, const uint32_t* q, int64_t n,
                    int64_t nnz, int32_t n_edges, int32_t neg, uint32_t step, uint64_t seed, int32_t* rows,
                    void* stream) {
    if (!c) return DRGB_ERR_INVALID;
    if (!row_ptr || !col || !q || !rows || n < 2 || nnz < 1 || n_edges < 1 || neg < 0 || neg > 8)
        return set_error(c, DRGB_ERR_INVALID, "mlp_sample: bad arguments");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int rc = ensure_scratch(c, 256, st);
    if (rc) return rc;
    uint32_t* step_dev = static_cast<uint32_t*>(c->scratch);
    const uint32_t before = step - 1;
    DRGB_CUDA(c, cudaMemcpyAsync(step_dev, &before, 4, cudaMemcpyHostToDevice, st));
    mlp_sample_kernel<<<grid_for(n_edges, 128, c->num_sms * 8), 128, 0, st>>>(row_ptr, col, q, n, nnz, n_edges, neg,
                                                                             step_dev, uint32_t(seed),
                                                                             uint32_t(seed >> 32), nullptr, rows);
    DRGB_CHECK_LAUNCH(c);
    return drgb_sync(c, stream);
}

int drgb_mlp_embed(drgb_ctx* c, const float* params, const float* X, int64_t n, int32_t d, float* Y, void* stream) {
    int rc = mlp_check(c, d);
    if (rc) return rc;
    if (!params || !X || !Y || n < 1) return set_error(c, DRGB_ERR_INVALID, "mlp_embed: bad arguments");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const size_t bytes = 2 * Carve::round(MLP_H * MLP_H * 2) + Carve::round(MLP_H * MLP_IN * 2) +
                         Carve::round(2 * MLP_H * 4) + 1024;
    if ((rc = ensure_scratch(c, bytes, st))) return rc;
    Carve cv(c->scratch);
    MlpWeights W;
    W.W2b = cv.take<bf16>(MLP_H * MLP_H);
    W.W2tb = cv.take<bf16>(MLP_H * MLP_H);
    W.W1b = cv.take<bf16>(MLP_H * MLP_IN);
    W.W3f = cv.take<float>(2 * MLP_H);
    mlp_cast_kernel<<<grid_for(MLP_P, 256, c->num_sms * 4), 256, 0, st>>>(params, W);
    DRGB_CHECK_LAUNCH(c);
    CUtensorMap m1, m2;
    if ((rc = make_map_k64(c, &m1, W.W1b, MLP_H, MLP_IN, MLP_H, false))) return rc;
    if ((rc = make_map_k64(c, &m2, W.W2b, MLP_H, MLP_H, MLP_H, false))) return rc;
    DRGB_CUDA(c, cudaFuncSetAttribute(mlp_embed_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(FE_SMEM)));
    mlp_embed_kernel<<<grid_for((n + G_BM - 1) / G_BM, 1, c->num_sms), FE_THREADS, FE_SMEM, st>>>(m1, m2, X, n, d, params,
                                                                                                W.W3f, Y, c->d_status);
    DRGB_CHECK_LAUNCH(c);
    return DRGB_OK;
}

}  // extern "C"
