// Exact k nearest database rows of a set of queries on the tensor cores, for
// rows of up to WD_MAX_D dimensions and any query set: the whole database (a
// graph of X on itself wider than the cell-ordered kernel of knn_tc.cu takes),
// listed rows of it, or another matrix.
//
// The operands, the candidate lists and the certificate are those of
// knn_tc.cu: FP16 operands [x~, C, C, C] and [-2 x~, h, m, l] whose product is
// s_ij = |x~_j|^2 - 2 x~_i . x~_j, the best 32 (s, j) of every query kept by
// the epilogue threads, their exact FP32 distances (the FP32 scan's
// arithmetic), and a bound that proves that no other row is among the k
// nearest; queries it cannot certify are scanned exactly.
//
// A CTA takes 128 queries and a contiguous share of the database tiles (256
// rows); K = d + 3 rounded up to 64 is streamed in steps of 64 columns of both
// operands through a 3-stage TMA ring, and two TMEM accumulators let the MMA
// of one tile run under the selection of the previous one.  The database is
// split over blockIdx.y so that few queries still fill the GPU: 235 blocks of
// 128 queries on 152 SMs leave a quarter of two waves idle, and a batch of
// 1,000 queries has 8 blocks.  The splits' lists are merged by the re-rank.
//
// Bound: the selection (about 250 list insertions a query for the first split
// and 30 for a later one, whose branches a warp of 32 rows takes on most chunks) up
// to K of about 256, the
// tensor pipe and the L2 reads of both operands (48 KB per 128 x 256 x 64
// step) above.
#include <cuda.h>
#include <cudaTypedefs.h>

#include "common.cuh"
#include "knn.cuh"
#include "knn_select.cuh"
#include "tc_ptx.cuh"

namespace drgb {

static constexpr int WD_BM = 128, WD_BN = 256, WD_STAGES = 3;
static constexpr int WD_THREADS = 64 + TC_EPI_WARPS * 32;
static constexpr int WD_A_BYTES = WD_BM * 64 * 2, WD_B_BYTES = WD_BN * 64 * 2;
static constexpr int WD_STAGE = WD_A_BYTES + WD_B_BYTES;
static constexpr size_t WD_SMEM =
    1024 + size_t(WD_STAGES) * WD_STAGE + 256 + TC_QUEUE_BYTES + size_t(2) * WD_BM * TC_NQ * 4;
static constexpr int WD_MAX_D = 1021;     // K <= 1024: the norms' split stays in FP16's range
static constexpr int WD_MAX_SPLITS = 64;
static constexpr int WD_STAT_BLOCKS = 256;  // row ranges of the database's column statistics (at most)
static constexpr int WD_STAT_QBLOCKS = 64;  // and of the queries'

// ------------------------------------------------------------------ staging
// Partial column sums (database only), minima and maxima (both sets): block b
// covers a range of rows, a thread per column.
__global__ void __launch_bounds__(256) wide_stats_kernel(const float* __restrict__ X, int64_t n,
                                                         const float* __restrict__ Q, int64_t nq, int d,
                                                         unsigned db_blocks, float* __restrict__ partial) {
    const bool db = blockIdx.x < db_blocks;
    const float* M = db ? X : Q;
    const int64_t rows = db ? n : nq, nb = db ? db_blocks : gridDim.x - db_blocks;
    const int64_t b = db ? blockIdx.x : blockIdx.x - db_blocks;
    const int64_t per = (rows + nb - 1) / nb, r0 = b * per, r1 = r0 + per < rows ? r0 + per : rows;
    for (int c = blockIdx.y * blockDim.x + threadIdx.x; c < d; c += gridDim.y * blockDim.x) {
        float s = 0.f, lo = INFINITY, hi = -INFINITY;
#pragma unroll 8
        for (int64_t r = r0; r < r1; ++r) {
            const float v = M[r * d + c];
            s += v;
            lo = fminf(lo, v);
            hi = fmaxf(hi, v);
        }
        float* p = partial + int64_t(blockIdx.x) * 3 * d + c;
        p[0] = s;
        p[d] = lo;
        p[2 * d] = hi;
    }
}

// Column means and the largest |x - mean| (maxbits[2]); 32 columns a block,
// eight threads a column.  Rounding is monotone, so fl(max - m) and fl(m - min)
// bound every |fl(x - m)| of the column.
__global__ void __launch_bounds__(256) wide_mean_kernel(const float* __restrict__ partial, int blocks, int db_blocks,
                                                        int64_t n, int d, float* __restrict__ mean,
                                                        unsigned int* __restrict__ maxbits) {
    __shared__ double s_s[8][32];
    __shared__ float s_lo[8][32], s_hi[8][32];
    const int c = blockIdx.x * 32 + threadIdx.x, g = threadIdx.y;
    double s = 0.0;
    float lo = INFINITY, hi = -INFINITY;
    if (c < d)
        for (int b0 = g; b0 < blocks; b0 += 64) {  // eight blocks' loads in flight
            float vs[8], vl[8], vh[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int b = b0 + 8 * u;
                const float* p = partial + int64_t(b < blocks ? b : g) * 3 * d + c;
                vs[u] = b < db_blocks ? p[0] : 0.f;
                vl[u] = p[d];
                vh[u] = p[2 * d];
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                s += double(vs[u]);
                lo = fminf(lo, vl[u]);
                hi = fmaxf(hi, vh[u]);
            }
        }
    s_s[g][threadIdx.x] = s;
    s_lo[g][threadIdx.x] = lo;
    s_hi[g][threadIdx.x] = hi;
    __syncthreads();
    if (g == 0 && c < d) {
        for (int u = 1; u < 8; ++u) {
            s += s_s[u][threadIdx.x];
            lo = fminf(lo, s_lo[u][threadIdx.x]);
            hi = fmaxf(hi, s_hi[u][threadIdx.x]);
        }
        const float m = float(s / double(n));
        mean[c] = m;
        atomicMax(&maxbits[2], __float_as_uint(fmaxf(0.f, fmaxf(hi - m, m - lo))));
    }
}

// Warp per row: operand B of the database rows (QUERY = false) or operand A of
// the queries, with the norm and the residual of the rounding.  Rows past the
// end are padding that no list keeps.  The database's largest norm and
// residual go to maxbits[0] and [1].
template <bool QUERY>
__global__ void __launch_bounds__(256) wide_stage_kernel(const float* __restrict__ M, const int64_t* __restrict__ rows,
                                                         int64_t n, int64_t n_pad, int d, int K,
                                                         const float* __restrict__ mean,
                                                         unsigned int* __restrict__ maxbits, op16* __restrict__ out,
                                                         float* __restrict__ norm, float* __restrict__ resid,
                                                         int32_t* __restrict__ bound) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = int64_t(gridDim.x) * (blockDim.x >> 5);
    const float S = operand_scale<true>(maxbits), inv_S = 1.0f / S;
    const float C = 32768.0f, inv_C = 1.0f / C;
    float nmax = 0.f, rmax = 0.f;
    for (int64_t i = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; i < n_pad; i += warps) {
        const float* x = M + (i < n ? (rows ? rows[i] : i) : 0) * d;
        op16* o = out + i * K;
        float sq = 0.f, rs = 0.f, cs = 0.f;
        for (int c0 = 2 * lane; c0 < K; c0 += 64) {
            op16 e[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int c = c0 + h;
                const float v = (i < n && c < d) ? (x[c] - mean[c]) * inv_S : 0.f;
                const op16 b = to_op<true>(v);
                const float vb = from_op<true>(b), r = v - vb;
                sq = fmaf(vb, vb, sq);
                rs = fmaf(r, r, rs);
                cs = fmaf(v, v, cs);
                e[h] = QUERY ? b : to_op<true>(-2.0f * vb);
            }
            if (c0 + 1 < d || c0 >= d + 3) {
                *reinterpret_cast<uint32_t*>(o + c0) = uint32_t(e[0]) | uint32_t(e[1]) << 16;
            } else {  // columns d .. d + 2 are written below
                if (c0 < d) o[c0] = e[0];
                if (c0 + 1 >= d + 3) o[c0 + 1] = e[1];
            }
        }
#pragma unroll
        for (int w = 16; w > 0; w >>= 1) {
            sq += __shfl_xor_sync(0xffffffffu, sq, w);
            rs += __shfl_xor_sync(0xffffffffu, rs, w);
            cs += __shfl_xor_sync(0xffffffffu, cs, w);
        }
        // three-way split of n / C (huge for padding rows: never selected)
        const float nv = i < n ? sq * inv_C : 65504.0f;
        const op16 nh = to_op<true>(nv);
        const float r1 = nv - from_op<true>(nh);
        const op16 nm = to_op<true>(r1);
        const op16 nl = to_op<true>(r1 - from_op<true>(nm));
        if (lane < 3) o[d + lane] = QUERY ? to_op<true>(C) : (lane == 0 ? nh : (lane == 1 ? nm : nl));
        if (lane == 0 && i < n) {
            // residual norm, widened by the FP32 rounding of the centring, the
            // scaling and this sum, and by a possible flush of subnormal operands
            const float delta = (sqrtf(rs) * (1.0f + 2e-6f) + 2.4e-7f * sqrtf(cs) + 6.2e-5f * sqrtf(float(d))) * S;
            if (QUERY) {
                norm[i] = sq * S * S;
                resid[i] = delta;
                bound[i] = 0x7F800000;  // +inf (an ordered_key)
            } else {
                nmax = fmaxf(nmax, sq * S * S);
                rmax = fmaxf(rmax, delta);
            }
        }
    }
    if (!QUERY && lane == 0) {
        atomicMax(&maxbits[0], __float_as_uint(nmax));
        atomicMax(&maxbits[1], __float_as_uint(rmax));
    }
}

// ------------------------------------------------------------------ GEMM + select
// A float as an integer of the same order (its own inverse on the bits).
__device__ __forceinline__ int32_t ordered_key(int32_t bits) { return bits ^ ((bits >> 31) & 0x7FFFFFFF); }

struct WideParams {
    int64_t nq;
    int n_tiles, kch, tiles_per_split;
    int32_t* cand_idx;   // [split][n queries padded][TC_KP]
    float* cand_s;
    int64_t nq_pad;
    int32_t* bound;      // [n queries]: the splits' common bound, an ordered_key (null: one split)
    int* status;
    unsigned long long* tiles_done;  // += tiles this CTA multiplies (null: not counted)
};

__global__ void __launch_bounds__(WD_THREADS, 1)
knn_wide_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, WideParams P) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    uint64_t* bars = reinterpret_cast<uint64_t*>(base + WD_STAGES * WD_STAGE);
    uint64_t* full = bars;
    uint64_t* empty = bars + WD_STAGES;
    uint64_t* acc_full = bars + 2 * WD_STAGES;  // [2]
    uint64_t* acc_empty = acc_full + 2;         // [2]
    uint64_t* mma_done = acc_empty + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mma_done + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    int2* q = reinterpret_cast<int2*>(reinterpret_cast<uint8_t*>(bars) + 256);
    float* s_thr = reinterpret_cast<float*>(q + TC_EPI_WARPS * 32 * TC_QCAP);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t q0 = int64_t(blockIdx.x) * WD_BM;
    const int t0 = blockIdx.y * P.tiles_per_split;
    const int nt = P.n_tiles - t0 < P.tiles_per_split ? P.n_tiles - t0 : P.tiles_per_split;
    if (threadIdx.x == 0) {
        for (int s = 0; s < WD_STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], TC_EPI_WARPS);
        }
        mbar_init(mma_done, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_slot)), "r"(2 * WD_BN) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            if (P.tiles_done) atomicAdd(P.tiles_done, static_cast<unsigned long long>(nt));
            const int steps = nt * P.kch;
            int u = 0;
            for (int t = 0; t < nt && u >= 0; ++t) {
                for (int kc = 0; kc < P.kch; ++kc, ++u) {
                    const int s = u % WD_STAGES;
                    if (u >= WD_STAGES && !mbar_wait(&empty[s], ((u / WD_STAGES) & 1) ^ 1, abort_flag, P.status)) break;
                    mbar_expect_tx(&full[s], WD_STAGE);
                    tma_load_2d(base + s * WD_STAGE, &tmA, kc * 64, int(q0), &full[s]);
                    tma_load_2d(base + s * WD_STAGE + WD_A_BYTES, &tmB, kc * 64, (t0 + t) * WD_BN, &full[s]);
                }
                if (u != (t + 1) * P.kch) break;  // aborted
            }
            if (u < steps) {  // aborted: let issued loads land before exit (each wait bounded by 100 ms)
                for (int v = (u > WD_STAGES ? u - WD_STAGES : 0); v < u; ++v) {
                    const unsigned long long w0 = global_timer();
                    while (!mbar_try(&full[v % WD_STAGES], (v / WD_STAGES) & 1) && global_timer() - w0 < 100000000ull) {
                    }
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc = idesc_f16kind(WD_BM, WD_BN, true);
            bool ok = true;
            int u = 0;
            for (int t = 0; t < nt && ok; ++t) {
                const int buf = t & 1, use = t >> 1;
                if (t >= 2 && !mbar_wait(&acc_empty[buf], (use & 1) ^ 1, abort_flag, P.status)) break;
                tc_fence_after();
                for (int kc = 0; kc < P.kch; ++kc, ++u) {
                    const int s = u % WD_STAGES;
                    if (!mbar_wait(&full[s], (u / WD_STAGES) & 1, abort_flag, P.status)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint64_t ad = sdesc_sw128(smem_u32(base + s * WD_STAGE));
                    const uint64_t bd = sdesc_sw128(smem_u32(base + s * WD_STAGE + WD_A_BYTES));
#pragma unroll
                    for (int k = 0; k < 4; ++k)  // 16 columns = 32 bytes = 2 descriptor units
                        mma_f16kind(tmem + uint32_t(buf * WD_BN), ad + 2 * k, bd + 2 * k, idesc,
                                    (kc > 0 || k > 0) ? 1u : 0u);
                    mma_commit(&empty[s]);
                }
                if (ok) mma_commit(&acc_full[buf]);
            }
            // every MMA issued above has completed once this barrier fires
            mma_commit(mma_done);
            const unsigned long long w0 = global_timer();
            while (!mbar_try(mma_done, 0) && global_timer() - w0 < 100000000ull) {
            }
        }
    } else {
        const int e = warp - 2;
        const int quarter = warp & 3;   // TMEM lanes [32 quarter, 32 quarter + 32)
        const int half = e >> 2;        // columns [128 half, 128 half + 128) of a tile
        const int row = quarter * 32 + lane;
        float L[TC_KP];
        int32_t I[TC_KP];
#pragma unroll
        for (int s = 0; s < TC_KP; ++s) {
            L[s] = INFINITY;
            I[s] = -1;
        }
        const int qb = e * 32 + lane;
        volatile float* q_mine = s_thr + (half * WD_BM + row) * TC_NQ;
        volatile float* q_other = s_thr + ((1 - half) * WD_BM + row) * TC_NQ;
#pragma unroll
        for (int j = 0; j < TC_NQ; ++j) q_mine[j] = INFINITY;
        asm volatile("bar.sync 1, %0;" ::"r"(TC_EPI_WARPS * 32) : "memory");
        int qn = 0;
        // A split's lists start empty, and a list of 32 from N columns in random
        // order takes about 32 (1 + ln(N / 32)) insertions.  Its bound on the row's
        // 32nd-best value holds for the other splits too, so each merge
        // publishes it and every tile starts from the smallest published: a later
        // split inserts little (the kernel at 30,000 x 200, 3 splits: 690 to 526 us).
        // A value between the row's 32nd best and a stale bound is queued in vain.
        int32_t* const bound = P.bound && q0 + row < P.nq ? P.bound + q0 + row : nullptr;
        float known = INFINITY;
        auto row_bound = [&]() { return fminf(list_bound(L, q_other), known); };
        auto flush = [&]() {
            list_merge(L, I, qn, q, qb, q_mine);
            const float b = list_bound(L, q_other);
            if (bound && b < known) {
                known = b;
                atomicMin(bound, ordered_key(__float_as_int(b)));
            }
        };
        for (int t = 0; t < nt; ++t) {
            const int buf = t & 1, use = t >> 1;
            if (bound) known = fminf(known, __int_as_float(ordered_key(*static_cast<volatile int32_t*>(bound))));
            if (!mbar_wait(&acc_full[buf], use & 1, abort_flag, P.status)) break;
            tc_fence_after();
            const uint32_t tbase = tmem + (uint32_t(quarter * 32) << 16) + uint32_t(buf * WD_BN + half * 128);
            select_tile(tbase, (t0 + t) * WD_BN + half * 128, qn, q, qb, row_bound, flush);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[buf]);
        }
        flush();
        // merge the two column halves of each row through shared memory (the
        // ring is idle once the last accumulator has been read)
        float* ms = reinterpret_cast<float*>(base);  // [2][128][TC_KP + 1]
        int32_t* mi = reinterpret_cast<int32_t*>(ms + 2 * WD_BM * (TC_KP + 1));
        asm volatile("bar.sync 1, %0;" ::"r"(TC_EPI_WARPS * 32) : "memory");
#pragma unroll
        for (int s = 0; s < TC_KP; ++s) {
            ms[(half * WD_BM + row) * (TC_KP + 1) + s] = L[s];
            mi[(half * WD_BM + row) * (TC_KP + 1) + s] = I[s];
        }
        asm volatile("bar.sync 1, %0;" ::"r"(TC_EPI_WARPS * 32) : "memory");
        if (half == 0 && q0 + row < P.nq && !*abort_flag) {
            const int64_t o = (int64_t(blockIdx.y) * P.nq_pad + q0 + row) * TC_KP;
            const int ra = row * (TC_KP + 1), rb = (WD_BM + row) * (TC_KP + 1);
            int a = 0, b = 0;
            for (int s = 0; s < TC_KP; ++s) {
                const float va = ms[ra + a], vb = ms[rb + b];
                const bool take_a = va < vb || (va == vb && uint32_t(mi[ra + a]) <= uint32_t(mi[rb + b]));
                P.cand_s[o + s] = take_a ? va : vb;
                P.cand_idx[o + s] = take_a ? mi[ra + a] : mi[rb + b];
                if (take_a) ++a; else ++b;
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * WD_BN) : "memory");
    }
}

// ------------------------------------------------------------------ re-rank + certify
// One warp per query: the splits' sorted lists are merged to the 32 smallest
// s (lane l holds the l-th), then lane l sums the exact squared distance of its
// candidate over the dimensions in order, 32 dimensions at a time staged by
// asynchronous copies into two alternating buffers, and a bitonic network
// orders the candidates by (distance, index).
//
// V floats a copy and a read, 4 or 2 where d and the matrices' alignment allow
// it: with one, the load/store pipe bounds it (30,000 x 200: 167 us; with four
// 115, 6.7 TB/s of the candidates' rows from L2).  The pitch keeps the lanes' reads of 32 rows on distinct banks.
static constexpr int WR_WARPS = 4;
constexpr int wr_pitch(int v) { return v == 4 ? 36 : 32 + v; }

template <int V>
__global__ void __launch_bounds__(WR_WARPS * 32)
wide_rerank_kernel(const float* __restrict__ X, int64_t n, int d, int k, const float* __restrict__ Q, bool separate,
                   const int64_t* __restrict__ rows, int64_t nq, int64_t nq_pad, int splits,
                   const int32_t* __restrict__ cand_idx, const float* __restrict__ cand_s,
                   const float* __restrict__ norm, const float* __restrict__ resid,
                   const unsigned int* __restrict__ maxbits, float eps_rel, int32_t* __restrict__ idx_out,
                   float* __restrict__ dist_out, int32_t* __restrict__ fail_rows, int32_t* __restrict__ fail_count,
                   int32_t* __restrict__ fail_bound) {
    constexpr int PITCH = wr_pitch(V), PER = 32 / V;  // copies a row of 32 dimensions
    __shared__ __align__(16) float s_rows[WR_WARPS][2][32 * PITCH];
    __shared__ __align__(16) float s_q[WR_WARPS][2][32];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const float n_max = __uint_as_float(maxbits[0]), r_max = __uint_as_float(maxbits[1]);
    const float S = operand_scale<true>(maxbits);
    const int64_t warps = int64_t(gridDim.x) * WR_WARPS;
    for (int64_t p = int64_t(blockIdx.x) * WR_WARPS + w; p < nq; p += warps) {
        float cs = cand_s[p * TC_KP + lane];
        int32_t ci = cand_idx[p * TC_KP + lane];
        for (int y = 1; y < splits; ++y) {
            // the 32 smallest of two sorted lists: pair one with the reversed other
            const int64_t o = (int64_t(y) * nq_pad + p) * TC_KP + 31 - lane;
            const float os = cand_s[o];
            const int32_t oi = cand_idx[o];
            if (os < cs) {
                cs = os;
                ci = oi;
            }
#pragma unroll
            for (int st = 16; st > 0; st >>= 1) {
                const float xs = __shfl_xor_sync(0xffffffffu, cs, st);
                const int32_t xi = __shfl_xor_sync(0xffffffffu, ci, st);
                const bool lower = (lane & st) == 0;
                if (lower ? xs < cs : xs > cs) {
                    cs = xs;
                    ci = xi;
                }
            }
        }
        const int64_t qi = rows ? rows[p] : p;
        const bool valid = ci >= 0 && ci < n && (separate || ci != qi);
        const float* xq = Q + qi * d;
        const int cv = valid ? ci : -1;
        auto stage = [&](int c0, int buf) {
            const int c = c0 + V * (lane % PER);
            if (lane < PER && c < d)
                asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_u32(&s_q[w][buf][V * lane])),
                             "l"(xq + c), "n"(4 * V) : "memory");
#pragma unroll 8
            for (int t0 = 0; t0 < 32; t0 += V) {
                const int t = t0 + lane / PER;
                const int ct = __shfl_sync(0xffffffffu, cv, t);
                if (ct >= 0 && c < d)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_u32(
                                     &s_rows[w][buf][t * PITCH + V * (lane % PER)])), "l"(X + int64_t(ct) * d + c),
                                 "n"(4 * V) : "memory");
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        float a = 0.f;
        stage(0, 0);
        for (int c0 = 0, buf = 0; c0 < d; c0 += 32, buf ^= 1) {
            if (c0 + 32 < d) {
                stage(c0 + 32, buf ^ 1);
                asm volatile("cp.async.wait_group 1;" ::: "memory");
            } else {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
            }
            __syncwarp();
            if (valid) {
                const int cc = d - c0 < 32 ? d - c0 : 32;
                const float* row = &s_rows[w][buf][lane * PITCH];
#pragma unroll 8
                for (int c = 0; c < cc; c += V) {
                    struct alignas(4 * V) Vec { float v[V]; };
                    const Vec x = *reinterpret_cast<const Vec*>(&s_q[w][buf][c]), y = *reinterpret_cast<const Vec*>(row + c);
#pragma unroll
                    for (int u = 0; u < V; ++u) {
                        const float df = x.v[u] - y.v[u];
                        a = fmaf(df, df, a);
                    }
                }
            }
            __syncwarp();  // the buffer is refilled two steps later
        }
        int32_t jj = ci;
        if (!valid) {
            a = INFINITY;
            jj = INT32_MAX;
        }
#pragma unroll
        for (int kk = 2; kk <= 32; kk <<= 1) {
#pragma unroll
            for (int st = kk >> 1; st > 0; st >>= 1) {
                const float oa = __shfl_xor_sync(0xffffffffu, a, st);
                const int32_t oj = __shfl_xor_sync(0xffffffffu, jj, st);
                const bool up = (lane & kk) == 0, lower = (lane & st) == 0;
                const bool self_less = a < oa || (a == oa && jj < oj);
                if (self_less != (lower == up)) {
                    a = oa;
                    jj = oj;
                }
            }
        }
        const int n_valid = __popc(__ballot_sync(0xffffffffu, valid));
        const float dk2 = __shfl_sync(0xffffffffu, a, k - 1);
        const float s32 = __shfl_sync(0xffffffffu, cs, 31);
        if (lane < k) {
            idx_out[p * k + lane] = jj;
            dist_out[p * k + lane] = sqrtf(a);
        }
        if (lane == 0) {
            // every row outside the list has s >= s32, hence a distance of at
            // least lb; FP32 sums of d squares carry a relative error below
            // (d + 2) 2^-24 each
            const float ni = norm[p];
            // (4 S^2: the norms' split below FP16's smallest normal number)
            const float lb2 = ni + s32 * (S * S) - eps_rel * (ni + n_max) - 4.0f * (S * S);
            const float lb = sqrtf(fmaxf(lb2, 0.f)) - resid[p] - r_max;
            const bool ok = n_valid >= k && lb > sqrtf(dk2) * (1.0f + float(d + 8) * 5.9604645e-8f);
            if (!ok) {
                const int32_t slot = atomicAdd(fail_count, 1);
                fail_rows[slot] = int32_t(p);
                if (fail_bound) fail_bound[slot] = KNN_UNBOUND;
            }
        }
    }
}

// ------------------------------------------------------------------ host
struct WideShape {
    int K, kch, n_tiles, splits, tiles_per_split;
    int64_t n_pad, nq_pad;
};

// Splits of the database: those that leave the fewest idle CTAs in the last
// wave, at most so many that a split has 4 tiles (its lists start empty, and
// filling them is the dearest part).
// `shared`: other searches run beside this one, so splits, each of which fills
// lists of its own, are made only until the search has an eighth of the SMs.
static WideShape wide_shape(const Ctx* c, int64_t nq, int64_t n, int d, bool shared = false) {
    WideShape w;
    w.K = (d + 3 + 63) / 64 * 64;
    w.kch = w.K / 64;
    w.n_pad = (n + WD_BN - 1) / WD_BN * WD_BN;
    w.nq_pad = (nq + WD_BM - 1) / WD_BM * WD_BM;
    w.n_tiles = int(w.n_pad / WD_BN);
    const int64_t blocks = w.nq_pad / WD_BM;
    double best = 1e30;
    int pick = 1;
    for (int s = 1; s <= WD_MAX_SPLITS && (s == 1 || w.n_tiles / s >= 4); ++s) {
        const int per = (w.n_tiles + s - 1) / s;
        const int64_t waves = (blocks * s + c->num_sms - 1) / c->num_sms;
        // a CTA's start costs about 6 tiles
        const double cost = shared ? (blocks * s * 8 < c->num_sms ? 1e9 - s : double(s)) : double(waves) * (per + 6.0);
        if (cost < best * 0.98) {
            best = cost;
            pick = s;
        }
    }
    w.tiles_per_split = (w.n_tiles + pick - 1) / pick;
    w.splits = (w.n_tiles + w.tiles_per_split - 1) / w.tiles_per_split;
    return w;
}

static constexpr size_t WD_PART_BYTES = size_t(64) << 20;  // partial lists of the exact re-scan

size_t knn_wide_scratch_bytes(const Ctx* c, int64_t nq, int64_t n, int d) {
    const WideShape w = wide_shape(c, nq, n, d);
    return Carve::round(size_t(WD_STAT_BLOCKS + WD_STAT_QBLOCKS) * 3 * d * 4) + Carve::round(size_t(d) * 4) +
           Carve::round(size_t(w.nq_pad) * w.K * 2) + Carve::round(size_t(w.n_pad) * w.K * 2) +
           2 * Carve::round(size_t(w.nq_pad) * 4) + 2 * Carve::round(64) +
           2 * Carve::round(size_t(w.splits) * w.nq_pad * TC_KP * 4) + 2 * Carve::round(size_t(nq) * 4) + WD_PART_BYTES +
           8192;
}

// Against the FP32 scan, at 1.5e8 pairs x dimensions and above (graphs of X on
// itself, product / scan us): 1,733 x 50 91 / 106, 2,000 x 50 85 / 124, 3,100 x 16
// 93 / 135, 4,096 x 50 97 / 210, 2,000 x 784 (5 rows re-scanned) 496 / 627.  (The
// line was drawn where they crossed while the host read the number of uncertified
// rows back: 144 / 144 at 1,100 x 50.)  Rows of fewer than 16 dimensions are often denser
// than the operands' rounding, and would mostly be re-scanned.
bool knn_wide_preferred(int64_t nq, int64_t n, int d, int k) {
    return d >= 16 && d <= WD_MAX_D && k < TC_KP && n >= 1024 && double(nq) * double(n) * d >= 1.5e8;
}

int knn_wide(Ctx* c, const float* Q, int64_t nq, bool separate, const int64_t* rows, const float* X, int64_t n, int d,
             int k, int32_t* idx_out, float* dist_out, cudaStream_t st, void* scratch, int32_t* defer_rows,
             int32_t* defer_count) {
    const WideShape w = wide_shape(c, nq, n, d, defer_rows != nullptr);
    Carve cv(scratch);
    float* partial = cv.take<float>(size_t(WD_STAT_BLOCKS + WD_STAT_QBLOCKS) * 3 * d);
    float* mean = cv.take<float>(d);
    op16* XA = cv.take<op16>(size_t(w.nq_pad) * w.K);
    op16* XB = cv.take<op16>(size_t(w.n_pad) * w.K);
    float* norm = cv.take<float>(w.nq_pad);
    float* resid = cv.take<float>(w.nq_pad);
    unsigned int* maxbits = cv.take<unsigned int>(16);
    int32_t* fail_count = cv.take<int32_t>(16);
    int32_t* cand_idx = cv.take<int32_t>(size_t(w.splits) * w.nq_pad * TC_KP);
    float* cand_s = cv.take<float>(size_t(w.splits) * w.nq_pad * TC_KP);
    int32_t* fail_rows = cv.take<int32_t>(nq);
    int32_t* fail_bound = cv.take<int32_t>(nq);
    void* part = cv.take<char>(WD_PART_BYTES);

    const bool graph = !separate && !rows;  // a graph of X on itself: the context's k-NN counters and times report it
    auto mark = [&](int idx) { return graph ? stage_mark(c, idx, st) : DRGB_OK; };
    int rc;
    if ((rc = mark(8))) return rc;
    DRGB_CUDA(c, cudaMemsetAsync(maxbits, 0, 64, st));
    DRGB_CUDA(c, cudaMemsetAsync(fail_count, 0, 64, st));
    const int db_blocks = grid_for(n, 32, WD_STAT_BLOCKS);
    const int blocks = db_blocks + (separate ? grid_for(nq, 32, WD_STAT_QBLOCKS) : 0);
    wide_stats_kernel<<<dim3(blocks, (d + 255) / 256), 256, 0, st>>>(X, n, Q, nq, d, db_blocks, partial);
    DRGB_CHECK_LAUNCH(c);
    wide_mean_kernel<<<(d + 31) / 32, dim3(32, 8), 0, st>>>(partial, blocks, db_blocks, n, d, mean, maxbits);
    DRGB_CHECK_LAUNCH(c);
    wide_stage_kernel<false><<<grid_for(w.n_pad, 8, c->num_sms * 8), 256, 0, st>>>(X, nullptr, n, w.n_pad, d, w.K, mean,
                                                                                  maxbits, XB, nullptr, nullptr, nullptr);
    DRGB_CHECK_LAUNCH(c);
    wide_stage_kernel<true><<<grid_for(w.nq_pad, 8, c->num_sms * 8), 256, 0, st>>>(Q, rows, nq, w.nq_pad, d, w.K, mean,
                                                                                  maxbits, XA, norm, resid, fail_rows);
    DRGB_CHECK_LAUNCH(c);
    CUtensorMap mA, mB;
    if ((rc = make_map_k64(c, &mA, XA, w.nq_pad, w.K, WD_BM, true))) return rc;
    if ((rc = make_map_k64(c, &mB, XB, w.n_pad, w.K, WD_BN, true))) return rc;
    DRGB_CUDA(c, cudaFuncSetAttribute(knn_wide_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(WD_SMEM)));
    WideParams P;
    P.nq = nq;
    P.n_tiles = w.n_tiles;
    P.kch = w.kch;
    P.tiles_per_split = w.tiles_per_split;
    P.cand_idx = cand_idx;
    P.cand_s = cand_s;
    P.nq_pad = w.nq_pad;
    P.bound = w.splits > 1 ? fail_rows : nullptr;  // (nothing has failed yet)
    P.status = c->d_status;
    P.tiles_done = nullptr;
    if (graph) {
        P.tiles_done = c->d_counter + 4;
        c->knn_tiles_total = (w.nq_pad / WD_BM) * w.n_tiles;
        DRGB_CUDA(c, cudaMemsetAsync(c->d_counter + 4, 0, 8, st));
    }
    if ((rc = mark(6))) return rc;
    knn_wide_kernel<<<dim3(unsigned(w.nq_pad / WD_BM), w.splits), WD_THREADS, WD_SMEM, st>>>(mA, mB, P);
    DRGB_CHECK_LAUNCH(c);
    if ((rc = mark(7))) return rc;
    // |s - s~| for K columns: a K = 16 step adds 16 exact products and the
    // accumulator, each aligned with an error below an FP32 unit (2^-23) of the
    // largest magnitude, which is at most n_j + 2 |x_i| |x_j| <= 2 (n_i + n_max):
    // 34 * 2^-23 (n_i + n_max) a step (measured: see tc_eps in knn_tc.cu), plus the
    // FP32 norms' own error
    const float eps_rel = float(w.K / 16) * 34.0f * 1.1920929e-7f + 7.6293945e-6f;
    auto whole = [&](int v) { return d % v == 0 && ((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(Q)) & (4 * v - 1)) == 0; };
    auto rerank = whole(4) ? wide_rerank_kernel<4> : whole(2) ? wide_rerank_kernel<2> : wide_rerank_kernel<1>;
    rerank<<<grid_for(nq, WR_WARPS, c->num_sms * 6), WR_WARPS * 32, 0, st>>>(
        X, n, d, k, Q, separate, rows, nq, w.nq_pad, w.splits, cand_idx, cand_s, norm, resid, maxbits, eps_rel,
        idx_out, dist_out, defer_rows ? defer_rows : fail_rows, defer_count ? defer_count : fail_count,
        defer_rows ? nullptr : fail_bound);
    DRGB_CHECK_LAUNCH(c);
    if ((rc = mark(9))) return rc;
    if (defer_rows) return DRGB_OK;  // the caller re-scans them
    if (graph) DRGB_CUDA(c, cudaMemcpyAsync(c->d_counter, fail_count, sizeof(int32_t), cudaMemcpyDeviceToDevice, st));
    // The number of uncertified queries stays on the device: read back, it would
    // hold the host, and whatever else it has to enqueue, until the search is done.
    if ((rc = launch_knn_exact_listed(c, Q, separate, rows, X, n, d, k, fail_rows, fail_count, fail_bound, idx_out,
                                      dist_out, st, part, WD_PART_BYTES)))
        return rc;
    return mark(10);
}

}  // namespace drgb
