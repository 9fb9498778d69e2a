// Per-row candidate selection shared by the tensor-core k-NN kernels: every
// epilogue thread keeps the best 32 (s, column) pairs of one row over one
// column half of the database tiles, sorted in registers.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace drgb {

static constexpr int TC_KP = 32;        // candidates kept per row
static constexpr int TC_EPI_WARPS = 8;  // epilogue warps (two per TMEM lane quarter, one per column half)
static constexpr int TC_QCAP = 32;      // per-thread candidate queue slots (one chunk)
static constexpr size_t TC_QUEUE_BYTES = size_t(TC_EPI_WARPS) * 32 * TC_QCAP * 8;
static constexpr int TC_NQ = 4;         // list quantiles a column half publishes

typedef uint16_t op16;  // raw 16-bit operand (BF16 or FP16 bits)

template <bool F16>
__device__ __forceinline__ op16 to_op(float v) {
    if constexpr (F16) return __half_as_ushort(__float2half_rn(v));
    else return __bfloat16_as_ushort(__float2bfloat16_rn(v));
}
template <bool F16>
__device__ __forceinline__ float from_op(op16 b) {
    if constexpr (F16) return __half2float(__ushort_as_half(b));
    else return __bfloat162float(__ushort_as_bfloat16(b));
}

// Power-of-two operand scale: FP16 maps max |x - mean| to at most 2^10.
template <bool F16>
__device__ __forceinline__ float operand_scale(const unsigned int* maxbits) {
    if constexpr (!F16) return 1.0f;
    const float amax = __uint_as_float(maxbits[2]);
    if (!(amax > 0.f)) return 1.0f;
    int e;
    frexpf(amax, &e);                      // amax < 2^e
    return ldexpf(1.0f, e - 10);
}

// Compare-exchange of (value, index) pairs i < l: afterwards the pair at i is
// the smaller (asc) or the larger (!asc) of the two values.
__device__ __forceinline__ void cas(float& vi, int32_t& ii, float& vl, int32_t& il, bool asc) {
    const bool sw = asc ? (vl < vi) : (vi < vl);
    const float a = vi, b = vl;
    const int32_t x = ii, y = il;
    vi = sw ? b : a;
    vl = sw ? a : b;
    ii = sw ? y : x;
    il = sw ? x : y;
}

// Bitonic merge of a bitonic sequence of N (power of two) into ascending order.
template <int N>
__device__ __forceinline__ void bitonic_merge_asc(float (&v)[N], int32_t (&ix)[N]) {
#pragma unroll
    for (int j = N / 2; j > 0; j >>= 1) {
#pragma unroll
        for (int i = 0; i < N; ++i)
            if ((i & j) == 0) cas(v[i], ix[i], v[i + j], ix[i + j], true);
    }
}

// Bitonic sort of N (power of two) into ascending order.
template <int N>
__device__ __forceinline__ void bitonic_sort_asc(float (&v)[N], int32_t (&ix)[N]) {
#pragma unroll
    for (int k = 2; k <= N; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const int l = i ^ j;
                if (l > i) cas(v[i], ix[i], v[l], ix[l], (i & k) == 0);
            }
        }
    }
}

// Three-input minimum (sm_100 and later).
__device__ __forceinline__ float min3f(float a, float b, float c) {
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Candidates below the row's threshold are appended to this thread's
// queue (slot s at q[s * 256 + tid], conflict-free).  The threshold
// is a bound on the row's 32nd-best value over both column halves:
// each half publishes the 8th, 16th, 24th and 32nd values of its
// sorted list, and for b in {0, 8, 16, 24, 32} the 32 - b smallest of
// this half's list together with the b smallest of the other's are 32
// distinct columns, so max(own[31 - b], other's b-th) bounds the
// row's 32nd-best; the threshold is the smallest of the five.  A value
// at or above it cannot be among the row's 32 best.  A stale (larger)
// published value still bounds correctly, since a list only improves.
__device__ __forceinline__ float list_bound(const float (&L)[TC_KP], const volatile float* q_other) {
    const float o8 = q_other[0], o16 = q_other[1], o24 = q_other[2], o32 = q_other[3];
    float t = fminf(L[TC_KP - 1], o32);
    t = fminf(t, fmaxf(L[23], o8));
    t = fminf(t, fmaxf(L[15], o16));
    t = fminf(t, fmaxf(L[7], o24));
    return t;
}

// When a chunk would overflow any lane's queue, all lanes merge their
// queues into their lists in lockstep: the queue (padded with +inf)
// is sorted by a bitonic network, the 32 smallest of list and queue
// are selected by pairing the list's upper half with the reversed
// queue, and a bitonic merge restores the order.
__device__ __forceinline__ void list_merge(float (&L)[TC_KP], int32_t (&I)[TC_KP], int& qn, const int2* q, int qb,
                                           volatile float* q_mine) {
    float qv[TC_QCAP];
    int32_t qi[TC_QCAP];
#pragma unroll
    for (int s = 0; s < TC_QCAP; ++s) {
        const int2 c = s < qn ? q[s * (TC_EPI_WARPS * 32) + qb] : make_int2(__float_as_int(INFINITY), -1);
        qv[s] = __int_as_float(c.x);
        qi[s] = c.y;
    }
    bitonic_sort_asc<TC_QCAP>(qv, qi);
    // the 32 smallest of L and Q: min(L[s], Q[31 - s]) is bitonic
#pragma unroll
    for (int s = 0; s < TC_KP; ++s) {
        const bool take = qv[TC_KP - 1 - s] < L[s];
        L[s] = take ? qv[TC_KP - 1 - s] : L[s];
        I[s] = take ? qi[TC_KP - 1 - s] : I[s];
    }
    bitonic_merge_asc<TC_KP>(L, I);
    qn = 0;
    q_mine[0] = L[7];
    q_mine[1] = L[15];
    q_mine[2] = L[23];
    q_mine[3] = L[TC_KP - 1];
}

// One thread's 128 columns (j0 ...) of a finished accumulator tile at TMEM
// address tbase.  bound() gives the row's threshold, flush() merges the queue.
template <class Bound, class Flush>
__device__ __forceinline__ void select_tile(uint32_t tbase, int32_t j0, int& qn, int2* q, int qb, Bound&& row_bound,
                                            Flush&& flush) {
    // the row's threshold, with the other half's quantiles read once
    // per tile (stale, larger, values still bound correctly)
    float thr_t = row_bound();
#pragma unroll 1
    for (int c = 0; c < 4; ++c) {
        float v[32];
        __syncwarp();
        tmem_ld32(tbase + c * 32, v);
        float thr = thr_t;
        float gm[4];
#pragma unroll
        for (int g = 0; g < 4; ++g)
            gm[g] = min3f(min3f(v[8 * g], v[8 * g + 1], v[8 * g + 2]),
                          min3f(v[8 * g + 3], v[8 * g + 4], v[8 * g + 5]), fminf(v[8 * g + 6], v[8 * g + 7]));
        const float m = fminf(min3f(gm[0], gm[1], gm[2]), gm[3]);
        if (__any_sync(0xffffffffu, m < thr)) {
            // room for this chunk's candidates: a bound from the groups
            // first, the exact count only when the bound overflows
            const int ub = 8 * ((gm[0] < thr) + (gm[1] < thr) + (gm[2] < thr) + (gm[3] < thr));
            if (__any_sync(0xffffffffu, qn + ub > TC_QCAP)) {
                int cnt = 0;
#pragma unroll
                for (int u = 0; u < 32; ++u) cnt += v[u] < thr ? 1 : 0;
                if (__any_sync(0xffffffffu, qn + cnt > TC_QCAP)) {
                    // the chunk is read again after the merge, which
                    // keeps its 32 values out of registers meanwhile
                    flush();
                    __syncwarp();
                    tmem_ld32(tbase + c * 32, v);
                    thr = thr_t = row_bound();
                }
            }
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                if (__any_sync(0xffffffffu, gm[g] < thr)) {
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        if (v[8 * g + u] < thr) {
                            q[qn * (TC_EPI_WARPS * 32) + qb] =
                                make_int2(__float_as_int(v[8 * g + u]), j0 + c * 32 + 8 * g + u);
                            ++qn;
                        }
                    }
                }
            }
        }
    }
}

}  // namespace drgb
