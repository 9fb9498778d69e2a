// Fuzzy simplicial-set graph: per-row rho/sigma and directed weights, then the
// fuzzy union of both directions as a head-sorted CSR with integer schedule
// words.  Everything is deterministic: the in-lists built with atomics are
// re-sorted by source before use, so the output does not depend on the order
// in which atomics resolved.
//
// Passes (n rows, k neighbours, m_j = in-degree of j):
//   1 rows      rho, sigma (64 bisection steps), w_{j|i}; out-list sorted by
//               column; histogram of tails, whose counts give each entry a slot
//   2 scan      in_ptr
//   3 scatter   in_src[in_ptr[j] + slot] = (i, w_{j|i})   (idx[i*k + s] = j)
//   4 sort      in-lists longer than a warp, by source
//   5 merge     union of out-list and in-list (sorted in the warp's registers)
//               by column -> tmp (cap k + m_i per row); entries kept
//               (T q >= 2^24)
//   6 scan      row_ptr
//   7 fill      col, w, q
// Passes 5 and 7 take a warp per row.  The largest weight of a graph is 1: a
// row's nearest neighbour has w = 1, and the union with 1 is 1; so q is
// round(2^24 w) without a pass for the maximum.
#include <mutex>

#include "common.cuh"
#include "graph.cuh"

namespace drgb {

static constexpr uint32_t Q_ONE = 1u << 24;

// ---------------------------------------------------------------- pass 1
// Rows are the n query points; neighbour indices lie in [0, db_n) and, when
// in_cnt is given (a graph of X on itself), must differ from the row.
//
// A thread per row, its k <= KM values in registers: the bisection is k
// exponentials and divides a step, in order.  Rows come and go through shared
// memory, so that global accesses are whole lines.  (With the values in
// indexable arrays, i.e. local memory: 136 us for 200,000 rows, 41 us for
// 2,000.)
static constexpr int FR_THREADS = 128;

// x / m, correctly rounded, from y = 1 / m correctly rounded (Markstein's
// theorem, IBM J. Res. Dev. 34, 1990: a quotient within one ulp, corrected by
// its exact remainder times y, is the correctly rounded one; two corrections,
// since x y itself may be off by more).  Straight-line code for quotients of
// one divisor: the general divide's branch keeps a row's k divides from
// overlapping (159 us for 200,000 rows, 46 us for 2,000).
__device__ __forceinline__ float quotient(float x, float m, float y) {
    float q = __fmul_rn(x, y);
    q = fmaf(fmaf(-q, m, x), y, q);
    return fmaf(fmaf(-q, m, x), y, q);
}

__device__ __forceinline__ float hw_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

template <int KM>
__global__ void __launch_bounds__(FR_THREADS)
fuzzy_rows_kernel(const int32_t* __restrict__ idx, const float* __restrict__ dist, int64_t n, int k, float target,
                  float* __restrict__ w_dir, int32_t* __restrict__ out_col, float* __restrict__ out_w,
                  float* __restrict__ rho_out, float* __restrict__ sigma_out, int* __restrict__ status, int64_t db_n,
                  int32_t* __restrict__ in_cnt, int32_t* __restrict__ slot) {
    extern __shared__ int32_t s_rows[];  // four arrays of FR_THREADS rows of `pitch` words
    const int pitch = k | 1;             // odd: the threads' rows start in distinct banks
    const int words = FR_THREADS * pitch;
    float* s_d = reinterpret_cast<float*>(s_rows);           // distances, then the weights in list order
    int32_t* s_j = s_rows + words;                           // neighbours, then the sorted columns
    float* s_w = reinterpret_cast<float*>(s_rows + 2 * words);  // their weights
    int32_t* s_s = s_rows + 3 * words;                       // slots
    const int tid = threadIdx.x;
    for (int64_t i0 = int64_t(blockIdx.x) * FR_THREADS; i0 < n; i0 += int64_t(gridDim.x) * FR_THREADS) {
        const int rows = n - i0 < FR_THREADS ? int(n - i0) : FR_THREADS;
        for (int t = tid; t < rows * k; t += FR_THREADS) {
            const int r = t / k, c = t - r * k;
            s_d[r * pitch + c] = dist[i0 * k + t];
            s_j[r * pitch + c] = idx[i0 * k + t];
        }
        __syncthreads();
        const int64_t i = i0 + tid;
        if (tid < rows) {
            float dr[KM];
            int32_t jr[KM];
            float mean = 0.f;
            bool bad = false;
#pragma unroll
            for (int s = 0; s < KM; ++s) {
                dr[s] = s < k ? s_d[tid * pitch + s] : 0.f;
                jr[s] = s < k ? s_j[tid * pitch + s] : -1;
                if (s < k) {
                    mean += dr[s];
                    bad |= !(dr[s] >= 0.f && dr[s] < INFINITY) || jr[s] < 0 || jr[s] >= db_n || (in_cnt && jr[s] == i);
                }
            }
            if (bad) report_status(status, DRGB_ERR_INVALID);
            mean /= float(k);
            const float rho = dr[0];
            // slots in the tails' in-lists (all requests in flight during the bisection)
            int32_t sl[KM];
            if (in_cnt) {
#pragma unroll
                for (int s = 0; s < KM; ++s)
                    sl[s] = s < k && jr[s] >= 0 && jr[s] < db_n && jr[s] != i ? atomicAdd(&in_cnt[jr[s]], 1) : -1;
            }
            float nx[KM];  // -max(0, d - rho)
#pragma unroll
            for (int s = 0; s < KM; ++s) nx[s] = -fmaxf(0.f, dr[s] - rho);
            // whether the quotients nx / mid (mid within 2^+-64) and their
            // remainders are all normal numbers
            bool tame = true;
#pragma unroll
            for (int s = 0; s < KM; ++s)
                if (s < k) tame = tame && (nx[s] == 0.f || (nx[s] < -8.67361738e-19f && nx[s] > -1.15292150e18f));
            float lo = 0.f, hi = INFINITY, mid = 1.f;
            for (int it = 0; it < 64; ++it) {
                float psum = 0.f;
                if (tame) {
                    const float y = __frcp_rn(mid);
                    // A sum of hardware exponentials is within 1e-4 of the
                    // precise one (each term within about 2^-20), so it decides
                    // the step unless it is that close to the target: about the
                    // first half of them.
                    const float z = 1.44269504f * y;
#pragma unroll
                    for (int s = 0; s < KM; ++s)
                        if (s < k) psum += hw_exp2(nx[s] * z);
                    if (fabsf(psum - target) <= 1e-4f) {
                        psum = 0.f;
#pragma unroll
                        for (int s = 0; s < KM; ++s)
                            if (s < k) psum += expf(quotient(nx[s], mid, y));
                    }
                } else {
#pragma unroll 1
                    for (int s = 0; s < k; ++s) psum += expf(-fmaxf(0.f, s_d[tid * pitch + s] - rho) / mid);
                }
                if (psum > target) {
                    hi = mid;
                } else {
                    lo = mid;
                }
                const float nxt = (hi == INFINITY) ? mid * 2.f : 0.5f * (lo + hi);
                // a step that leaves mid unchanged repeats itself (same test, same
                // bound): every later step would too, so the 64-step result is mid
                if (nxt == mid) break;
                mid = nxt;
            }
            const float sigma = fmaxf(mid, 1e-3f * mean);
            if (rho_out) rho_out[i] = rho;
            if (sigma_out) sigma_out[i] = sigma;
            bool dup = false;
#pragma unroll
            for (int s = 0; s < KM; ++s) {
                if (s < k) {
                    const float ex = dr[s] - rho;
                    const float w = ex > 0.f ? expf(-ex / sigma) : 1.f;
                    int rank = 0;  // place in the list sorted by column
#pragma unroll
                    for (int t = 0; t < KM; ++t) {
                        if (t < k && t != s) {
                            rank += jr[t] < jr[s] || (t < s && jr[t] == jr[s]);
                            dup |= jr[t] == jr[s];
                        }
                    }
                    s_d[tid * pitch + s] = w;
                    s_j[tid * pitch + rank] = jr[s];
                    s_w[tid * pitch + rank] = w;
                    if (in_cnt) s_s[tid * pitch + s] = sl[s];
                }
            }
            if (dup) report_status(status, DRGB_ERR_INVALID);  // a neighbour listed twice
        }
        __syncthreads();
        for (int t = tid; t < rows * k; t += FR_THREADS) {
            const int r = t / k, c = t - r * k;
            w_dir[i0 * k + t] = s_d[r * pitch + c];
            out_col[i0 * k + t] = s_j[r * pitch + c];
            out_w[i0 * k + t] = s_w[r * pitch + c];
            if (in_cnt) slot[i0 * k + t] = s_s[r * pitch + c];
        }
        __syncthreads();
    }
}

static int launch_fuzzy_rows(Ctx* c, const int32_t* idx, const float* dist, int64_t n, int k, int64_t db_n,
                             float* w_dir, int32_t* out_col, float* out_w, float* rho, float* sigma, int32_t* in_cnt,
                             int32_t* slot, cudaStream_t st) {
    const float target = float(std::log2(double(k)));
    const auto bytes = [](int list) { return size_t(4) * FR_THREADS * (list | 1) * 4; };
    const size_t smem = bytes(k);
    auto kernel = k <= 8 ? fuzzy_rows_kernel<8> : (k <= 16 ? fuzzy_rows_kernel<16> : fuzzy_rows_kernel<32>);
    // (the same for every call: a setting of the process, read by other threads' launches)
    DRGB_CUDA(c, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(bytes(DRGB_MAX_K))));
    kernel<<<grid_for(n, FR_THREADS, c->num_sms * 16), FR_THREADS, smem, st>>>(
        idx, dist, n, k, target, w_dir, out_col, out_w, rho, sigma, c->d_status, db_n, in_cnt, slot);
    DRGB_CHECK_LAUNCH(c);
    return DRGB_OK;
}

// ---------------------------------------------------------------- pass 3
// In-lists in the order of their slots (any order).  Lists longer than a warp
// are noted for pass 4: those a warp ranks from the front of long_rows, those
// a CTA sorts from its back (long_cnt counts both).
static constexpr int IS_WARP_MAX = 128;
static constexpr int IS_BIG_MAX = 8192;
static constexpr int IS_THREADS = 256;

__global__ void in_scatter_kernel(const int32_t* __restrict__ idx, int64_t n, int k,
                                  const int32_t* __restrict__ in_ptr, const int32_t* __restrict__ slot,
                                  const float* __restrict__ w_dir, int2* __restrict__ in_src,
                                  int32_t* __restrict__ long_rows, unsigned int* __restrict__ long_cnt) {
    const int64_t nk = n * k;
    for (int64_t p = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; p < nk;
         p += int64_t(gridDim.x) * blockDim.x) {
        const int32_t s = slot[p];
        if (s >= 0) in_src[in_ptr[idx[p]] + s] = make_int2(int32_t(p / k), __float_as_int(w_dir[p]));
        if (p < n) {
            const int32_t m = in_ptr[p + 1] - in_ptr[p];
            if (m > IS_WARP_MAX && m <= IS_BIG_MAX) long_rows[n - 1 - atomicAdd(&long_cnt[1], 1u)] = int32_t(p);
            else if (m > 32) long_rows[atomicAdd(&long_cnt[0], 1u)] = int32_t(p);
        }
    }
}

// ---------------------------------------------------------------- pass 4
// Ascending order of the (distinct) sources of the in-lists longer than 32, in
// place.  Up to IS_WARP_MAX: a warp ranks its elements against the whole list.
// Longer ones (hubs: at 70K the in-degree reaches 620), padded with INT32_MAX to
// a power of two, are sorted by a CTA's bitonic network in shared memory; beyond
// IS_BIG_MAX a warp ranks them in global memory (through tmp, as large as src).
__global__ void __launch_bounds__(IS_THREADS)
in_sort_kernel(const int32_t* __restrict__ in_ptr, int2* __restrict__ src, int2* __restrict__ tmp, int64_t n,
               const int32_t* __restrict__ long_rows, const unsigned int* __restrict__ long_cnt) {
    extern __shared__ __align__(16) int2 s_row[];  // [IS_BIG_MAX]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned warps = gridDim.x * (IS_THREADS / 32), few = long_cnt[0], many = long_cnt[1];
    for (unsigned r = blockIdx.x * (IS_THREADS / 32) + warp; r < few; r += warps) {
        const int32_t j = long_rows[r], b = in_ptr[j], m = in_ptr[j + 1] - b;
        if (m <= IS_WARP_MAX) {
            int32_t* list = reinterpret_cast<int32_t*>(s_row) + warp * IS_WARP_MAX;
            int2 x[IS_WARP_MAX / 32];
            int32_t rank[IS_WARP_MAX / 32];
#pragma unroll
            for (int u = 0; u < IS_WARP_MAX / 32; ++u) {
                const int a = lane + 32 * u;
                x[u] = a < m ? src[b + a] : make_int2(INT32_MAX, 0);
                list[a] = x[u].x;
                rank[u] = 0;
            }
            __syncwarp();
#pragma unroll 4
            for (int t = 0; t < m; ++t) {
                const int32_t y = list[t];
#pragma unroll
                for (int u = 0; u < IS_WARP_MAX / 32; ++u) rank[u] += y < x[u].x;
            }
#pragma unroll
            for (int u = 0; u < IS_WARP_MAX / 32; ++u)
                if (lane + 32 * u < m) src[b + rank[u]] = x[u];
            __syncwarp();
        } else {
            for (int32_t a = lane; a < m; a += 32) {
                const int2 x = src[b + a];
                int32_t rank = 0;
                for (int32_t t = 0; t < m; ++t) rank += src[b + t].x < x.x;
                tmp[b + rank] = x;
            }
            __syncwarp();
            for (int32_t a = lane; a < m; a += 32) src[b + a] = tmp[b + a];
        }
    }
    for (unsigned r = blockIdx.x; r < many; r += gridDim.x) {
        const int32_t j = long_rows[n - 1 - r], b = in_ptr[j], m = in_ptr[j + 1] - b;
        int P = 2 * IS_WARP_MAX;
        while (P < m) P <<= 1;
        __syncthreads();  // the previous lists are done with
        for (int a = threadIdx.x; a < P; a += IS_THREADS) s_row[a] = a < m ? src[b + a] : make_int2(INT32_MAX, 0);
        __syncthreads();
        for (int kk = 2; kk <= P; kk <<= 1) {
            for (int jj = kk >> 1; jj > 0; jj >>= 1) {
                for (int a = threadIdx.x; a < P; a += IS_THREADS) {
                    const int l = a ^ jj;
                    if (l > a) {
                        const int2 x = s_row[a], y = s_row[l];
                        if ((x.x > y.x) == ((a & kk) == 0)) {
                            s_row[a] = y;
                            s_row[l] = x;
                        }
                    }
                }
                __syncthreads();
            }
        }
        for (int a = threadIdx.x; a < m; a += IS_THREADS) src[b + a] = s_row[a];
    }
}

// ---------------------------------------------------------------- pass 5
__device__ __forceinline__ float fuzzy_union(float a, float b) {
    // a + b - ab, written symmetrically in (a, b) so that w_ij == w_ji exactly
    // and exactly 1 whenever either side is 1.
    const float hi = fmaxf(a, b), lo = fminf(a, b);
    return fmaf(lo, 1.0f - hi, hi);
}

__device__ __forceinline__ uint32_t schedule_word(float w) { return __float2uint_rn(float(Q_ONE) * w); }
__device__ __forceinline__ bool word_fires(uint32_t q, int T) { return uint64_t(T) * q >= Q_ONE; }

// First lane of a sorted list (one element a lane, INT32_MAX past its end)
// whose element is >= x: 0 .. 32.
__device__ __forceinline__ int warp_lower_bound(int32_t list, int32_t x) {
    int r = 0;
#pragma unroll
    for (int st = 16; st > 0; st >>= 1) {
        const int32_t y = __shfl_sync(0xffffffffu, list, r + st - 1);
        if (y < x) r += st;
    }
    const int32_t y = __shfl_sync(0xffffffffu, list, r);
    return r + (y < x);
}

// Warp per row.  Out-list entry a (lane a < k; sorted by column, entries
// reported invalid by pass 1 skipped) and in-list entry b (sorted by source,
// hence by column) go straight to their place in the union sorted by column:
// for a column x that place is #(valid out columns < x) + #(in columns < x)
// - #(columns < x present in both), and a column present in both is written
// once, by its out entry, with the fuzzy union of the two weights.  Columns
// are distinct within each list.  The counts are binary searches among the
// lanes (a walk over the other list by shuffles took 150 us for 200,000 rows,
// and a sort of every in-list before it 57).
// The next row's bounds and out-list are loaded while this one is merged.
__global__ void __launch_bounds__(256)
merge_kernel(const int32_t* __restrict__ out_col, const float* __restrict__ out_w, const int32_t* __restrict__ in_ptr,
             const int2* __restrict__ in_src, int64_t n, int k, int T, int32_t* __restrict__ tcol,
             float* __restrict__ tw, int32_t* __restrict__ tcnt, int32_t* __restrict__ keep_cnt) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const int64_t warps = int64_t(gridDim.x) * (blockDim.x >> 5);
    int64_t i = int64_t(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
    int32_t ib_n = 0, ie_n = 0, oc_n = INT32_MAX;
    float ow_n = 0.f;
    auto prefetch = [&](int64_t r) {
        if (r < n) {
            ib_n = in_ptr[r];
            ie_n = in_ptr[r + 1];
            oc_n = lane < k ? out_col[r * k + lane] : INT32_MAX;
            ow_n = lane < k ? out_w[r * k + lane] : 0.f;
        }
    };
    prefetch(i);
    for (; i < n; i += warps) {
        const int32_t ib = ib_n, m = ie_n - ib, c0 = oc_n;
        const float wa = ow_n;
        const int64_t base = i * k + ib;
        // the first 32 in entries, sorted
        int2 p = lane < m ? in_src[ib + lane] : make_int2(INT32_MAX, 0);
        prefetch(i + warps);
        if (m <= 32) {
#pragma unroll
            for (int kk = 2; kk <= 32; kk <<= 1) {
                if (kk > 16 && m <= 16) break;  // the first 16 lanes hold the list, ascending
#pragma unroll
                for (int st = kk >> 1; st > 0; st >>= 1) {
                    const int32_t o = __shfl_xor_sync(0xffffffffu, p.x, st), ow = __shfl_xor_sync(0xffffffffu, p.y, st);
                    // (the padding's keys are equal, and so are their weights)
                    const bool keep_min = ((lane & kk) == 0) == ((lane & st) == 0);
                    if (keep_min == (o < p.x)) {
                        p.x = o;
                        p.y = ow;
                    }
                }
            }
        }
        const bool va = lane < k && c0 >= 0 && c0 < n && c0 != i;
        const unsigned vmask = __ballot_sync(0xffffffffu, va);
        int32_t in_less = 0, kept = 0;
        float w_in = 0.f;
        bool matched = false;
        // out entries: in columns below c0, and c0's in weight if present
        for (int32_t t0 = 0; t0 < m; t0 += 32) {
            if (t0) p = t0 + lane < m ? in_src[ib + t0 + lane] : make_int2(INT32_MAX, 0);
            const int32_t cb = p.x;
            const float wb = __int_as_float(p.y);
            const int at = warp_lower_bound(cb, c0);
            in_less += at;
            const int32_t cm = __shfl_sync(0xffffffffu, cb, at & 31);
            const float wm = __shfl_sync(0xffffffffu, wb, at & 31);
            if (at < 32 && cm == c0 && va) {
                matched = true;
                w_in = wm;
            }
            if (m <= 32) {  // the common case: the in entries are at hand
                const unsigned mmask = __ballot_sync(0xffffffffu, matched);
                const int ao = warp_lower_bound(c0, cb);
                const int32_t co = __shfl_sync(0xffffffffu, c0, ao & 31);
                const unsigned below = ao >= 32 ? 0xffffffffu : (1u << ao) - 1u;
                const bool mine = lane < m && !(ao < 32 && co == cb && (vmask >> ao & 1u));
                if (mine) {
                    const int32_t pos = lane + __popc(vmask & below) - __popc(mmask & below);
                    tcol[base + pos] = cb;
                    tw[base + pos] = wb;
                }
                kept += __popc(__ballot_sync(0xffffffffu, mine && word_fires(schedule_word(wb), T)));
            }
        }
        const unsigned mmask = __ballot_sync(0xffffffffu, matched);
        float wv = 0.f;
        if (va) {
            const int32_t pos = __popc(vmask & lt) + in_less - __popc(mmask & lt);
            wv = matched ? fuzzy_union(wa, w_in) : wa;
            tcol[base + pos] = c0;
            tw[base + pos] = wv;
        }
        kept += __popc(__ballot_sync(0xffffffffu, va && word_fires(schedule_word(wv), T)));
        if (m > 32) {  // in entries without an out partner
            for (int32_t t0 = 0; t0 < m; t0 += 32) {
                const int32_t t = t0 + lane;
                const int2 e = t < m ? in_src[ib + t] : make_int2(INT32_MAX, 0);
                const int32_t cb = e.x;
                const float wb = __int_as_float(e.y);
                const int ao = warp_lower_bound(c0, cb);
                const int32_t co = __shfl_sync(0xffffffffu, c0, ao & 31);
                const unsigned below = ao >= 32 ? 0xffffffffu : (1u << ao) - 1u;
                const bool mine = t < m && !(ao < 32 && co == cb && (vmask >> ao & 1u));
                if (mine) {
                    const int32_t pos = t + __popc(vmask & below) - __popc(mmask & below);
                    tcol[base + pos] = cb;
                    tw[base + pos] = wb;
                }
                kept += __popc(__ballot_sync(0xffffffffu, mine && word_fires(schedule_word(wb), T)));
            }
        }
        if (lane == 0) {
            tcnt[i] = __popc(vmask) + m - __popc(mmask);
            keep_cnt[i] = kept;
        }
    }
}

// ---------------------------------------------------------------- pass 7
// Warp per row; the kept entries keep their order.  A warp loads the bounds
// and first 32 entries of FILL_ROWS rows before it writes any.
static constexpr int FILL_ROWS = 4;

__global__ void __launch_bounds__(256)
fill_kernel(const int32_t* __restrict__ in_ptr, const int32_t* __restrict__ tcol, const float* __restrict__ tw,
            const int32_t* __restrict__ tcnt, int64_t n, int k, int T, const int32_t* __restrict__ row_ptr,
            int32_t* __restrict__ col, float* __restrict__ w, uint32_t* __restrict__ q) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const int64_t warps = int64_t(gridDim.x) * (blockDim.x >> 5);
    for (int64_t i0 = (int64_t(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5)) * FILL_ROWS; i0 < n;
         i0 += warps * FILL_ROWS) {
        int64_t base[FILL_ROWS];
        int32_t cnt[FILL_ROWS], o[FILL_ROWS], cv[FILL_ROWS];
        float wv[FILL_ROWS];
#pragma unroll
        for (int u = 0; u < FILL_ROWS; ++u) {
            const int64_t i = i0 + u;
            base[u] = i < n ? i * k + in_ptr[i] : 0;
            cnt[u] = i < n ? tcnt[i] : 0;
            o[u] = i < n ? row_ptr[i] : 0;
        }
#pragma unroll
        for (int u = 0; u < FILL_ROWS; ++u) {
            wv[u] = lane < cnt[u] ? tw[base[u] + lane] : 0.f;
            cv[u] = lane < cnt[u] ? tcol[base[u] + lane] : 0;
        }
#pragma unroll
        for (int u = 0; u < FILL_ROWS; ++u) {
            for (int32_t t0 = 0; t0 < cnt[u]; t0 += 32) {
                const int32_t t = t0 + lane;
                if (t0) {
                    wv[u] = t < cnt[u] ? tw[base[u] + t] : 0.f;
                    cv[u] = t < cnt[u] ? tcol[base[u] + t] : 0;
                }
                const uint32_t qt = schedule_word(wv[u]);
                const bool keep = t < cnt[u] && word_fires(qt, T);
                const unsigned km = __ballot_sync(0xffffffffu, keep);
                if (keep) {
                    const int64_t d = o[u] + __popc(km & lt);
                    col[d] = cv[u];
                    w[d] = wv[u];
                    q[d] = qt;
                }
                o[u] += __popc(km);
            }
        }
    }
}

int launch_directed_weights(Ctx* c, const int32_t* idx, const float* dist, int64_t n, int k, int64_t db_n,
                            float* w_dir, int32_t* out_col, float* out_w, cudaStream_t st) {
    return launch_fuzzy_rows(c, idx, dist, n, k, db_n, w_dir, out_col, out_w, nullptr, nullptr, nullptr, nullptr, st);
}

size_t fuzzy_scratch_bytes(int64_t n, int k) {
    const size_t nk = size_t(n) * k;
    size_t b = 0;
    b += Carve::round(nk * 4) * 3;          // w_dir, out_col, out_w
    b += Carve::round((n + 1) * 4) * 4;     // in_cnt, in_ptr, long_rows, keep_cnt
    b += Carve::round(nk * 4) * 2;          // in_src (pairs)
    b += Carve::round(2 * nk * 4) * 2;      // tcol, tw
    b += Carve::round(n * 4);               // tcnt
    b += Carve::round(256);                 // long_cnt
    b += Carve::round(scan_scratch_elems(n) * 4);
    return b + 4096;
}

int build_fuzzy_graph(Ctx* c, const int32_t* idx, const float* dist, int64_t n, int k, int T,
                      int32_t* row_ptr, int32_t* col, float* w, uint32_t* q, float* rho,
                      float* sigma, void* scratch, cudaStream_t st) {
    const size_t nk = size_t(n) * k;
    Carve cv(scratch);
    float* w_dir = cv.take<float>(nk);
    int32_t* out_col = cv.take<int32_t>(nk);
    float* out_w = cv.take<float>(nk);
    int32_t* in_cnt = cv.take<int32_t>(n + 1);
    int32_t* in_ptr = cv.take<int32_t>(n + 1);
    int32_t* long_rows = cv.take<int32_t>(n + 1);
    int32_t* keep_cnt = cv.take<int32_t>(n + 1);
    int2* in_src = cv.take<int2>(nk);
    int32_t* tcol = cv.take<int32_t>(2 * nk);
    float* tw = cv.take<float>(2 * nk);
    int32_t* tcnt = cv.take<int32_t>(n);
    unsigned int* long_cnt = cv.take<unsigned int>(64);
    int32_t* scan_tmp = cv.take<int32_t>(scan_scratch_elems(n));
    int32_t* slot = tcol;  // free until the merge, as is the sort's
    int2* sort_tmp = reinterpret_cast<int2*>(tw);

    const int TB = 256;
    const int gmax = c->num_sms * 16;
    DRGB_CUDA(c, cudaMemsetAsync(in_cnt, 0, (n + 1) * 4, st));
    DRGB_CUDA(c, cudaMemsetAsync(long_cnt, 0, 8, st));
    int rc = launch_fuzzy_rows(c, idx, dist, n, k, n, w_dir, out_col, out_w, rho, sigma, in_cnt, slot, st);
    if (rc || (rc = exclusive_scan(c, in_cnt, in_ptr, n, scan_tmp, st))) return rc;
    in_scatter_kernel<<<grid_for(int64_t(nk), TB, gmax), TB, 0, st>>>(idx, n, k, in_ptr, slot, w_dir, in_src, long_rows,
                                                                       long_cnt);
    DRGB_CHECK_LAUNCH(c);
    DRGB_CUDA(c, cudaFuncSetAttribute(in_sort_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, IS_BIG_MAX * 8));
    in_sort_kernel<<<c->num_sms * 2, IS_THREADS, size_t(IS_BIG_MAX) * 8, st>>>(in_ptr, in_src, sort_tmp, n, long_rows,
                                                                               long_cnt);
    DRGB_CHECK_LAUNCH(c);
    merge_kernel<<<grid_for(n, TB / 32, gmax), TB, 0, st>>>(out_col, out_w, in_ptr, in_src, n, k, T, tcol, tw,
                                                           tcnt, keep_cnt);
    DRGB_CHECK_LAUNCH(c);
    if ((rc = exclusive_scan(c, keep_cnt, row_ptr, n, scan_tmp, st))) return rc;
    fill_kernel<<<grid_for(n, FILL_ROWS * TB / 32, gmax), TB, 0, st>>>(in_ptr, tcol, tw, tcnt, n, k, T, row_ptr, col, w, q);
    DRGB_CHECK_LAUNCH(c);
    return DRGB_OK;
}

}  // namespace drgb

using namespace drgb;

extern "C" int drgb_fuzzy_weights(drgb_ctx* c, const int32_t* idx, const float* dist, int64_t n,
                                  int32_t k, int32_t n_epochs, int32_t* row_ptr, int32_t* col,
                                  float* w, uint32_t* q, int64_t cap, float* rho, float* sigma,
                                  void* stream) {
    if (!c) return DRGB_ERR_INVALID;
    if (!idx || !dist || !row_ptr || !col || !w || !q)
        return set_error(c, DRGB_ERR_INVALID, "fuzzy_weights: NULL pointer");
    if (k < 1 || k > DRGB_MAX_K || n < k + 1 || n > (INT32_MAX / 2) / k || n_epochs < 1)
        return set_error(c, DRGB_ERR_INVALID, "fuzzy_weights: bad n=%lld k=%d n_epochs=%d",
                         (long long)n, k, n_epochs);
    if (cap < 2 * n * k)
        return set_error(c, DRGB_ERR_WORKSPACE, "fuzzy_weights: cap %lld < 2nk = %lld",
                         (long long)cap, (long long)(2 * n * k));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int rc = ensure_scratch(c, fuzzy_scratch_bytes(n, k), st);
    if (rc) return rc;
    return build_fuzzy_graph(c, idx, dist, n, k, n_epochs, row_ptr, col, w, q, rho, sigma,
                             c->scratch, st);
}

// ---------------------------------------------------------------------------
// Allocation-free variant.  Its scratch is this file-scope device array: every
// device that loads the library reserves it for the life of the process.  The
// first 256 bytes hold the device status word, the rest is carved exactly as
// the context scratch of drgb_fuzzy_weights.
static __device__ __align__(256) unsigned char g_fuzzy_static_scratch[DRGB_STATIC_SCRATCH_BYTES];

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_static_mutex;
void* g_static_ptr[kMaxDevices] = {};
int g_static_sms[kMaxDevices] = {};
}  // namespace

extern "C" int drgb_fuzzy_weights_static(const int32_t* idx, const float* dist, int64_t n, int32_t k,
                                         int32_t n_epochs, int32_t* row_ptr, int32_t* col, float* w,
                                         uint32_t* q, int64_t cap, float* rho, float* sigma,
                                         void* stream) {
    if (!idx || !dist || !row_ptr || !col || !w || !q) return DRGB_ERR_INVALID;
    if (k < 1 || k > DRGB_MAX_K || n < k + 1 || n > (INT32_MAX / 2) / k || n_epochs < 1) return DRGB_ERR_INVALID;
    if (cap < 2 * n * k) return DRGB_ERR_WORKSPACE;
    if (256 + fuzzy_scratch_bytes(n, k) > size_t(DRGB_STATIC_SCRATCH_BYTES)) return DRGB_ERR_WORKSPACE;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return DRGB_ERR_DEVICE;
    void* base = nullptr;
    int sms = 0;
    {
        // one-time set-up per device, with that device current: look up the
        // device address of the array (the host-side symbol is only a handle)
        std::lock_guard<std::mutex> lock(g_static_mutex);
        if (!g_static_ptr[dev]) {
            void* p = nullptr;
            if (cudaGetSymbolAddress(&p, g_fuzzy_static_scratch) != cudaSuccess || !p) {
                cudaGetLastError();
                return DRGB_ERR_CUDA;
            }
            int count = 0;
            if (cudaDeviceGetAttribute(&count, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
                cudaGetLastError();
                return DRGB_ERR_CUDA;
            }
            g_static_ptr[dev] = p;
            g_static_sms[dev] = count;
        }
        base = g_static_ptr[dev];
        sms = g_static_sms[dev];
    }
    // a stack context: no device memory of its own, status word in the array
    Ctx c;
    c.device = dev;
    c.num_sms = sms;
    c.d_status = static_cast<int*>(base);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (cudaMemsetAsync(c.d_status, 0, sizeof(int), st) != cudaSuccess) return DRGB_ERR_CUDA;
    int rc = build_fuzzy_graph(&c, idx, dist, n, k, n_epochs, row_ptr, col, w, q, rho, sigma,
                               static_cast<unsigned char*>(base) + 256, st);
    if (rc) return rc;
    if (cudaStreamSynchronize(st) != cudaSuccess) return DRGB_ERR_CUDA;
    int status = 0;
    if (cudaMemcpy(&status, c.d_status, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return DRGB_ERR_CUDA;
    return status ? status : DRGB_OK;
}
