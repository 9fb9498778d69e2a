// Exact k-NN by an FP32 scan (SIMT), and the FP32 rank counts used by the
// trustworthiness metric.
//
// Both are one kernel (but for small databases, scan_small_kernel): a CTA takes 64 query rows and streams a chunk of the
// database through shared memory, 128 points by 32 dimensions at a time
// (transposed, two buffers filled by cp.async), and each of its 256 threads
// accumulates the squared distances of 4 queries to 8 points in registers as
// packed pairs (add.f32x2, fma.f32x2).  Squared distances are evaluated
// directly as sum_c (x_qc - x_pc)^2 in dimension order, so the result is the
// exact FP32 ranking.  A finished 64 x 128 tile goes to shared memory, where a
// warp per row compares it with the row's current k-th distance and inserts
// the few that pass into the row's sorted list (one entry per lane), ordered
// by (distance, index).
//
// Bound: FP32 issue and shared-memory reads, two packed operations per two
// pairs of points and dimension.  The earlier form, one thread per query with
// its whole list in registers, filled the GPU only from about 80,000 queries
// on; splitting the database over blockIdx.y fills it from a few hundred, and
// the partial lists are merged afterwards.  Measured, earlier form -> this one:
// 3,000 ranks and neighbours of 20,000 x 50 and its 2-D image 40.2 -> 2.4 ms, and
// 1.36 with the lists below and wider searches on the tensor cores (knn_wide.cu);
// all pairs of 30,011 x 200 40.5 -> 22.5 ms.
#include "common.cuh"
#include "knn.cuh"

namespace drgb {

static constexpr int SC_Q = 64;         // queries per CTA
static constexpr int SC_P = 128;        // points per tile
static constexpr int SC_DC = 32;        // dimensions per stage
static constexpr int SC_THREADS = 256;  // 16 x 16: 4 queries x 8 points each
static constexpr int SC_PITCH = 132;    // floats per staged dimension (128 points): transposing stores hit distinct banks
static constexpr int SC_QPITCH = 66;    // float pairs per dimension of the queries
static constexpr int SC_WARPS = SC_THREADS / 32;
static constexpr int SC_ROWS = SC_Q / SC_WARPS;  // rows a warp selects

// The cell order a SCAN_CELLS scan works on (see launch_knn_cells).
struct CellScan {
    const int32_t* rows;       // listed rows (point indices)
    const int32_t* perm;       // point at a position
    int K;
    const int32_t* cell_beg;   // [K + 1] positions
    const int32_t* chunk_beg;  // [K + 1] chunks
    const int32_t* cell_cnt;   // [K] listed rows that reach the cell
    const int32_t* cell_rows;  // [K][number of listed rows] which
};
static constexpr int64_t CELL_CHUNK = 1024;  // positions per chunk of a cell (at least)

struct ScanArgs {
    const float* X;          // n x d database
    int64_t n;
    int d;
    int k;
    const float* Q;          // query matrix (X itself unless `separate`)
    bool separate;           // Q is another matrix: no self to exclude
    const int32_t* list;     // queries scanned: list[r], or r
    const int64_t* rows;     // query p is row rows[p] of Q, or row p
    int64_t n_rows;
    int64_t chunk;           // points per blockIdx.y (a multiple of SC_P)
    const float* ub;         // see launch_knn_exact_rows_n (nullable)
    // nearest: the list of query p goes to row p of idx/dist, or (partial) to
    // list blockIdx.y of r as squared distances
    int32_t* idx;
    float* dist;
    bool partial;
    int32_t* bound;          // partial: [n_rows], the chunks' common bound as float bits (nullable)
    // listed: see scan_listed_kernel
    const int32_t* count;
    char* part;
    size_t part_bytes;
    int64_t slots;
    // cells: see launch_knn_cells
    CellScan cells;
    // ranks: targets and their squared distances (n_rows x k), counts added to
    const int32_t* tgt;
    const float* td;
    int32_t* cnt;
};

static size_t scan_smem(int d, int k, bool ranks) {
    const int qd = d <= 2 * SC_DC ? d : 2 * SC_DC, kl = k <= 16 ? 16 : 32;
    return size_t(2) * SC_DC * SC_PITCH * 4 + size_t(qd) * SC_QPITCH * 8 + size_t(SC_Q) * SC_PITCH * 4 +
           size_t(SC_Q) * kl * 8 + (SC_Q * 4) + (ranks ? size_t(SC_Q) * kl * 4 : 0);
}

// The most a scan may take.  The limit is a setting of the process: each call sets
// the same value, so that none is lowered before another thread's launch.
static int scan_smem_max(bool ranks) { return int(scan_smem(2 * SC_DC, DRGB_MAX_K, ranks)); }

__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

static constexpr int32_t SC_UNBOUND = KNN_UNBOUND;
static constexpr int SC_RANK_FEW = 24;  // points near enough to matter up to which they are walked one by one
static constexpr int SC_BULK = 6;  // candidates of 32 from which sorting them beats inserting them one by one

// One step of a sorting network over the lanes: keep the smaller (keep_min) or
// the larger, by (distance, index), of this lane's pair and lane ^ st's.
__device__ __forceinline__ void cmp_swap(float& d, int32_t& i, int st, bool keep_min) {
    const float od = __shfl_xor_sync(0xffffffffu, d, st);
    const int32_t oi = __shfl_xor_sync(0xffffffffu, i, st);
    const bool less = od < d || (od == d && oi < i);
    const bool same = od == d && oi == i;
    if (!same && less == keep_min) {
        d = od;
        i = oi;
    }
}

// The 32 smallest, by (distance, index), of a sorted list and 32 candidates, one of
// each a lane: sort the candidates, pair them with the list reversed, merge.
__device__ __forceinline__ void sorted_insert(float cd, int32_t ci, int lane, float& D, int32_t& I) {
#pragma unroll
    for (int kk = 2; kk <= 32; kk <<= 1) {
#pragma unroll
        for (int st = kk >> 1; st > 0; st >>= 1) cmp_swap(cd, ci, st, ((lane & kk) == 0) == ((lane & st) == 0));
    }
    const float od = __shfl_sync(0xffffffffu, cd, 31 - lane);
    const int32_t oi = __shfl_sync(0xffffffffu, ci, 31 - lane);
    if (od < D || (od == D && oi < I)) {
        D = od;
        I = oi;
    }
#pragma unroll
    for (int st = 16; st > 0; st >>= 1) cmp_swap(D, I, st, (lane & st) == 0);
}

// NEAREST: the k nearest of every query row in the chunk.  RANKS: for every
// target s of row r, the number of points of the chunk that precede it in the
// FP32 (distance, index) order.  CELLS: the k nearest among chunk blockIdx.y of
// a cell for the listed rows that reach the cell; X is in cell order, and a
// point's index is cells.perm of its position (ascending within a cell, so the
// order by position is the order by index).
enum { SCAN_NEAREST = 0, SCAN_RANKS = 1, SCAN_CELLS = 2 };

template <int MODE>
__device__ __forceinline__ void scan_block(const ScanArgs& A, const unsigned bx, const unsigned by) {
    constexpr bool RANK = MODE == SCAN_RANKS, CELLS = MODE == SCAN_CELLS;
    extern __shared__ __align__(16) unsigned char sc_raw[];
    const int d = A.d, k = A.k, kl = k <= 16 ? 16 : 32;
    const bool q_all = d <= 2 * SC_DC;  // the queries stay in shared memory
    float* s_x = reinterpret_cast<float*>(sc_raw);                            // [2][SC_DC][SC_PITCH]
    float2* s_q = reinterpret_cast<float2*>(s_x + 2 * SC_DC * SC_PITCH);      // [dims][SC_QPITCH], (-q, -q)
    float* s_d = reinterpret_cast<float*>(s_q + (q_all ? d : 2 * SC_DC) * SC_QPITCH);  // [SC_Q][SC_PITCH]
    float* s_ld = s_d + SC_Q * SC_PITCH;                                      // [SC_Q][kl] list (or target) distances
    int32_t* s_li = reinterpret_cast<int32_t*>(s_ld + SC_Q * kl);             // [SC_Q][kl] their indices
    int32_t* s_qi = s_li + SC_Q * kl;                                         // [SC_Q] point excluded (-1: none)
    int32_t* s_cnt = s_qi + SC_Q;                                             // RANKS: [SC_Q][kl] counts
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tx = tid & 15, ty = tid >> 4;
    const int64_t r0 = int64_t(bx) * SC_Q;
    int64_t p_begin = int64_t(by) * A.chunk;
    int64_t p_end = p_begin + A.chunk < A.n ? p_begin + A.chunk : A.n;
    int64_t n_rows = A.n_rows;
    const int32_t* list = A.list;
    if constexpr (CELLS) {
        const CellScan& S = A.cells;
        if (int(by) >= S.chunk_beg[S.K]) return;
        int C = 0;  // the cell holding this chunk: the last C with chunk_beg[C] <= by
        for (int lo = 0, hi = S.K - 1; lo <= hi;) {
            const int mid = (lo + hi) >> 1;
            if (S.chunk_beg[mid] <= int(by)) {
                C = mid;
                lo = mid + 1;
            } else {
                hi = mid - 1;
            }
        }
        n_rows = S.cell_cnt[C];
        if (r0 >= n_rows) return;
        list = S.cell_rows + int64_t(C) * A.n_rows;
        p_begin = S.cell_beg[C] + (int64_t(by) - S.chunk_beg[C]) * A.chunk;
        p_end = S.cell_beg[C + 1] - p_begin < A.chunk ? S.cell_beg[C + 1] : p_begin + A.chunk;
    }
    // where query q of this CTA goes in the outputs, and its row of Q
    auto place_of = [&](int q) -> int64_t {
        const int64_t r = r0 + q < n_rows ? r0 + q : n_rows - 1;
        return list ? int64_t(list[r]) : r;
    };
    auto query_of = [&](int q) -> int64_t {
        const int64_t p = place_of(q);
        if constexpr (CELLS) return A.cells.rows[p];
        return A.rows ? A.rows[p] : p;
    };
    // dimensions [c0, c0 + cc) of the queries, negated and doubled
    auto load_q = [&](int c0, int cc, float2* dst) {
        for (int t = tid; t < SC_Q * ((cc + 7) & ~7); t += SC_THREADS) {
            const int c = (t & 7) | ((t >> 9) << 3), q = (t >> 3) & (SC_Q - 1);
            if (c < cc) {
                const float v = -A.Q[query_of(q) * d + c0 + c];
                dst[c * SC_QPITCH + q] = make_float2(v, v);
            }
        }
    };
    static_assert(SC_Q * 8 == 512, "load_q index split");
    for (int t = tid; t < SC_Q * kl; t += SC_THREADS) {
        const int q = t / kl, s = t - q * kl;
        if (RANK) {
            const bool in = s < k && r0 + q < n_rows;
            s_cnt[t] = 0;
            s_ld[t] = in ? A.td[(r0 + q) * k + s] : -1.f;
            s_li[t] = in ? A.tgt[(r0 + q) * k + s] : -1;
        } else {
            // admission bound: the square of the k-th listed distance, rounded
            // up past the rounding of the square root and of this square, plus
            // the smallest normal number so that a k-th distance of 0 (k or
            // more exact copies of the query) still admits the points at
            // distance 0 (the test is strict)
            float T = INFINITY;
            if (A.ub) {
                const float u = A.ub[(CELLS ? query_of(q) : place_of(q)) * k + k - 1];
                T = fmaf(u * u, 1.0f + 1e-6f, 1.17549435e-38f);
                if (!(T < INFINITY)) T = INFINITY;
            }
            s_ld[t] = T;
            s_li[t] = INT32_MAX;
        }
    }
    if (tid < SC_Q) s_qi[tid] = A.separate ? -1 : int32_t(query_of(tid));
    const int nch = (d + SC_DC - 1) / SC_DC;
    const int64_t tiles = p_end > p_begin ? (p_end - p_begin + SC_P - 1) / SC_P : 0;
    const int64_t stages = tiles * nch;
    if (q_all) load_q(0, d, s_q);
    // a warp copies 8 dimensions of 4 points per instruction: whole sectors in
    // global memory, distinct banks in shared memory.  Points past the chunk
    // repeat its last point (their distances are not looked at).
    auto load_x = [&](int64_t st) {
        const int64_t tile = st / nch;
        const int c0 = int(st - tile * nch) * SC_DC;
        const int cc = d - c0 < SC_DC ? d - c0 : SC_DC;
        const int64_t p0 = p_begin + tile * SC_P;
        float* dst = s_x + (st & 1) * SC_DC * SC_PITCH;
        const int cl = tid & 7, pl = tid >> 3;
#pragma unroll
        for (int pb = 0; pb < SC_P; pb += SC_THREADS / 8) {
            const int p = pb + pl;
            const int64_t gp = p0 + p < p_end ? p0 + p : p_end - 1;
            const float* src = A.X + gp * d + c0;
#pragma unroll
            for (int cb = 0; cb < SC_DC; cb += 8) {
                const int c = cb + cl;
                if (c < cc)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(static_cast<uint32_t>(
                                     __cvta_generic_to_shared(dst + c * SC_PITCH + p))),
                                 "l"(src + c)
                                 : "memory");
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        if (!q_all) load_q(c0, cc, s_q + (st & 1) * SC_DC * SC_QPITCH);
    };
    uint64_t acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
    if (stages > 0) load_x(0);
    int ch = 0;
    int64_t p0 = p_begin;
    for (int64_t st = 0; st < stages; ++st) {
        if (st + 1 < stages) {
            load_x(st + 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        // The chunks' lists all start empty; a chunk's k-th distance bounds the
        // row's, so each chunk publishes its own and a tile admits nothing beyond the
        // smallest (points at the same distance are admitted: the index decides).
        // Read here, a lane per row of the warp, before the tile's distances.
        float known = INFINITY;
        if (MODE == SCAN_NEAREST && A.bound && ch == nch - 1 && lane < SC_ROWS && r0 + warp * SC_ROWS + lane < n_rows) {
            const int32_t b = *static_cast<volatile int32_t*>(A.bound + r0 + warp * SC_ROWS + lane);
            if (b != SC_UNBOUND) known = __int_as_float(b);
        }
        const int c0 = ch * SC_DC;
        const int cc = d - c0 < SC_DC ? d - c0 : SC_DC;
        const float* xs = s_x + (st & 1) * SC_DC * SC_PITCH + 4 * tx;
        const float2* qs = s_q + (q_all ? c0 : int(st & 1) * SC_DC) * SC_QPITCH + 4 * ty;
#pragma unroll 4
        for (int c = 0; c < cc; ++c) {
            const ulonglong2 xa = *reinterpret_cast<const ulonglong2*>(xs + c * SC_PITCH);
            const ulonglong2 xb = *reinterpret_cast<const ulonglong2*>(xs + c * SC_PITCH + 64);
            const ulonglong2 qa = *reinterpret_cast<const ulonglong2*>(qs + c * SC_QPITCH);
            const ulonglong2 qb = *reinterpret_cast<const ulonglong2*>(qs + c * SC_QPITCH + 2);
            const uint64_t xv[4] = {xa.x, xa.y, xb.x, xb.y}, qv[4] = {qa.x, qa.y, qb.x, qb.y};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint64_t df = add2(xv[j], qv[i]);
                    acc[i][j] = fma2(df, df, acc[i][j]);
                }
        }
        if (++ch == nch) {  // the tile is complete
            ch = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float* row = s_d + (4 * ty + i) * SC_PITCH + 4 * tx;
                *reinterpret_cast<ulonglong2*>(row) = make_ulonglong2(acc[i][0], acc[i][1]);
                *reinterpret_cast<ulonglong2*>(row + 64) = make_ulonglong2(acc[i][2], acc[i][3]);
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
            }
            __syncthreads();
            const int64_t left = p_end - p0;
            for (int rr = 0; rr < SC_ROWS; ++rr) {
                const int q = warp * SC_ROWS + rr;
                const float4 v4 = *reinterpret_cast<const float4*>(s_d + q * SC_PITCH + 4 * lane);
                float v[4] = {v4.x, v4.y, v4.z, v4.w};
                const int64_t self = CELLS ? -1 : s_qi[q] - p0;
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (4 * lane + j >= left || 4 * lane + j == self) v[j] = __int_as_float(0x7fc00000);  // compares false
                float* ld = s_ld + q * kl;
                int32_t* li = s_li + q * kl;
                const int32_t gp = int32_t(p0) + 4 * lane;
                if constexpr (RANK) {
                    const float tl = lane < k ? ld[lane] : -1.f;
                    float tmax = tl;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, o));
                    if (!__any_sync(0xffffffffu, v[0] <= tmax || v[1] <= tmax || v[2] <= tmax || v[3] <= tmax)) continue;
                    const int32_t jl = lane < k ? li[lane] : -1;
                    int32_t mine = 0;
                    unsigned near[4];
                    int few = 0;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        near[j] = __ballot_sync(0xffffffffu, v[j] <= tmax);
                        few += __popc(near[j]);
                    }
                    if (few <= SC_RANK_FEW) {
                        // lane s compares the few points that can precede any
                        // target with target s
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            unsigned todo = near[j];
                            while (todo) {
                                const int src = __ffs(todo) - 1;
                                todo &= todo - 1;
                                const float cd = __shfl_sync(0xffffffffu, v[j], src);
                                mine += cd < tl || (cd == tl && int32_t(p0) + 4 * src + j < jl);
                            }
                        }
                    } else {
                        for (int s = 0; s < k; ++s) {
                            const float t = __shfl_sync(0xffffffffu, tl, s);
                            const int32_t tj = __shfl_sync(0xffffffffu, jl, s);
                            int c = 0;
                            if (tj < p0) {  // every point of the tile comes after the target's index
#pragma unroll
                                for (int j = 0; j < 4; ++j) c += v[j] < t;
                            } else if (tj >= p0 + SC_P) {
#pragma unroll
                                for (int j = 0; j < 4; ++j) c += v[j] <= t;
                            } else {
#pragma unroll
                                for (int j = 0; j < 4; ++j) c += v[j] < t || (v[j] == t && gp + j < tj);
                            }
                            c = __reduce_add_sync(0xffffffffu, c);
                            if (lane == s) mine = c;
                        }
                    }
                    if (lane < k) s_cnt[q * kl + lane] += mine;  // (the warp's own rows)
                } else {
                    const float shared_k = MODE == SCAN_NEAREST ? __shfl_sync(0xffffffffu, known, rr) : INFINITY;
                    // (just above it, and no subnormal)
                    const float thr = shared_k < INFINITY
                        ? fminf(ld[k - 1], fmaxf(__int_as_float(__float_as_int(shared_k) + 1), 1.17549435e-38f)) : ld[k - 1];
                    const float m = fminf(fminf(v[0], v[1]), fminf(v[2], v[3]));  // ignores the NaN marks
                    if (!__any_sync(0xffffffffu, m < thr)) continue;
                    float D = lane < kl ? ld[lane] : INFINITY;
                    int32_t I = lane < kl ? li[lane] : INT32_MAX;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        unsigned todo = __ballot_sync(0xffffffffu, v[j] < thr);
                        if (__popc(todo) > SC_BULK) {
                            // many at once (a list that is still filling): sort
                            // the 32 and keep the 32 smallest of them and the list
                            const bool in = v[j] < thr;
                            float cd = in ? v[j] : INFINITY;
                            int32_t ci = in ? int32_t(p0) + 4 * lane + j : INT32_MAX;
                            if constexpr (CELLS) {
                                if (in) ci = A.cells.perm[ci];
                                if (ci == s_qi[q]) {
                                    cd = INFINITY;
                                    ci = INT32_MAX;
                                }
                            }
                            sorted_insert(cd, ci, lane, D, I);
                            todo = 0;
                        }
                        while (todo) {
                            const int src = __ffs(todo) - 1;
                            todo &= todo - 1;
                            const float cd = __shfl_sync(0xffffffffu, v[j], src);
                            int32_t ci = int32_t(p0) + 4 * src + j;
                            if constexpr (CELLS) {
                                ci = A.cells.perm[ci];
                                if (ci == s_qi[q]) continue;
                            }
                            // (written out: as a function this took 6% longer)
                            const bool less = D < cd || (D == cd && I < ci);
                            const int pos = __popc(__ballot_sync(0xffffffffu, less));
                            if (pos >= k) continue;  // overtaken by this tile's other points
                            const float Du = __shfl_up_sync(0xffffffffu, D, 1);
                            const int32_t Iu = __shfl_up_sync(0xffffffffu, I, 1);
                            if (lane > pos) {
                                D = Du;
                                I = Iu;
                            }
                            if (lane == pos) {
                                D = cd;
                                I = ci;
                            }
                        }
                    }
                    if (lane < kl) {
                        ld[lane] = D;
                        li[lane] = I;
                    }
                    if (MODE == SCAN_NEAREST && A.bound && lane == k - 1 && D < shared_k && r0 + q < n_rows)
                        atomicMin(A.bound + r0 + q, __float_as_int(D));
                    __syncwarp();
                }
            }
            p0 += SC_P;
        }
        __syncthreads();  // the buffer and the tile may be overwritten
    }
    if constexpr (RANK) {
        __syncthreads();
        for (int t = tid; t < SC_Q * k; t += SC_THREADS) {
            const int q = t / k, s = t - q * k;
            const int32_t c = s_cnt[q * kl + s];
            if (r0 + q < n_rows && c) atomicAdd(&A.cnt[(r0 + q) * k + s], c);
        }
    } else {
        __syncthreads();
        for (int t = tid; t < SC_Q * k; t += SC_THREADS) {
            const int q = t / k, s = t - q * k;
            const int64_t r = r0 + q;
            if (r >= n_rows) continue;
            const int64_t o = CELLS ? int64_t(by) * A.n_rows + place_of(q)
                                    : (A.partial ? int64_t(by) * A.n_rows + r : place_of(q));
            const float D = s_ld[q * kl + s];
            const int32_t I = s_li[q * kl + s];
            A.idx[o * k + s] = I == INT32_MAX ? -1 : I;
            A.dist[o * k + s] = A.partial ? D : sqrtf(D);
        }
    }
}

template <int MODE>
__global__ void __launch_bounds__(SC_THREADS, 2) scan_kernel(const ScanArgs A) {
    scan_block<MODE>(A, blockIdx.x, blockIdx.y);
}

// The k nearest of every query row in a small database: a warp a query, a point a
// lane, the list one entry a lane.
//
// Why: the tiled scan gives a CTA 64 queries, and a warp selects eight of them one
// after the other; with a few hundred points that is a chain on a few SMs.  This
// is a chain over the tiles of 32 points.  Measured (graphs, us a call, tiled / this):
// 40 x 8 46 / 15, 200 x 50 66 / 19, 512 x 50 89 / 39, 1,000 x 61 111 / 68, 1,500 x
// 61 116 / 101 (89 / 95 with 5 neighbours), 200 x 300 148 / 63, 512 x 784 323 / 351.  With
// many queries the tiles' sharing of the points tells: 20,000 queries of 1,000 x 61 and
// all that follows 578 / 512, 60,000 865 / 1,165; of 300 x 200 4,000 queries 325 / 249,
// 8,000 326 / 367.
static bool scan_is_small(int64_t n_rows, int64_t n, int d) {
    return d <= 64 ? n <= 1200 && n_rows <= 20000 : n <= 400 && n_rows <= 2000;
}
static constexpr int SS_WARPS = 4, SS_DC = 64, SS_PITCH = SS_DC + 1;

__global__ void __launch_bounds__(SS_WARPS * 32) scan_small_kernel(const ScanArgs A) {
    __shared__ float s_x[32 * SS_PITCH];          // 32 points' dimensions of a step
    __shared__ float s_q[SS_WARPS][SS_DC];
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const int d = A.d, k = A.k, n = int(A.n);
    const int64_t p = int64_t(blockIdx.x) * SS_WARPS + w;  // (the last CTA's spare warps repeat its last query)
    const int64_t r = p < A.n_rows ? p : A.n_rows - 1, q = A.rows ? A.rows[r] : r;
    const int self = A.separate ? -1 : int(q);
    float D = INFINITY;
    int32_t I = INT32_MAX;
    for (int p0 = 0; p0 < n; p0 += 32) {
        const int pts = n - p0 < 32 ? n - p0 : 32;
        float a = 0.f;
        for (int c0 = 0; c0 < d; c0 += SS_DC) {
            const int cc = d - c0 < SS_DC ? d - c0 : SS_DC;
            __syncthreads();  // the previous step has been read
            for (int t = tid; t < pts * SS_DC; t += SS_WARPS * 32) {
                const int u = t / SS_DC, c = t % SS_DC;
                if (c < cc) s_x[u * SS_PITCH + c] = A.X[int64_t(p0 + u) * d + c0 + c];
            }
            if (d > SS_DC || p0 == 0)
                for (int c = lane; c < cc; c += 32) s_q[w][c] = A.Q[q * d + c0 + c];
            __syncthreads();
#pragma unroll 8
            for (int c = 0; c < cc; ++c) {
                const float df = s_x[lane * SS_PITCH + c] - s_q[w][c];
                a = fmaf(df, df, a);
            }
        }
        const float thr = __shfl_sync(0xffffffffu, D, k - 1);
        const bool in = lane < pts && p0 + lane != self && a < thr;
        unsigned todo = __ballot_sync(0xffffffffu, in);
        if (__popc(todo) > SC_BULK) {
            sorted_insert(in ? a : INFINITY, in ? p0 + lane : INT32_MAX, lane, D, I);
            continue;
        }
        while (todo) {
            const int src = __ffs(todo) - 1;
            todo &= todo - 1;
            const float cd = __shfl_sync(0xffffffffu, a, src);
            const int32_t ci = p0 + src;
            const bool less = D < cd || (D == cd && I < ci);
            const int pos = __popc(__ballot_sync(0xffffffffu, less));
            if (pos >= k) continue;  // overtaken by this tile's other points
            const float Du = __shfl_up_sync(0xffffffffu, D, 1);
            const int32_t Iu = __shfl_up_sync(0xffffffffu, I, 1);
            if (lane > pos) {
                D = Du;
                I = Iu;
            }
            if (lane == pos) {
                D = cd;
                I = ci;
            }
        }
    }
    if (p < A.n_rows && lane < k) {
        A.idx[p * k + lane] = I == INT32_MAX ? -1 : I;
        A.dist[p * k + lane] = sqrtf(D);
    }
}

// Database chunks of a scan: enough (row block, chunk) CTAs for one to four
// whole waves of `slots` CTAs, whichever leaves the fewest idle, chunks of at
// least two tiles, the partial lists within part_bytes.
__host__ __device__ inline int scan_split(int64_t slots, int64_t n_rows, int64_t n, int k, size_t part_bytes, bool lists) {
    const int64_t blocks = (n_rows + SC_Q - 1) / SC_Q;
    int64_t best = 1;
    double best_use = 0.0;
    for (int w = 1; w <= 4; ++w) {
        const int64_t C = slots * w / blocks;
        const double use = double(blocks * C) / double(slots * w);
        if (C >= 1 && use > best_use + 0.02) {
            best = C;
            best_use = use;
        }
    }
    const int64_t most = n / (2 * SC_P);
    if (best > most) best = most;
    if (best > 128) best = 128;
    if (lists) {
        const int64_t fit = part_bytes > 1024 ? int64_t((part_bytes / 2 - 512) / (size_t(n_rows) * k * 4)) : 0;
        if (best > fit) best = fit;
    }
    return best > 1 ? int(best) : 1;
}

// Points of a chunk when the database is cut into C.
__host__ __device__ inline int64_t scan_chunk(int64_t n, int C) { return ((n + C - 1) / C + SC_P - 1) / SC_P * SC_P; }

// A scan of *A.count listed rows, a number that only the device knows: every CTA
// and the merge after it derive the split from it.  Unsplit, the lists are the
// outputs.
__device__ __forceinline__ int listed_split(ScanArgs& A, int32_t count) {
    A.n_rows = count;
    const int C = scan_split(A.slots, count, A.n, A.k, A.part_bytes, true);
    A.chunk = scan_chunk(A.n, C);
    A.partial = C > 1;
    if (!A.partial) {
        A.bound = nullptr;
        return 1;
    }
    A.idx = reinterpret_cast<int32_t*>(A.part);
    A.dist = reinterpret_cast<float*>(A.part + ((size_t(count) * C * A.k * 4 + 255) & ~size_t(255)));
    return int((A.n + A.chunk - 1) / A.chunk);
}

// CTAs take the (row block, chunk) pairs in turn; none are left where nothing is listed.
__global__ void __launch_bounds__(SC_THREADS, 2) scan_listed_kernel(const ScanArgs A0) {
    const int32_t count = *A0.count;
    if (count <= 0) return;
    ScanArgs A = A0;
    const int lists = listed_split(A, count);
    const int64_t blocks = (count + SC_Q - 1) / SC_Q;
    for (int64_t t = blockIdx.x; t < blocks * lists; t += gridDim.x) {
        scan_block<SCAN_NEAREST>(A, unsigned(t % blocks), unsigned(t / blocks));
        __syncthreads();  // the lists in shared memory have been written out
    }
}

// Merge the C partial k-lists (squared distances, ascending) of each listed
// row into its final k nearest, ordered by (distance, index).  One warp per
// row: lane l keeps the best K of the lists l, l + 32, ...; then k rounds each
// take the warp-wide smallest head by (distance, index).  The chunks cover
// disjoint index ranges, so no index appears twice.
template <int K>
__device__ __forceinline__ bool lex_less(float a, int32_t i, float b, int32_t j) {
    return a < b || (a == b && i < j);
}

template <int K>
__device__ __forceinline__ void merge_lists(const int32_t* __restrict__ pidx, const float* __restrict__ pd2,
                                            int64_t cnt, int C, int k, const int32_t* __restrict__ rows32,
                                            int32_t none, int32_t* __restrict__ idx_out, float* __restrict__ dist_out) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = int64_t(gridDim.x) * (blockDim.x >> 5);
    for (int64_t r = int64_t(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5); r < cnt; r += warps) {
        float D[K];
        int32_t I[K];
#pragma unroll
        for (int s = 0; s < K; ++s) {
            D[s] = INFINITY;
            I[s] = INT32_MAX;
        }
        for (int c0 = lane; c0 < C; c0 += 4 * 32) {
          // the heads of four lists are loaded together; a list whose head
          // is empty (-1) or not better than the current K-th is skipped
          int32_t hj[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
              const int c = c0 + u * 32;
              hj[u] = c < C ? pidx[(int64_t(c) * cnt + r) * k] : -1;
          }
#pragma unroll 1
          for (int u = 0; u < 4; ++u) {
            if (hj[u] < 0) continue;
            const int64_t base = (int64_t(c0 + u * 32) * cnt + r) * k;
            for (int s = 0; s < k; ++s) {
                const float a = pd2[base + s];
                const int32_t j = s ? pidx[base + s] : hj[u];
                if (j < 0 || !lex_less<K>(a, j, D[K - 1], I[K - 1])) break;  // each list is ascending
#pragma unroll
                for (int t = K - 1; t > 0; --t) {
                    const bool shift = lex_less<K>(a, j, D[t - 1], I[t - 1]);
                    const bool place = !shift && lex_less<K>(a, j, D[t], I[t]);
                    D[t] = shift ? D[t - 1] : (place ? a : D[t]);
                    I[t] = shift ? I[t - 1] : (place ? j : I[t]);
                }
                if (lex_less<K>(a, j, D[0], I[0])) {
                    D[0] = a;
                    I[0] = j;
                }
            }
          }
        }
        const int64_t row = rows32 ? int64_t(rows32[r]) : r;
        for (int s = 0; s < k; ++s) {
            float bd = D[0];
            int32_t bi = I[0];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const float od = __shfl_xor_sync(0xffffffffu, bd, o);
                const int32_t oi = __shfl_xor_sync(0xffffffffu, bi, o);
                if (lex_less<K>(od, oi, bd, bi)) {
                    bd = od;
                    bi = oi;
                }
            }
            if (lane == 0) {
                idx_out[row * k + s] = bi == INT32_MAX ? none : bi;
                dist_out[row * k + s] = sqrtf(bd);
            }
            if (I[0] == bi && D[0] == bd) {  // the owner pops its head
#pragma unroll
                for (int t = 0; t < K - 1; ++t) {
                    D[t] = D[t + 1];
                    I[t] = I[t + 1];
                }
                D[K - 1] = INFINITY;
                I[K - 1] = INT32_MAX;
            }
        }
    }
}

template <int K>
__global__ void merge_partials_kernel(const int32_t* __restrict__ pidx, const float* __restrict__ pd2,
                                      int64_t cnt, int C, int k, const int32_t* __restrict__ rows32,
                                      int32_t none, int32_t* __restrict__ idx_out, float* __restrict__ dist_out) {
    merge_lists<K>(pidx, pd2, cnt, C, k, rows32, none, idx_out, dist_out);
}

// The partial lists of scan_listed_kernel with the same arguments (idx and dist: the outputs).
template <int K>
__global__ void merge_listed_kernel(const ScanArgs A0, int32_t none) {
    const int32_t count = *A0.count;
    if (count <= 0) return;
    ScanArgs A = A0;
    const int lists = listed_split(A, count);
    if (A.partial) merge_lists<K>(A.idx, A.dist, count, lists, A.k, A.list, none, A0.idx, A0.dist);
}

// Two CTAs an SM.
static int scan_chunks(const Ctx* c, int64_t n_rows, int64_t n, int k, size_t part_bytes, bool lists) {
    return scan_split(2 * int64_t(c->num_sms), n_rows, n, k, part_bytes, lists);
}

size_t knn_scan_scratch_bytes(const Ctx* c, int64_t n_rows, int64_t n, int d, int k) {
    if (scan_is_small(n_rows, n, d)) return 0;
    const int C = scan_chunks(c, n_rows, n, k, ~size_t(0) >> 1, true);
    return C > 1 ? 2 * (size_t(n_rows) * C * k * 4 + 512) + size_t(n_rows) * 4 + 512 : 0;
}

template <int MODE>
static int scan_launch(Ctx* c, ScanArgs& A, int C, cudaStream_t st) {
    A.chunk = scan_chunk(A.n, C);
    const size_t smem = scan_smem(A.d, A.k, MODE == SCAN_RANKS);
    DRGB_CUDA(c, cudaFuncSetAttribute(scan_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      scan_smem_max(MODE == SCAN_RANKS)));
    const dim3 grid(unsigned((A.n_rows + SC_Q - 1) / SC_Q), unsigned((A.n + A.chunk - 1) / A.chunk));
    scan_kernel<MODE><<<grid, SC_THREADS, smem, st>>>(A);
    DRGB_CHECK_LAUNCH(c);
    return DRGB_OK;
}

// The k nearest of the queries of A, through partial lists when `part` holds
// them; `none`: the index written where a row has fewer than k.
static int scan_nearest(Ctx* c, ScanArgs& A, int32_t* idx_out, float* dist_out, void* part, size_t part_bytes,
                        int32_t none, cudaStream_t st) {
    if (A.n_rows <= 0) return DRGB_OK;
    if (scan_is_small(A.n_rows, A.n, A.d) && !A.ub && !A.list) {
        A.idx = idx_out;
        A.dist = dist_out;
        scan_small_kernel<<<unsigned((A.n_rows + SS_WARPS - 1) / SS_WARPS), SS_WARPS * 32, 0, st>>>(A);
        DRGB_CHECK_LAUNCH(c);
        return DRGB_OK;
    }
    const int C = scan_chunks(c, A.n_rows, A.n, A.k, part ? part_bytes : 0, true);
    if (C <= 1) {
        A.idx = idx_out;
        A.dist = dist_out;
        A.partial = false;
        return scan_launch<SCAN_NEAREST>(c, A, 1, st);
    }
    Carve cv(part);
    A.idx = cv.take<int32_t>(size_t(A.n_rows) * C * A.k);
    A.dist = cv.take<float>(size_t(A.n_rows) * C * A.k);
    A.partial = true;
    // with room beside the lists the chunks share their bounds
    const size_t lists_end = size_t(reinterpret_cast<char*>(cv.take<char>(0)) - static_cast<char*>(part));
    A.bound = lists_end + size_t(A.n_rows) * 4 <= part_bytes ? cv.take<int32_t>(A.n_rows) : nullptr;
    if (A.bound) DRGB_CUDA(c, cudaMemsetAsync(A.bound, SC_UNBOUND & 0xFF, size_t(A.n_rows) * 4, st));
    int rc = scan_launch<SCAN_NEAREST>(c, A, C, st);
    if (rc) return rc;
    const int lists = int((A.n + A.chunk - 1) / A.chunk);
    return launch_merge_partials(c, A.idx, A.dist, A.n_rows, lists, A.k, A.list, idx_out,
                                 dist_out, st, none);
}

// chunk_beg[C] = sum over cells c < C of ceil(|c| / CH) (one warp, K <= 128);
// the cells' row counts start at 0.
__global__ void cell_chunks_kernel(const int32_t* __restrict__ cell_beg, int K, int32_t CH,
                                   int32_t* __restrict__ chunk_beg, int32_t* __restrict__ cell_cnt) {
    int32_t carry = 0;
    for (int c0 = 0; c0 < K; c0 += 32) {
        const int c = c0 + threadIdx.x;
        const int32_t v = c < K ? (cell_beg[c + 1] - cell_beg[c] + CH - 1) / CH : 0;
        int32_t incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (int(threadIdx.x) >= o) incl += y;
        }
        if (c < K) {
            chunk_beg[c] = carry + incl - v;
            cell_cnt[c] = 0;
        }
        carry += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (threadIdx.x == 0) chunk_beg[K] = carry;
}

// The listed rows that can have one of their k nearest in cell C, for every C
// (in any order).  For a point p of C, |x_q - p| >= |x_q - c_C| - |p - c_C|;
// the FP32 values D~ of |x_q - c_C| and r~_C >= max |p - c_C| carry a relative
// error below 1e-5 each (sums of at most 61 squares), and a point that can
// enter the row's k nearest has FP32 distance <= u, exact distance <= u (1 +
// 1.1e-5).  So C is left out when D~ - r~_C - 1e-5 (D~ + r~_C) > u (1 + 2e-5).
// One warp per row, a cell per lane.
__global__ void cell_reach_kernel(const float* __restrict__ X, int d, int k, const int32_t* __restrict__ rows,
                                  int64_t cnt, int K, const float* __restrict__ cell_c,
                                  const float* __restrict__ cell_r, const float* __restrict__ dist_in,
                                  int32_t* __restrict__ cell_cnt, int32_t* __restrict__ cell_rows) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t(gridDim.x) * blockDim.x) >> 5;
    for (int64_t r = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; r < cnt; r += warps) {
        const int64_t q = rows[r];
        const float u = dist_in[q * k + k - 1];
        for (int C = lane; C < K; C += 32) {
            float sq = 0.f;
#pragma unroll 8
            for (int c = 0; c < d; ++c) {
                const float df = X[q * d + c] - cell_c[int64_t(C) * d + c];
                sq = fmaf(df, df, sq);
            }
            const float Dc = sqrtf(sq), rc = cell_r[C];
            if (Dc - rc - 1e-5f * (Dc + rc) > u * (1.0f + 2e-5f)) continue;  // false for u = INFINITY
            cell_rows[int64_t(C) * cnt + atomicAdd(&cell_cnt[C], 1)] = int32_t(r);
        }
    }
}

// Below this the five short kernels cost more than scanning all points for the
// uncertified rows does (us a call with that re-scan / this one, about a tenth of
// the rows uncertified: 4,096 x 3 263 / 325, 9,000 x 15 330 / 379, 16,500 x 61 554 / 605,
// 20,000 x 3 660 / 654, 30,000 x 2 1,122 / 965).
static constexpr int64_t CELLS_MIN_ROWS = 16384;

int launch_knn_cells(Ctx* c, const float* X, const float* Xp, int64_t n, int d, int k, const int32_t* rows,
                     int64_t cnt, int K, const int32_t* perm, const int32_t* cell_beg, const float* cell_c,
                     const float* cell_r, int32_t* idx_out, float* dist_out, cudaStream_t st, void* part,
                     size_t part_bytes, bool* done) {
    *done = false;
    // chunks of at least CELL_CHUNK positions, as many as the partial lists'
    // scratch holds (at most n / CH + K chunks in all)
    const size_t fixed = 3 * Carve::round(size_t(K + 1) * 4) + Carve::round(size_t(K) * cnt * 4) + 4096;
    const size_t per_list = size_t(cnt) * k * 8;
    if (K <= 1 || n < CELLS_MIN_ROWS || fixed >= part_bytes) return DRGB_OK;
    const int64_t max_lists = int64_t((part_bytes - fixed) / per_list) - K;
    if (max_lists <= 0) return DRGB_OK;
    int64_t CH = CELL_CHUNK;
    if (CH * max_lists < n) CH = (n + max_lists - 1) / max_lists;
    CH = (CH + SC_P - 1) / SC_P * SC_P;
    const int64_t nchunk = (n + CH - 1) / CH + K;
    if (nchunk > 65535) return DRGB_OK;
    Carve pc(part);
    int32_t* chunk_beg = pc.take<int32_t>(K + 1);
    int32_t* cell_cnt = pc.take<int32_t>(K);
    int32_t* cell_rows = pc.take<int32_t>(size_t(K) * cnt);
    ScanArgs A = {};
    A.idx = pc.take<int32_t>(size_t(cnt) * nchunk * k);
    A.dist = pc.take<float>(size_t(cnt) * nchunk * k);
    cell_chunks_kernel<<<1, 32, 0, st>>>(cell_beg, K, int32_t(CH), chunk_beg, cell_cnt);
    DRGB_CHECK_LAUNCH(c);
    DRGB_CUDA(c, cudaMemsetAsync(A.idx, 0xFF, size_t(cnt) * nchunk * k * 4, st));  // lists that no CTA writes are empty
    cell_reach_kernel<<<grid_for(cnt, 4, c->num_sms * 16), 128, 0, st>>>(X, d, k, rows, cnt, K, cell_c, cell_r, dist_out,
                                                                       cell_cnt, cell_rows);
    DRGB_CHECK_LAUNCH(c);
    A.X = Xp;
    A.Q = X;
    A.n = n;
    A.d = d;
    A.k = k;
    A.n_rows = cnt;
    A.chunk = CH;
    A.ub = dist_out;
    A.partial = true;
    A.cells = CellScan{rows, perm, K, cell_beg, chunk_beg, cell_cnt, cell_rows};
    const size_t smem = scan_smem(d, k, false);
    DRGB_CUDA(c, cudaFuncSetAttribute(scan_kernel<SCAN_CELLS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      scan_smem_max(false)));
    scan_kernel<SCAN_CELLS><<<dim3(unsigned((cnt + SC_Q - 1) / SC_Q), unsigned(nchunk)), SC_THREADS, smem, st>>>(A);
    DRGB_CHECK_LAUNCH(c);
    *done = true;
    return launch_merge_partials(c, A.idx, A.dist, cnt, int(nchunk), k, rows, idx_out, dist_out, st);
}

int launch_knn_exact_rows_n(Ctx* c, const float* X, int64_t n, int d, int k, const int32_t* rows32, int64_t cnt,
                            int32_t* idx_out, float* dist_out, cudaStream_t st, void* part_scratch,
                            size_t part_bytes) {
    ScanArgs A = {};
    A.X = A.Q = X;
    A.n = n;
    A.d = d;
    A.k = k;
    A.list = rows32;
    A.n_rows = cnt;
    A.ub = dist_out;
    return scan_nearest(c, A, idx_out, dist_out, part_scratch, part_bytes, INT32_MAX, st);
}

int launch_knn_exact_listed(Ctx* c, const float* Q, bool separate, const int64_t* rows, const float* X, int64_t n,
                            int d, int k, const int32_t* list, const int32_t* count, int32_t* bound, int32_t* idx_out,
                            float* dist_out, cudaStream_t st, void* part, size_t part_bytes) {
    ScanArgs A = {};
    A.X = X;
    A.Q = Q;
    A.separate = separate;
    A.n = n;
    A.d = d;
    A.k = k;
    A.list = list;
    A.rows = rows;
    A.count = count;
    A.ub = dist_out;
    A.idx = idx_out;
    A.dist = dist_out;
    A.bound = bound;
    A.part = static_cast<char*>(part);
    A.part_bytes = part_bytes;
    A.slots = 2 * int64_t(c->num_sms);
    const size_t smem = scan_smem(d, k, false);
    DRGB_CUDA(c, cudaFuncSetAttribute(scan_listed_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, scan_smem_max(false)));
    scan_listed_kernel<<<int(A.slots), SC_THREADS, smem, st>>>(A);
    DRGB_CHECK_LAUNCH(c);
    const int mb = c->num_sms * 4;
    if (k <= 16) merge_listed_kernel<16><<<mb, 128, 0, st>>>(A, -1);
    else merge_listed_kernel<32><<<mb, 128, 0, st>>>(A, -1);
    DRGB_CHECK_LAUNCH(c);
    return DRGB_OK;
}

int launch_merge_partials(Ctx* c, const int32_t* pidx, const float* pd2, int64_t cnt, int C, int k,
                          const int32_t* rows32, int32_t* idx_out, float* dist_out, cudaStream_t st, int32_t none) {
    if (cnt <= 0) return DRGB_OK;
    const int mb = grid_for(cnt, 4, c->num_sms * 8);   // one warp per row, 4 warps per CTA
    if (k <= 16)
        merge_partials_kernel<16><<<mb, 128, 0, st>>>(pidx, pd2, cnt, C, k, rows32, none, idx_out, dist_out);
    else
        merge_partials_kernel<32><<<mb, 128, 0, st>>>(pidx, pd2, cnt, C, k, rows32, none, idx_out, dist_out);
    DRGB_CHECK_LAUNCH(c);
    return DRGB_OK;
}

int launch_knn_scan(Ctx* c, const float* Q, int64_t nq, bool separate, const int64_t* rows, const float* X, int64_t n,
                    int d, int k, int32_t* idx_out, float* dist_out, cudaStream_t st, void* part, size_t part_bytes) {
    ScanArgs A = {};
    A.X = X;
    A.Q = Q;
    A.separate = separate;
    A.n = n;
    A.d = d;
    A.k = k;
    A.rows = rows;
    A.n_rows = nq;
    return scan_nearest(c, A, idx_out, dist_out, part, part_bytes, -1, st);
}

size_t knn_queries_scratch_bytes(const Ctx* c, int64_t nq, int64_t n, int d, int k) {
    return knn_wide_preferred(nq, n, d, k) ? knn_wide_scratch_bytes(c, nq, n, d) : knn_scan_scratch_bytes(c, nq, n, d, k);
}

int knn_queries(Ctx* c, const float* Q, int64_t nq, bool separate, const int64_t* rows, const float* X, int64_t n,
                int d, int k, int32_t* idx_out, float* dist_out, cudaStream_t st, void* scratch,
                size_t scratch_bytes) {
    if (knn_wide_preferred(nq, n, d, k) && scratch && scratch_bytes >= knn_wide_scratch_bytes(c, nq, n, d))
        return knn_wide(c, Q, nq, separate, rows, X, n, d, k, idx_out, dist_out, st, scratch);
    return launch_knn_scan(c, Q, nq, separate, rows, X, n, d, k, idx_out, dist_out, st, scratch, scratch_bytes);
}

// Squared distances of the targets, by the scan's formula and order (-1 for a
// missing target, which then precedes nothing).
__global__ void target_dist_kernel(const float* __restrict__ X, int d, int k, const int64_t* __restrict__ rows,
                                   int64_t n_rows, const int32_t* __restrict__ tgt, float* __restrict__ td,
                                   int32_t* __restrict__ cnt) {
    for (int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; t < n_rows * k;
         t += int64_t(gridDim.x) * blockDim.x) {
        const int64_t r = t / k, qi = rows ? rows[r] : r;
        const int32_t j = tgt[t];
        float a = -1.f;
        if (j >= 0) {
            a = 0.f;
#pragma unroll 8
            for (int c = 0; c < d; ++c) {
                const float df = X[qi * d + c] - X[int64_t(j) * d + c];
                a = fmaf(df, df, a);
            }
        }
        td[t] = a;
        cnt[t] = 0;
    }
}

__global__ void rank_excess_kernel(const int32_t* __restrict__ cnt, const int32_t* __restrict__ tgt, int64_t n_rows,
                                   int k, int64_t* __restrict__ excess_out) {
    for (int64_t r = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; r < n_rows; r += int64_t(gridDim.x) * blockDim.x) {
        int64_t ex = 0;
        for (int s = 0; s < k; ++s)
            if (tgt[r * k + s] >= 0 && cnt[r * k + s] + 1 > k) ex += cnt[r * k + s] + 1 - k;
        excess_out[r] = ex;
    }
}

int launch_rank(Ctx* c, const float* X, int64_t n, int d, int k, const int64_t* rows, int64_t n_rows,
                const int32_t* tgt, float* td, int32_t* cnt, int64_t* excess_out, cudaStream_t st) {
    if (n_rows <= 0) return DRGB_OK;
    target_dist_kernel<<<grid_for(n_rows * k, 128, c->num_sms * 16), 128, 0, st>>>(X, d, k, rows, n_rows, tgt, td, cnt);
    DRGB_CHECK_LAUNCH(c);
    ScanArgs A = {};
    A.X = A.Q = X;
    A.n = n;
    A.d = d;
    A.k = k;
    A.rows = rows;
    A.n_rows = n_rows;
    A.tgt = tgt;
    A.td = td;
    A.cnt = cnt;
    int rc = scan_launch<SCAN_RANKS>(c, A, scan_chunks(c, n_rows, n, k, 0, false), st);
    if (rc) return rc;
    rank_excess_kernel<<<grid_for(n_rows, 128, c->num_sms * 8), 128, 0, st>>>(cnt, tgt, n_rows, k, excess_out);
    DRGB_CHECK_LAUNCH(c);
    return DRGB_OK;
}

__global__ void nonfinite_scan_kernel(const float* __restrict__ X, int64_t count, int* status) {
    bool bad = false;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < count;
         i += int64_t(gridDim.x) * blockDim.x)
        bad |= !isfinite(X[i]);
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) report_status(status, DRGB_ERR_NONFINITE);
}

int launch_nonfinite_scan(Ctx* c, const float* X, int64_t count, cudaStream_t st) {
    nonfinite_scan_kernel<<<grid_for(count, 256, c->num_sms * 8), 256, 0, st>>>(X, count, c->d_status);
    DRGB_CHECK_LAUNCH(c);
    return DRGB_OK;
}

int check_knn_args(Ctx* c, const float* X, int64_t n, int d, int k, const void* idx_out,
                   const void* dist_out) {
    if (!c) return DRGB_ERR_INVALID;
    if (!X || !idx_out || !dist_out) return set_error(c, DRGB_ERR_INVALID, "knn_graph: NULL pointer");
    if (!aligned(X, 4)) return set_error(c, DRGB_ERR_INVALID, "knn_graph: X must be 4-byte aligned");
    if (k < 1 || k > DRGB_MAX_K || d < 1 || n < int64_t(k) + 1 || n > INT32_MAX)
        return set_error(c, DRGB_ERR_INVALID, "knn_graph: bad sizes n=%lld d=%d k=%d", (long long)n, d, k);
    return DRGB_OK;
}

}  // namespace drgb

using namespace drgb;

namespace drgb {

int knn_resolve_mode(int64_t n, int d, int k, int mode) {
    if (mode != 0) return mode;
    // The cell-ordered product (knn_tc) spends about 150 us on the order and its
    // bounds, and wins from between 16,000 and 20,000 rows on where the data has fewer
    // clusters than the order has cells (n / 2,048, at least 16): 10 clusters in 50
    // dimensions, wide / cells us: 8,000 rows 148 / 258, 16,000 265 / 301, 20,000
    // 366 / 322, 30,000 591 / 471.  With 100 clusters the bounds rule out little and
    // it loses (268 / 459 at 16,000, 886 / 1,278 at 40,000).  The clusters are not
    // known before the search, so the line is drawn by n for data of few.
    if (knn_tc_preferred(n, d, k) && (n > 16000 || !knn_wide_preferred(n, n, d, k))) return 3;
    return knn_wide_preferred(n, n, d, k) ? KNN_WIDE : 1;
}

size_t knn_scratch_bytes(const Ctx* c, int64_t n, int d, int k, int mode, size_t* least) {
    const int m = knn_resolve_mode(n, d, k, mode);
    const bool cells = m == 2 || m == 3 || (m == KNN_WIDE && knn_tc_preferred(n, d, k));
    const size_t tb = cells ? knn_tc_scratch_bytes(n, d) : 0;
    const size_t b = m == KNN_WIDE ? knn_wide_scratch_bytes(c, n, n, d) : (m == 1 ? knn_scan_scratch_bytes(c, n, n, d, k) : 0);
    if (least) *least = tb;
    return b > tb ? b : tb;
}

int knn_run(Ctx* c, const float* X, int64_t n, int d, int k, int mode, int32_t* idx_out, float* dist_out,
            cudaStream_t st, void* scratch, size_t scratch_bytes, int32_t* defer_rows, int32_t* defer_count) {
    int m = knn_resolve_mode(n, d, k, mode);
    if (m == KNN_WIDE && knn_tc_preferred(n, d, k) && scratch_bytes < knn_wide_scratch_bytes(c, n, n, d)) m = 3;
    if (m == 2 || m == 3)
        return knn_tc(c, X, n, d, k, m == 3, idx_out, dist_out, st, scratch, defer_rows, defer_count);
    if (m == KNN_WIDE && scratch && scratch_bytes >= knn_wide_scratch_bytes(c, n, n, d))
        return knn_wide(c, X, n, false, nullptr, X, n, d, k, idx_out, dist_out, st, scratch, defer_rows, defer_count);
    if (m != 1 && m != KNN_WIDE) return set_error(c, DRGB_ERR_INVALID, "knn_graph: bad mode %d", mode);
    return launch_knn_scan(c, X, n, false, nullptr, X, n, d, k, idx_out, dist_out, st, scratch, scratch_bytes);
}

}  // namespace drgb

extern "C" int drgb_knn_graph(drgb_ctx* c, const float* X, int64_t n, int32_t d, int32_t k,
                              int32_t mode, int32_t* idx_out, float* dist_out, void* stream) {
    int rc = check_knn_args(c, X, n, d, k, idx_out, dist_out);
    if (rc) return rc;
    if (mode < 0 || mode > 3) return set_error(c, DRGB_ERR_INVALID, "knn_graph: bad mode %d", mode);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int m = knn_resolve_mode(n, d, k, mode);
    auto by_cells = [&](int how) -> int {
        size_t least = 0, bytes = knn_scratch_bytes(c, n, d, k, how, &least);
        int r = ensure_scratch_within(c, &bytes, least, st);
        return r ? r : knn_run(c, X, n, d, k, how, idx_out, dist_out, st, c->scratch, c->scratch_bytes);
    };
    if (m == 2 || m == 3) return by_cells(m);
    // Sizes that the cell-ordered form takes as well fall back on it, and are refused
    // where it is (its scratch above the limit, a captured stream).
    const bool cells = m == KNN_WIDE && knn_tc_preferred(n, d, k);
    const bool captured = stream_captures(st);
    if (cells && (captured || (c->scratch_limit && knn_tc_scratch_bytes(n, d) > c->scratch_limit))) return by_cells(3);
    // The other forms can do without scratch, and what they want is a buffer of
    // their own, so that one enqueued on one stream may overlap other calls' use of
    // the context's scratch, and other searches, on another.  A captured call
    // scans unsplit (its graph may outlive the buffer); so does one that the scratch
    // limit or the device leaves no room for.
    const size_t want = captured ? 0 : (m == KNN_WIDE ? knn_wide_scratch_bytes(c, n, n, d) : knn_scan_scratch_bytes(c, n, n, d, k));
    KnnBuf* buf = nullptr;
    if (want && (rc = take_knn_buf(c, want, st, &buf))) return rc;
    if (!buf) return cells ? by_cells(3) : knn_run(c, X, n, d, k, 1, idx_out, dist_out, st, nullptr, 0);
    const bool profiling = c->profiling;
    c->profiling = false;  // the stage times are a fit's
    rc = knn_run(c, X, n, d, k, m, idx_out, dist_out, st, buf->p, want);
    c->profiling = profiling;
    DRGB_CUDA(c, cudaEventRecord(buf->ev, st));
    return rc;
}
