// Initialisation and the synchronous SGD epoch (the method's per-epoch step:
// attraction along active CSR entries, repulsion from Philox negatives, clip
// to +-4, Y' = Y + lr g), plus the epoch loop: one cooperative launch for small
// graphs, else a CUDA graph of one launch per epoch.
//
// Layout: Y is n x 2 FP32 read as float2 (one 8-byte gather per point); the
// CSR is head-sorted (row_ptr int32, col int32, q uint32 schedule words).
// All reads come from Y^(t); there are no atomics.
//
// An epoch is one kernel.  The rows of an instance are cut into windows by
// their first entry: window w holds the rows whose first entry lies in
// [w EPOCH_WIN, (w + 1) EPOCH_WIN) (counted from the instance's first entry).
// One warp takes a window: it compacts the active entries of the window's
// rows into shared memory, computes their forces 32 at a time (one entry per
// lane), adds each head's terms and writes Y' = Y + lr * sum for every row of
// the window.  No row crosses a window, so no row needs a second writer.
//
// Summation order of a row's force (a fixed function of the row's instance
// CSR, so results do not depend on the launch shape, the tuning or on other
// instances of a batch):
//   term(e)    = (((0 + attraction) + repulsion_0) + ...) + repulsion_{neg-1}
//   group sum  = the window's active entries, in entry order, form groups of
//                32; the terms of one head in one group are added by the
//                5-step segmented inclusive scan over the group's lanes (step d
//                adds the partial d lanes to the left)
//   force      = 0 + (((group sum_0) + group sum_1) + ...) over the groups that
//                hold the head, in order
#include <type_traits>

#include "common.cuh"
#include "epoch.cuh"
#include "knn.cuh"  // launch_nonfinite_scan

namespace drgb {

__device__ __forceinline__ unsigned long long loop_timer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__global__ void init_embedding_kernel(float2* __restrict__ Y, int64_t n, float range, uint32_t k0,
                                      uint32_t k1) {
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
         i += int64_t(gridDim.x) * blockDim.x) {
        U4 r = philox4x32_10(U4{uint32_t(i), 0u, 0u, TAG_INIT}, k0, k1);
        const float s = 5.9604644775390625e-08f;  // 2^-24
        float ux = float(r.x >> 8) * s, uy = float(r.y >> 8) * s;
        Y[i] = make_float2(fmaf(ux, 2.0f * range, -range), fmaf(uy, 2.0f * range, -range));
    }
}

__global__ void init_batched_kernel(float2* __restrict__ Y, int64_t n, float range, int count,
                                    const int64_t* __restrict__ inst_off, const uint64_t* __restrict__ inst_seed) {
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
         i += int64_t(gridDim.x) * blockDim.x) {
        int lo = 0, hi = count - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (inst_off[mid] <= i) lo = mid; else hi = mid - 1;
        }
        const uint64_t seed = inst_seed[lo];
        U4 r = philox4x32_10(U4{uint32_t(i - inst_off[lo]), 0u, 0u, TAG_INIT}, uint32_t(seed), uint32_t(seed >> 32));
        const float s = 5.9604644775390625e-08f;  // 2^-24
        float ux = float(r.x >> 8) * s, uy = float(r.y >> 8) * s;
        Y[i] = make_float2(fmaf(ux, 2.0f * range, -range), fmaf(uy, 2.0f * range, -range));
    }
}

__device__ __forceinline__ float clip4(float v) { return fminf(4.0f, fmaxf(-4.0f, v)); }

__device__ __forceinline__ float hw_ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float hw_lg2(float x) {
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// a / b as a * (1 / b) for normal b (subnormal operands count as 0).
__device__ __forceinline__ float hw_div(float a, float b) {
    float y;
    asm("div.approx.ftz.f32 %0, %1, %2;" : "=f"(y) : "f"(a), "f"(b));
    return y;
}

// Both components of a point in one packed operation.
__device__ __forceinline__ uint64_t pack2(float2 v) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(v.x), "f"(v.y));
    return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t r) {
    float2 v;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(r));
    return v;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
    return unpack2(r);
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
    return unpack2(r);
}
// a - b: the product by -1 is exact, so one rounding
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(pack2(b)), "l"(pack2(make_float2(-1.f, -1.f))), "l"(pack2(a)));
    return unpack2(r);
}

// d^b for d > 0 via the hardware base-2 logarithm and exponential.
__device__ __forceinline__ float pow_pos(float d, float b) { return hw_ex2(b * hw_lg2(d)); }

static constexpr unsigned FULL = 0xffffffffu;

// Read of one point of Y^(t).  (Read-only-path and L1 evict-last loads were
// measured and made no difference; epoch_loop_kernel must not take the former.)
__device__ __forceinline__ float2 load_y(const float2* p) { return *p; }

// Instance-local view of a row: rows [off, off + n) with entries from eoff on,
// negatives drawn under Philox key (k0, k1).  A single instance has off = 0,
// n = A.n (or the anchored negative range), eoff = 0 and the call's key.
struct RowInst {
    int64_t off;
    uint32_t n;
    int32_t eoff;
    uint32_t k0, k1;
};

// What changes from one epoch to the next: the positions read and written,
// the learning rate and the epoch number.
struct EpochStep {
    const float2* Y_in;
    float2* Y_out;
    float lr;
    uint32_t t;
};

// Negative words of entry e32 at epoch t, group g (negatives 4g .. 4g+3):
// Philox4x32-10 at counter (e, t, g, 0) under the row's key.  A single
// instance takes the precomputed round keys from the kernel parameters.
template <bool BATCHED>
__device__ __forceinline__ U4 negative_words(const EpochArgs& A, const EpochStep& S, const RowInst& R, uint32_t e32,
                                             uint32_t g) {
    if (BATCHED) return philox4x32_10(U4{e32, S.t, g, TAG_NEGATIVE}, R.k0, R.k1);
    return philox4x32_10_rk(U4{e32, S.t, g, TAG_NEGATIVE}, A.rk);
}

// Force on head i from one active entry e = (i, j) and its negatives, summed in
// the fixed order: attraction, then negatives j' = 0 .. neg-1.  NEG is the
// negative count when fixed at compile time (5, the method's default), or -1
// for any count up to 64 (A.neg).
//
// It is split in two so that a warp can gather one group's points while it
// computes the previous group's forces: draw_entry draws the first (up to
// eight) negatives, gather_entry issues the loads of Y_i, Y_j and Y_m, and
// entry_math does the arithmetic (and, for more than eight negatives, draws and gathers the
// rest itself).
//
// A skipped negative (m = i) is evaluated with Y_m = Y_i: its difference vector
// is zero, so it adds exactly +0 and needs no branch (a sum that starts at +0
// never becomes -0).  A zero distance takes d^b = 0, so coincident points
// repel with zero force as well.
template <int NEG>
struct EntryInputs {
    static constexpr int NP = NEG >= 0 ? (NEG < 8 ? NEG : 8) : 8;  // negatives drawn with the fetch
    float2 yi, yj;
    float2 ym[NP > 0 ? NP : 1];
    int32_t e;
    int32_t i;   // head row; -1 - lane for a lane without a valid entry
    bool ok;
};

// Which points an entry reads: everything that does not need Y.
template <int NEG>
struct EntryPlan {
    static constexpr int NP = EntryInputs<NEG>::NP;
    int32_t e, i;      // as in EntryInputs
    int32_t ii, jj;    // rows of Y_i and Y_j (a valid row for an invalid entry)
    uint32_t m[NP > 0 ? NP : 1];  // negatives (instance-local; a skipped one names row i)
    bool ok;
};

template <int NEG, bool BATCHED>
__device__ __forceinline__ void draw_entry(const EpochArgs& A, const EpochStep& S, const RowInst& R, bool valid,
                                           int32_t e, int32_t j, int32_t i, int64_t h_lo, int64_t h_hi, int lane,
                                           EntryPlan<NEG>& pl) {
    constexpr int NP = EntryInputs<NEG>::NP;
    const int neg = NEG >= 0 ? NEG : A.neg;
    const bool ok = valid && i >= h_lo && i < h_hi && uint64_t(uint32_t(j)) < uint64_t(A.n);
    if (valid && !ok) report_status(A.status, DRGB_ERR_INVALID);  // malformed CSR: skip the entry
    pl.ok = ok;
    pl.e = e;
    pl.i = ok ? i : -1 - lane;
    pl.ii = ok ? i : int32_t(h_lo);
    pl.jj = ok ? j : pl.ii;
    const uint32_t n32 = R.n, i32 = uint32_t(pl.ii - R.off), e32 = uint32_t(e - R.eoff);
    U4 r0{0u, 0u, 0u, 0u}, r1{0u, 0u, 0u, 0u};
    if (NP > 0 && neg > 0) r0 = negative_words<BATCHED>(A, S, R, e32, 0u);
    if (NP > 4 && neg > 4) r1 = negative_words<BATCHED>(A, S, R, e32, 1u);
    const uint32_t u[8] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
#pragma unroll
    for (int w = 0; w < NP; ++w) {
        const uint32_t m = __umulhi(u[w], n32);  // floor(u n / 2^32)
        const bool take = ok && (NEG >= 0 || w < neg) && (m != i32);
        pl.m[w] = take ? m : i32;  // a skipped negative reads Y_i
    }
}

template <int NEG>
__device__ __forceinline__ void gather_entry(const EpochStep& S, const RowInst& R, const EntryPlan<NEG>& pl,
                                             EntryInputs<NEG>& in) {
    in.ok = pl.ok;
    in.e = pl.e;
    in.i = pl.i;
    in.yi = load_y(S.Y_in + pl.ii);
    in.yj = load_y(S.Y_in + pl.jj);
    const float2* Yb = S.Y_in + R.off;
#pragma unroll
    for (int w = 0; w < EntryInputs<NEG>::NP; ++w) in.ym[w] = load_y(Yb + pl.m[w]);
}

template <int NEG, bool BATCHED>
__device__ __forceinline__ float2 entry_math(const EpochArgs& A, const EpochStep& S, const RowInst& R,
                                             const EntryInputs<NEG>& in, float two_ab, float two_b) {
    constexpr int NP = EntryInputs<NEG>::NP;
    const float2 yi = in.yi;
    float2 g = make_float2(0.f, 0.f);
    // the clipped step c (dx, dy) added to the sum, both components at once
    auto add_clipped = [&](float c, float2 df) {
        const float2 v = mul2(make_float2(c, c), df);
        g = add2(g, make_float2(clip4(v.x), clip4(v.y)));
    };
    {
        const float2 df = sub2(yi, in.yj);
        const float d = fmaf(df.x, df.x, df.y * df.y);
        // (below the smallest normal number d^b is 0, and so is the force)
        const bool far = d >= 1.17549435e-38f;
        const float pb = far ? pow_pos(d, A.b) : 0.f;
        const float c = far ? hw_div(-two_ab * pb, d * fmaf(A.a, pb, 1.0f)) : 0.f;
        add_clipped(c, df);
    }
    auto repel = [&](float2 y) {
        const float2 df = sub2(yi, y);
        const float dm = fmaf(df.x, df.x, df.y * df.y);
        // for b > 0 the hardware's log2 and exp2 give 0^b = 0 by themselves
        const float pb = (NEG >= 0 || dm > 0.f) ? pow_pos(dm, A.b) : 0.f;
        const float c = hw_div(two_b, (0.001f + dm) * fmaf(A.a, pb, 1.0f));
        add_clipped(c, df);
    };
#pragma unroll
    for (int w = 0; w < NP; ++w) repel(in.ym[w]);
    if (NEG < 0 || NEG > 8) {
        const int neg = NEG >= 0 ? NEG : A.neg;
        const uint32_t n32 = R.n, i32 = uint32_t(in.i - R.off), e32 = uint32_t(in.e - R.eoff);
        const float2* Yb = S.Y_in + R.off;
        for (int g = 2; g * 4 < neg; ++g) {
            const U4 r = negative_words<BATCHED>(A, S, R, e32, uint32_t(g));
            const uint32_t v[4] = {r.x, r.y, r.z, r.w};
            float2 yg[4];
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                const uint32_t m = __umulhi(v[w], n32);
                const bool ok = (g * 4 + w < neg) && (m != i32);
                yg[w] = ok ? load_y(Yb + m) : yi;
            }
#pragma unroll
            for (int w = 0; w < 4; ++w) repel(yg[w]);
        }
    }
    return g;
}

// ------------------------------------------------------------------ per-call preparation
// Head row of every CSR entry of rows [row_begin, n).  Entries not covered by
// any row keep -1; a row whose bounds leave [0, nnz_cap] is reported.  A warp
// takes 32 rows: where their bounds ascend, as in any well-formed CSR, it
// writes their entries 32 at a time, each lane finding its entry's row among
// the 32 by five shuffles (a thread per row, each writing its own run of
// entries, took 115 us for a million rows; now 21); otherwise each lane writes
// its own row's entries.
__global__ void epoch_heads_kernel(const int32_t* __restrict__ rp, int64_t n_rows, int64_t row_begin,
                                   int64_t nnz_cap, int32_t* __restrict__ row_of, int* status) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t(gridDim.x) * blockDim.x) >> 5;
    for (int64_t l0 = ((int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5) * 32; l0 < n_rows; l0 += warps * 32) {
        const int64_t lr = l0 + lane;
        const bool in = lr < n_rows;
        const int32_t beg = in ? rp[lr] : INT32_MAX, end = in ? rp[lr + 1] : INT32_MAX;
        const bool bad = in && (beg < 0 || end < beg || end > nnz_cap);
        if (bad) report_status(status, DRGB_ERR_INVALID);
        if (__any_sync(FULL, bad)) {
            if (in && !bad)
                for (int32_t e = beg; e < end; ++e) row_of[e] = int32_t(row_begin + lr);
            continue;
        }
        const int rows = n_rows - l0 < 32 ? int(n_rows - l0) : 32;
        const int32_t b = __shfl_sync(FULL, beg, 0), z = __shfl_sync(FULL, end, rows - 1);
        for (int32_t e0 = b; e0 < z; e0 += 32) {
            const int32_t e = e0 + lane;
            int r = 0;  // the last row of the 32 that starts at or before e
#pragma unroll
            for (int st = 16; st > 0; st >>= 1) {
                const int32_t v = __shfl_sync(FULL, beg, r + st);
                if (v <= e) r += st;
            }
            if (e < z) row_of[e] = int32_t(row_begin + l0 + r);
        }
    }
}

// Entry offsets of the instances and their window counts.
__global__ void epoch_instances_kernel(const int32_t* __restrict__ rp, const int64_t* __restrict__ inst_off,
                                       int count, int32_t* __restrict__ inst_eoff, int32_t* __restrict__ win_cnt) {
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b <= count; b += gridDim.x * blockDim.x) {
        inst_eoff[b] = rp[inst_off[b]];
        if (b < count) {
            // an instance without entries still takes one (empty) window, so
            // that its rows are written (Y + lr * 0) and no other instance's
            // window reaches into them
            const int32_t ne = rp[inst_off[b + 1]] - rp[inst_off[b]];
            win_cnt[b] = ne > 0 ? (ne + EPOCH_WIN - 1) / EPOCH_WIN : 1;
        }
    }
}

// First row of every window: window w of an instance holds the rows whose
// first entry lies in [eoff + w EPOCH_WIN, eoff + (w + 1) EPOCH_WIN) (relative
// to the instance's first entry), plus, in the instance's last window, its
// trailing empty rows.  win_row[w + 1] ends window w.
__global__ void epoch_windows_kernel(const int32_t* __restrict__ rp, int64_t n, int64_t row_begin, int count,
                                     const int64_t* __restrict__ inst_off, const int32_t* __restrict__ inst_eoff,
                                     const int32_t* __restrict__ win_base, int64_t win_cap,
                                     int32_t* __restrict__ win_row) {
    const int64_t n_rows = n - row_begin;
    const int32_t n_win = count > 0 ? win_base[count] : (rp[n_rows] + EPOCH_WIN - 1) / EPOCH_WIN;
    for (int64_t w = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; w <= win_cap;
         w += int64_t(gridDim.x) * blockDim.x) {
        if (w >= n_win) {
            win_row[w] = int32_t(n);
            continue;
        }
        int64_t lo, hi;     // rows searched (relative to row_begin), the target entry
        int32_t target;
        if (count > 0) {
            int a = 0, z = count - 1;  // instance whose windows hold w
            while (a < z) {
                const int mid = (a + z + 1) >> 1;
                if (win_base[mid] <= w) a = mid; else z = mid - 1;
            }
            lo = inst_off[a];
            hi = inst_off[a + 1];
            target = inst_eoff[a] + int32_t(w - win_base[a]) * EPOCH_WIN;
        } else {
            lo = 0;
            hi = n_rows;
            target = int32_t(w) * EPOCH_WIN;
        }
        while (lo < hi) {  // first row whose first entry is >= target
            const int64_t mid = (lo + hi) >> 1;
            if (rp[mid] < target) lo = mid + 1; else hi = mid;
        }
        win_row[w] = int32_t(row_begin + lo);
    }
}

size_t epoch_scratch_bytes(int64_t n, int64_t nnz_cap, int count) {
    const int64_t win_cap = (nnz_cap + EPOCH_WIN - 1) / EPOCH_WIN + count;
    size_t b = Carve::round(size_t(nnz_cap > 0 ? nnz_cap : 1) * 4) + Carve::round(size_t(win_cap + 2) * 4);
    if (count > 0)
        b += 3 * Carve::round(size_t(count + 1) * 4) + Carve::round(scan_scratch_elems(count) * 4);
    (void)n;
    return b + 1024;
}

int epoch_prepare(Ctx* c, const int32_t* rp, int64_t n, int64_t row_begin, int64_t nnz_cap, int count,
                  const int64_t* inst_off, void* scratch, EpochScratch* es, cudaStream_t st) {
    Carve cv(scratch);
    es->nnz_cap = nnz_cap;
    es->win_cap = (nnz_cap + EPOCH_WIN - 1) / EPOCH_WIN + count;
    es->row_of = cv.take<int32_t>(size_t(nnz_cap > 0 ? nnz_cap : 1));
    es->win_row = cv.take<int32_t>(size_t(es->win_cap + 2));
    es->sync = cv.take<unsigned int>(2);
    DRGB_CUDA(c, cudaMemsetAsync(es->row_of, 0xFF, size_t(nnz_cap > 0 ? nnz_cap : 1) * 4, st));
    const int64_t n_rows = n - row_begin;
    if (n_rows > 0) {
        epoch_heads_kernel<<<grid_for(n_rows, 256, c->num_sms * 16), 256, 0, st>>>(rp, n_rows, row_begin, nnz_cap,
                                                                                 es->row_of, c->d_status);
        DRGB_CHECK_LAUNCH(c);
    }
    if (count > 0) {
        es->inst_eoff = cv.take<int32_t>(count + 1);
        int32_t* win_cnt = cv.take<int32_t>(count + 1);
        es->win_base = cv.take<int32_t>(count + 1);
        int32_t* tmp = cv.take<int32_t>(scan_scratch_elems(count));
        epoch_instances_kernel<<<grid_for(count + 1, 256, c->num_sms), 256, 0, st>>>(rp, inst_off, count,
                                                                                    es->inst_eoff, win_cnt);
        DRGB_CHECK_LAUNCH(c);
        int rc = exclusive_scan(c, win_cnt, es->win_base, count, tmp, st);
        if (rc) return rc;
    }
    epoch_windows_kernel<<<grid_for(es->win_cap + 1, 256, c->num_sms * 4), 256, 0, st>>>(
        rp, n, row_begin, count, inst_off, es->inst_eoff, es->win_base, es->win_cap, es->win_row);
    DRGB_CHECK_LAUNCH(c);
    return DRGB_OK;
}

// ------------------------------------------------------------------ epoch kernel
// Programmatic dependent launch: an epoch launched right after another one
// may start while that one finishes.  Everything before grid_dep_wait() reads
// only the CSR and the prepared tables (which no epoch writes); Y is read and
// written only after it, when the previous epoch's grid has completed and its
// writes are visible.

// CSR chunks (of 32 entries) a warp loads at once before testing them.  The
// window's CSR words are streamed in bursts so that several loads are in
// flight per lane; the active entries of a burst wait in a per-warp queue of
// at most 31 + 32 * burst entries.  The queue is kept this small on
// purpose: shared memory left unused goes to the L1 cache, and the random
// 8-byte gathers of Y run at about 2.5x the rate with the largest L1 (the
// misses in flight per SM are bounded by L1 capacity).
static constexpr int EPOCH_BURST = 4;
constexpr int epoch_qcap(int burst) { return 32 * burst + 32; }
// Warps per SM each form's register budget is sized for: the pipelined form
// holds two groups' gathered points (about 80 registers a thread), the flat
// form one (about 48).
static constexpr int epoch_warps_per_sm(bool pipe) { return pipe ? 24 : 40; }

// Where a window's CSR words come from: global memory, streamed with
// evict-first loads (they are read once per epoch, so L2 keeps the gathered
// positions Y instead).
struct CsrGlobal {
    const uint32_t* __restrict__ q;
    const int32_t* __restrict__ col;
    const int32_t* __restrict__ row_of;
    __device__ __forceinline__ void load(int32_t e, bool in, uint32_t& qv, int32_t& jv, int32_t& hv) const {
        qv = in ? __ldcs(q + e) : 0u;  // q = 0 never fires
        jv = in ? __ldcs(col + e) : 0;
        hv = in ? __ldcs(row_of + e) : -1;
    }
};
// The instance that window W belongs to and the rows [h_lo, h_hi) of its heads.
template <bool BATCHED>
__device__ __forceinline__ void window_instance(const EpochArgs& A, int32_t W, RowInst& R, int64_t& h_lo, int64_t& h_hi) {
    R = RowInst{0, A.neg_n ? A.neg_n : uint32_t(A.n), 0, A.k0, A.k1};
    h_lo = A.row_begin;
    h_hi = A.n;
    if (BATCHED) {
        int lo = 0, hi = A.count - 1;  // the instance whose windows hold W
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (A.win_base[mid] <= W) lo = mid; else hi = mid - 1;
        }
        R.off = A.inst_off[lo];
        R.n = uint32_t(A.inst_off[lo + 1] - R.off);
        R.eoff = A.inst_eoff[lo];
        R.k0 = uint32_t(A.inst_seed[lo]);
        R.k1 = uint32_t(A.inst_seed[lo] >> 32);
        h_lo = R.off;
        h_hi = R.off + R.n;
    }
}

// One window W of epoch S, by one warp.  No row crosses a window, so the warp
// writes the final Y' of every row of the window.
//
// The warp streams the window's CSR in bursts of BURST chunks of 32 entries
// (one entry per lane and chunk, coalesced) and appends each burst's active
// entries to its queue, in entry order.  Every 32 waiting entries form a
// group: one entry per lane, its negatives drawn and its points gathered
// (fetch), then its force computed and the group's terms added by head
// (segmented scan, carry between groups).  The window's last group may be
// partial.
//
// PIPE: the gathers of a group are issued before the previous group's forces
// are computed, so one warp keeps two groups' loads in flight (for grids with
// few windows per SM); the next burst's CSR loads are issued before the held
// group is finished.  Without PIPE each group is finished before the next is
// fetched, and latency is hidden by more warps per SM (for grids with many
// windows).  Both forms form the same groups and add in the same order, so
// they give the same bits.
template <bool BATCHED, int NEG, bool PIPE, int BURST, class Csr>
__device__ __forceinline__ void epoch_window(const EpochArgs& A, const EpochStep& S, const Csr& csr, int32_t W,
                                             int lane, int2* act_w, int32_t* head_w, float4* carry_w,
                                             int32_t* chead_w, float two_ab, float two_b) {
    const unsigned lt_mask = (1u << lane) - 1u;
    const int32_t rA = A.win_row[W], rB = A.win_row[W + 1];
    if (rA >= rB) return;  // a long row started in an earlier window covers this one
    RowInst R;
    int64_t h_lo, h_hi;  // rows a head may take (the instance's rows)
    window_instance<BATCHED>(A, W, R, h_lo, h_hi);
    if (rA < h_lo || rB > h_hi) {
        if (lane == 0) report_status(A.status, DRGB_ERR_INVALID);
        return;
    }
    const int32_t es = A.row_ptr[rA - A.row_begin], ee = A.row_ptr[rB - A.row_begin];
    // Negatives and gathers of `cnt` waiting entries from queue position p.
    auto fetch_group = [&](int p, int cnt, EntryInputs<NEG>& in) {
        const bool v = lane < cnt;
        const int2 ej = v ? act_w[p + lane] : make_int2(es, 0);
        EntryPlan<NEG> pl;
        draw_entry<NEG, BATCHED>(A, S, R, v, ej.x, ej.y, v ? head_w[p + lane] : -1, h_lo, h_hi, lane, pl);
        gather_entry<NEG>(S, R, pl, in);
    };
    // Forces of a fetched group of `cnt` entries, added by head.
    auto finish_group = [&](const EntryInputs<NEG>& cur, int cnt) {
        float fx = 0.f, fy = 0.f;
        if (cur.ok) {
            const float2 f = entry_math<NEG, BATCHED>(A, S, R, cur, two_ab, two_b);
            fx = f.x;
            fy = f.y;
        }
        const int32_t i = cur.i;
        const int32_t chead = *chead_w;
        // the carried head ends unless this group starts with it
        if (chead >= 0 && lane == 0 && i != chead) {
            const float4 cv = *carry_w;
            S.Y_out[chead] = make_float2(fmaf(S.lr, 0.f + cv.x, cv.z), fmaf(S.lr, 0.f + cv.y, cv.w));
        }
        // segmented inclusive scan over runs of equal heads
        const int32_t i_prev = __shfl_up_sync(FULL, i, 1);
        const unsigned starts = __ballot_sync(FULL, lane == 0 || i_prev != i);
        const int seg0 = 31 - __clz(starts & (FULL >> (31 - lane)));
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const float ox = __shfl_up_sync(FULL, fx, d), oy = __shfl_up_sync(FULL, fy, d);
            if (lane - d >= seg0) {
                fx = ox + fx;
                fy = oy + fy;
            }
        }
        if (seg0 == 0 && i == chead) {
            const float4 cv = *carry_w;
            fx = cv.x + fx;
            fy = cv.y + fy;
        }
        // a run that ends inside the group is the row's last: write it; the
        // group's last run is carried
        const int32_t i_next = __shfl_down_sync(FULL, i, 1);
        if (cur.ok && lane < cnt - 1 && i_next != i)
            S.Y_out[i] = make_float2(fmaf(S.lr, 0.f + fx, cur.yi.x), fmaf(S.lr, 0.f + fy, cur.yi.y));
        __syncwarp();
        if (lane == cnt - 1) {
            *carry_w = make_float4(fx, fy, cur.yi.x, cur.yi.y);
            *chead_w = cur.ok ? i : -1;
        }
        __syncwarp();
    };
    EntryInputs<NEG> held;  // PIPE: the fetched group waiting for its forces
    int held_cnt = 0;
    int qn = 0;             // active entries waiting at the front of the queue
    // (a window whose rows are all empty still takes one, empty, burst)
    for (int32_t c0 = es; c0 == es || c0 < ee; c0 += 32 * BURST) {
        // the burst's CSR words, all loads in flight before any test
        uint32_t qv[BURST];
        int32_t jv[BURST], hv[BURST];
#pragma unroll
        for (int b = 0; b < BURST; ++b) {
            const int32_t e = c0 + 32 * b + lane;
            csr.load(e, e < ee, qv[b], jv[b], hv[b]);
        }
        if (PIPE && held_cnt) {  // the previous burst's last group, while the loads fly
            finish_group(held, held_cnt);
            held_cnt = 0;
        }
#pragma unroll
        for (int b = 0; b < BURST; ++b) {
            // floor((t+1) q / 2^24) > floor(t q / 2^24)  <=>  (t q mod 2^24) + q >= 2^24
            const bool act = qv[b] >= 0x1000000u - ((S.t * qv[b]) & 0xFFFFFFu);
            const unsigned m = __ballot_sync(FULL, act);
            if (act) {
                const int pos = qn + __popc(m & lt_mask);
                act_w[pos] = make_int2(c0 + 32 * b + lane, jv[b]);
                head_w[pos] = hv[b];
            }
            qn += __popc(m);
        }
        __syncwarp();
        if (c0 == es) {
            // every row of the window first gets Y + lr * 0; rows with active
            // entries are rewritten with their force below.  The wait for the
            // previous epoch comes here, after the first burst has been loaded
            // and tested.
            grid_dep_wait();
            for (int64_t r = rA + lane; r < rB; r += 32) {
                const float2 y = load_y(S.Y_in + r);
                S.Y_out[r] = make_float2(fmaf(S.lr, 0.f, y.x), fmaf(S.lr, 0.f, y.y));
            }
            if (lane == 0) *chead_w = -1;
            __syncwarp();
        }
        const bool last = c0 + 32 * BURST >= ee;
        const int ng = last ? (qn + 31) / 32 : qn / 32;
        for (int g = 0; g < ng; ++g) {
            const int cnt = qn - 32 * g < 32 ? qn - 32 * g : 32;
            EntryInputs<NEG> in;
            fetch_group(32 * g, cnt, in);
            if (PIPE) {
                if (held_cnt) finish_group(held, held_cnt);
                held = in;
                held_cnt = cnt;
            } else {
                finish_group(in, cnt);
            }
        }
        // move the waiting partial group to the front
        const int left = qn - 32 * ng > 0 ? qn - 32 * ng : 0;
        int2 lv = make_int2(0, 0);
        int32_t lh = -1;
        if (lane < left) {
            lv = act_w[32 * ng + lane];
            lh = head_w[32 * ng + lane];
        }
        __syncwarp();
        if (lane < left) {
            act_w[lane] = lv;
            head_w[lane] = lh;
        }
        qn = left;
        __syncwarp();
    }
    if (PIPE && held_cnt) finish_group(held, held_cnt);
    if (lane == 0 && *chead_w >= 0) {
        const float4 cv = *carry_w;
        S.Y_out[*chead_w] = make_float2(fmaf(S.lr, 0.f + cv.x, cv.z), fmaf(S.lr, 0.f + cv.y, cv.w));
    }
    __syncwarp();
}

// Entries and windows of the call, checked against the prepared tables.
__device__ __forceinline__ bool epoch_extent(const EpochArgs& A, int32_t& nnz, int32_t& n_win) {
    if (A.count > 0) {
        nnz = A.inst_eoff[A.count];
        n_win = A.win_base[A.count];
    } else {
        nnz = A.row_ptr[A.n - A.row_begin];
        n_win = (nnz + EPOCH_WIN - 1) / EPOCH_WIN;
    }
    return nnz >= 0 && nnz <= A.nnz_cap && n_win <= A.win_cap;
}

// One epoch: one warp per window (grid-stride over windows).
template <bool BATCHED, int NEG, int NW, bool PIPE>
__global__ void __launch_bounds__(NW * 32, epoch_warps_per_sm(PIPE) / NW)
    epoch_force_kernel(const __grid_constant__ EpochArgs A) {
    constexpr int QCAP = epoch_qcap(EPOCH_BURST);
    __shared__ int2 s_ej[NW][QCAP];     // (entry, tail) of the waiting active entries
    __shared__ int32_t s_hd[NW][QCAP];  // their heads
    // carry of each warp: running sum of the previous group's last head and
    // that head's position; the head itself (-1 when none)
    __shared__ float4 s_carry[NW];
    __shared__ int32_t s_chead[NW];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const float two_ab = 2.0f * A.a * A.b, two_b = 2.0f * A.b;
    const EpochStep S{A.Y_in, A.Y_out, A.lr, A.t};
    grid_dep_launch();
    int32_t nnz = 0, n_win = 0;
    if (!epoch_extent(A, nnz, n_win)) {
        if (threadIdx.x == 0 && blockIdx.x == 0) report_status(A.status, DRGB_ERR_INVALID);
        return;
    }
    if (n_win == 0) {  // no entries at all: every row keeps its position
        grid_dep_wait();
        for (int64_t r = A.row_begin + int64_t(blockIdx.x) * blockDim.x + threadIdx.x; r < A.n;
             r += int64_t(gridDim.x) * blockDim.x) {
            const float2 y = A.Y_in[r];
            A.Y_out[r] = make_float2(fmaf(A.lr, 0.f, y.x), fmaf(A.lr, 0.f, y.y));
        }
        return;
    }
    const CsrGlobal csr{A.q, A.col, A.row_of};
    // Single instances in the pipelined form deal the windows out over all CTAs (to
    // every CTA's first warp first), so that fewer windows than warps load every
    // SM alike (us an epoch, CTAs of consecutive windows / dealt out: 50,000 rows
    // 18.8 / 15.9, 60,000 19.3 / 17.5, 130,000 35.5 / 34.4).  Batches keep an
    // instance's windows together, whose positions stay in L1 (48 us, dealt out
    // 56), and so does the flat form for large instances (a million rows 193, dealt
    // out 198).
    constexpr bool DEAL = PIPE && !BATCHED;
    const int32_t grid = int32_t(gridDim.x), blk = int32_t(blockIdx.x);
    for (int32_t W = DEAL ? blk + w * grid : blk * NW + w; W < n_win; W += grid * NW)
        epoch_window<BATCHED, NEG, PIPE, EPOCH_BURST>(A, S, csr, W, lane, s_ej[w], s_hd[w], &s_carry[w], &s_chead[w],
                                                      two_ab, two_b);
}

// ------------------------------------------------------------------ loop of epochs in one launch
// All epochs [t_begin, t_end) in one cooperative launch, for graphs of few
// windows: a CTA takes a window (or every gridDim-th one) with all its warps,
// and the CTAs meet at a barrier after every epoch.
//
// Why: with one warp per window and one launch per epoch an epoch of a small
// graph is one chain of dependent steps (a warp's 16 CSR chunks, five groups of
// gathers and forces, the next launch) on a few SMs: 8 us for 2,000 rows (15
// CTAs), 13 us for the anchored epochs of 5,000 new points.  Here the
// window's entries are tested by all warps at once and every group of 32
// active entries has its own warp, so the chain is one group; the test of the
// next epoch's first window runs while the CTA waits at the barrier.
//
// Bound: the latency of the barrier and of one group's gathers up to about
// 5,000 rows (3.2 us an epoch at 2,000), then the windows a CTA takes in turn.
//
// The groups and the order of every sum are those of epoch_window: a group's
// runs that start and end inside it are final, and the first and last run of
// each group are joined to their neighbours in group order by one thread.
static constexpr int LOOP_ROUND = 768;  // entries tested per round (a window has about 512)
static constexpr int LOOP_QCAP = LOOP_ROUND + 32;
static constexpr int LOOP_LR = 128;     // learning rates computed at a time
// CTAs of 8 warps while two per SM hold every window, else of 4 warps, which
// keep more windows in flight (16,000 rows: 9.8 us an epoch with 4 warps and 5
// CTAs per SM, 11.8 with 8; 6 CTAs per SM spill registers, 13.2 against 11.3
// at 20,000 rows; CTAs of 2 warps 14.0 against 12.0 at 30,000).
constexpr int loop_ctas_per_sm(int nw) { return nw == 8 ? 2 : 5; }
static constexpr int LOOP_WINDOWS = 16;  // windows a CTA may hold

// A CTA's window: its rows, entries and instance.
struct LoopWindow {
    int32_t rA, rB, es, ee;
    RowInst R;
    int64_t h_lo, h_hi;
};

struct LoopArgs {
    float2* buf[2];        // positions of even and odd steps
    int t_begin, t_end, T;
    float lr0;
    unsigned int* arrived;  // barrier counter (0 at the start)
    int* stop;              // raised by a CTA whose wait ran out (0 at the start)
};

// The first and the last run of a group.
struct GroupEnds {
    int32_t head0, head1;  // their heads (negative: an invalid entry); equal when the group is one run
    float2 sum0, sum1, y0, y1;
    bool one;              // the group is one run
};

template <bool BATCHED, int NEG, int LOOP_WARPS>
__global__ void __launch_bounds__(LOOP_WARPS * 32, loop_ctas_per_sm(LOOP_WARPS))
    epoch_loop_kernel(const __grid_constant__ EpochArgs A, const __grid_constant__ LoopArgs P) {
    constexpr int LOOP_THREADS = LOOP_WARPS * 32;
    constexpr int LOOP_CHUNKS = LOOP_ROUND / LOOP_THREADS;  // chunks of 32 entries a warp tests per round
    __shared__ int32_t s_e[LOOP_QCAP];  // active entries
    __shared__ int s_cnt[LOOP_WARPS];
    __shared__ GroupEnds s_end[LOOP_QCAP / 32];
    __shared__ float s_lr[LOOP_LR];
    __shared__ int32_t s_chead;
    __shared__ float4 s_carry;
    __shared__ int s_stop, s_nw;
    __shared__ LoopWindow s_win[LOOP_WINDOWS];
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const unsigned lt_mask = (1u << lane) - 1u;
    const float two_ab = 2.0f * A.a * A.b, two_b = 2.0f * A.b;
    int32_t nnz = 0, n_win = 0;
    if (!epoch_extent(A, nnz, n_win)) {
        if (tid == 0 && blockIdx.x == 0) report_status(A.status, DRGB_ERR_INVALID);
        return;
    }
    if (n_win == 0) {  // no entries at all: every row keeps its position
        const int last = (P.t_end - P.t_begin) & 1;
        for (int64_t r = A.row_begin + int64_t(blockIdx.x) * blockDim.x + tid; r < A.n; r += int64_t(gridDim.x) * blockDim.x) {
            const float2 y = P.buf[0][r];
            P.buf[last][r] = make_float2(fmaf(P.lr0, 0.f, y.x), fmaf(P.lr0, 0.f, y.y));
        }
        return;
    }
    const unsigned ctas = unsigned(n_win) < gridDim.x ? unsigned(n_win) : gridDim.x;
    if (blockIdx.x >= ctas) return;
    unsigned arrivals = 0;  // epochs this CTA has finished
    if (tid == 0) {  // this CTA's windows (host: at most LOOP_WINDOWS)
        s_stop = 0;
        s_chead = -1;
        s_carry = make_float4(0.f, 0.f, 0.f, 0.f);
        int k = 0;
        for (int32_t W = int32_t(blockIdx.x); W < n_win && k < LOOP_WINDOWS; W += int32_t(ctas)) {
            LoopWindow d;
            d.rA = A.win_row[W];
            d.rB = A.win_row[W + 1];
            if (d.rA >= d.rB) continue;  // a long row started in an earlier window covers this one
            window_instance<BATCHED>(A, W, d.R, d.h_lo, d.h_hi);
            if (d.rA < d.h_lo || d.rB > d.h_hi) {
                report_status(A.status, DRGB_ERR_INVALID);
                continue;
            }
            d.es = A.row_ptr[d.rA - A.row_begin];
            d.ee = A.row_ptr[d.rB - A.row_begin];
            s_win[k++] = d;
        }
        s_nw = k;
    }
    __syncthreads();
    const int n_mine = s_nw;
    // Schedule words of one round of a window, in this thread's registers.
    // They are loaded a window ahead, when the previous ones have been
    // compacted; tails and heads are read for the active entries alone.
    uint32_t qv[LOOP_CHUNKS];
    auto load_round = [&](int32_t c0, int32_t ee) {
        const int32_t e0 = c0 + w * (32 * LOOP_CHUNKS) + lane;
#pragma unroll
        for (int b = 0; b < LOOP_CHUNKS; ++b) qv[b] = e0 + 32 * b < ee ? A.q[e0 + 32 * b] : 0u;  // 0 never fires
    };
    if (n_mine > 0) load_round(s_win[0].es, s_win[0].ee);
    // Every CTA has finished the previous epoch (bounded; false: give up).  A CTA's
    // barrier and its first thread's release order the epoch's writes of Y before
    // the count; the acquire here and the barrier after it order the count before the
    // other threads' reads, plain loads included (the acquire drops the L1's older
    // lines).  Loads that are not coherent (ld.global.nc, __restrict__) would not be
    // ordered.
    auto wait_epoch = [&]() -> bool {
        if (tid == 0 && arrivals) {
            const unsigned target = arrivals * ctas;
            const unsigned long long t0 = loop_timer();
            for (;;) {
                unsigned v;
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(P.arrived) : "memory");
                if (v >= target) break;
                if (loop_timer() - t0 > 2000000000ull || *static_cast<volatile int*>(P.stop)) {
                    *static_cast<volatile int*>(P.stop) = 1;
                    report_status(A.status, DRGB_ERR_TIMEOUT);
                    s_stop = 1;
                    break;
                }
            }
        }
        __syncthreads();
        return s_stop == 0;
    };
    for (int t = P.t_begin; t < P.t_end; ++t) {
        const int step = t - P.t_begin;
        if (step % LOOP_LR == 0) {  // learning rates of the next epochs
            __syncthreads();
            for (int u = tid; u < LOOP_LR; u += LOOP_THREADS)
                s_lr[u] = float(double(P.lr0) * (1.0 - double(t + u) / double(P.T)));
            __syncthreads();
        }
        const EpochStep S{P.buf[step & 1], P.buf[(step & 1) ^ 1], s_lr[step % LOOP_LR], uint32_t(t)};
        bool waited = false;
        for (int k = 0; k < n_mine; ++k) {
            const int32_t rA = s_win[k].rA, rB = s_win[k].rB, es = s_win[k].es, ee = s_win[k].ee;
            const RowInst R = s_win[k].R;
            const int64_t h_lo = s_win[k].h_lo, h_hi = s_win[k].h_hi;
            int qn = 0;  // active entries waiting at the front of the list
            for (int32_t c0 = es; c0 == es || c0 < ee; c0 += LOOP_ROUND) {
                const int32_t e0 = c0 + w * (32 * LOOP_CHUNKS) + lane;
                unsigned m[LOOP_CHUNKS];
                int cnt = 0;
#pragma unroll
                for (int b = 0; b < LOOP_CHUNKS; ++b) {
                    // floor((t+1) q / 2^24) > floor(t q / 2^24)  <=>  (t q mod 2^24) + q >= 2^24
                    m[b] = __ballot_sync(FULL, qv[b] >= 0x1000000u - ((S.t * qv[b]) & 0xFFFFFFu));
                    cnt += __popc(m[b]);
                }
                if (lane == 0) s_cnt[w] = cnt;
                __syncthreads();
                int pos = qn, total = 0;
#pragma unroll
                for (int u = 0; u < LOOP_WARPS; ++u) {
                    const int v = s_cnt[u];
                    pos += u < w ? v : 0;
                    total += v;
                }
#pragma unroll
                for (int b = 0; b < LOOP_CHUNKS; ++b) {
                    if (m[b] >> lane & 1u) {
                        const int p = pos + __popc(m[b] & lt_mask);
                        s_e[p] = e0 + 32 * b;
                    }
                    pos += __popc(m[b]);
                }
                qn += total;
                const bool last = c0 + LOOP_ROUND >= ee;
                if (!last) {
                    load_round(c0 + LOOP_ROUND, ee);
                } else if (n_mine > 1 || c0 != es) {  // (a lone window of one round stays in registers)
                    const int kn = k + 1 < n_mine ? k + 1 : 0;
                    load_round(s_win[kn].es, s_win[kn].ee);
                }
                if (c0 == es && tid == 0) s_chead = -1;
                __syncthreads();
                const int ng = last ? (qn + 31) / 32 : qn / 32;
                auto draw = [&](int g, EntryPlan<NEG>& pl) {
                    const int p = 32 * g + lane;
                    const bool v = p < qn;
                    const int32_t e = v ? s_e[p] : es;
                    draw_entry<NEG, BATCHED>(A, S, R, v, e, v ? A.col[e] : 0, v ? A.row_of[e] : -1, h_lo, h_hi, lane, pl);
                };
                EntryPlan<NEG> pl;
                if (w < ng) draw(w, pl);
                if (!waited) {  // the first read of Y
                    if (!wait_epoch()) return;
                    waited = true;
                }
                EntryInputs<NEG> in;
                if (w < ng) gather_entry<NEG>(S, R, pl, in);
                if (c0 == es) {
                    // every row of the window first gets Y + lr * 0; rows with
                    // active entries are rewritten with their force below
                    for (int64_t r = rA + tid; r < rB; r += LOOP_THREADS) {
                        const float2 y = load_y(S.Y_in + r);
                        S.Y_out[r] = make_float2(fmaf(S.lr, 0.f, y.x), fmaf(S.lr, 0.f, y.y));
                    }
                    __syncthreads();
                }
                for (int g = w; g < ng; g += LOOP_WARPS) {
                    if (g != w) {
                        draw(g, pl);
                        gather_entry<NEG>(S, R, pl, in);
                    }
                    const int gn = qn - 32 * g < 32 ? qn - 32 * g : 32;
                    float fx = 0.f, fy = 0.f;
                    if (in.ok) {
                        const float2 f = entry_math<NEG, BATCHED>(A, S, R, in, two_ab, two_b);
                        fx = f.x;
                        fy = f.y;
                    }
                    const int32_t i = in.i;
                    const int32_t i_prev = __shfl_up_sync(FULL, i, 1), i_next = __shfl_down_sync(FULL, i, 1);
                    const unsigned starts = __ballot_sync(FULL, lane == 0 || i_prev != i);
                    const int seg0 = 31 - __clz(starts & (FULL >> (31 - lane)));
#pragma unroll
                    for (int d = 1; d < 32; d <<= 1) {
                        const float ox = __shfl_up_sync(FULL, fx, d), oy = __shfl_up_sync(FULL, fy, d);
                        if (lane - d >= seg0) {
                            fx = ox + fx;
                            fy = oy + fy;
                        }
                    }
                    const bool ends = lane == gn - 1 || (lane < gn - 1 && i_next != i);
                    if (ends && lane < gn - 1 && seg0 > 0 && in.ok)  // inside the group: final
                        S.Y_out[i] = make_float2(fmaf(S.lr, 0.f + fx, in.yi.x), fmaf(S.lr, 0.f + fy, in.yi.y));
                    if (ends && seg0 == 0) {
                        s_end[g].head0 = in.ok ? i : -1;
                        s_end[g].sum0 = make_float2(fx, fy);
                        s_end[g].y0 = in.yi;
                        s_end[g].one = lane == gn - 1;
                    }
                    if (lane == gn - 1) {
                        s_end[g].head1 = in.ok ? i : -1;
                        s_end[g].sum1 = make_float2(fx, fy);
                        s_end[g].y1 = in.yi;
                    }
                }
                // entries of an incomplete group go to the front for the next round
                const int left = qn - 32 * ng > 0 ? qn - 32 * ng : 0;
                const int32_t le = !last && w == 0 && lane < left ? s_e[32 * ng + lane] : 0;
                __syncthreads();
                if (!last && w == 0 && lane < left) s_e[lane] = le;
                qn = left;
                if (w == 0) {
                    auto put = [&](int32_t h, float2 f, float2 y) {
                        if (h >= 0) S.Y_out[h] = make_float2(fmaf(S.lr, 0.f + f.x, y.x), fmaf(S.lr, 0.f + f.y, y.y));
                    };
                    // Lane g joins group g's first run to the run before it
                    // (the previous group's last, or the carry of the previous
                    // round).  A group that is one run passes its join on, so
                    // with one of those before the last group (rare: a row with
                    // more than 32 active entries) one lane walks the groups.
                    static_assert(LOOP_QCAP / 32 <= 32, "a lane per group");
                    GroupEnds E;
                    E.head0 = E.head1 = -1;
                    E.one = false;
                    if (lane < ng) E = s_end[lane];
                    int32_t chead = s_chead;
                    float4 cv = s_carry;
                    if (__any_sync(FULL, lane < ng - 1 && E.one)) {
                        if (lane == 0) {
                            for (int g = 0; g < ng; ++g) {
                                E = s_end[g];
                                float2 f = E.sum0;
                                if (chead >= 0 && E.head0 == chead) {
                                    f.x = cv.x + f.x;
                                    f.y = cv.y + f.y;
                                } else {
                                    put(chead, make_float2(cv.x, cv.y), make_float2(cv.z, cv.w));
                                }
                                if (E.one) {
                                    chead = E.head0;
                                    cv = make_float4(f.x, f.y, E.y0.x, E.y0.y);
                                } else {
                                    put(E.head0, f, E.y0);
                                    chead = E.head1;
                                    cv = make_float4(E.sum1.x, E.sum1.y, E.y1.x, E.y1.y);
                                }
                            }
                            if (last) put(chead, make_float2(cv.x, cv.y), make_float2(cv.z, cv.w));
                            s_chead = chead;
                            s_carry = cv;
                        }
                    } else if (ng > 0) {
                        const int32_t ph = __shfl_up_sync(FULL, E.head1, 1);
                        const float4 pv = make_float4(__shfl_up_sync(FULL, E.sum1.x, 1), __shfl_up_sync(FULL, E.sum1.y, 1),
                                                      __shfl_up_sync(FULL, E.y1.x, 1), __shfl_up_sync(FULL, E.y1.y, 1));
                        if (lane > 0) {
                            chead = ph;
                            cv = pv;
                        }
                        if (lane < ng) {
                            float2 f = E.sum0;
                            if (chead >= 0 && E.head0 == chead) {
                                f.x = cv.x + f.x;
                                f.y = cv.y + f.y;
                            } else {
                                put(chead, make_float2(cv.x, cv.y), make_float2(cv.z, cv.w));
                            }
                            if (E.one) {  // the last group
                                E.head1 = E.head0;
                                E.sum1 = f;
                                E.y1 = E.y0;
                            } else {
                                put(E.head0, f, E.y0);
                            }
                            if (lane == ng - 1) {
                                if (last) put(E.head1, E.sum1, E.y1);
                                s_chead = E.head1;
                                s_carry = make_float4(E.sum1.x, E.sum1.y, E.y1.x, E.y1.y);
                            }
                        }
                    } else if (last && lane == 0) {
                        put(chead, make_float2(cv.x, cv.y), make_float2(cv.z, cv.w));
                    }
                    __syncwarp();
                }
            }
        }
        if (!waited && !wait_epoch()) return;  // (a CTA whose windows were all skipped)
        __syncthreads();
        ++arrivals;
        if (tid == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(P.arrived) : "memory");
    }
}

static constexpr int64_t EPOCH_FLAT_ROWS = 200000, EPOCH_FLAT_ROWS_END = 9000000;

bool epoch_warps_supported(int warps) { return warps == 4 || warps == 8; }

int launch_epoch(Ctx* c, const EpochArgs& A_in, int warps, cudaStream_t st, bool after_epoch) {
    if (warps <= 0) warps = c->epoch_warps;
    if (!epoch_warps_supported(warps))
        return set_error(c, DRGB_ERR_INVALID, "epoch: unsupported force-kernel width %d", warps);
    if (!A_in.row_of || !A_in.win_row) return set_error(c, DRGB_ERR_INVALID, "epoch: state not prepared");
    EpochArgs A = A_in;
    philox_round_keys(A.k0, A.k1, A.rk);
    const bool bat = A.count > 0, n5 = A.neg == 5 && A.b > 0.f;
    // Untuned, a large single instance takes the flat form: its gathers miss L1,
    // and 40 warps an SM hide that better than 24 with two groups each, until the
    // gathers miss L2 as well, between 8 and 10 million rows (us an
    // epoch, pipelined / flat: 70,000 rows 19.1 / 26.6, 130,000 34.0 / 36.4, 250,000
    // 58.3 / 55.0, a million 213 / 204, eight million 1,708 / 1,632, ten million 2,282 /
    // 2,371; batches of small instances 48.0 / 49.8).
    const bool pipe = c->epoch_pipe != 0 &&
                      (c->epoch_pipe_set || bat || A.n < EPOCH_FLAT_ROWS || A.n >= EPOCH_FLAT_ROWS_END);
    const int per_sm = epoch_warps_per_sm(pipe) / warps;
    const int fgrid = grid_for(A.win_cap, pipe && !bat ? 1 : warps, c->num_sms * per_sm);
    auto go = [&](auto kernel) -> int {
        // Ask for no more shared memory than the resident CTAs hold (their
        // queues plus the 1 KB the hardware reserves per CTA); the rest of the
        // SM's 256 KB stays L1 cache for the gathers of Y.
        cudaFuncAttributes fa;
        DRGB_CUDA(c, cudaFuncGetAttributes(&fa, kernel));
        const size_t need = size_t(per_sm) * (fa.sharedSizeBytes + 1024);
        int pct = int((need * 100 + c->smem_per_sm - 1) / (c->smem_per_sm ? c->smem_per_sm : 1));
        pct = pct < 1 ? 1 : (pct > 100 ? 100 : pct);
        DRGB_CUDA(c, cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, pct));
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(fgrid);
        cfg.blockDim = dim3(warps * 32);
        cfg.dynamicSmemBytes = 0;
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = after_epoch ? 1 : 0;  // only an epoch may precede with overlap
        DRGB_CUDA(c, cudaLaunchKernelEx(&cfg, kernel, A));
        return DRGB_OK;
    };
    auto pick = [&](auto nw, auto pp) -> int {
        constexpr int NW = decltype(nw)::value;
        constexpr bool P = decltype(pp)::value;
        return bat ? (n5 ? go(epoch_force_kernel<true, 5, NW, P>) : go(epoch_force_kernel<true, -1, NW, P>))
                   : (n5 ? go(epoch_force_kernel<false, 5, NW, P>) : go(epoch_force_kernel<false, -1, NW, P>));
    };
    using I4 = std::integral_constant<int, 4>;
    using I8 = std::integral_constant<int, 8>;
    using PT = std::true_type;
    using PF = std::false_type;
    int rc = warps == 4 ? (pipe ? pick(I4{}, PT{}) : pick(I4{}, PF{})) : (pipe ? pick(I8{}, PT{}) : pick(I8{}, PF{}));
    if (rc) return rc;
    DRGB_CHECK_LAUNCH(c);
    return DRGB_OK;
}

int launch_init_batched(Ctx* c, float2* Y, int64_t n_total, float range, int count,
                        const int64_t* inst_off, const uint64_t* inst_seed, cudaStream_t st) {
    int blocks = grid_for(n_total, 256, c->num_sms * 16);
    init_batched_kernel<<<blocks, 256, 0, st>>>(Y, n_total, range, count, inst_off, inst_seed);
    DRGB_CHECK_LAUNCH(c);
    return DRGB_OK;
}

int launch_init(Ctx* c, float2* Y, int64_t n, float range, uint64_t seed, cudaStream_t st) {
    int blocks = grid_for(n, 256, c->num_sms * 16);
    init_embedding_kernel<<<blocks, 256, 0, st>>>(Y, n, range, uint32_t(seed), uint32_t(seed >> 32));
    DRGB_CHECK_LAUNCH(c);
    return DRGB_OK;
}

static void fill_args(EpochArgs& A, const int32_t* rp, const int32_t* col, const uint32_t* q, int64_t n, float a,
                      float b, int neg, uint64_t seed, int* status, const EpochScratch& es, int count,
                      const int64_t* inst_off, const uint64_t* inst_seed, int64_t row_begin, uint32_t neg_n) {
    A.row_ptr = rp;
    A.col = col;
    A.q = q;
    A.n = n;
    A.a = a;
    A.b = b;
    A.neg = neg;
    A.k0 = uint32_t(seed);
    A.k1 = uint32_t(seed >> 32);
    A.status = status;
    A.row_of = es.row_of;
    A.win_row = es.win_row;
    A.nnz_cap = es.nnz_cap;
    A.win_cap = es.win_cap;
    A.count = count;
    A.inst_off = inst_off;
    A.inst_seed = inst_seed;
    A.inst_eoff = es.inst_eoff;
    A.win_base = es.win_base;
    A.row_begin = row_begin;
    A.neg_n = neg_n;
}

// Windows (by capacity) up to which an epoch loop runs as one cooperative launch
// (epoch_loop_kernel): microseconds an epoch against the chained launches, 15
// neighbours: 2,000 rows 3.2 / 9.2, 8,000 5.1 / 13.4, 12,000 6.3 / 15.0, 20,000
// 10.9 / 11.5, 30,000 11.8 / 14.2, 35,000 14.5 / 14.5, 40,000 15.1 / 14.7, 50,000
// 19.0 / 15.9 (35,000 rows are 11.5 windows an SM).
static constexpr int64_t LOOP_MAX_WINDOWS_PER_SM = 11;
// A short loop over more than a few windows an SM takes launches too: the graph's
// launches are prepared while the device works on the call's tables, and the loop's
// CTAs take their windows in turn (us a call, loop / launches: 20,000 rows 3
// epochs 75 / 66, 6 103 / 100, 10 139 / 148; with 20 negatives 108 / 94, 167 / 166, 251 /
// 265; 10,000 rows, 3 windows an SM, 60 / 66 and 72 / 93).
static constexpr int64_t LOOP_FEW_WINDOWS_PER_SM = 4;
static constexpr int LOOP_MIN_EPOCHS = 8;
static constexpr int LOOP_MAX_EPOCHS = 1000000;  // the barrier counts epochs x CTAs in 32 bits

// *done is false, and no epoch has run, where the device, or the part of it that
// the stream may use, does not hold the grid at once: the caller chains launches.
static int run_epoch_loop(Ctx* c, float2* Y, float2* Y_tmp, EpochArgs& A, float lr0, int t_begin, int t_end, int T,
                          unsigned int* sync, cudaStream_t st, bool* done) {
    *done = false;
    DRGB_CUDA(c, cudaMemsetAsync(sync, 0, 2 * sizeof(unsigned int), st));
    LoopArgs P;
    P.buf[0] = Y;
    P.buf[1] = Y_tmp;
    P.t_begin = t_begin;
    P.t_end = t_end;
    P.T = T;
    P.lr0 = lr0;
    P.arrived = sync;
    P.stop = reinterpret_cast<int*>(sync + 1);
    philox_round_keys(A.k0, A.k1, A.rk);
    const bool bat = A.count > 0, n5 = A.neg == 5 && A.b > 0.f;
    auto pick = [&](auto nw) {
        constexpr int NW = decltype(nw)::value;
        return bat ? (n5 ? epoch_loop_kernel<true, 5, NW> : epoch_loop_kernel<true, -1, NW>)
                   : (n5 ? epoch_loop_kernel<false, 5, NW> : epoch_loop_kernel<false, -1, NW>);
    };
    const int64_t per = A.win_cap * 5 / 6;  // (about a sixth of the capacity is pruned or merged away)
    const int nw = per <= int64_t(c->num_sms) * loop_ctas_per_sm(8) ? 8 : 4;
    auto kernel = nw == 8 ? pick(std::integral_constant<int, 8>{}) : pick(std::integral_constant<int, 4>{});
    int per_sm = 0;
    DRGB_CUDA(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, nw * 32, 0));
    if (per_sm > loop_ctas_per_sm(nw)) per_sm = loop_ctas_per_sm(nw);
    // as for the force kernel: shared memory for the resident CTAs, L1 for the rest
    cudaFuncAttributes fa;
    DRGB_CUDA(c, cudaFuncGetAttributes(&fa, kernel));
    const size_t need = size_t(per_sm) * (fa.sharedSizeBytes + 1024);
    const int pct = int((need * 100 + c->smem_per_sm - 1) / (c->smem_per_sm ? c->smem_per_sm : 1));
    DRGB_CUDA(c, cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, pct < 100 ? pct : 100));
    const int64_t ctas = per_sm > 0 ? grid_for(A.win_cap, 1, c->num_sms * per_sm) : 0;
    if (A.win_cap > ctas * LOOP_WINDOWS) return DRGB_OK;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned(ctas));
    cfg.blockDim = dim3(nw * 32);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<const EpochArgs&>(A), static_cast<const LoopArgs&>(P));
    if (e == cudaErrorCooperativeLaunchTooLarge) {
        cudaGetLastError();
        return DRGB_OK;
    }
    DRGB_CUDA(c, e);
    DRGB_CHECK_LAUNCH(c);
    *done = true;
    if ((t_end - t_begin) & 1)
        DRGB_CUDA(c, cudaMemcpyAsync(Y, Y_tmp, size_t(A.n) * sizeof(float2), cudaMemcpyDeviceToDevice, st));
    return DRGB_OK;
}

// Epochs [t_begin, t_end) of a T-epoch schedule, ping-ponging between Y and
// Y_tmp; the result is left in Y.  A small graph's run in one launch.  Else, and
// where that launch is refused, the launches are captured into a CUDA
// graph (on a private stream) and the graph is launched on `st`.  Building an
// executable graph of hundreds of nodes costs milliseconds of host time, so
// the context keeps the last one and refreshes it in place
// (cudaGraphExecUpdate: same nodes, new parameters) whenever the new loop has
// the same shape; a launch already enqueued keeps the parameters it had.
int run_epochs(Ctx* c, float2* Y, float2* Y_tmp, const int32_t* rp, const int32_t* col, const uint32_t* q,
               int64_t n, float a, float b, float lr0, int neg, int t_begin, int t_end, int T, uint64_t seed,
               cudaStream_t st, int64_t nnz_cap, void* scratch, int count, const int64_t* inst_off,
               const uint64_t* inst_seed, int64_t row_begin, uint32_t neg_n) {
    if (t_end <= t_begin) return DRGB_OK;
    EpochScratch es;
    int rc = epoch_prepare(c, rp, n, row_begin, nnz_cap, count, inst_off, scratch, &es, st);
    if (rc) return rc;
    const int few = es.win_cap <= LOOP_FEW_WINDOWS_PER_SM * c->num_sms ? 2 : LOOP_MIN_EPOCHS;
    if (t_end - t_begin >= few && t_end - t_begin <= LOOP_MAX_EPOCHS &&
        es.win_cap <= LOOP_MAX_WINDOWS_PER_SM * c->num_sms) {
        EpochArgs A;
        fill_args(A, rp, col, q, n, a, b, neg, seed, c->d_status, es, count, inst_off, inst_seed, row_begin, neg_n);
        bool done = false;
        rc = run_epoch_loop(c, Y, Y_tmp, A, lr0, t_begin, t_end, T, es.sync, st, &done);
        if (rc || done) return rc;
    }
    cudaStream_t cap;
    DRGB_CUDA(c, cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
    cudaGraph_t graph = nullptr;
    cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) {
        cudaStreamDestroy(cap);
        return set_error(c, DRGB_ERR_CUDA, "begin capture: %s", cudaGetErrorString(e));
    }
    float2* src = Y;
    float2* dst = Y_tmp;
    for (int t = t_begin; t < t_end && rc == DRGB_OK; ++t) {
        EpochArgs A;
        fill_args(A, rp, col, q, n, a, b, neg, seed, c->d_status, es, count, inst_off, inst_seed, row_begin, neg_n);
        A.Y_in = src;
        A.Y_out = dst;
        A.lr = float(double(lr0) * (1.0 - double(t) / double(T)));
        A.t = uint32_t(t);
        rc = launch_epoch(c, A, 0, cap, t > t_begin);
        float2* tmp = src;
        src = dst;
        dst = tmp;
    }
    if (rc == DRGB_OK && src != Y)
        cudaMemcpyAsync(Y, src, size_t(n) * sizeof(float2), cudaMemcpyDeviceToDevice, cap);
    e = cudaStreamEndCapture(cap, &graph);
    if (rc == DRGB_OK && e != cudaSuccess)
        rc = set_error(c, DRGB_ERR_CUDA, "end capture: %s", cudaGetErrorString(e));
    if (rc == DRGB_OK && c->epoch_exec) {
        cudaGraphExecUpdateResultInfo info;
        if (cudaGraphExecUpdate(c->epoch_exec, graph, &info) != cudaSuccess) {
            cudaGetLastError();  // a different shape: build a new executable graph
            cudaGraphExecDestroy(c->epoch_exec);
            c->epoch_exec = nullptr;
        }
    }
    if (rc == DRGB_OK && !c->epoch_exec) {
        e = cudaGraphInstantiate(&c->epoch_exec, graph, 0);
        if (e != cudaSuccess) {
            c->epoch_exec = nullptr;
            rc = set_error(c, DRGB_ERR_CUDA, "instantiate: %s", cudaGetErrorString(e));
        }
    }
    if (rc == DRGB_OK) {
        e = cudaGraphLaunch(c->epoch_exec, st);
        if (e != cudaSuccess) rc = set_error(c, DRGB_ERR_CUDA, "graph launch: %s", cudaGetErrorString(e));
    }
    if (graph) cudaGraphDestroy(graph);
    cudaStreamDestroy(cap);
    return rc;
}

// Force-kernel widths and forms tried by the tuner.
static const int kWarpChoices[] = {4, 8};
static const int kPipeChoices[] = {1, 0};

int autotune_epoch(Ctx* c, const float2* Y, float2* Ya, float2* Yb, const int32_t* rp, const int32_t* col,
                   const uint32_t* q, int64_t n, float a, float b, int neg, int T, uint64_t seed, int trials,
                   cudaStream_t st, const EpochScratch& es, int count, const int64_t* inst_off,
                   const uint64_t* inst_seed, float* best_us) {
    cudaEvent_t e0, e1;
    DRGB_CUDA(c, cudaEventCreate(&e0));
    DRGB_CUDA(c, cudaEventCreate(&e1));
    const int saved_pipe = c->epoch_pipe;
    const bool saved_set = c->epoch_pipe_set;
    c->epoch_pipe_set = true;
    int best_w = c->epoch_warps, best_p = c->epoch_pipe, rc = DRGB_OK;
    float best = 1e30f;
    const int t0 = T / 4 < T - trials ? T / 4 : (T - trials > 0 ? T - trials : 0);
    for (int pipe : kPipeChoices) {
        c->epoch_pipe = pipe;
        for (int warps : kWarpChoices) {
            EpochArgs A;
            fill_args(A, rp, col, q, n, a, b, neg, seed, c->d_status, es, count, inst_off, inst_seed, 0, 0);
            if (cudaMemcpyAsync(Ya, Y, size_t(n) * 8, cudaMemcpyDeviceToDevice, st) != cudaSuccess) {
                rc = set_error(c, DRGB_ERR_CUDA, "autotune: copy failed");
                break;
            }
            float ms = 0.f;
            for (int pass = 0; pass < 2 && rc == DRGB_OK; ++pass) {  // pass 0 warms up
                cudaEventRecord(e0, st);
                for (int k = 0; k < trials && rc == DRGB_OK; ++k) {
                    A.Y_in = (k & 1) ? Yb : Ya;
                    A.Y_out = (k & 1) ? Ya : Yb;
                    A.t = uint32_t(t0 + k);
                    A.lr = 1.0f - float(t0 + k) / float(T);
                    rc = launch_epoch(c, A, warps, st, k > 0);
                }
                cudaEventRecord(e1, st);
                if (cudaEventSynchronize(e1) != cudaSuccess) rc = set_error(c, DRGB_ERR_CUDA, "autotune: sync failed");
                cudaEventElapsedTime(&ms, e0, e1);
            }
            if (rc) break;
            const float us = ms * 1000.f / trials;
            if (us < best) {
                best = us;
                best_w = warps;
                best_p = pipe;
            }
        }
        if (rc) break;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    c->epoch_pipe = saved_pipe;
    c->epoch_pipe_set = saved_set;
    if (rc) return rc;
    c->epoch_pipe_set = true;
    c->epoch_warps = best_w;
    c->epoch_pipe = best_p;
    if (best_us) *best_us = best;
    return DRGB_OK;
}

}  // namespace drgb

using namespace drgb;

extern "C" {

int drgb_init_embedding(drgb_ctx* c, int64_t n, float init_range, uint64_t seed, float* Y,
                        void* stream) {
    if (!c || !Y || n < 1 || !aligned(Y, 8) || !(init_range > 0.f))
        return set_error(c, DRGB_ERR_INVALID, "init_embedding: invalid argument");
    return launch_init(c, reinterpret_cast<float2*>(Y), n, init_range, seed,
                       static_cast<cudaStream_t>(stream));
}

static int check_epoch_args(drgb_ctx* c, const float* Y_in, const float* Y_out, const int32_t* rp,
                            const int32_t* col, const uint32_t* q, int64_t n, int32_t neg) {
    if (!c) return DRGB_ERR_INVALID;
    if (!Y_in || !Y_out || !rp || !col || !q)
        return set_error(c, DRGB_ERR_INVALID, "embed_epoch: NULL pointer");
    if (Y_in == Y_out) return set_error(c, DRGB_ERR_INVALID, "embed_epoch: Y_out aliases Y_in");
    if (!aligned(Y_in, 8) || !aligned(Y_out, 8))
        return set_error(c, DRGB_ERR_INVALID, "embed_epoch: Y must be 8-byte aligned");
    if (!aligned(rp, 4) || !aligned(col, 4) || !aligned(q, 4))
        return set_error(c, DRGB_ERR_INVALID, "embed_epoch: CSR arrays must be 4-byte aligned");
    if (n < 1 || n > INT32_MAX) return set_error(c, DRGB_ERR_INVALID, "embed_epoch: bad n");
    if (neg < 0 || neg > 64) return set_error(c, DRGB_ERR_INVALID, "embed_epoch: neg out of range");
    return DRGB_OK;
}

// Entry count row_ptr[n] (read back to size the per-call state) and that state.
static int epoch_state_for(drgb_ctx* c, const int32_t* rp, int64_t n, cudaStream_t st, EpochScratch* es) {
    int32_t nnz = 0;
    DRGB_CUDA(c, cudaMemcpyAsync(&nnz, rp + n, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    DRGB_CUDA(c, cudaStreamSynchronize(st));
    if (nnz < 0) return set_error(c, DRGB_ERR_INVALID, "embed_epoch: row_ptr[n] < 0");
    int rc = ensure_scratch(c, epoch_scratch_bytes(n, nnz, 0), st);
    if (rc) return rc;
    return epoch_prepare(c, rp, n, 0, nnz, 0, nullptr, c->scratch, es, st);
}

int drgb_embed_epoch(drgb_ctx* c, const float* Y_in, float* Y_out, const int32_t* row_ptr,
                     const int32_t* col, const uint32_t* q, int64_t n, float a, float b, float lr,
                     int32_t neg, int32_t epoch, uint64_t seed, void* stream) {
    int rc = check_epoch_args(c, Y_in, Y_out, row_ptr, col, q, n, neg);
    if (rc) return rc;
    if (epoch < 0) return set_error(c, DRGB_ERR_INVALID, "embed_epoch: epoch < 0");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    EpochScratch es;
    if ((rc = epoch_state_for(c, row_ptr, n, st, &es))) return rc;
    if ((rc = launch_nonfinite_scan(c, Y_in, 2 * n, st))) return rc;  // reported by the next synchronising call
    EpochArgs A;
    fill_args(A, row_ptr, col, q, n, a, b, neg, seed, c->d_status, es, 0, nullptr, nullptr, 0, 0);
    A.Y_in = reinterpret_cast<const float2*>(Y_in);
    A.Y_out = reinterpret_cast<float2*>(Y_out);
    A.lr = lr;
    A.t = uint32_t(epoch);
    return launch_epoch(c, A, 0, st);
}

int drgb_embed_epochs(drgb_ctx* c, float* Y, float* Y_tmp, const int32_t* row_ptr,
                      const int32_t* col, const uint32_t* q, int64_t n, float a, float b,
                      float lr0, int32_t neg, int32_t t_begin, int32_t t_end, int32_t n_epochs,
                      uint64_t seed, void* stream) {
    int rc = check_epoch_args(c, Y, Y_tmp, row_ptr, col, q, n, neg);
    if (rc) return rc;
    if (!(0 <= t_begin && t_begin <= t_end && t_end <= n_epochs) || n_epochs < 1)
        return set_error(c, DRGB_ERR_INVALID, "embed_epochs: bad epoch range");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int32_t nnz = 0;
    DRGB_CUDA(c, cudaMemcpyAsync(&nnz, row_ptr + n, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    DRGB_CUDA(c, cudaStreamSynchronize(st));
    if (nnz < 0) return set_error(c, DRGB_ERR_INVALID, "embed_epochs: row_ptr[n] < 0");
    if ((rc = ensure_scratch(c, epoch_scratch_bytes(n, nnz, 0), st))) return rc;
    if ((rc = launch_nonfinite_scan(c, Y, 2 * n, st))) return rc;  // reported by the next synchronising call
    return run_epochs(c, reinterpret_cast<float2*>(Y), reinterpret_cast<float2*>(Y_tmp), row_ptr, col, q, n, a,
                      b, lr0, neg, t_begin, t_end, n_epochs, seed, st, nnz, c->scratch);
}

}  // extern "C"
