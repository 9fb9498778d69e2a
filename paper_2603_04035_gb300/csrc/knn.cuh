// Internal interface of the k-NN kernels.
#pragma once
#include "common.cuh"

namespace drgb {

int check_knn_args(Ctx* c, const float* X, int64_t n, int d, int k, const void* idx_out,
                   const void* dist_out);
// Exact FP32 k-NN scan: query p is row rows[p] (null: p) of Q; `separate`: Q is
// another matrix than X, so no row is excluded as the query itself.
// This and the other scans split the database into chunks when `part` (part_bytes
// of scratch, knn_scan_scratch_bytes for the preferred split) holds the partial
// lists, and take it whole when it is null or too small; the results are the same.
int launch_knn_scan(Ctx* c, const float* Q, int64_t nq, bool separate, const int64_t* rows, const float* X, int64_t n,
                    int d, int k, int32_t* idx_out, float* dist_out, cudaStream_t st, void* part, size_t part_bytes);
size_t knn_scan_scratch_bytes(const Ctx* c, int64_t n_rows, int64_t n, int d, int k);
// Exact FP32 scan of the rows listed in rows32[0 .. cnt).  On entry each listed
// row of idx_out/dist_out must already hold k
// distinct points other than the row in ascending order of their FP32
// distances (the direct sum over dimensions), INFINITY where it has fewer:
// the scan keeps only points within the listed k-th distance.  Results are
// written to the listed rows.
int launch_knn_exact_rows_n(Ctx* c, const float* X, int64_t n, int d, int k, const int32_t* rows32, int64_t cnt,
                            int32_t* idx_out, float* dist_out, cudaStream_t st, void* part_scratch,
                            size_t part_bytes);
// The same over the cells that each listed row can reach: Xp holds the points
// in cell order (cell C: positions [cell_beg[C], cell_beg[C+1]), in the sphere
// (cell_c[C], cell_r[C]); position p holds point perm[p]; indices ascend within
// a cell).  *done is false, and nothing was enqueued, when there is one cell, the
// points are few or part_bytes do not hold the lists.
int launch_knn_cells(Ctx* c, const float* X, const float* Xp, int64_t n, int d, int k, const int32_t* rows,
                     int64_t cnt, int K, const int32_t* perm, const int32_t* cell_beg, const float* cell_c,
                     const float* cell_r, int32_t* idx_out, float* dist_out, cudaStream_t st, void* part,
                     size_t part_bytes, bool* done);
// The same for the queries list[0 .. *count) of a query set (as for knn_wide),
// a count that stays on the device; bound[0 .. *count): KNN_UNBOUND.
static constexpr int32_t KNN_UNBOUND = 0x7F7F7F7F;  // no bound published yet (every byte the same)
int launch_knn_exact_listed(Ctx* c, const float* Q, bool separate, const int64_t* rows, const float* X, int64_t n,
                            int d, int k, const int32_t* list, const int32_t* count, int32_t* bound, int32_t* idx_out,
                            float* dist_out, cudaStream_t st, void* part, size_t part_bytes);
// Merge C partial k-lists per listed row: list l of row r at
// (l * cnt + r) * k in pidx/pd2 (squared distances, ascending by (distance,
// index), ended early by index -1); the k best by (distance, index) go to
// row rows32[r] (null: r) of idx_out/dist_out (Euclidean distances); `none`
// is the index written where a row has fewer than k.
int launch_merge_partials(Ctx* c, const int32_t* pidx, const float* pd2, int64_t cnt, int C, int k,
                          const int32_t* rows32, int32_t* idx_out, float* dist_out, cudaStream_t st,
                          int32_t none = INT32_MAX);
// Per query row: sum over its k targets of max(0, rank_X - k); td, cnt: n_rows x k scratch.
int launch_rank(Ctx* c, const float* X, int64_t n, int d, int k, const int64_t* rows, int64_t n_rows,
                const int32_t* tgt, float* td, int32_t* cnt, int64_t* excess_out, cudaStream_t st);
int launch_nonfinite_scan(Ctx* c, const float* X, int64_t count, cudaStream_t st);

// BF16 tensor-core candidate generation + FP32 re-rank (knn_tc.cu).
bool knn_tc_preferred(int64_t n, int d, int k);
size_t knn_tc_scratch_bytes(int64_t n, int d);
// `scratch` must hold knn_tc_scratch_bytes(n, d) bytes (256-byte aligned).
// With defer_rows/defer_count (device; *defer_count zeroed by the caller) the
// uncertified rows are appended there (row indices of X) and not re-scanned:
// the caller re-scans them later (launch_knn_exact_rows_n), which lets many
// k-NN runs be enqueued without a host synchronisation.
int knn_tc(Ctx* c, const float* X, int64_t n, int d, int k, bool f16, int32_t* idx_out, float* dist_out,
           cudaStream_t st, void* scratch, int32_t* defer_rows = nullptr, int32_t* defer_count = nullptr);
// Bytes of scratch a deferred re-scan may use for its partial lists.
size_t knn_rescan_part_bytes();

// The same for larger problems on the tensor cores (knn_wide.cu).
// Uncertified queries are re-scanned without their number being read back, unless
// that is deferred to the caller (as for knn_tc).  `scratch` holds knn_wide_scratch_bytes.
bool knn_wide_preferred(int64_t nq, int64_t n, int d, int k);
size_t knn_wide_scratch_bytes(const Ctx* c, int64_t nq, int64_t n, int d);
int knn_wide(Ctx* c, const float* Q, int64_t nq, bool separate, const int64_t* rows, const float* X, int64_t n, int d,
             int k, int32_t* idx_out, float* dist_out, cudaStream_t st, void* scratch, int32_t* defer_rows = nullptr,
             int32_t* defer_count = nullptr);
// Whichever of the two is preferred and has its scratch.
size_t knn_queries_scratch_bytes(const Ctx* c, int64_t nq, int64_t n, int d, int k);
int knn_queries(Ctx* c, const float* Q, int64_t nq, bool separate, const int64_t* rows, const float* X, int64_t n,
                int d, int k, int32_t* idx_out, float* dist_out, cudaStream_t st, void* scratch, size_t scratch_bytes);

// Spatial order for the tensor-core k-NN (knn_order.cu): K cells from
// farthest-point pivots; perm[p] = point at position p (p < n), cell c holds
// positions [cell_beg[c], cell_beg[c+1]) inside the sphere (centre[c], radius[c]).
int knn_order_cells(int64_t n);
size_t knn_order_scratch_bytes(int64_t n, int d, int K);
int knn_order(Ctx* c, const float* X, int64_t n, int d, int K, int32_t* perm, int32_t* cell_beg, float* centre,
              float* radius, void* scratch, cudaStream_t st);

// k-NN graph with the mode resolved (0 = auto).  `scratch` holds scratch_bytes;
// knn_scratch_bytes gives what the mode wants and in *least what it cannot do
// without (0 for the scans, which then run unsplit).
static constexpr int KNN_WIDE = 5;  // knn_wide (auto mode only)
int knn_resolve_mode(int64_t n, int d, int k, int mode);
size_t knn_scratch_bytes(const Ctx* c, int64_t n, int d, int k, int mode, size_t* least);
// defer_rows/defer_count: as for knn_tc (the exact-scan modes leave no
// uncertified rows).
int knn_run(Ctx* c, const float* X, int64_t n, int d, int k, int mode, int32_t* idx_out, float* dist_out,
            cudaStream_t st, void* scratch, size_t scratch_bytes, int32_t* defer_rows = nullptr,
            int32_t* defer_count = nullptr);

}  // namespace drgb
