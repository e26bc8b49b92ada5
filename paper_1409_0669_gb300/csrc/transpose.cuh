// Shared by the CSR transpose's two forms (k_grad.cu, k_transpose.cu).
#pragma once

#include "lak_internal.cuh"

namespace lak {

// Inclusive scan of v[0..len) in place; sums: scan_scratch_ints(len) ints.
int64_t scan_scratch_ints(int64_t len);
void launch_scan_i32(int32_t *v, int64_t len, int32_t *sums, cudaStream_t s);

// Columns the stable partition takes (two passes over column blocks of 2^10).
constexpr int64_t kTransposeMaxCols = 1LL << 30;
// CSC form (and, where vals is given, the values in its order; vbytes 2 or 4) by
// stable partitioning; n, nnz >= 1, n <= kTransposeMaxCols
// (the workspace is 0 beyond).
size_t transpose_workspace(int64_t n, int64_t nnz);
lak_status launch_transpose(int32_t *col_ptr, int32_t *row_idx, int32_t *perm, void *vals_t,
                            const int32_t *rp, const int32_t *ci, const void *vals, int64_t m,
                            int64_t n, int64_t nnz, int vbytes, void *ws, cudaStream_t s);

}  // namespace lak
