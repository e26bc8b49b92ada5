// The CSR transpose's stable partition (k_transpose.cu) for its entry points (k_grad.cu).
#pragma once

#include "lak_internal.cuh"

namespace lak {

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
