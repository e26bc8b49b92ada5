// CSR sparse matrix-vector product y = A x (the textbook product; the paper
// leaves sparse formats out of its study, Sec. 1).  Two kernels, three
// variants chosen on the host from the mean row length:
//
// Group per row (spmv_kernel): a group of G lanes (a power of two <= 32) owns
// one row; the lanes stride through the row's stored entries G at a time,
// each issuing U independent loads per step before using any of them,
// multiply by the gathered x[col] (cached load: neighbouring rows share x
// entries), and the group reduces with shuffles.  Short rows (stencils, mean
// <= 12) take one or two lanes per row with U covering the row, so a warp
// keeps 16-32 rows' loads in flight; their col_idx / vals loads are strided
// across the warp and go through L1 (one miss brings the lines the next lanes
// need).  In FP64 each lane keeps one accumulator chain.  Long rows (mean > 64) take
// spmv_long_kernel below; with an explicit configuration they take this kernel with
// more lanes per row, col_idx / vals streamed past L1.
//
// Warp-segmented (spmv_seg_kernel, 13 <= mean <= 64): a warp owns 32
// consecutive rows, whose entries are contiguous, and walks them in chunks of
// 32*U entries with coalesced (16-byte when aligned) loads; rows that cross
// lanes are joined by a segmented shuffle scan, rows that cross chunks in a
// per-warp shared accumulator with one writer per row per chunk -- no atomics,
// deterministic (the body lives in spmv_seg.cuh, shared with the batched
// kernel).
#include <type_traits>

#include "lak_internal.cuh"
#include "spmv_seg.cuh"

namespace lak {
namespace {

template <typename T, int U, int P>
__global__ void __launch_bounds__(512)
spmv_kernel(T *__restrict__ y, const int32_t *__restrict__ rp, const int32_t *__restrict__ ci,
            const T *__restrict__ vals, const T *__restrict__ x, int64_t m, int G, int inc) {
    LAK_PDL_WAIT();
    using Ac = typename Acc<T>::type;
    const int R = blockDim.x / G;
    const int grp = threadIdx.x / G;
    const int lg = threadIdx.x % G;
    int64_t row0, row_end, step;
    if (inc == LAK_INC_GLOBAL) {
        row0 = (int64_t)blockIdx.x * R;
        row_end = m;
        step = (int64_t)gridDim.x * R;
    } else {
        int64_t per = (m + gridDim.x - 1) / gridDim.x;
        per = (per + R - 1) / R * R;
        row0 = (int64_t)blockIdx.x * per;
        row_end = row0 + per < m ? row0 + per : m;
        step = R;
    }
    for (int64_t rb = row0; rb < row_end; rb += step) {   // block-uniform trip count
        const int64_t row = rb + grp;
        Ac acc[U];
#pragma unroll
        for (int u = 0; u < U; ++u) acc[u] = Ac(0);
        if (row < row_end) {
            const int64_t k0 = __ldg(rp + row);
            const int64_t k1 = __ldg(rp + row + 1);
            for (int64_t k = k0 + lg; k < k1; k += (int64_t)G * U) {
                int32_t col[U];
                T val[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int64_t kk = k + (int64_t)u * G;
                    if (kk < k1) {
                        ld_raw<4, P>(&col[u], ci + kk);
                        ld_raw<(int)sizeof(T), P>(&val[u], vals + kk);
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int64_t kk = k + (int64_t)u * G;
                    // FP64: one chain (GB300's FP64 pipe, not latency, is the limit,
                    // and U partial sums would cost U - 1 extra adds per row)
                    constexpr bool one_chain = sizeof(Ac) == 8;
                    if (kk < k1) {
                        Ac &a = one_chain ? acc[0] : acc[u];
                        a = fma_acc(widen(val[u]), widen(ld_cached(x + col[u])), a);
                    }
                }
            }
        }
        if constexpr (sizeof(Ac) != 8) {
#pragma unroll
            for (int w = 1; w < U; w <<= 1) {
#pragma unroll
                for (int u = 0; u + w < U; u += 2 * w) acc[u] += acc[u + w];
            }
        }
        const Ac s = group_sum(acc[0], G);
        if (lg == 0 && row < row_end) y[row] = narrow<T>(s);
    }
}

// One lane group's row: the G lanes of a group stride through its entries U at a time,
// `longest` (uniform over the warp) bounding the steps so that slots no row of the warp
// fills are not issued -- in FP64 a predicated-off FMA costs as much as a full one.
// S partial sums per lane, at most U: FP32 two, FP64 as many as leave its chains no longer
// than those of the one-row form, which has more lanes per row (with one chain in 4 lanes
// rows of 81 were 30 % further off).  All 32 lanes call it; every lane of a group returns
// the row's sum.
// Pos, of positions in the row: the step past a row of nearly 2^31 entries must not wrap, so
// signed ones leave the loop before it and unsigned ones have the room.
template <typename T, int G, int U, int P, int S, typename Pos>
__device__ __forceinline__ typename Acc<T>::type group_row(const int32_t *__restrict__ c,
                                                           const T *__restrict__ v,
                                                           const T *__restrict__ x, int32_t len,
                                                           int32_t longest, int lg) {
    using Ac = typename Acc<T>::type;
    constexpr bool wide = std::is_unsigned_v<Pos>;
    static_assert(wide ? (Pos)0x7fffffff + 32u * U > 0x7fffffffu : 0x80000000u % (G * U) == 0,
                  "no position of the last step wraps");
    Ac acc[S];
#pragma unroll
    for (int i = 0; i < S; ++i) acc[i] = Ac(0);
    for (Pos base = 0; base < (Pos)longest; base += G * U) {
        int32_t col[U];
        T val[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const Pos k = base + u * G + lg;
            if (k < (Pos)len) {
                ld_raw<4, P>(&col[u], c + k);
                ld_raw<(int)sizeof(T), P>(&val[u], v + k);
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const Pos k = base + u * G + lg;
            if (base + u * G < (Pos)longest && k < (Pos)len) {    // the first part is uniform
                Ac &a = acc[u % S];
                a = fma_acc(widen(val[u]), widen(ld_cached(x + col[u])), a);
            }
        }
        if constexpr (!wide)
            if (longest - base <= G * U) break;
    }
#pragma unroll
    for (int w = 1; w < S; w <<= 1) {
#pragma unroll
        for (int i = 0; i + w < S; i += 2 * w) acc[i] += acc[i + w];
    }
    return group_sum(acc[0], G);
}

// Long rows (mean > 64): G lanes per row, 32 / G rows per warp (group_row).  A warp
// whose longest row is far from the mean of its rows takes them one by one with all
// its lanes instead.  FP64 is bound by the pipe's warp instructions, so fewer lanes per
// row than the one-row form's serve it: 81 entries in 16 lanes took 8 FMAs (2 of them
// for slots no row fills) and 4 adds for two rows, in 4 lanes 21 and 5 for eight.
// Measured (us, one-row groups -> this; 41 M entries in rows of 81 near the diagonal, L2
// cold): FP64 187 -> 116, FP32 87 -> 65, BF16 106 -> 56; random columns FP64 186 -> 190,
// FP32 167 -> 166; rows with a heavy tail (up to 50000 entries, mean 76) as before (FP64 899 -> 865, FP32
// 441 -> 411).
template <typename T, int G, int S>
__global__ void __launch_bounds__(kSpmvLongBlock)
spmv_long_kernel(T *__restrict__ y, const int32_t *__restrict__ rp,
                 const int32_t *__restrict__ ci, const T *__restrict__ vals,
                 const T *__restrict__ x, int64_t m) {
    LAK_PDL_WAIT();
    using Ac = typename Acc<T>::type;
    // FP64 in less than a warp measured faster with unsigned positions (500000 rows of 81:
    // 116 against 120 us), the others with signed ones (FP32 65, 75; FP64 rows of 2500 68, 70)
    using Pos = std::conditional_t<sizeof(Ac) == 8 && G < 32, uint32_t, int32_t>;
    constexpr int U = 4, rows = 32 / G;
    const int lane = threadIdx.x & 31, lg = lane % G;
    const int64_t row0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * rows;
    if (row0 >= m) return;                                   // warp-uniform
    const int64_t row = row0 + lane / G;
    const int64_t last = row0 + rows < m ? row0 + rows : m;
    int32_t k0 = 0, len = 0;
    if (row < m) {
        k0 = __ldg(rp + row);
        len = __ldg(rp + row + 1) - k0;
    }
    const int32_t longest = __reduce_max_sync(0xffffffffu, len);
    const int64_t total = (int64_t)__ldg(rp + last) - __ldg(rp + row0);
    constexpr int F = rows == 2 ? 3 : 4;                    // twice the factor on the mean
    if (2 * (int64_t)longest * rows <= F * total + 64 * rows) {
        const Ac t = group_row<T, G, U, CACHED, S, Pos>(ci + k0, vals + k0, x, len, longest, lg);
        if (lg == 0 && row < m) y[row] = narrow<T>(t);
    } else {
        for (int r = 0; r < rows && row0 + r < m; ++r) {
            const int32_t a = __shfl_sync(0xffffffffu, k0, r * G);
            const int32_t n = __shfl_sync(0xffffffffu, len, r * G);
            const Ac t = group_row<T, 32, U, STREAM, sizeof(Ac) == 8 ? 1 : 2, Pos>(ci + a, vals + a, x, n, n, lane);
            if (lane == 0) y[row0 + r] = narrow<T>(t);
        }
    }
}

// Warp-segmented variant: the 32-row block body lives in spmv_seg.cuh (shared
// with the batched kernel); this kernel hands each warp its 32-row blocks.
template <typename T, int U, bool VLOAD, int WMAX = 16>
__global__ void __launch_bounds__(512)
spmv_seg_kernel(T *__restrict__ y, const int32_t *__restrict__ rp,
                const int32_t *__restrict__ ci, const T *__restrict__ vals,
                const T *__restrict__ x, int64_t m, int inc) {
    LAK_PDL_WAIT();
    using Ac = typename Acc<T>::type;
    const int warp = threadIdx.x >> 5;
    const int wpb = blockDim.x >> 5;
    uint32_t *rs_w;
    Ac *racc_w;
    if constexpr (sizeof(Ac) == 8) {
        __shared__ uint32_t rs_all[WMAX][33];
        __shared__ Ac racc_all[WMAX][32];
        rs_w = rs_all[warp];
        racc_w = racc_all[warp];
    } else {
        // sized to the block's warps (the launch passes the bytes), which leaves
        // more of the unified L1 to the x gathers: FP32 power-law 142.0 -> 140.0-
        // 141.0 us.  FP64 keeps static arrays, sized for WMAX warps (2 for its
        // 64-thread default blocks: 178.8 -> 176.8 us); the dynamic form cost it
        // two registers and 2 % (178.9 -> 182.9 us).
        extern __shared__ __align__(16) unsigned char seg_smem[];
        racc_w = reinterpret_cast<Ac *>(seg_smem) + (size_t)warp * 32;
        rs_w = reinterpret_cast<uint32_t *>(seg_smem + (size_t)wpb * 32 * sizeof(Ac)) + (size_t)warp * 33;
    }
    const int64_t nrb = (m + 31) / 32;               // 32-row blocks
    const int64_t gw = (int64_t)blockIdx.x * wpb + warp;
    const int64_t nw = (int64_t)gridDim.x * wpb;
    int64_t b0, b_end, b_step;
    if (inc == LAK_INC_GLOBAL) {
        b0 = gw;
        b_end = nrb;
        b_step = nw;
    } else {
        const int64_t per = (nrb + nw - 1) / nw;
        b0 = gw * per;
        b_end = b0 + per < nrb ? b0 + per : nrb;
        b_step = 1;
    }
    const int64_t nnz = __ldg(rp + m);
    for (int64_t b = b0; b < b_end; b += b_step)     // warp-uniform trip count
        seg_rows32<T, U, VLOAD>(y, rp, ci, vals, x, m, nnz, b, rs_w, racc_w);
}

template <typename T, int U>
lak_status spmv_seg_launch(T *yp, const int32_t *rp, const int32_t *ci, const T *vp,
                           const T *xp, int64_t m, const Launch &L, cudaStream_t s) {
    const bool vload = U % 4 == 0 && (uintptr_t)ci % 16 == 0 && (uintptr_t)vp % 16 == 0;
    using Ac = typename Acc<T>::type;
    const size_t smem = sizeof(Ac) == 8 ? 0 : (size_t)(L.block / 32) * (32 * sizeof(Ac) + 33 * 4);
    if constexpr (U % 4 == 0) {
        if (vload) {
            if (sizeof(Ac) == 8 && L.block <= 64)
                launch_k(spmv_seg_kernel<T, U, true, 2>, L.grid, L.block, smem, s, yp, rp, ci, vp, xp, m, L.inc);
            else
                launch_k(spmv_seg_kernel<T, U, true>, L.grid, L.block, smem, s, yp, rp, ci, vp, xp, m, L.inc);
            return check_launch("csr_spmv (warp-segmented)");
        }
    }
    launch_k(spmv_seg_kernel<T, U, false>, L.grid, L.block, smem, s, yp, rp, ci, vp, xp, m, L.inc);
    return check_launch("csr_spmv (warp-segmented)");
}

template <typename T>
lak_status spmv_t(void *y, const int32_t *rp, const int32_t *ci, const void *vals, const void *x,
                  int64_t m, const Launch &L, int G, cudaStream_t s) {
    T *yp = static_cast<T *>(y);
    const T *vp = static_cast<const T *>(vals);
    const T *xp = static_cast<const T *>(x);
    if (G == 0) {
        switch (L.vec) {
        case 1: return spmv_seg_launch<T, 1>(yp, rp, ci, vp, xp, m, L, s);
        case 2: return spmv_seg_launch<T, 2>(yp, rp, ci, vp, xp, m, L, s);
        case 4: return spmv_seg_launch<T, 4>(yp, rp, ci, vp, xp, m, L, s);
        case 8: return spmv_seg_launch<T, 8>(yp, rp, ci, vp, xp, m, L, s);
        case 16: return spmv_seg_launch<T, 16>(yp, rp, ci, vp, xp, m, L, s);
        default: return fail(LAK_EINVAL, "csr_spmv: unsupported vec %d", L.vec);
        }
    }
#define LAK_SPMV(UU)                                                                      \
    do {                                                                                  \
        if (G <= 4)                                                                       \
            launch_k(spmv_kernel<T, UU, CACHED>, L.grid, L.block, 0, s, yp, rp, ci, vp, xp, m, G, \
                                                                  L.inc);                 \
        else                                                                              \
            launch_k(spmv_kernel<T, UU, STREAM>, L.grid, L.block, 0, s, yp, rp, ci, vp, xp, m, G, \
                                                                  L.inc);                 \
    } while (0)
    switch (L.vec) {
    case 1: LAK_SPMV(1); break;
    case 2: LAK_SPMV(2); break;
    case 4: LAK_SPMV(4); break;
    case 8: LAK_SPMV(8); break;
    case 16: LAK_SPMV(16); break;
    default: return fail(LAK_EINVAL, "csr_spmv: unsupported vec %d", L.vec);
    }
#undef LAK_SPMV
    return check_launch("csr_spmv");
}

}  // namespace

namespace {

template <typename T>
lak_status spmv_long_t(void *y, const int32_t *rp, const int32_t *ci, const void *vals,
                       const void *x, int64_t m, int G, bool longer, cudaStream_t s) {
    T *yp = static_cast<T *>(y);
    const T *vp = static_cast<const T *>(vals);
    const T *xp = static_cast<const T *>(x);
    const unsigned grid = (unsigned)ceil_div(m * G, kSpmvLongBlock);
#define LAK_LONG(GG, SS)                                                                    \
    launch_k(spmv_long_kernel<T, GG, SS>, grid, kSpmvLongBlock, 0, s, yp, rp, ci, vp, xp, m)
    if constexpr (sizeof(T) == 8) {
        // chains as long as the general kernel's: 8 lanes of rows up to 100 need two of them
        switch (G) {
        case 4: LAK_LONG(4, 4); break;
        case 8: if (longer) LAK_LONG(8, 4); else LAK_LONG(8, 2); break;
        case 16: LAK_LONG(16, 2); break;
        default: LAK_LONG(32, 1); break;
        }
    } else {
        switch (G) {
        case 8: LAK_LONG(8, 2); break;
        case 16: LAK_LONG(16, 2); break;
        default: LAK_LONG(32, 2); break;
        }
    }
#undef LAK_LONG
    return check_launch("csr_spmv (long rows)");
}

}  // namespace

lak_status launch_spmv_long(lak_dtype dt, void *y, const int32_t *rp, const int32_t *ci,
                            const void *vals, const void *x, int64_t m, int group,
                            bool longer, cudaStream_t s) {
    switch (dt) {
    case LAK_F32: return spmv_long_t<float>(y, rp, ci, vals, x, m, group, longer, s);
    case LAK_F64: return spmv_long_t<double>(y, rp, ci, vals, x, m, group, longer, s);
    case LAK_BF16: return spmv_long_t<__nv_bfloat16>(y, rp, ci, vals, x, m, group, longer, s);
    case LAK_F16: return spmv_long_t<__half>(y, rp, ci, vals, x, m, group, longer, s);
    }
    return fail(LAK_EDTYPE, "csr_spmv: unknown dtype %d", (int)dt);
}

lak_status launch_spmv(lak_dtype dt, void *y, const int32_t *rp, const int32_t *ci,
                       const void *vals, const void *x, int64_t m, const Launch &L, int group,
                       cudaStream_t s) {
    switch (dt) {
    case LAK_F32: return spmv_t<float>(y, rp, ci, vals, x, m, L, group, s);
    case LAK_F64: return spmv_t<double>(y, rp, ci, vals, x, m, L, group, s);
    case LAK_BF16: return spmv_t<__nv_bfloat16>(y, rp, ci, vals, x, m, L, group, s);
    case LAK_F16: return spmv_t<__half>(y, rp, ci, vals, x, m, L, group, s);
    }
    return fail(LAK_EDTYPE, "csr_spmv: unknown dtype %d", (int)dt);
}

}  // namespace lak
