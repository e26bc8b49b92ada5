// Dense products whose shape or alignment the one-group-per-row and the
// tile-per-block kernels of k_gemv.cu serve badly:
//
//   gemv_rows_kernel   row-major: R rows of one alignment share every load of x,
//                      their columns can be split over blocks, and x may start at
//                      any offset against the rows
//   gemv_tall_kernel   column-major with very many rows: a thread owns its rows
//                      over all columns, no combine at all
//   gemv_col_off_kernel  column-major, columns off 16 bytes: every warp takes columns
//                      of one offset and shifts its rows by it
//
// All compute y = alpha * A x + beta * y (y is not read when beta == 0).
#include "lak_internal.cuh"

namespace lak {
namespace {

template <typename T>
__device__ __forceinline__ T epilogue(typename Acc<T>::type t, typename Acc<T>::type alpha,
                                      typename Acc<T>::type beta, typename Acc<T>::type yold) {
    using Ac = typename Acc<T>::type;
    if (beta == Ac(0)) return narrow<T>(alpha * t);
    return narrow<T>(fma_acc(alpha, t, beta * yold));
}

// acc + <a, x> over one pack, as one FMA chain
template <typename T, int V>
__device__ __forceinline__ typename Acc<T>::type pack_dot(typename Acc<T>::type acc,
                                                          const Pack<T, V> &a,
                                                          const Pack<T, V> &x) {
#pragma unroll
    for (int v = 0; v < V; ++v) acc = fma_wide(a.e[v], x.e[v], acc);
    return acc;
}

// ---- row-major: R rows per block, columns split over blocks ------------------------
//
// What bounds the shapes this serves: few long rows left the GPU idle (one block per
// row: 30 rows of 2,097,152 FP64 ran as 30 warps), and rows whose length is not a
// multiple of 16 bytes start at other offsets than x, so the one-row kernel loads x
// one element at a time.
//
// Layout.  Rows r, r + P, ..., r + (R-1) P with P the smallest stride (a power of two,
// at most 16 bytes / element) at which rows start at the same offset modulo 16 bytes:
// a block takes one such set, so one head, one aligned body and ONE load of x serve R
// rows, with R 16-byte loads of A in flight per lane and step.  x is read through two
// aligned 16-byte loads whose 32 bytes are shifted in registers by the set's offset
// (uniform over the block; the second load hits L1).  blockIdx.y is the column split:
// with more than one, partial sums go to the workspace and the last block of a set to
// arrive adds them in split order (deterministic).  No load leaves [x, x + n) or the
// rows: packs whose window would are done one element at a time.
//
// Dependents may launch once every block is past its body, not at entry: a grid that
// starts while SMs of this one are still busy puts most of its few blocks on the SMs
// that are free first (4096 x 16384 FP64 by two rows: 208 us with the trigger at
// entry, 127 us here).
//
// Measured (us, before -> with row sets): 30 x 2097152 FP64 12110 -> 121 (FP64 pipe: 100),
// FP32 3780 -> 45 (5.6 TB/s); BF16 12007 x 11003 79 -> 45.6 (5.8 TB/s); FP32 16384 x
// 16383 252 -> 155 (6.9 TB/s); FP64 4096 x 16384 150 -> 122.
template <typename T, int R>
__global__ void __launch_bounds__(256, R == 1 ? 4 : 2)
gemv_rows_kernel(T *__restrict__ y, const T *__restrict__ A, const T *__restrict__ x, int64_t m,
                 int64_t n, int64_t lda, int P, typename Acc<T>::type alpha,
                 typename Acc<T>::type beta, typename Acc<T>::type *__restrict__ partials,
                 unsigned int *__restrict__ tickets) {
    LAK_PDL_WAIT();
    using Ac = typename Acc<T>::type;
    constexpr int ES = (int)sizeof(T);
    constexpr int V = 16 / ES;
    __shared__ Ac red[8][R];
    __shared__ int am_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    const int64_t set = blockIdx.x;
    const int64_t row0 = (set / P) * ((int64_t)R * P) + set % P;
    if (row0 >= m) return;                                  // block-uniform
    const int64_t left = (m - row0 + P - 1) / P;            // rows from row0 on, P apart
    const int nr = left < R ? (int)left : R;
    const int split = blockIdx.y, nsplit = gridDim.y;

    const T *a = A + row0 * lda;
    const int64_t step = (int64_t)P * lda;                  // from row to row of the set
    const int64_t mis = (int64_t)((uintptr_t)a % 16) / ES;
    int64_t h = mis ? V - mis : 0;
    if (h > n) h = n;
    int64_t b0 = 0, b1 = (n - h) / V;                       // packs of the body
    const uint32_t sb = (uint32_t)((uintptr_t)(x + h) % 16);
    if (sb) {
        // the window of pack c: 32 bytes from x + h + c V - sb/ES
        if (h * ES < sb) b0 = 1;
        if (h + b1 * V + V - (int64_t)sb / ES > n) --b1;
        if (b1 < b0) b1 = b0 = 0;
    }
    const int64_t head = b1 > b0 ? h + b0 * V : n;          // elements done one by one
    const int64_t tail = b1 > b0 ? h + b1 * V : n;

    Ac acc[R];
#pragma unroll
    for (int j = 0; j < R; ++j) acc[j] = Ac(0);
    if (split == 0)
        for (int64_t k = tid; k < head; k += blockDim.x) {
            const T xv = ld_cached(x + k);
#pragma unroll
            for (int j = 0; j < R; ++j)
                if (j < nr) acc[j] = fma_wide(a[j * step + k], xv, acc[j]);
        }
    if (split == nsplit - 1)
        for (int64_t k = tail + tid; k < n; k += blockDim.x) {
            const T xv = ld_cached(x + k);
#pragma unroll
            for (int j = 0; j < R; ++j)
                if (j < nr) acc[j] = fma_wide(a[j * step + k], xv, acc[j]);
        }
    const int64_t per = (b1 - b0 + nsplit - 1) / nsplit;
    const int64_t s0 = b0 + split * per;
    const int64_t s1 = s0 + per < b1 ? s0 + per : b1;
    const T *ab = a + h;
    const T *xb = x + h;
    auto body = [&](auto shifted, auto full) {
        // U packs a step: their loads are issued together and summed before the one add to the
        // running sum, in FP32 each pack by itself (one chain over both was 4 % further off;
        // 16-bit results round that away, and BF16 12007 x 11003 takes 44.7 us, not 45.1)
        constexpr int U = R == 1 ? 4 : 2;
        auto load_x = [&](Pack<T, V> &px, int64_t c) {
            if constexpr (shifted.value)
                load_window<T, CACHED>(px, xb + c * V, sb);
            else
                load_pack<T, V, CACHED>(px, xb + c * V);
        };
        int64_t c = s0 + tid;
        for (; c + (U - 1) * (int64_t)blockDim.x < s1; c += U * (int64_t)blockDim.x) {
            Pack<T, V> px[U], pa[U][R];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t cu = c + u * (int64_t)blockDim.x;
#pragma unroll
                for (int j = 0; j < R; ++j)
                    if (full.value || j < nr)
                        load_pack<T, V, STREAM>(pa[u][j], ab + j * step + cu * V);
                load_x(px[u], cu);
            }
#pragma unroll
            for (int j = 0; j < R; ++j) {
                if (!full.value && j >= nr) continue;
                if constexpr (sizeof(Ac) == 8) {
#pragma unroll
                    for (int u = 0; u < U; ++u) acc[j] = pack_dot<T, V>(acc[j], pa[u][j], px[u]);
                } else {
                    Ac t = pack_dot<T, V>(Ac(0), pa[0][j], px[0]);
#pragma unroll
                    for (int u = 1; u < U; ++u) {
                        if constexpr (ES == 4)
                            t += pack_dot<T, V>(Ac(0), pa[u][j], px[u]);
                        else
                            t = pack_dot<T, V>(t, pa[u][j], px[u]);
                    }
                    acc[j] += t;
                }
            }
        }
        for (; c < s1; c += blockDim.x) {
            Pack<T, V> px;
            load_x(px, c);
#pragma unroll
            for (int j = 0; j < R; ++j) {
                if (!full.value && j >= nr) continue;
                Pack<T, V> pa;
                load_pack<T, V, STREAM>(pa, ab + j * step + c * V);
                acc[j] += pack_dot<T, V>(Ac(0), pa, px);
            }
        }
    };
    using Yes = Flag<true>;
    using No = Flag<false>;
    if (nr == R) {
        if (sb) body(Yes{}, Yes{}); else body(No{}, Yes{});
    } else {
        if (sb) body(Yes{}, No{}); else body(No{}, No{});
    }

    LAK_PDL_TRIGGER();
    // block sums of the set's rows, held by thread j for row j
#pragma unroll
    for (int j = 0; j < R; ++j) acc[j] = group_sum(acc[j], 32);
    Ac t = Ac(0);
    if (nw == 1) {
#pragma unroll
        for (int j = 0; j < R; ++j)
            if (lane == j) t = acc[j];
    } else {
        if (lane == 0) {
#pragma unroll
            for (int j = 0; j < R; ++j) red[warp][j] = acc[j];
        }
        __syncthreads();
        if (tid < nr)
            for (int w = 0; w < nw; ++w) t += red[w][tid];
    }
    if (nsplit == 1) {
        if (tid < nr) {
            const int64_t row = row0 + (int64_t)tid * P;
            const Ac yold = beta != Ac(0) ? widen(y[row]) : Ac(0);
            y[row] = epilogue<T>(t, alpha, beta, yold);
        }
        return;
    }
    if (tid < nr) partials[(int64_t)split * m + row0 + (int64_t)tid * P] = t;
    __threadfence();
    __syncthreads();
    if (tid == 0) am_last = ticket_acq_rel(tickets + set, nsplit - 1) == (unsigned)nsplit - 1;
    __syncthreads();
    if (!am_last) return;
    for (int j = warp; j < nr; j += nw) {
        const int64_t row = row0 + (int64_t)j * P;
        double f = 0.0;                                     // split order per lane, then a tree
#pragma unroll 8
        for (int q = lane; q < nsplit; q += 32) f += (double)__ldcg(partials + (int64_t)q * m + row);
        f = group_sum(f, 32);
        if (lane == 0) {
            const Ac yold = beta != Ac(0) ? widen(y[row]) : Ac(0);
            y[row] = epilogue<T>((Ac)f, alpha, beta, yold);
        }
    }
}

// ---- column-major with very many rows ----------------------------------------------
//
// A thread owns V consecutive rows and walks all columns: every warp load is 32 V
// consecutive entries of one column, and nothing is combined between threads (the
// tile-per-block kernel splits its columns over the block's warps and adds their sums
// in shared memory).  Sums of kGemvTallOneSum columns are added to a running one, so that the
// chains of roundings are no longer than the tile-per-block kernel's (one chain over 30
// FP32 columns was 22 % further off, over 64 columns 64 %).  FP64 is bound by its pipe, on
// which those additions cost what the form saves (2097152 x 30: 118 us with one chain, 134
// with sums, 125 by tiles), so it comes here only with one such sum.
// SHIFT: columns start at other offsets than a multiple of 16 bytes; each pack is
// then read through two aligned loads and shifted by the column's offset (uniform
// over the grid; the second load hits L1).  The first and the last column, whose
// windows could leave the matrix, are read one element at a time.  FP32 is held to 32
// registers there, for a full SM (999983 x 17 20.6 -> 15.8 us).
// Tile-per-block -> this (us, L2 cold): FP32 1000000 x 8 16.0 -> 6.2, 2000000 x 30 49.9 ->
// 36.8 (6.5 TB/s), odd 999983 x 17 82 -> 15.8; BF16 2000000 x 30 34.5 -> 19.2; FP64 odd
// 700001 x 8 63 -> 18.5.
template <typename T, int V, bool SHIFT>
__global__ void __launch_bounds__(kGemvTallBlock, SHIFT && sizeof(T) == 4 ? 8 : 4)
gemv_tall_kernel(T *__restrict__ y, const T *__restrict__ A, const T *__restrict__ x, int64_t m,
                 int64_t n, int64_t lda, typename Acc<T>::type alpha,
                 typename Acc<T>::type beta, bool y_ok) {
    LAK_PDL_WAIT();
    using Ac = typename Acc<T>::type;
    const int64_t r0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * V;
    if (r0 >= m) return;
    const T *a = A + r0;
    if (r0 + V > m) {                                       // the last rows
        for (int64_t r = r0; r < m; ++r) {
            Ac t = Ac(0);
            for (int64_t j = 0; j < n; ++j) t = fma_wide(A[j * lda + r], ld_cached(x + j), t);
            const Ac yold = beta != Ac(0) ? widen(y[r]) : Ac(0);
            y[r] = epilogue<T>(t, alpha, beta, yold);
        }
        return;
    }
    Ac acc[V];
#pragma unroll
    for (int v = 0; v < V; ++v) acc[v] = Ac(0);
    auto scalar_column = [&](int64_t j) {
        const T xj = ld_cached(x + j);
#pragma unroll
        for (int v = 0; v < V; ++v) acc[v] = fma_wide(a[j * lda + v], xj, acc[v]);
    };
    int64_t j = 0, j1 = n;
    if constexpr (SHIFT) {
        scalar_column(0);
        j = 1;
        j1 = n - 1;
    }
    if constexpr (sizeof(T) == 2 || !SHIFT) {
        // K columns' loads together, then their sum
        constexpr int K = SHIFT ? 4 : kGemvTallOneSum;
        auto columns = [&](int64_t j, int count, auto whole) {
            Pack<T, V> pa[K];
            T xj[K];
#pragma unroll
            for (int i = 0; i < K; ++i) {
                if (!whole.value && i >= count) break;
                const T *p = a + (j + i) * lda;
                xj[i] = ld_cached(x + j + i);
                if constexpr (SHIFT)
                    load_window<T, CACHED>(pa[i], p, (uint32_t)((uintptr_t)p % 16));
                else
                    load_pack<T, V, STREAM>(pa[i], p);
            }
            Ac t[V];
#pragma unroll
            for (int v = 0; v < V; ++v) t[v] = Ac(0);
#pragma unroll
            for (int i = 0; i < K; ++i) {
                if (!whole.value && i >= count) break;
#pragma unroll
                for (int v = 0; v < V; ++v) t[v] = fma_wide(pa[i].e[v], xj[i], t[v]);
            }
#pragma unroll
            for (int v = 0; v < V; ++v) acc[v] += t[v];
        };
        for (; j + K <= j1; j += K) columns(j, K, Flag<true>{});
        if (j < j1) columns(j, (int)(j1 - j), Flag<false>{});
    } else {
        while (j < j1) {
            const int64_t je = j + kGemvTallOneSum < j1 ? j + kGemvTallOneSum : j1;
            Ac t[V];
#pragma unroll
            for (int v = 0; v < V; ++v) t[v] = Ac(0);
#pragma unroll 4
            for (; j < je; ++j) {
                Pack<T, V> pa;
                const T *p = a + j * lda;
                load_window<T, CACHED>(pa, p, (uint32_t)((uintptr_t)p % 16));
                const T xj = ld_cached(x + j);
#pragma unroll
                for (int v = 0; v < V; ++v) t[v] = fma_wide(pa.e[v], xj, t[v]);
            }
#pragma unroll
            for (int v = 0; v < V; ++v) acc[v] += t[v];
        }
    }
    if constexpr (SHIFT)
        if (n > 1) scalar_column(n - 1);
    LAK_PDL_TRIGGER();
    Pack<T, V> py;
    if (beta != Ac(0)) {
        if (y_ok) {
            load_pack<T, V, COHERENT>(py, y + r0);
        } else {
#pragma unroll
            for (int v = 0; v < V; ++v) py.e[v] = y[r0 + v];
        }
    }
#pragma unroll
    for (int v = 0; v < V; ++v)
        py.e[v] = epilogue<T>(acc[v], alpha, beta, beta != Ac(0) ? widen(py.e[v]) : Ac(0));
    if (y_ok) {
        store_pack<T, V>(y + r0, py);
    } else {
#pragma unroll
        for (int v = 0; v < V; ++v) y[r0 + v] = py.e[v];
    }
}

// ---- column-major, columns off 16 bytes ---------------------------------------------
//
// Where the columns do not start on 16-byte boundaries the tile-per-block kernel reads
// one element at a time.  Columns j and j + nw, nw warps per block, start at the same
// offset modulo 16 bytes (nw is a multiple of every such period), so each warp takes
// columns of one offset and shifts its window of 32 V rows down by it: all its loads are
// aligned 16-byte ones, and its sums are added to the block's rows at that shift.  A
// block owns 31 V rows, which every window covers; the rows read twice (1 / 32) are the
// neighbouring block's, in L2.  No load leaves a column's rows.  Splits over columns
// as in the tile-per-block kernel.  Tile-per-block -> this (us, back to back, L2 cold):
// FP32 7999 x 8000 117 -> 50 (5.1 TB/s), 3001 x 5000 39.6 -> 15.5; BF16 74 -> 33 and 26.5
// -> 13.1; FP64 208 -> 139 and 54.4 -> 40.4.  With the matrix in L2: FP32 3001 x 5000 20 ->
// 9.9, BF16 15.2 -> 9.9.
template <typename T>
__global__ void __launch_bounds__(kGemvOffBlock)
gemv_col_off_kernel(T *__restrict__ y, const T *__restrict__ A, const T *__restrict__ x, int64_t m,
                    int64_t n, int64_t lda, int64_t cols_per_split,
                    typename Acc<T>::type *__restrict__ partials,
                    unsigned int *__restrict__ tickets, typename Acc<T>::type alpha,
                    typename Acc<T>::type beta) {
    LAK_PDL_WAIT();
    using Ac = typename Acc<T>::type;
    constexpr int V = 16 / (int)sizeof(T), TILE = 32 * V, OWN = 31 * V;
    constexpr int NW = kGemvOffBlock / 32;
    __shared__ Ac red[NW * TILE];
    __shared__ int shift[NW];
    __shared__ int am_last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t tile0 = (int64_t)blockIdx.x * OWN;
    const int nsplit = gridDim.y;
    const int64_t c0 = (int64_t)blockIdx.y * cols_per_split;
    const int64_t c1 = c0 + cols_per_split < n ? c0 + cols_per_split : n;
    int sh = 0;
    if (c0 + warp < c1) sh = (int)((uintptr_t)(A + (c0 + warp) * lda + tile0) % 16) / (int)sizeof(T);
    if (lane == 0) shift[warp] = sh;
    const int64_t r = tile0 - sh + (int64_t)lane * V;        // this lane's rows r .. r + V - 1

    Ac acc[V];
#pragma unroll
    for (int v = 0; v < V; ++v) acc[v] = Ac(0);
    if (r >= 0 && r + V <= m) {
#pragma unroll 4
        for (int64_t j = c0 + warp; j < c1; j += NW) {
            Pack<T, V> pa;
            load_pack<T, V, STREAM>(pa, A + j * lda + r);
            const T xj = ld_cached(x + j);
#pragma unroll
            for (int v = 0; v < V; ++v) acc[v] = fma_wide(pa.e[v], xj, acc[v]);
        }
    } else if (r > -V && r < m) {
        for (int64_t j = c0 + warp; j < c1; j += NW) {
            const T xj = ld_cached(x + j);
#pragma unroll
            for (int v = 0; v < V; ++v)
                if (r + v >= 0 && r + v < m) acc[v] = fma_wide(A[j * lda + r + v], xj, acc[v]);
        }
    }
    if constexpr (sizeof(Ac) != 8) LAK_PDL_TRIGGER();
#pragma unroll
    for (int v = 0; v < V; ++v) red[warp * TILE + lane * V + v] = acc[v];
    __syncthreads();
    for (int rr = threadIdx.x; rr < OWN; rr += kGemvOffBlock) {
        const int64_t row = tile0 + rr;
        if (row >= m) break;
        Ac t = Ac(0);
#pragma unroll
        for (int w = 0; w < NW; ++w) t += red[w * TILE + rr + shift[w]];
        if (nsplit == 1)
            y[row] = epilogue<T>(t, alpha, beta, beta != Ac(0) ? widen(y[row]) : Ac(0));
        else
            partials[(int64_t)blockIdx.y * m + row] = t;
    }
    if (nsplit == 1) return;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0)
        am_last = ticket_acq_rel(tickets + blockIdx.x, nsplit - 1) == (unsigned)nsplit - 1;
    __syncthreads();
    if (!am_last) return;
    for (int rr = threadIdx.x; rr < OWN; rr += kGemvOffBlock) {
        const int64_t row = tile0 + rr;
        if (row >= m) break;
        // eight splits at a time, their loads together: one by one and in FP64 this tail was
        // a third of a product of 46 splits
        const Ac *p = partials + row;
        Ac t = Ac(0);
        int q = 0;
        for (; q + 8 <= nsplit; q += 8) {
            Ac u[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) u[i] = __ldcg(p + (int64_t)(q + i) * m);
            t += ((u[0] + u[1]) + (u[2] + u[3])) + ((u[4] + u[5]) + (u[6] + u[7]));
        }
        Ac u[7];
#pragma unroll
        for (int i = 0; i < 7; ++i) u[i] = q + i < nsplit ? __ldcg(p + (int64_t)(q + i) * m) : Ac(0);
        t += ((u[0] + u[1]) + (u[2] + u[3])) + ((u[4] + u[5]) + u[6]);
        y[row] = epilogue<T>(t, alpha, beta, beta != Ac(0) ? widen(y[row]) : Ac(0));
    }
}

template <typename T>
lak_status col_off_t(void *y, const void *A, const void *x, int64_t m, int64_t n, int64_t lda,
                     int splits, void *ws, double alpha, double beta, cudaStream_t s) {
    using Ac = typename Acc<T>::type;
    const int64_t tiles = ceil_div(m, 31 * (16 / (int64_t)sizeof(T)));
    Ac *partials = nullptr;
    if (splits > 1)
        partials = reinterpret_cast<Ac *>(static_cast<char *>(ws) + LAK_WS_COUNTER_BYTES);
    launch_k(gemv_col_off_kernel<T>, dim3((unsigned)tiles, (unsigned)splits), kGemvOffBlock, 0, s,
             static_cast<T *>(y), static_cast<const T *>(A), static_cast<const T *>(x), m, n, lda,
             ceil_div(n, splits), partials, static_cast<unsigned int *>(ws), (Ac)alpha, (Ac)beta);
    return check_launch("dense_gemv (column-major, unaligned columns)");
}

template <typename T>
lak_status rows_t(void *y, const void *A, const void *x, int64_t m, int64_t n, int64_t lda,
                  const RowsLaunch &L, void *ws, double alpha, double beta, cudaStream_t s) {
    using Ac = typename Acc<T>::type;
    T *yp = static_cast<T *>(y);
    const T *Ap = static_cast<const T *>(A);
    const T *xp = static_cast<const T *>(x);
    unsigned int *tickets = static_cast<unsigned int *>(ws);
    Ac *partials = nullptr;
    if (L.splits > 1)
        partials = reinterpret_cast<Ac *>(static_cast<char *>(ws) + LAK_WS_COUNTER_BYTES);
    const dim3 grid((unsigned)L.sets, (unsigned)L.splits);
#define LAK_ROWS(RR)                                                                           \
    launch_k(gemv_rows_kernel<T, RR>, grid, L.block, 0, s, yp, Ap, xp, m, n, lda, L.period,    \
             (Ac)alpha, (Ac)beta, partials, tickets)
    if (L.rows == 1)
        LAK_ROWS(1);
    else
        LAK_ROWS(4);
#undef LAK_ROWS
    return check_launch("dense_gemv (row-major, row sets)");
}

template <typename T>
lak_status tall_t(void *y, const void *A, const void *x, int64_t m, int64_t n, int64_t lda,
                  double alpha, double beta, cudaStream_t s) {
    using Ac = typename Acc<T>::type;
    constexpr int V = 16 / (int)sizeof(T);
    constexpr int block = kGemvTallBlock;
    T *yp = static_cast<T *>(y);
    const T *Ap = static_cast<const T *>(A);
    const T *xp = static_cast<const T *>(x);
    const bool aligned = (uintptr_t)A % 16 == 0 && (lda * (int64_t)sizeof(T)) % 16 == 0;
    const bool y_ok = (uintptr_t)y % 16 == 0;
    const unsigned grid = (unsigned)ceil_div(m, (int64_t)V * block);
    if (aligned)
        launch_k(gemv_tall_kernel<T, V, false>, grid, block, 0, s, yp, Ap, xp, m, n, lda,
                 (Ac)alpha, (Ac)beta, y_ok);
    else
        launch_k(gemv_tall_kernel<T, V, true>, grid, block, 0, s, yp, Ap, xp, m, n, lda,
                 (Ac)alpha, (Ac)beta, y_ok);
    return check_launch("dense_gemv (column-major, many rows)");
}

}  // namespace

lak_status launch_gemv_rows(lak_dtype dt, void *y, const void *A, const void *x, int64_t m,
                            int64_t n, int64_t lda, const RowsLaunch &L, void *ws, double alpha,
                            double beta, cudaStream_t s) {
    switch (dt) {
    case LAK_F32: return rows_t<float>(y, A, x, m, n, lda, L, ws, alpha, beta, s);
    case LAK_F64: return rows_t<double>(y, A, x, m, n, lda, L, ws, alpha, beta, s);
    case LAK_BF16: return rows_t<__nv_bfloat16>(y, A, x, m, n, lda, L, ws, alpha, beta, s);
    case LAK_F16: return rows_t<__half>(y, A, x, m, n, lda, L, ws, alpha, beta, s);
    }
    return fail(LAK_EDTYPE, "dense_gemv: unknown dtype %d", (int)dt);
}

lak_status launch_gemv_tall(lak_dtype dt, void *y, const void *A, const void *x, int64_t m,
                            int64_t n, int64_t lda, double alpha, double beta, cudaStream_t s) {
    switch (dt) {
    case LAK_F32: return tall_t<float>(y, A, x, m, n, lda, alpha, beta, s);
    case LAK_F64: return tall_t<double>(y, A, x, m, n, lda, alpha, beta, s);
    case LAK_BF16: return tall_t<__nv_bfloat16>(y, A, x, m, n, lda, alpha, beta, s);
    case LAK_F16: return tall_t<__half>(y, A, x, m, n, lda, alpha, beta, s);
    }
    return fail(LAK_EDTYPE, "dense_gemv: unknown dtype %d", (int)dt);
}

lak_status launch_gemv_col_off(lak_dtype dt, void *y, const void *A, const void *x, int64_t m,
                               int64_t n, int64_t lda, int splits, void *ws, double alpha,
                               double beta, cudaStream_t s) {
    switch (dt) {
    case LAK_F32: return col_off_t<float>(y, A, x, m, n, lda, splits, ws, alpha, beta, s);
    case LAK_F64: return col_off_t<double>(y, A, x, m, n, lda, splits, ws, alpha, beta, s);
    case LAK_BF16: return col_off_t<__nv_bfloat16>(y, A, x, m, n, lda, splits, ws, alpha, beta, s);
    case LAK_F16: return col_off_t<__half>(y, A, x, m, n, lda, splits, ws, alpha, beta, s);
    }
    return fail(LAK_EDTYPE, "dense_gemv: unknown dtype %d", (int)dt);
}

}  // namespace lak
