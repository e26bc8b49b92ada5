// CSC form of a CSR pattern by stable partitioning (csr_transpose and
// csr_transpose_vals of include/lak.h).
//
// What bounds it: moving nnz entries into column order.  Serving each entry's place
// from an atomic cursor scatters 4-byte stores over the whole output (one DRAM sector
// each) and leaves every column to be sorted afterwards; 32 M entries of a power-law
// matrix took 3.6 ms that way, and bringing the values into that order by a gather
// another 0.57 ms.  Here the entries move twice, as 16-byte records (column, row, CSR
// position, value):
//
//   1. partition by column block (2^s columns, about 4600 entries), a tile of
//      consecutive entries per thread block: counts per tile and column block, a scan
//      over the tiles of each column block, then every tile orders its records by
//      column block in shared memory and stores them as runs behind those of the
//      tiles before it.  Tiles run in order, so the stores of the tiles in flight lie
//      side by side and L2 completes the sectors.
//   2. one thread block per column block orders its records by column on chip the same
//      way (the scan also gives col_ptr) and writes the outputs consecutively.
//
// Ranks are stable: a warp ranks its 32 entries against counters of its own, and the
// warps' counters are scanned in warp order.  So every column keeps its entries in CSR
// order: the result of a stable counting sort, independent of scheduling, with no
// global atomics.  More than 1024 column blocks take the partition twice (low half of
// the block number, then high half).  Blocks are half an SM, so that one's loads and
// stores run under the other's ranking.
//
// Values of 16 and 32 bits travel in the records; 64-bit ones are gathered afterwards
// (beside the records they cost more than the gather: 3D Laplacian 128^3 666 against
// 548 us, power law about equal).
//
// Patterns with far fewer entries than rows or columns take the same passes: the cost of
// an empty row is its share of row_ptr (chunk_rows_kernel), that of a block of empty
// columns its part of col_ptr.  Atomic scatter -> this (us): 1000 entries in 10 M x 10 M
// 125 -> 71, 1 M in 50 M x 1 M 159 -> 144, 1 M in 64 M x 64 M 816 -> 613; 1000 in
// 1000 x 1000 17 -> 22 (launches).
//
// Measured (32 M entries of a power-law matrix, 2 M columns, FP32 values carried along):
// 0.89 ms against 3.3 ms for the atomic scatter, the columns' sort and the gather; three
// passes of 0.9-1.0 GB each, 0.45 ms at the copy rate.  Blocks of a whole SM
// (1024 threads, tiles of 8192) took 1.42 ms, ten-bit digits in one pass with column
// blocks of 32 K entries gathered through L2 1.30 ms, per-warp fronts without the
// exchange 2.1 ms.
#include "lak_internal.cuh"
#include "transpose.cuh"

namespace lak {
namespace {

constexpr int kDigitBits = 10;
constexpr int kMaxBlocks = 1 << kDigitBits;     // digits of a partition pass, at most
constexpr int kMaxColBits = 10;         // columns per block: at most 2^10 (or 2^12, make_plan)
constexpr int kTileWarps = 16;          // warps per block of the partition kernels
constexpr int kTileThreads = 32 * kTileWarps;
constexpr int kItems = 8;               // entries a lane takes of a tile
constexpr int kTile = kTileThreads * kItems;
constexpr int kOrderWarps = 16;         // warps per block of the ordering kernel

struct __align__(16) Rec {
    int32_t col, row, k;
    uint32_t v;                         // 16- or 32-bit value
};

// Stable rank of this lane's entry among the entries of digit d that the warp has seen:
// the warp's counter plus the number of lower lanes with that digit; the counter
// advances by the lanes'.  The lanes with equal digits are found with one ballot per
// bit of the digit (match.any measured about 100 cycles of an SM per warp here).
// All 32 lanes call it.
template <typename C>
__device__ __forceinline__ int32_t warp_rank(C *counter, int32_t d, int bits, bool valid,
                                             int lane) {
    unsigned same = __ballot_sync(0xffffffffu, valid);
    auto split = [&](int from, int to) {
#pragma unroll
        for (int i = from; i < to; ++i) {
            const bool one = d & (1 << i);
            const unsigned ones = __ballot_sync(0xffffffffu, one);
            same &= one ? ones : ~ones;
        }
    };
    split(0, 4);
    if (bits > 4) split(4, 6);          // warp-uniform
    if (bits > 6) split(6, 7);
    if (bits > 7) split(7, 8);
    if (bits > 8) split(8, 10);
    if (bits > 10) split(10, 12);
    const int leader = __ffs((int)same) - 1;        // of an invalid lane: any
    int32_t base = 0;
    if (valid && lane == leader) {
        base = counter[d];
        counter[d] = (C)(base + __popc(same));
    }
    base = __shfl_sync(0xffffffffu, base, leader < 0 ? 0 : leader);
    __syncwarp();                       // the next entry's leader may be another lane
    return base + __popc(same & ((1u << lane) - 1u));
}

// first[c] = row of entry c << bits, by the rows (every non-empty row holds the chunk
// starts that lie in it).  A warp reads kRowsPerLane rows per lane at a time; few of them
// hold a chunk start.  The whole warp fills in the chunks of a hub row (one thread's
// stores took 31 us for a power-law matrix of 2 M rows, all of it waiting for the longest).
constexpr int kChunkBits = 7, kChunk = 1 << kChunkBits;
constexpr int kRowsPerLane = 8;
__global__ void __launch_bounds__(256)
chunk_rows_kernel(int32_t *__restrict__ first, const int32_t *__restrict__ rp, int64_t m,
                  int bits) {
    LAK_PDL_ENTRY();
    constexpr int N = kRowsPerLane;
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * blockDim.x / 32;
    const int64_t up = (1LL << bits) - 1;
    for (int64_t r0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32 * (32 * N); r0 < m;
         r0 += warps * (32 * N)) {                          // warp-uniform
        int32_t at[N + 1];
#pragma unroll
        for (int j = 0; j <= N; ++j) {
            const int64_t r = r0 + 32 * j + (j < N ? lane : 0);
            at[j] = __ldg(rp + (r < m ? r : m));
        }
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const int32_t down = __shfl_down_sync(0xffffffffu, at[j], 1);
            const int32_t over = __shfl_sync(0xffffffffu, at[j + 1], 0);
            int32_t c = (int32_t)((at[j] + up) >> bits);
            const int32_t e = (int32_t)(((lane < 31 ? down : over) + up) >> bits);
            if (!__any_sync(0xffffffffu, c < e)) continue;
            const int64_t r = r0 + 32 * j;
            for (unsigned hubs = __ballot_sync(0xffffffffu, e - c > 8); hubs; hubs &= hubs - 1) {
                const int src = __ffs((int)hubs) - 1;
                const int32_t c0 = __shfl_sync(0xffffffffu, c, src);
                const int32_t e0 = __shfl_sync(0xffffffffu, e, src);
                for (int32_t i = c0 + lane; i < e0; i += 32) first[i] = (int32_t)(r + src);
                if (lane == src) c = e;
            }
            for (; c < e; ++c) first[c] = (int32_t)(r + lane);
        }
    }
}

// cells[b * tiles + tile] = entries of the tile with digit b.  Keys: columns, of which
// the digit is (column >> shift) & mask, or the digits that an earlier pass left.
template <typename K>
__global__ void __launch_bounds__(kTileThreads)
part_count_kernel(int32_t *__restrict__ cells, const K *__restrict__ keys, int64_t nnz, int shift,
                  int mask, int nb) {
    LAK_PDL_ENTRY();
    extern __shared__ int32_t part_smem[];
    for (int b = threadIdx.x; b < nb; b += blockDim.x) part_smem[b] = 0;
    __syncthreads();
    const int64_t t0 = (int64_t)blockIdx.x * kTile;
    int32_t c[kItems];
    if constexpr (sizeof(K) == 2) {
        // 16-byte aligned, and readable to the end of its 16 bytes
        Pack<uint16_t, 8> p;
        static_assert(kItems == 8, "digits of a thread");
        const int64_t k = t0 + threadIdx.x * kItems;
        if (k < nnz) load_pack<uint16_t, 8, STREAM>(p, keys + k);
#pragma unroll
        for (int i = 0; i < kItems; ++i)
            if (k + i < nnz) atomicAdd(part_smem + p.e[i], 1);
    } else {
        const int64_t k0 = t0 + threadIdx.x;
#pragma unroll
        for (int i = 0; i < kItems; ++i) {
            const int64_t k = k0 + i * kTileThreads;
            if (k < nnz) c[i] = __ldg(keys + k);
        }
#pragma unroll
        for (int i = 0; i < kItems; ++i)
            if (k0 + i * kTileThreads < nnz) atomicAdd(part_smem + ((c[i] >> shift) & mask), 1);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < nb; b += blockDim.x)
        cells[(int64_t)b * gridDim.x + blockIdx.x] = part_smem[b];
}

// Sum over a block of 1024 threads up to this one (inclusive); wtot: 32 ints, free again
// after the next barrier
__device__ __forceinline__ int32_t block_scan(int32_t v, int32_t *wtot) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t up = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += up;
    }
    if (lane == 31) wtot[warp] = v;
    __syncthreads();
    int32_t before = lane < warp ? wtot[lane] : 0;
    before = __reduce_add_sync(0xffffffffu, before);
    return v + before;
}

// Scan over the tiles of each digit, a block per digit: cells[b][tile] -> entries of the
// digit in the tiles before; totals[b].  (Three kernels over segments of tiles, one
// thread per digit, took 35 us a pass for 8000 tiles; this one and the next 9.)
__global__ void __launch_bounds__(1024)
cell_scan_kernel(int32_t *__restrict__ cells, int32_t *__restrict__ totals, int64_t tiles) {
    LAK_PDL_ENTRY();
    __shared__ int32_t wtot[32];
    __shared__ int32_t chunk;
    int32_t *v = cells + (int64_t)blockIdx.x * tiles;
    int32_t carry = 0;
    for (int64_t base = 0; base < tiles; base += 1024 * 8) {
        const int64_t i0 = base + threadIdx.x * 8;
        int32_t c[8], sum = 0;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            c[u] = i0 + u < tiles ? v[i0 + u] : 0;
            sum += c[u];
        }
        const int32_t incl = block_scan(sum, wtot);
        int32_t at = carry + incl - sum;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            if (i0 + u < tiles) v[i0 + u] = at;
            at += c[u];
        }
        if (threadIdx.x == 1023) chunk = incl;
        __syncthreads();
        carry += chunk;
        __syncthreads();
    }
    if (threadIdx.x == 0) totals[blockIdx.x] = carry;
}

// starts[b] = entries with digits below b (nb <= 1024)
__global__ void __launch_bounds__(1024)
starts_kernel(int32_t *__restrict__ starts, const int32_t *__restrict__ totals, int nb) {
    LAK_PDL_ENTRY();
    __shared__ int32_t wtot[32];
    const int b = threadIdx.x;
    const int32_t v = b < nb ? totals[b] : 0;
    const int32_t incl = block_scan(v, wtot);
    if (b < nb) starts[b] = incl - v;
}

// Threads per digit of a tile's scan over (digit, warp): as many as the block has, so that
// few digits don't leave most of it waiting for 16 counts in turn (the moves of 32 M
// entries by 7 and 6 bits: 284 -> 273 and 288 -> 241 us)
__device__ __forceinline__ int scan_split(int nb) {
    int q = 1;
    while (q * 2 <= kTileWarps && q * 2 * nb <= kTileThreads) q *= 2;
    return q;
}

// counts v[w * ld], w < n, replaced by `at` plus the sum of those before; returns the total
__device__ __forceinline__ int32_t run_counts(uint16_t *v, int ld, int n, int32_t at) {
    for (int w = 0; w < n; w += 4) {
        int32_t c[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) c[u] = w + u < n ? v[(w + u) * ld] : 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (w + u < n) v[(w + u) * ld] = (uint16_t)at;
            at += c[u];
        }
    }
    return at;
}

__device__ __forceinline__ int32_t sum_counts(const uint16_t *v, int ld, int n) {
    int32_t s = 0;
#pragma unroll 4
    for (int w = 0; w < n; ++w) s += v[w * ld];
    return s;
}

// Rows that a warp walks through to find those of its entries (32 a step, a step's loads
// behind the one before); beyond that every entry searches for its own.  1 M entries in the
// first and last of 16 M rows: 179 ms by walking only, 84 us.
constexpr int kWalkRows = 512;

constexpr size_t move_smem(int nb) {
    return (size_t)kTile * 16 + (size_t)nb * 4 + (size_t)kTileWarps * nb * 2;
}

// Orders a tile's records by column block in shared memory and stores them as runs.
// From the CSR arrays, or (CSR false) from the records of an earlier pass.
// E: the values' type (uint16_t, uint32_t; vals may be null).
// digits (may be null): the digit from bit `above` of the column on, for a later pass.
// rows: the entries' rows; where null they are found from row_ptr, `first` giving that of
// every kChunk-th entry.
template <typename E, bool CSR>
__global__ void __launch_bounds__(kTileThreads, 2)
part_move_kernel(Rec *__restrict__ out, uint16_t *__restrict__ digits, int above,
                 const int32_t *__restrict__ rp,
                 const int32_t *__restrict__ ci, const E *__restrict__ vals,
                 const Rec *__restrict__ in, const int32_t *__restrict__ cells,
                 const int32_t *__restrict__ starts, const int32_t *__restrict__ first,
                 const int32_t *__restrict__ rows, int64_t m, int64_t nnz, int shift, int mask,
                 int nb, int bits) {
    LAK_PDL_ENTRY();
    constexpr int ITEMS = kItems, TILE = kTile;
    extern __shared__ __align__(16) unsigned char move_raw[];
    Rec *stage = reinterpret_cast<Rec *>(move_raw);
    int32_t *delta = reinterpret_cast<int32_t *>(move_raw + (size_t)TILE * 16);
    uint16_t *count = reinterpret_cast<uint16_t *>(delta + nb);        // [warp][nb]
    __shared__ int32_t wtot[kTileWarps];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t t0 = (int64_t)blockIdx.x * TILE;
    const int64_t t1 = t0 + TILE < nnz ? t0 + TILE : nnz;
    for (int i = tid; i < kTileWarps * nb / 2; i += kTileThreads)
        reinterpret_cast<uint32_t *>(count)[i] = 0;
    __syncthreads();

    // 1. ranks within the warp; a lane keeps (digit, rank) and the row of its entries
    const int64_t w0 = t0 + (int64_t)warp * 32 * ITEMS;
    const int have = (int)(t1 - w0) - lane;         // item i is there where 32 i < have
    const int32_t k0 = (int32_t)w0 + lane;
    uint16_t *mine = count + warp * nb;
    uint32_t where[ITEMS];
    int32_t row[ITEMS];
    Rec rec[ITEMS];
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        rec[i].col = 0;
        rec[i].v = 0;
        if (32 * i < have) {
            if constexpr (CSR) {
                rec[i].col = __ldg(ci + w0 + lane + 32 * i);
                if (vals) rec[i].v = __ldg(vals + w0 + lane + 32 * i);
            } else {
                ld_raw<16, STREAM>(&rec[i], in + w0 + lane + 32 * i);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const int32_t d = (rec[i].col >> shift) & mask;
        const int32_t r = warp_rank(mine, d, bits, 32 * i < have, lane);
        where[i] = (uint32_t)d << 16 | (uint32_t)r;
    }
    if constexpr (CSR) {
        // the rows that the warp's entries lie in: run .. top
        int32_t run = 0, top = 0;
        const int64_t w1 = w0 + 32 * ITEMS < t1 ? w0 + 32 * ITEMS : t1;
        if (w0 < t1 && !rows) {
            run = __ldg(first + w0 / kChunk);
            const int64_t c1 = (w1 + kChunk - 1) / kChunk;
            top = c1 * kChunk < nnz ? __ldg(first + c1) : (int32_t)(m - 1);
        }
        if (rows) {                                         // grid-uniform
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) row[i] = 32 * i < have ? __ldg(rows + k0 + 32 * i) : 0;
        } else if (top - run <= kWalkRows) {                // warp-uniform
            // every non-empty row that begins inside the warp's entries leaves its number
            // at its first entry; an entry's row is the last such number up to it
            int32_t *marks = reinterpret_cast<int32_t *>(stage) + warp * 32 * ITEMS;
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) marks[32 * i + lane] = 0;
            __syncwarp();
            for (int64_t rb = run + 1; rb <= top; rb += 32) {
                const int64_t r = rb + lane;
                const int64_t a = r <= top ? (int64_t)__ldg(rp + r) : w1;
                const int64_t b = r <= top ? (int64_t)__ldg(rp + r + 1) : w1;
                if (a < w1 && b > a) marks[a - w0] = (int32_t)r;
                if (__any_sync(0xffffffffu, a >= w1)) break;
            }
            __syncwarp();
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) {
                const int32_t v = marks[32 * i + lane];
                const unsigned begun = __ballot_sync(0xffffffffu, v) & (0xffffffffu >> (31 - lane));
                const int32_t r = __shfl_sync(0xffffffffu, v, begun ? 31 - __clz((int)begun) : 0);
                row[i] = begun ? r : run;
                run = __shfl_sync(0xffffffffu, row[i], 31);
            }
        } else {
            // runs of empty rows: the last row in run .. top that begins at or before the
            // entry, by halving (all entries of the warp in step)
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) row[i] = run;
            for (int32_t len = top - run + 1; len > 1; len -= len / 2) {
                const int32_t half = len / 2;
#pragma unroll
                for (int i = 0; i < ITEMS; ++i)
                    if (32 * i < have && __ldg(rp + row[i] + half) <= k0 + 32 * i) row[i] += half;
            }
        }
    }
    __syncthreads();

    // 2. counts -> places in the tile (by column block, then warp); delta: from a place
    // in the tile to the place in the output
    {
        const int per = (nb + kTileThreads - 1) / kTileThreads;
        const int q = scan_split(nb), wn = kTileWarps / q;
        const int b0 = tid / q * per, b1 = b0 + per < nb ? b0 + per : nb;
        uint16_t *from = count + tid % q * wn * nb;
        int32_t sum = 0;
        for (int b = b0; b < b1; ++b) sum += sum_counts(from + b, nb, wn);
        int32_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t up = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += up;
        }
        if (lane == 31) wtot[warp] = incl;
        __syncthreads();
        int32_t at = incl - sum;
        for (int w = 0; w < warp; ++w) at += wtot[w];
        const int32_t *cell = cells + blockIdx.x;
        for (int b = b0; b < b1; ++b) {
            if (tid % q == 0)
                delta[b] = __ldg(starts + b) + __ldg(cell + (int64_t)b * gridDim.x) - at;
            at = run_counts(from + b, nb, wn, at);
        }
    }
    __syncthreads();

    // 3. records to their places in the tile
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        if (32 * i >= have) break;
        if constexpr (CSR) {
            rec[i].row = row[i];
            rec[i].k = k0 + 32 * i;
        }
        const int place = (int)mine[where[i] >> 16] + (int)(where[i] & 0xffffu);
        stage[place] = rec[i];
    }
    __syncthreads();

    // 4. runs to the output
    const int len = (int)(t1 - t0);
    for (int q = tid; q < len; q += kTileThreads) {
        const Rec rec = stage[q];
        const int32_t pos = delta[(rec.col >> shift) & mask] + q;
        st_raw<16>(out + pos, &rec);
        if (CSR && digits) digits[pos] = (uint16_t)(rec.col >> above);
    }
}

// bounds[b] = first record with a column of block b or later (records in block order); a
// warp per block, 33 ways at a time (25 dependent loads of a binary search took 25 us)
__global__ void __launch_bounds__(128)
bounds_kernel(int32_t *__restrict__ bounds, const Rec *__restrict__ recs, int64_t nnz,
              int64_t blocks, int s) {
    LAK_PDL_ENTRY();
    const int lane = threadIdx.x & 31;
    const int64_t b = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (b >= blocks) return;                                // warp-uniform
    const int64_t c = b << s;
    int64_t lo = 0, hi = nnz;
    while (hi - lo > 32) {
        const int64_t at = lo + (hi - lo) * (lane + 1) / 33;
        const int below = __popc(__ballot_sync(0xffffffffu, __ldg(&recs[at].col) < c));
        const int64_t l = __shfl_sync(0xffffffffu, at, below > 0 ? below - 1 : 0);
        const int64_t h = __shfl_sync(0xffffffffu, at, below < 32 ? below : 0);
        if (below > 0) lo = l + 1;
        if (below < 32) hi = h;
    }
    const bool is = lo + lane < hi && __ldg(&recs[lo + lane].col) < c;
    lo += __popc(__ballot_sync(0xffffffffu, is));
    if (lane == 0) bounds[b] = (int32_t)lo;
}

// Warps that rank the records of a column block of 2^s columns, so that their counters
// take 32 KB
constexpr int rank_warps(int s) { return s > kMaxColBits ? kOrderWarps >> 2 : kOrderWarps; }
// Records of a column block that are ordered on chip, 12 bytes each beside the counters
constexpr int kOrderItems = 12;
constexpr int order_cap(int s) { return 32 * rank_warps(s) * kOrderItems; }

constexpr size_t order_smem(int s) {
    return (size_t)rank_warps(s) * (1 << s) * 2 + 16 + (size_t)order_cap(s) * 12;
}

// One block per column block: orders its records by column and writes the CSC arrays.
// bounds: first record of every column block.
// The usual column block fits on chip: its records are read, ranked, placed in shared
// memory and written out consecutively.  A larger one (hub columns) is counted and
// ranked in place, its entries stored one by one.
template <typename E, int RW>
__global__ void __launch_bounds__(32 * kOrderWarps, 2)
order_kernel(int32_t *__restrict__ col_ptr, int32_t *__restrict__ row_idx,
             int32_t *__restrict__ perm, E *__restrict__ vals_t, const Rec *__restrict__ recs,
             const int32_t *__restrict__ bounds, int64_t n, int64_t nnz, int s) {
    LAK_PDL_ENTRY();
    constexpr int ITEMS = kOrderItems, CAP = 32 * RW * ITEMS, BIG = RW / 2;
    extern __shared__ __align__(16) unsigned char order_raw[];
    __shared__ int32_t wtot[kOrderWarps];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nc = 1 << s;
    const int64_t c0 = (int64_t)blockIdx.x << s;
    const int64_t b0 = bounds[blockIdx.x];
    const int64_t len = (blockIdx.x + 1 == gridDim.x ? nnz : bounds[blockIdx.x + 1]) - b0;
    if (len == 0) {                                         // block-uniform
        for (int j = tid; j < nc; j += 32 * kOrderWarps)
            if (c0 + j < n) col_ptr[c0 + j] = (int32_t)b0;
        if (blockIdx.x == gridDim.x - 1 && tid == 0) col_ptr[n] = (int32_t)nnz;
        return;
    }
    // counters per warp and column: 16 bits for the records on chip, 32 bits and half
    // the warps for more
    const bool small = len <= CAP;
    const int nw = small ? RW : BIG;
    uint16_t *half = reinterpret_cast<uint16_t *>(order_raw);
    int32_t *full = reinterpret_cast<int32_t *>(order_raw);
    for (int i = tid; i < RW * nc / 2; i += 32 * kOrderWarps) full[i] = 0;
    __syncthreads();
    const int64_t per = (len + nw * 32 - 1) / (nw * 32) * 32;
    const int64_t e0 = warp < nw ? warp * per : len;
    const int64_t e1 = e0 + per < len ? e0 + per : len;
    uint16_t *mine16 = half + warp * nc;
    int32_t *mine32 = full + warp * nc;
    uint32_t where[ITEMS];
    // on chip: item i of this lane is from[32 i] where 32 i < have (32-bit counts: with
    // 64-bit positions throughout, 32 M entries took 293 us here, now 282)
    const Rec *from = recs + b0 + e0 + lane;
    const int have = small ? (int)(e1 - e0) - lane : 0;
    const int32_t first = (int32_t)c0;
    if (small) {
        int32_t c[ITEMS];
#pragma unroll
        for (int i = 0; i < ITEMS; ++i)
            c[i] = 32 * i < have ? __ldg(&from[32 * i].col) - first : 0;
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            if (32 * i >= have + lane) break;               // warp-uniform
            const int32_t r = warp_rank(mine16, c[i], s, 32 * i < have, lane);
            where[i] = (uint32_t)c[i] << 16 | (uint32_t)r;
        }
    } else {
        for (int64_t k = e0 + lane; k < e1; k += 32)
            atomicAdd(mine32 + (int)(__ldg(&recs[b0 + k].col) - c0), 1);
    }
    __syncthreads();
    // exclusive scan over (column, warp); thread t takes columns [t cpt, t cpt + cpt)
    const int cpt = (nc + 32 * kOrderWarps - 1) / (32 * kOrderWarps);
    int32_t total = 0;
    for (int j = tid * cpt; j < (tid + 1) * cpt && j < nc; ++j) {
        if (small) {
#pragma unroll(RW < 8 ? RW : 8)
            for (int w = 0; w < RW; ++w) total += half[w * nc + j];
        } else {
            for (int w = 0; w < BIG; ++w) total += full[w * nc + j];
        }
    }
    int32_t incl = total;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t up = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += up;
    }
    if (lane == 31) wtot[warp] = incl;
    __syncthreads();
    int32_t at = incl - total;
    for (int w = 0; w < warp; ++w) at += wtot[w];
    for (int j = tid * cpt; j < (tid + 1) * cpt && j < nc; ++j) {
        if (c0 + j < n) col_ptr[c0 + j] = (int32_t)(b0 + at);
        if (small) {
#pragma unroll
            for (int w = 0; w < RW; w += 4) {
                int32_t c[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) c[u] = half[(w + u) * nc + j];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    half[(w + u) * nc + j] = (uint16_t)at;
                    at += c[u];
                }
            }
        } else {
            for (int w = 0; w < BIG; ++w) {
                const int32_t c = full[w * nc + j];
                full[w * nc + j] = at;
                at += c;
            }
        }
    }
    if (blockIdx.x == gridDim.x - 1 && tid == 0) col_ptr[n] = (int32_t)nnz;
    __syncthreads();
    if (small) {
        int32_t *srow = reinterpret_cast<int32_t *>(order_raw + ((size_t)RW * nc * 2 + 15) / 16 * 16);
        int32_t *sk = srow + CAP;
        uint32_t *sv = reinterpret_cast<uint32_t *>(sk + CAP);
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            if (32 * i >= have) break;
            Rec r;
            ld_raw<16, CACHED>(&r, from + 32 * i);
            const int place = (int)mine16[where[i] >> 16] + (int)(where[i] & 0xffffu);
            srow[place] = r.row;
            sk[place] = r.k;
            sv[place] = r.v;
        }
        __syncthreads();
        row_idx += b0;
        perm += b0;
        for (int q = tid; q < (int)len; q += 32 * kOrderWarps) {
            row_idx[q] = srow[q];
            perm[q] = sk[q];
        }
        if (vals_t) {
            vals_t += b0;
            for (int q = tid; q < (int)len; q += 32 * kOrderWarps) vals_t[q] = (E)sv[q];
        }
        return;
    }
    for (int64_t kb = e0; kb < e1; kb += 32) {              // warp-uniform
        const int64_t k = kb + lane;
        const bool valid = k < e1;
        Rec r{};
        if (valid) ld_raw<16, CACHED>(&r, recs + b0 + k);
        const int32_t pos = warp_rank(mine32, valid ? (int32_t)(r.col - c0) : 0, s, valid, lane);
        if (valid) {
            row_idx[b0 + pos] = r.row;
            perm[b0 + pos] = r.k;
            if (vals_t) vals_t[b0 + pos] = (E)r.v;
        }
    }
}

struct Plan {
    int s;                  // log2 of the columns per block
    int64_t blocks;         // column blocks
    int passes;             // partition passes (1 or 2)
    int bits[2], nb[2];     // of each pass: bits of its digit, number of digits
    int64_t tiles;
    size_t off_cells, off_totals, off_starts, off_first, off_rec[2], bytes;
};

size_t up256(size_t b) { return (b + 255) / 256 * 256; }

Plan make_plan(int64_t n, int64_t nnz) {
    Plan p{};
    // columns per block: as many as leave the mean column block three quarters of what
    // the ordering kernel holds on chip, and two blocks per SM or more where they would
    // still have 2048 entries
    const int64_t mean = order_cap(kMaxColBits) / 4 * 3;
    int s = kMaxColBits;
    auto blocks = [&](int bits) { return ((n - 1) >> bits) + 1; };
    while (s > 0 && blocks(s - 1) <= (int64_t)kMaxBlocks * kMaxBlocks &&
           (blocks(s) * mean < nnz || (blocks(s) < 304 && blocks(s) * 2048 < nnz)))
        --s;
    // four columns and more per entry: blocks of four times the columns, two thirds of their
    // room filled in the mean at most, where that saves the second pass or many blocks with
    // little to do (us: 1 M entries 4 M columns 104 -> 89, 64 M 612 -> 514; 100,000 entries
    // 1.6 M columns 53 -> 40)
    if (s == kMaxColBits && ((n / 4 >= nnz && blocks(s) > kMaxBlocks) ||
                             (n / 16 >= nnz && blocks(s) > 304)))
        s = kMaxColBits + 2;
    p.s = s;
    p.blocks = ((n - 1) >> s) + 1;
    int bits = 0;
    while ((1LL << bits) < p.blocks) ++bits;
    p.passes = bits > kDigitBits ? 2 : 1;
    p.bits[0] = p.passes == 1 ? bits : (bits + 1) / 2;
    p.bits[1] = bits - p.bits[0];
    p.nb[0] = p.passes == 1 ? (int)p.blocks : 1 << p.bits[0];
    p.nb[1] = p.passes == 1 ? 0 : (int)((p.blocks - 1) >> p.bits[0]) + 1;
    p.tiles = ceil_div(nnz, kTile);
    const int64_t nb = p.nb[0] > p.nb[1] ? p.nb[0] : p.nb[1];
    size_t at = 0;
    p.off_cells = at;
    at += up256((size_t)(p.tiles * nb) * 4);
    p.off_totals = at;
    at += up256((size_t)nb * 4);
    p.off_starts = at;
    at += up256((size_t)(p.blocks > nb ? p.blocks : nb) * 4);
    p.off_first = at;
    at += up256((size_t)ceil_div(nnz, kChunk) * 4);
    for (int i = 0; i < p.passes; ++i) {
        p.off_rec[i] = at;
        at += up256((size_t)nnz * 16);
    }
    p.bytes = at;
    return p;
}

template <typename E>
lak_status run(const Plan &p, int32_t *col_ptr, int32_t *row_idx, int32_t *perm, E *vals_t,
               const int32_t *rp, const int32_t *ci, const E *vals, int64_t m, int64_t n,
               int64_t nnz, char *w, cudaStream_t st) {
    int32_t *cells = reinterpret_cast<int32_t *>(w + p.off_cells);
    int32_t *totals = reinterpret_cast<int32_t *>(w + p.off_totals);
    int32_t *starts = reinterpret_cast<int32_t *>(w + p.off_starts);
    int32_t *first = reinterpret_cast<int32_t *>(w + p.off_first);
    Rec *rec[2];
    for (int i = 0; i < 2; ++i)
        rec[i] = reinterpret_cast<Rec *>(w + p.off_rec[i < p.passes ? i : 0]);
    const int move_most = (int)move_smem(kMaxBlocks);
    const int order_most = (int)order_smem(kMaxColBits);
    const bool wide = p.s > kMaxColBits;
    auto *order = wide ? order_kernel<E, rank_warps(kMaxColBits + 2)>
                       : order_kernel<E, rank_warps(kMaxColBits)>;
    cudaError_t e = cudaFuncSetAttribute(part_move_kernel<E, true>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, move_most);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(part_move_kernel<E, false>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, move_most);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(order, cudaFuncAttributeMaxDynamicSharedMemorySize, order_most);
    if (e != cudaSuccess)
        return fail(LAK_ECUDA, "csr_transpose: shared memory: %s", cudaGetErrorString(e));
    // more rows than entries: the rows of all entries, kept in row_idx until order_kernel
    // writes it (64 M rows of 1 M entries, 1 M columns: 265 us where each entry searches)
    int32_t *rows = m > nnz ? row_idx : nullptr;
    const int64_t row_blocks = ceil_div(m, 256 * kRowsPerLane);
    launch_k(chunk_rows_kernel, (unsigned)(row_blocks < 65535 ? row_blocks : 65535), 256, 0, st,
             rows ? rows : first, rp, m, rows ? 0 : kChunkBits);
    for (int i = 0; i < p.passes; ++i) {
        const int nb = p.nb[i];
        const int shift = p.s + (i ? p.bits[0] : 0);
        const int mask = p.passes == 2 && i == 0 ? nb - 1 : 0x7fffffff;
        const int bits = p.bits[i];
        // the second pass counts digits that the first left where its own records will go
        uint16_t *digits = p.passes == 2 ? reinterpret_cast<uint16_t *>(rec[1]) : nullptr;
        if (i == 0)
            launch_k(part_count_kernel<int32_t>, (unsigned)p.tiles, kTileThreads, (size_t)nb * 4,
                     st, cells, ci, nnz, shift, mask, nb);
        else
            launch_k(part_count_kernel<uint16_t>, (unsigned)p.tiles, kTileThreads, (size_t)nb * 4,
                     st, cells, (const uint16_t *)digits, nnz, shift, mask, nb);
        launch_k(cell_scan_kernel, (unsigned)nb, 1024, 0, st, cells, totals, p.tiles);
        launch_k(starts_kernel, 1, 1024, 0, st, starts, (const int32_t *)totals, nb);
        if (i == 0)
            launch_k(part_move_kernel<E, true>, (unsigned)p.tiles, kTileThreads, move_smem(nb),
                     st, rec[0], digits, p.s + p.bits[0], rp, ci, vals, (const Rec *)nullptr,
                     (const int32_t *)cells, (const int32_t *)starts, (const int32_t *)first,
                     (const int32_t *)rows, m, nnz, shift, mask, nb, bits);
        else
            launch_k(part_move_kernel<E, false>, (unsigned)p.tiles, kTileThreads, move_smem(nb),
                     st, rec[1], (uint16_t *)nullptr, 0, rp, ci, (const E *)nullptr,
                     (const Rec *)rec[0], (const int32_t *)cells, (const int32_t *)starts,
                     (const int32_t *)first, (const int32_t *)nullptr, m, nnz, shift, mask, nb, bits);
    }
    if (p.passes == 2)
        launch_k(bounds_kernel, (unsigned)ceil_div(p.blocks, 4), 128, 0, st, starts,
                 (const Rec *)rec[1], nnz, p.blocks, p.s);
    launch_k(order, (unsigned)p.blocks, 32 * kOrderWarps, order_smem(p.s), st,
             col_ptr, row_idx, perm, vals ? vals_t : (E *)nullptr, (const Rec *)rec[p.passes - 1],
             (const int32_t *)starts, n, nnz, p.s);
    return check_launch("csr_transpose");
}

}  // namespace

size_t transpose_workspace(int64_t n, int64_t nnz) {
    return n < 1 || nnz < 1 || n > kTransposeMaxCols ? 0 : make_plan(n, nnz).bytes;
}

lak_status launch_transpose(int32_t *col_ptr, int32_t *row_idx, int32_t *perm, void *vals_t,
                            const int32_t *rp, const int32_t *ci, const void *vals, int64_t m,
                            int64_t n, int64_t nnz, int vbytes, void *ws, cudaStream_t s) {
    const Plan p = make_plan(n, nnz);
    char *w = static_cast<char *>(ws);
    if (vbytes == 2)
        return run<uint16_t>(p, col_ptr, row_idx, perm, (uint16_t *)vals_t, rp, ci,
                             (const uint16_t *)vals, m, n, nnz, w, s);
    return run<uint32_t>(p, col_ptr, row_idx, perm, (uint32_t *)vals_t, rp, ci,
                         (const uint32_t *)vals, m, n, nnz, w, s);
}

}  // namespace lak
