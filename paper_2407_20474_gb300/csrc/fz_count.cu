// fz_count.cu -- the exact counting table of the factorization sets.
//
//   C[j][r] = |Z(r, (g_{j+1}, ..., g_d))|,  j = 0..d (0-based), r = 0..n,
//   C[d][r] = [r == 0],   C[j][r] = sum_{t >= 0} C[j+1][r - t g_{j+1}].
//
// By the disjoint recurrence of Section 2 (Lemma "disjdyn") C[i-1][r] is
// |Z_{>=i}(r)|, the size of the block incr_i(Z_{>=i}(r)) = Z_{=i}(r + g_i)
// whose saving the paper describes in Section 2.3.  It gives every block's
// size and start, hence exact output offsets for every warp.
//
// Each row is a strided inclusive prefix sum of the row below it (stride
// g_{j+1}): for every residue class rho mod g the entries rho, rho + g, ...
// are summed in order.  Short chains are scanned by a warp or a lane each or
// tile by tile; long chains are cut into blocks of RB entries, the block sums
// are scanned by the same routine (they form a strided array of the same
// shape), and the blocks are then re-walked with their carries.  All sums
// saturate at 2^64 - 1.
#include <cstdlib>
#include <cstring>

#include "fz_internal.cuh"

namespace fz {

namespace {

constexpr int64_t DIRECT_T = 4096;  // chains up to this length: one warp each
constexpr int64_t LANE_T = 256;     // chains up to this length, 32 or more: one lane each
constexpr int64_t CHAIN_T = 128;    // fewer than 32 chains up to this length: one warp each
constexpr int LANE_ILP = 8;
constexpr int64_t TILE_MAX_T = 16384;  // fewer than 8 chains up to this length: a tile each
constexpr int RB = 32;              // entries per block in the blocked scan
constexpr int THREADS = 256;

// ---------------------------------------------------------------------------
// Tile scan: a block scans `width` (1, 8 or 32) neighbouring residue chains, its
// threads cut into 256 / width segments of TILE_U consecutive chain entries (16
// for a row on its own, 8 in the batched scans' 64 registers), so that loads
// cover neighbouring entries of the row, all of a chunk's entries are in
// flight at once, and each is read once.
// The segments' sums meet by shuffles and in shared memory.  For chains longer
// than 256 entries, where a warp or a lane a chain takes dozens of dependent
// rounds of loads (six rows of 39065 entries, chains of 200 to 600: 47 us by a
// warp a chain, 34 by tiles of 8; twelve rows of 1106 entries, chains of 25 to
// 70: 44 and 57).  Entry r of the chains is entry off + r es of the row.
// ---------------------------------------------------------------------------
template <int TILE_U, class In>
__device__ __forceinline__ void tile_scan(In input, uint64_t *__restrict__ out, int64_t len,
                                          int64_t g, int64_t first, int width,
                                          int64_t ones_below, int64_t off = 0, int64_t es = 1) {
    __shared__ uint64_t part[2][8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int cls = threadIdx.x & (width - 1), seg = threadIdx.x / width;
    const int nseg = THREADS / width;
    const int64_t rho = first + cls;
    const int64_t chains = g < len ? g : len;
    const int64_t T = rho < chains ? (len - rho + g - 1) / g : 0;
    const int64_t Tmax = (len - first + g - 1) / g;  // the tile's longest chain
    uint64_t carry = 0;
    int buf = 0;
    for (int64_t t0 = 0; t0 < Tmax; t0 += (int64_t)nseg * TILE_U, buf ^= 1) {
        const int64_t tb = t0 + (int64_t)seg * TILE_U;
        uint64_t v[TILE_U];
#pragma unroll
        for (int u = 0; u < TILE_U; ++u)
            v[u] = tb + u < T ? input(off + (rho + (tb + u) * g) * es) : 0ull;
#pragma unroll
        for (int u = 1; u < TILE_U; ++u) v[u] = sat_add(v[u], v[u - 1]);
        uint64_t x = v[TILE_U - 1];  // inclusive over the warp's segments of the class
        for (int o = width; o < 32; o <<= 1) {
            const uint64_t y = __shfl_up_sync(FULL, x, o);
            if (lane >= o) x = sat_add(x, y);
        }
        if (lane >= 32 - width) part[buf][warp][cls] = x;
        uint64_t before = __shfl_up_sync(FULL, x, width & 31);
        if (lane < width) before = 0;
        __syncthreads();
        before = sat_add(before, carry);
#pragma unroll
        for (int w = 0; w < THREADS / 32; ++w) {
            const uint64_t y = part[buf][w][cls];
            if (w < warp) before = sat_add(before, y);
            carry = sat_add(carry, y);
        }
#pragma unroll
        for (int u = 0; u < TILE_U; ++u) {
            const int64_t x = off + (rho + (tb + u) * g) * es;
            if (tb + u < T) out[x] = x < ones_below ? 1ull : sat_add(before, v[u]);
        }
    }
}

__global__ void __launch_bounds__(THREADS, 4)
row_tile_kernel(const uint64_t *__restrict__ in, uint64_t *__restrict__ out, int64_t len, int64_t g,
                int width) {
    tile_scan<16>([&](int64_t r) { return __ldg(in + r); }, out, len, g,
              (int64_t)blockIdx.x * width, width, 0);
}

// One warp per residue chain; 4 x 32 entries loaded ahead of the scan.
__global__ void __launch_bounds__(THREADS)
chain_scan_direct_kernel(const uint64_t *__restrict__ in, uint64_t *__restrict__ out,
                         int64_t len, int64_t g) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t chains = g < len ? g : len;
    for (int64_t rho = warp; rho < chains; rho += nwarps) {
        const int64_t T = (len - rho + g - 1) / g;
        uint64_t carry = 0;
        for (int64_t t0 = 0; t0 < T; t0 += 128) {
            uint64_t v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                int64_t t = t0 + u * 32 + lane;
                v[u] = t < T ? __ldg(in + rho + t * g) : 0ull;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                int64_t t = t0 + u * 32 + lane;
                uint64_t s = sat_add(warp_incl_scan_sat(v[u], lane), carry);
                if (t < T) out[rho + t * g] = s;
                carry = shfl_u64(s, 31);
            }
        }
    }
}

// S[b*g + rho] = sum of the RB entries of chain rho in block b.
__global__ void __launch_bounds__(THREADS)
block_sum_kernel(const uint64_t *__restrict__ in, uint64_t *__restrict__ S, int64_t len,
                 int64_t g, int64_t slen) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (; i < slen; i += stride) {
        const int64_t b = i / g, rho = i - b * g;
        const int64_t r0 = (b * RB) * g + rho;
        uint64_t acc = 0;
#pragma unroll 8
        for (int t = 0; t < RB; ++t) {
            int64_t r = r0 + (int64_t)t * g;
            if (r < len) acc = sat_add(acc, __ldg(in + r));
        }
        S[i] = acc;
    }
}

// out[r] = carry(block) + running sum inside the block.  At most 64
// registers (4 blocks per SM), so that it fits beside an enumeration capped
// at 3 blocks per SM.
__global__ void __launch_bounds__(THREADS, 4)
block_apply_kernel(const uint64_t *__restrict__ in, uint64_t *__restrict__ out,
                   const uint64_t *__restrict__ Sincl, int64_t len, int64_t g, int64_t slen) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (; i < slen; i += stride) {
        const int64_t b = i / g, rho = i - b * g;
        uint64_t acc = b > 0 ? Sincl[i - g] : 0ull;
        const int64_t r0 = (b * RB) * g + rho;
#pragma unroll 4
        for (int t = 0; t < RB; ++t) {
            int64_t r = r0 + (int64_t)t * g;
            if (r < len) {
                acc = sat_add(acc, __ldg(in + r));
                out[r] = acc;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Short tables (n <= SMALL_N): all rows of a table in one launch, one block,
// the row in hand in shared memory.  A row is scanned by doubling: log2(n / g)
// steps add the entry s = g, 2 g, 4 g, ... below.  Block 0: the count table
// (or its row 0 only), block 1: the candidates table.  Row by row these are a
// launch each of which the GPU runs in 3 us, 12 launches for a set of width 9.
// A plan's two tables take it up to SMALL_N (rebuild of 1e6 rows of width 6: 86
// us, 90 row by row), one table alone up to SMALL_ONE_N: its d - 2 scans row by
// row beside it at n = 3500, 6000, 11500: 18, 19, 21 us against 23, 29, 63 for
// width 5, 13, 14, 14 against 14, 18, 36 for width 3.
// ---------------------------------------------------------------------------
constexpr int SMALL_N = 12000, SMALL_ONE_N = 3000;
constexpr int SMALL_THREADS = 1024;
struct SmallTables {
    uint64_t *C;      // rows 0..d, or null
    uint64_t *C0;     // row 0 only, or null
    uint64_t *RT;     // rows 0..lam, or null
    uint64_t *sums;   // sums[j] of row j's entries (each clamped to 2^32), or null
    int d, n, lam, clamp_row, clamp_top;
    int g[FZ_MAX_D];
};

__global__ void __launch_bounds__(SMALL_THREADS)
    small_tables_kernel(const __grid_constant__ SmallTables P) {
    extern __shared__ __align__(16) uint64_t small_smem[];
    __shared__ uint64_t part[SMALL_THREADS / 32];
    const bool runs = P.C == nullptr && P.C0 == nullptr ? true : blockIdx.x == 1;
    const int len = P.n + 1, rows = runs ? P.lam : P.d;
    uint64_t *a = small_smem, *b = small_smem + len;
    uint64_t *out = runs ? P.RT : P.C;
    for (int r = threadIdx.x; r < len; r += SMALL_THREADS) {
        const uint64_t v = runs || r == 0 ? 1ull : 0ull;
        a[r] = v;
        if (out) out[(int64_t)rows * len + r] = v;
    }
    __syncthreads();
    for (int j = rows - 1;; --j) {
        if (!runs && P.sums) {  // of row j + 1, in hand
            uint64_t acc = 0;
            for (int r = threadIdx.x; r < len; r += SMALL_THREADS)
                acc += a[r] < (1ull << 32) ? a[r] : (1ull << 32);
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1) acc += __shfl_xor_sync(FULL, acc, o);
            if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
            __syncthreads();
            if (threadIdx.x == 0) {
                for (int w = 1; w < SMALL_THREADS / 32; ++w) acc += part[w];
                P.sums[j + 1] = acc;
            }
            __syncthreads();
        }
        if (j < 0) break;
        for (int64_t s = P.g[j]; s < len; s *= 2) {
            for (int r = threadIdx.x; r < len; r += SMALL_THREADS)
                b[r] = r >= s ? sat_add(a[r], a[r - s]) : a[r];
            __syncthreads();
            uint64_t *t = a;
            a = b;
            b = t;
        }
        if (runs && j == P.clamp_row) {
            for (int r = threadIdx.x; r < len && r < P.clamp_top; r += SMALL_THREADS) a[r] = 1ull;
            __syncthreads();
        }
        if (out)
            for (int r = threadIdx.x; r < len; r += SMALL_THREADS) out[(int64_t)j * len + r] = a[r];
    }
    if (!runs && P.C0)
        for (int r = threadIdx.x; r < len; r += SMALL_THREADS) P.C0[r] = a[r];
}

int launch_small_tables(const SmallTables &P, cudaStream_t s) {
    static DeviceOnce attr_set;
    int dev = 0;
    FZ_CUDA_TRY(cudaGetDevice(&dev));
    if (!attr_set.is_set(dev)) {
        FZ_CUDA_TRY(cudaFuncSetAttribute(small_tables_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         2 * (SMALL_N + 1) * 8));
        attr_set.set(dev);
    }
    const int blocks = (P.C || P.C0 ? 1 : 0) + (P.RT ? 1 : 0);
    small_tables_kernel<<<blocks, SMALL_THREADS, 2 * ((size_t)P.n + 1) * 8, s>>>(P);
    note_launch();
    FZ_CUDA_TRY(cudaGetLastError());
    return FZ_OK;
}

int grid_for(int64_t work, int per_block) {
    int64_t b = (work + per_block - 1) / per_block;
    if (b < 1) b = 1;
    if (b > 65535LL * 16) b = 65535LL * 16;
    return (int)b;
}

// Scratch words the blocked scan needs for an array of `len` entries, stride g.
int64_t scan_tmp_words(int64_t len, int64_t g) {
    int64_t T = (len + g - 1) / g;
    if (len <= 0 || T <= DIRECT_T) return 0;
    int64_t nrb = (T + RB - 1) / RB;
    int64_t slen = nrb * g;
    return 2 * slen + scan_tmp_words(slen, g);
}

// out[r] = sum_{t >= 0, r - t g >= 0} in[r - t g], for r < len.
int strided_scan(const uint64_t *in, uint64_t *out, int64_t len, int64_t g, uint64_t *tmp,
                 cudaStream_t s) {
    if (len <= 0) return FZ_OK;
    const int64_t T = (len + g - 1) / g;
    if (T <= DIRECT_T) {
        int64_t chains = g < len ? g : len;
        if (chains >= 8 && T > LANE_T) {
            // 8 chains a block: a single row has few, and latency bounds it.  A
            // block has one tile, so every tile has a block (chains of more
            // than LANE_T entries: at most 2^20 of them).
            row_tile_kernel<<<(unsigned)((chains + 7) / 8), THREADS, 0, s>>>(in, out, len, g, 8);
            note_launch();
            FZ_CUDA_TRY(cudaGetLastError());
            return FZ_OK;
        }
        int blocks = grid_for(chains * 32, THREADS);
        chain_scan_direct_kernel<<<blocks, THREADS, 0, s>>>(in, out, len, g);
        note_launch();
        FZ_CUDA_TRY(cudaGetLastError());
        return FZ_OK;
    }
    const int64_t nrb = (T + RB - 1) / RB;
    const int64_t slen = nrb * g;
    uint64_t *S = tmp, *Sincl = tmp + slen;
    block_sum_kernel<<<grid_for(slen, THREADS), THREADS, 0, s>>>(in, S, len, g, slen);
    note_launch();
    FZ_CUDA_TRY(cudaGetLastError());
    int rc = strided_scan(S, Sincl, slen, g, tmp + 2 * slen, s);
    if (rc != FZ_OK) return rc;
    block_apply_kernel<<<grid_for(slen, THREADS), THREADS, 0, s>>>(in, out, Sincl, len, g, slen);
    note_launch();
    FZ_CUDA_TRY(cudaGetLastError());
    return FZ_OK;
}

}  // namespace

int64_t count_table_tmp_words(const int32_t *g, int d, int32_t n) {
    int64_t w = 0;
    for (int j = 0; j < d; ++j) {
        int64_t t = scan_tmp_words((int64_t)n + 1, g[j]);
        if (t > w) w = t;
    }
    return w;
}

int64_t exclusive_scan_tmp_words(int64_t len) { return scan_tmp_words(len, 1); }

bool small_tables(int32_t n) { return n <= SMALL_N; }

int launch_tables_small(const int32_t *g, int d, int32_t n, uint64_t *C, uint64_t *RT, int lam,
                        int clamp_row, int64_t clamp_top, uint64_t *sums, cudaStream_t s) {
    SmallTables P{};
    P.C = C;
    P.RT = RT;
    P.sums = sums;
    P.d = d;
    P.n = n;
    P.lam = lam;
    P.clamp_row = clamp_top > 0 ? clamp_row : -1;
    P.clamp_top = (int)(clamp_top < (int64_t)n + 1 ? clamp_top : (int64_t)n + 1);
    for (int i = 0; i < d; ++i) P.g[i] = g[i];
    return launch_small_tables(P, s);
}

// The last rows of a count table from their closed forms: C[d] the delta row,
// C[d-1][r] = [g_d | r], C[d-2][r] = |Z(r, (g_{d-1}, g_d))|; null rows are not
// written.  Bound by the stores: three rows of 2e6 entries in one launch and no
// scan (count table of width 4: 109 us with four scans, 69 with two; all counts
// to 39064 for width 6: 86, 71).
__global__ void __launch_bounds__(THREADS)
    tail_rows_kernel(const __grid_constant__ PairForm F, FastDiv last, uint64_t *__restrict__ pair,
                     uint64_t *__restrict__ one, uint64_t *__restrict__ delta, int64_t len) {
    const int64_t step = (int64_t)gridDim.x * THREADS;
    for (int64_t r = (int64_t)blockIdx.x * THREADS + threadIdx.x; r < len; r += step) {
        const uint32_t x = (uint32_t)r;
        if (delta) delta[r] = r == 0 ? 1ull : 0ull;
        if (one) one[r] = fd_mod(x, last) == 0u ? 1ull : 0ull;
        if (pair) pair[r] = pair_form_count(F, x);
    }
}

// pair needs d >= 2.
int launch_tail_rows(const int32_t *g, int d, uint64_t *pair, uint64_t *one, uint64_t *delta,
                     int64_t len, cudaStream_t s) {
    const PairForm F = d >= 2 ? make_pair_form(g[d - 2], g[d - 1]) : PairForm{};
    tail_rows_kernel<<<grid_for(len, THREADS), THREADS, 0, s>>>(
        F, make_fastdiv((uint32_t)g[d - 1]), pair, one, delta, len);
    note_launch();
    FZ_CUDA_TRY(cudaGetLastError());
    return FZ_OK;
}

int launch_count_table_tmp(const int32_t *g, int d, int32_t n, uint64_t *table, uint64_t *tmp,
                           cudaStream_t s, bool one_block) {
    if (one_block && n <= SMALL_ONE_N)
        return launch_tables_small(g, d, n, table, nullptr, 0, -1, 0, nullptr, s);
    const int64_t len = (int64_t)n + 1;
    uint64_t *last = table + (int64_t)d * len;
    int rc = launch_tail_rows(g, d, d >= 2 ? last - 2 * len : nullptr, last - len, last, len, s);
    if (rc != FZ_OK) return rc;
    for (int j = d - 3; j >= 0; --j) {
        rc = strided_scan(table + (int64_t)(j + 1) * len, table + (int64_t)j * len, len,
                              g[j], tmp, s);
        if (rc != FZ_OK) return rc;
    }
    return FZ_OK;
}

// The last rows of a candidates table: ones, and x div g + 1 above them (1 below
// `clamp`).
__global__ void __launch_bounds__(THREADS)
    head_rows_kernel(FastDiv g, uint64_t *__restrict__ lin, uint64_t *__restrict__ ones,
                     int64_t clamp, int64_t len) {
    const int64_t step = (int64_t)gridDim.x * THREADS;
    for (int64_t r = (int64_t)blockIdx.x * THREADS + threadIdx.x; r < len; r += step) {
        ones[r] = 1ull;
        if (lin) lin[r] = r < clamp ? 1ull : (uint64_t)fd_div((uint32_t)r, g) + 1ull;
    }
}

__global__ void row_ones_kernel(uint64_t *__restrict__ row, int64_t len) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (; i < len; i += stride) row[i] = 1ull;
}

// Number of depth-lam nodes (runs of sibling leaves) under a node at depth j
// with remainder x: RT[lam][x] = 1 and RT[j] = RT[j+1] strided-summed with
// stride g_j -- the count-table recurrence over the leading generators.
int launch_runs_table(const int32_t *g, int lam, int32_t n, uint64_t *RT, uint64_t *tmp,
                      int clamp_row, int64_t clamp_top, cudaStream_t s, bool one_block) {
    if (one_block && n <= SMALL_ONE_N)
        return launch_tables_small(g, lam, n, nullptr, RT, lam, clamp_row, clamp_top, nullptr, s);
    const int64_t len = (int64_t)n + 1;
    uint64_t *ones = RT + (int64_t)lam * len;
    head_rows_kernel<<<grid_for(len, THREADS), THREADS, 0, s>>>(
        make_fastdiv(lam >= 1 ? (uint32_t)g[lam - 1] : 1u), lam >= 1 ? ones - len : nullptr, ones,
        clamp_row == lam - 1 ? clamp_top : 0, len);
    note_launch();
    FZ_CUDA_TRY(cudaGetLastError());
    for (int j = lam - 2; j >= 0; --j) {
        int rc = strided_scan(RT + (int64_t)(j + 1) * len, RT + (int64_t)j * len, len, g[j],
                              tmp, s);
        if (rc != FZ_OK) return rc;
        if (j == clamp_row && clamp_top > 0) {
            const int64_t m = clamp_top < len ? clamp_top : len;
            row_ones_kernel<<<grid_for(m, THREADS), THREADS, 0, s>>>(RT + (int64_t)j * len, m);
            note_launch();
            FZ_CUDA_TRY(cudaGetLastError());
        }
    }
    return FZ_OK;
}

// ---------------------------------------------------------------------------
// Batched strided scans: many independent rows (of many instances' count and
// runs tables) in one launch.  Each CTA executes one task: a range of chains
// scanned directly (one warp per chain), a range of block sums, a range of
// chains of block sums, a range of block applications, or a range of a row
// initialisation (delta or ones).
// ---------------------------------------------------------------------------
// Logical entry r of a job's rows is entry off + r * es of the table row
// (es = 1, off = 0: the whole row; es = g_1, off = n mod g_1: the one chain
// of row 0 that is ever read).
__device__ __forceinline__ uint64_t scan_input(const ScanJob &J, const uint64_t *in, int64_t x) {
    if (J.input == SCAN_LOAD) return __ldg(in + x);
    if (J.input == SCAN_PAIR) return pair_form_count(J.pair, (uint32_t)x);
    return (uint64_t)fd_div((uint32_t)x, J.lin) + 1ull;
}

// One chain by a warp, input(x) -> out (or S -> Sincl with a plain view).
template <class In>
__device__ __forceinline__ void chain_scan_warp(In input, uint64_t *__restrict__ out, int64_t len,
                                                int64_t g, int64_t rho, int lane,
                                                int64_t ones_below = 0, int64_t off = 0,
                                                int64_t es = 1) {
    const int64_t T = (len - rho + g - 1) / g;
    uint64_t carry = 0;
    for (int64_t t0 = 0; t0 < T; t0 += 128) {
        uint64_t v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            int64_t t = t0 + u * 32 + lane;
            v[u] = t < T ? input(off + (rho + t * g) * es) : 0ull;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            int64_t t = t0 + u * 32 + lane;
            uint64_t sc = sat_add(warp_incl_scan_sat(v[u], lane), carry);
            const int64_t x = off + (rho + t * g) * es;
            if (t < T) out[x] = x < ones_below ? 1ull : sc;
            carry = shfl_u64(sc, 31);
        }
    }
}

// One chain by a lane, walked down with its own running sum; a warp's loads and
// stores cover 32 neighbouring entries of a row (one 256-byte span when es =
// 1).  `input` without a branch on where the entries come from keeps LANE_ILP
// loads in flight: a batch of 512 partial memos rebuilds in 224 us, 256 with
// the branch at every entry.
template <class In>
__device__ __forceinline__ void chain_scan_lane(In input, const ScanJob &J, int64_t rho, int64_t off,
                                                int64_t es) {
    uint64_t *__restrict__ out = J.out;
    const int64_t T = (J.len - rho + J.g - 1) / J.g;
    uint64_t acc = 0;
    for (int64_t t0 = 0; t0 < T; t0 += LANE_ILP) {
        uint64_t v[LANE_ILP];
#pragma unroll
        for (int u = 0; u < LANE_ILP; ++u)
            v[u] = t0 + u < T ? input(off + (rho + (t0 + u) * J.g) * es) : 0ull;
#pragma unroll
        for (int u = 0; u < LANE_ILP; ++u) {
            if (t0 + u < T) {
                const int64_t x = off + (rho + (t0 + u) * J.g) * es;
                acc = sat_add(acc, v[u]);
                out[x] = x < J.ones_below ? 1ull : acc;
            }
        }
    }
}

constexpr int SCAN_MINB_DEFAULT = 4;

// MINB: CTAs per SM the register budget is set for (3 fit without a bound:
// 76 registers; 4 at 64 registers; 6 at 40 registers with a few spills).
template <int MINB>
__global__ void __launch_bounds__(THREADS, MINB) scan_tasks_kernel(const ScanJob *__restrict__ jobs,
                                                                   const ScanTask *__restrict__ tasks) {
    const ScanTask t = tasks[blockIdx.x];
    const ScanJob J = jobs[t.job];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int nwarps = blockDim.x >> 5;
    const int64_t es = J.es ? J.es : 1, off = J.off;
    switch (t.kind) {
        case TK_TILE:  // t.end: chains of the tile
            tile_scan<8>([&](int64_t x) { return scan_input(J, J.in, x); }, J.out, J.len, J.g, t.begin,
                      (int)t.end, J.ones_below, off, es);
            break;
        case TK_CHAIN:
            for (int64_t rho = t.begin + warp; rho < t.end; rho += nwarps)
                chain_scan_warp([&](int64_t x) { return scan_input(J, J.in, x); }, J.out, J.len, J.g, rho,
                                lane, J.ones_below, off, es);
            break;
        case TK_LANES: {
            // lane l of warp w: chain begin + 32 w + l
            const int64_t rho = t.begin + (int64_t)warp * 32 + lane;
            if (rho >= t.end) break;
            if (J.input == SCAN_LOAD)
                chain_scan_lane([&](int64_t x) { return __ldg(J.in + x); }, J, rho, off, es);
            else
                chain_scan_lane([&](int64_t x) { return scan_input(J, J.in, x); }, J, rho, off, es);
            break;
        }
        case TK_SSCAN:
            for (int64_t rho = t.begin + warp; rho < t.end; rho += nwarps)
                chain_scan_warp([&](int64_t x) { return __ldg(J.S + x); }, J.Sincl, J.slen, J.g, rho,
                                lane);
            break;
        case TK_BSUM: {
            const int64_t rb = J.rb > 0 ? J.rb : RB;
            for (int64_t i = t.begin + threadIdx.x; i < t.end; i += blockDim.x) {
                const int64_t b = i / J.g, rho = i - b * J.g;
                const int64_t r0 = (b * rb) * J.g + rho;
                uint64_t acc = 0;
                for (int64_t u0 = 0; u0 < rb; u0 += 8) {
                    uint64_t v[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int64_t r = r0 + (u0 + u) * J.g;
                        v[u] = (u0 + u < rb && r < J.len) ? scan_input(J, J.in, off + r * es) : 0ull;
                    }
#pragma unroll
                    for (int u = 0; u < 8; ++u) acc = sat_add(acc, v[u]);
                }
                J.S[i] = acc;
            }
            break;
        }
        case TK_APPLY: {
            const int64_t rb = J.rb > 0 ? J.rb : RB;
            for (int64_t i = t.begin + threadIdx.x; i < t.end; i += blockDim.x) {
                const int64_t b = i / J.g, rho = i - b * J.g;
                uint64_t acc = b > 0 ? J.Sincl[i - J.g] : 0ull;
                const int64_t r0 = (b * rb) * J.g + rho;
                for (int64_t u0 = 0; u0 < rb; u0 += 8) {
                    uint64_t v[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int64_t r = r0 + (u0 + u) * J.g;
                        v[u] = (u0 + u < rb && r < J.len) ? scan_input(J, J.in, off + r * es) : 0ull;
                    }
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int64_t r = r0 + (u0 + u) * J.g;
                        if (u0 + u < rb && r < J.len) {
                            const int64_t x = off + r * es;
                            acc = sat_add(acc, v[u]);
                            J.out[x] = x < J.ones_below ? 1ull : acc;
                        }
                    }
                }
            }
            break;
        }
        case TK_DELTA:
            for (int64_t i = t.begin + threadIdx.x; i < t.end; i += blockDim.x)
                J.out[off + i * es] = (off + i * es == 0) ? 1ull : 0ull;
            break;
        case TK_ONES:
            for (int64_t i = t.begin + threadIdx.x; i < t.end; i += blockDim.x)
                J.out[off + i * es] = 1ull;
            break;
        case TK_PAIR:
            // row d-2 in closed form, and row d-1 when a memo is built from it
            // (whole rows only: es == 1)
            for (int64_t i = t.begin + threadIdx.x; i < t.end; i += blockDim.x) {
                const uint32_t r = (uint32_t)(off + i * es);
                J.out[r] = pair_form_count(J.pair, r);
                if (J.ones_below && es == 1)
                    J.out[J.len + r] = fd_mod(r, J.pair.fh) == 0 ? 1ull : 0ull;
            }
            break;
        case TK_LINEAR:
            for (int64_t i = t.begin + threadIdx.x; i < t.end; i += blockDim.x) {
                const int64_t x = off + i * es;
                J.out[x] = x < J.ones_below ? 1ull : (uint64_t)((uint32_t)x / (uint32_t)J.g + 1u);
            }
            break;
        default:
            break;
    }
}

// FZ_SCAN_MINB=1|4|6: the register budget of the batched scans (tuning only).
static int scan_minb() {
    static const int v = [] {
        const char *e = getenv("FZ_SCAN_MINB");
        const int x = e ? atoi(e) : 0;
        return (x == 1 || x == 4 || x == 6) ? x : SCAN_MINB_DEFAULT;
    }();
    return v;
}

int launch_scan_tasks(const ScanJob *jobs, const ScanTask *tasks, int ntasks, cudaStream_t s) {
    if (ntasks <= 0) return FZ_OK;
    switch (scan_minb()) {
        case 1: scan_tasks_kernel<1><<<ntasks, THREADS, 0, s>>>(jobs, tasks); break;
        case 6: scan_tasks_kernel<6><<<ntasks, THREADS, 0, s>>>(jobs, tasks); break;
        default: scan_tasks_kernel<4><<<ntasks, THREADS, 0, s>>>(jobs, tasks); break;
    }
    note_launch();
    FZ_CUDA_TRY(cudaGetLastError());
    return FZ_OK;
}

// How the chains of a row (`chains` of them, the longest T entries) are
// scanned: 0 = a lane each, -2 = a warp each, else tiles of that width; -1 =
// blocked.  A few chains of one round of a warp's loads are not worth a tile's
// two meetings (256 sets of width 9: 471 us a rebuild, 478 with tiles).
int scan_plan(int64_t chains, int64_t T) {
    if (T <= CHAIN_T && chains < 32) return -2;
    if (chains < 8) return T <= TILE_MAX_T ? 1 : -1;
    if (T > DIRECT_T) return -1;
    if (chains >= 32 && T <= LANE_T) return 0;
    return chains >= 32 && T <= 512 ? 32 : 8;
}
int64_t scan_direct_limit() { return DIRECT_T; }
// Block sums a task of a blocked scan covers: one a thread (256).
// FZ_SCAN_BS_TASK=2048 gives a thread eight (tuning only).
int64_t scan_blocks_per_task() {
    static const int64_t v = [] {
        const char *e = getenv("FZ_SCAN_BS_TASK");
        const long x = e ? atol(e) : 0;
        return (x >= 256 && x <= 65536 && x % 256 == 0) ? (int64_t)x : (int64_t)THREADS;
    }();
    return v;
}

int scan_block_rows() { return RB; }

int launch_count_rolling(const int32_t *g, int d, int32_t n, uint64_t *a, uint64_t *b,
                         uint64_t *tmp, uint64_t **result, cudaStream_t s) {
    const int64_t len = (int64_t)n + 1;
    if (n <= SMALL_ONE_N) {
        SmallTables P{};
        P.C0 = a;
        P.d = d;
        P.n = n;
        for (int i = 0; i < d; ++i) P.g[i] = g[i];
        *result = a;
        return launch_small_tables(P, s);
    }
    int rc = launch_tail_rows(g, d, d >= 2 ? a : nullptr, d >= 2 ? nullptr : a, nullptr, len, s);
    if (rc != FZ_OK) return rc;
    uint64_t *below = a, *cur = b;
    for (int j = d - 3; j >= 0; --j) {
        rc = strided_scan(below, cur, len, g[j], tmp, s);
        if (rc != FZ_OK) return rc;
        uint64_t *t = below;
        below = cur;
        cur = t;
    }
    *result = below;
    return FZ_OK;
}

// in: len entries; out: len + 1 entries, out[0] = 0, out[r+1] = sum_{r' <= r} in[r'].
int launch_exclusive_scan_tmp(const uint64_t *in, uint64_t *out, int64_t len, uint64_t *tmp,
                              cudaStream_t s) {
    FZ_CUDA_TRY(cudaMemsetAsync(out, 0, sizeof(uint64_t), s));
    return strided_scan(in, out + 1, len, 1, tmp, s);
}

// ---------------------------------------------------------------------------
// Write probe (fz_write_probe): distinct words, 16-byte stores, a grid of
// 8 CTAs of 256 threads per SM striding over the buffer.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) write_probe_kernel(int4 *__restrict__ out, uint64_t n16,
                                                          int32_t *__restrict__ tail,
                                                          uint64_t tail_words, uint64_t tail_w0) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n16; i += stride) {
        const int32_t w = (int32_t)(i * 4);
        out[i] = make_int4(w, w + 1, w + 2, w + 3);
    }
    if (blockIdx.x == 0 && threadIdx.x < tail_words)
        tail[threadIdx.x] = (int32_t)(tail_w0 + threadIdx.x);
}

int launch_write_probe(int32_t *out, uint64_t words, cudaStream_t s) {
    int dev = 0, sms = 1;
    FZ_CUDA_TRY(cudaGetDevice(&dev));
    FZ_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const uint64_t n16 = words / 4;
    const uint64_t tail_words = words - n16 * 4;  // < 4
    uint64_t grid = (uint64_t)sms * 8;
    const uint64_t want = (n16 + 255) / 256;
    if (want < grid) grid = want < 1 ? 1 : want;
    write_probe_kernel<<<(unsigned)grid, 256, 0, s>>>(reinterpret_cast<int4 *>(out), n16,
                                                      out + n16 * 4, tail_words, n16 * 4);
    note_launch();
    FZ_CUDA_TRY(cudaGetLastError());
    return FZ_OK;
}

}  // namespace fz
