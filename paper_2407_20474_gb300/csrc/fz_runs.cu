// fz_runs.cu -- run-order tables and the memo of tail sets, built level by
// level.
//
// For generators (t_0..t_{k-1}) the run-order table S_j holds the rows of
// Z(p, (t_{j+1}..t_{k-1})) for the elements p = c, c + t_j, c + 2 t_j, ... of
// each residue class c mod t_j, classes in increasing order, each row with
// its quotient p div t_j in front.  The rows of a class up to p are exactly
// Z(p, (t_j..t_{k-1})) with a_j = p div t_j - quotient: by the disjoint
// recurrence of Section 2 (Lemma "disjlex"), Z(p, (t_j..)) is the
// concatenation over a_j, greatest first, of Z(p - a_j t_j, (t_{j+1}..)).  So
// every list of the next level is ONE contiguous range of this one,
//
//   Z(p, (t_j..)) = S_j[cls_j[p mod t_j], + |Z(p, (t_j..))|),
//
// and S_{j-1} is S_j read element by element in the class order of t_{j-1}.
// The chain starts at the closed form of the last two generators and takes
// k - 2 fully parallel launches; the dependent elementwise batches of the
// dynamic pass (Section 2.2, fz_memo.cu), thousands of them for long memos,
// are not needed.  The memo in element order is the last step with the
// elements taken in increasing order.
//
// Measured on one GB300 (kernel times under ncu): all Z(r), r < 1155, of
// (7, 10, 11, 19, 39), 3.6e7 rows: 238 us for the four launches (the last one
// writes 720 MB at 3.6 TB/s) against 1244 us for the dynamic pass and its
// gather map; the depth-3 memo of (115, 176, 195) up to 39845 in run order,
// 2.7e6 rows: 52 us against 857 us.
#include "fz_walk.cuh"

namespace fz {

namespace {

constexpr int BW = 8;                  // warps a block
constexpr int BT = BW * 32;
constexpr int WARP_BYTES = 5632;       // leaf descriptors + ring per warp (44 KB a block)

extern __shared__ __align__(128) unsigned char build_smem[];

// The block's job, kept after the warps' rings; its address is hidden at every
// use (see flat_rows).
struct JobRef {
    __device__ __forceinline__ const RunBuild &operator()() const {
        uint32_t o = BW * WARP_BYTES;
        asm volatile("" : "+r"(o));
        return *reinterpret_cast<const RunBuild *>(build_smem + o);
    }
    __device__ __forceinline__ const LeafSource &src() const { return (*this)().src; }
    __device__ __forceinline__ int32_t *out() const { return (*this)().dst; }
    __device__ __forceinline__ bool aligned() const { return ((uintptr_t)out() & 15u) == 0; }
    int *st;
    __device__ __forceinline__ int *status() const { return st; }
};

// The elements of a class-ordered table: flat index f -> (class c, step t),
// element c + t g.  Classes 0..rr have qn + 1 elements, the rest qn.
struct ClassWalk {
    JobRef job;
    uint32_t f;
    uint32_t t = 0;
    __device__ __forceinline__ int word(int) const { return (int)t; }
    __device__ __forceinline__ bool leaf(uint32_t &p, uint64_t &E) {
        const RunBuild &J = job();
        if (f > (uint32_t)J.n) return false;
        const uint32_t q1 = J.qn + 1u, lim = (J.rr + 1u) * q1;
        uint32_t c;
        if (f < lim) {
            c = fd_div(f, J.fq1);
            t = f - c * q1;
        } else {
            const uint32_t y = fd_div(f - lim, J.fq);
            c = J.rr + 1u + y;
            t = f - lim - y * J.qn;
        }
        p = c + t * (uint32_t)J.g;
        E = __ldg(J.cls + c) + __ldg(J.F + p);
        return true;
    }
    __device__ __forceinline__ void next() { f = f <= 0x7fffffffu ? f + 32u : f; }
};

// Elements in increasing order.
struct ElementWalk {
    JobRef job;
    uint32_t f;
    __device__ __forceinline__ int word(int) const { return 0; }
    __device__ __forceinline__ bool leaf(uint32_t &p, uint64_t &E) const {
        const RunBuild &J = job();
        if (f > (uint32_t)J.n) return false;
        p = f;
        E = __ldg(J.F + f);
        return true;
    }
    __device__ __forceinline__ void next() { f = f <= 0x7fffffffu ? f + 32u : f; }
};

// The job of this block into shared memory: jobs own consecutive block ranges
// from blk0 on (jobs owning no block have equal starts).
__device__ __forceinline__ void load_job(const RunBuild *jobs, int njobs, RunBuild &sj) {
    __shared__ int s_id;
    if (threadIdx.x < 32) {
        uint64_t first;
        const uint32_t id = warp_last_le((uint32_t)njobs, blockIdx.x, (int)threadIdx.x, &first,
                                         [&](uint32_t u) { return (uint64_t)jobs[u].blk0; });
        if (threadIdx.x == 0) s_id = (int)id;
    }
    __syncthreads();
    const uint32_t *src = reinterpret_cast<const uint32_t *>(jobs + s_id);
    uint32_t *dst = reinterpret_cast<uint32_t *>(&sj);
    for (int w = threadIdx.x; w < (int)(sizeof(RunBuild) / 4); w += blockDim.x) dst[w] = src[w];
    __syncthreads();
}

// A place in a table: leaf f, which starts at row `base`, and a row of it.
struct TablePlace {
    uint32_t f;
    uint64_t base, row;
};

// The row that cost x of a table falls on.  An element costs FLAT_LEAF_COST
// and a row 1, so tables of far more elements than rows (short tails of long
// ranges: 324 rows of 1106 elements) still spread over many warps.
__device__ __forceinline__ TablePlace table_place(const RunBuild &J, uint64_t x, int lane) {
    const uint32_t q1 = J.qn + 1u;
    auto first = [&](uint32_t c) {  // flat index of class c's first element
        return c <= J.rr ? c * q1 : (J.rr + 1u) * q1 + (c - J.rr - 1u) * J.qn;
    };
    uint64_t cc, ct;
    const uint32_t c = warp_last_le((uint32_t)J.G, x, lane, &cc, [&](uint32_t u) {
        return __ldg(J.cls + u) + FLAT_LEAF_COST * first(u);
    });
    const uint64_t *F = J.F + c;
    const uint32_t g = (uint32_t)J.g, cnt = J.qn + (c <= J.rr ? 1u : 0u);
    auto before = [&](uint32_t u) { return u == 0 ? 0ull : __ldg(F + (uint64_t)(u - 1) * g); };
    const uint32_t t = warp_last_le(cnt, x - cc, lane, &ct, [&](uint32_t u) {
        return before(u) + FLAT_LEAF_COST * u;
    });
    const uint64_t in = x - cc - ct, b = before(t);
    const uint64_t size = __ldg(F + (uint64_t)t * g) - b;
    const uint64_t o = in > FLAT_LEAF_COST ? in - FLAT_LEAF_COST : 0ull;
    TablePlace pl;
    pl.f = first(c) + t;
    pl.base = cc - FLAT_LEAF_COST * first(c) + b;
    pl.row = pl.base + (o < size ? o : size);
    return pl;
}

// Rows of one level: a warp writes an even share (per_warp) of its job.  K:
// coordinates a row; CSR: the memo in element order (K packed words a row),
// else a run-order table (quotient first).
template <int K, int SRC, bool CSR>
__global__ void __launch_bounds__(BT, 4)
    run_build_kernel(const RunBuild *__restrict__ jobs, int njobs, int *status) {
    load_job(jobs, njobs, *reinterpret_cast<RunBuild *>(build_smem + BW * WARP_BYTES));
    const JobRef job{status};
    const RunBuild &J = job();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint64_t item = (uint64_t)(blockIdx.x - J.blk0) * BW + wid;
    constexpr int NP = CSR ? 0 : 1;
    constexpr int W = K;
    constexpr int DS = CSR ? K : run_stride(K + 1);
    constexpr uint32_t B = flat_half_rows<NP, SRC, DS>(WARP_BYTES);
    int4 *desc = reinterpret_cast<int4 *>(build_smem + (size_t)wid * WARP_BYTES);
    int32_t *ring = reinterpret_cast<int32_t *>(build_smem + (size_t)wid * WARP_BYTES +
                                                leaf_bytes<NP, SRC>());
    const uint64_t pol = policy_evict_normal();
    uint64_t base = 0;
    if constexpr (CSR) {
        // equal rows, in multiples of 32 (16-byte aligned bulk stores)
        const uint64_t row0 = item * J.per_warp;
        if (row0 >= J.rows) return;
        const uint64_t rest = J.rows - row0;
        const uint32_t left = rest < J.per_warp ? (uint32_t)rest : J.per_warp;
        const uint64_t *F = J.F;
        const uint32_t f = warp_last_le((uint32_t)J.n + 1u, row0, lane, &base, [&](uint32_t u) {
            return u == 0 ? 0ull : __ldg(F + u - 1);
        });
        ElementWalk wk{job, f + (uint32_t)lane};
        flat_rows<NP, W, DS, SRC>(wk, base, (uint32_t)(row0 - base), job, row0, left, desc, ring,
                                  B, pol, lane);
    } else {
        // equal cost; a warp starts at any row of a table whose rows are whole
        // 16-byte vectors, at an even one of 24-byte rows (bulk stores)
        __shared__ uint64_t s_row[BW + 1];
        const uint64_t total = J.rows + FLAT_LEAF_COST * ((uint64_t)J.n + 1u);
        const uint64_t x = item * J.per_warp;
        TablePlace pl{0, 0, J.rows};
        auto even = [&](uint64_t r) {
            if (DS % 4 != 0) r = (r + 1) & ~1ull;
            return r < J.rows ? r : J.rows;
        };
        if (x < total) pl = table_place(J, x, lane);
        pl.row = even(pl.row);
        if (lane == 0) s_row[wid] = pl.row;
        if (wid == 0) {
            const uint64_t xe = (item + BW) * J.per_warp;
            const uint64_t re = xe < total ? even(table_place(J, xe, lane).row) : J.rows;
            if (lane == 0) s_row[BW] = re;
        }
        __syncthreads();
        const uint64_t end = s_row[wid + 1];
        if (end <= pl.row) return;
        ClassWalk wk{job, pl.f + (uint32_t)lane};
        flat_rows<NP, W, DS, SRC>(wk, pl.base, (uint32_t)(pl.row - pl.base), job, pl.row,
                                  (uint32_t)(end - pl.row), desc, ring, B, pol, lane);
    }
    if (lane == 0) bulk_wait_all();
    __syncwarp();
}

// Tables of depth 1: the element p = m ta holds the one row (p div g, m).
__global__ void __launch_bounds__(BT)
    run_build1_kernel(const RunBuild *__restrict__ jobs, int njobs, int *status) {
    __shared__ RunBuild sj;
    load_job(jobs, njobs, sj);
    const RunBuild &J = sj;
    const uint32_t ta = J.src.fg.g;
    const uint64_t m = (uint64_t)(blockIdx.x - J.blk0) * BT + threadIdx.x;
    if (m * ta > (uint64_t)J.n) return;
    const uint32_t p = (uint32_t)(m * ta), g = (uint32_t)J.g;
    const uint32_t q = p / g;
    const uint64_t row = __ldg(J.cls + (p - q * g)) + __ldg(J.F + p) - 1ull;
    if (row >= J.rows) {
        atomicExch(status, (int)DEV_INTERNAL);
        return;
    }
    reinterpret_cast<int4 *>(J.dst)[row] = make_int4((int)q, (int)m, 0, 0);
}

// Tables of depth 2 with fewer rows than elements: a thread per lattice point
// (x, y), element p = x t0 + y t1 <= n, writes its one row.  The points of the
// columns x and X - x (X = n div t0) share one line of `wide` threads, about as
// many as both hold.  The row's place inside its element counts the points
// with a greater x; all rows of an element below p are its class's count.
//
// 4096 instances of widths 3..8 (4.1e7 elements, 1.1e7 rows): 270 us with the
// dense tables' flat walk, against 613 us by the flat walk alone, which reads a
// count for every element.
__global__ void __launch_bounds__(BT)
    run_build2_kernel(const RunBuild *__restrict__ jobs, int njobs, int *status) {
    __shared__ RunBuild sj;
    load_job(jobs, njobs, sj);
    const RunBuild &J = sj;
    const PairForm &F = J.src.pair;
    const uint32_t t0 = F.g, t1 = F.fh.g, n = (uint32_t)J.n;
    const uint32_t wide = (n + t0) / t1 + 2u, X = fd_div(n, F.fg);
    const uint64_t i = (uint64_t)(blockIdx.x - J.blk0) * BT + threadIdx.x;
    uint32_t x = (uint32_t)(i / wide);
    uint32_t y = (uint32_t)(i - (uint64_t)x * wide);
    if (x > X / 2u) return;
    const uint32_t len = fd_div(n - x * t0, F.fh) + 1u;
    if (y >= len) {
        y -= len;
        const uint32_t other = X - x;
        if (other == x || y > fd_div(n - other * t0, F.fh)) return;
        x = other;
    }
    const uint32_t p = x * t0 + y * t1;
    const uint32_t top = pair_form_top(F, p);
    const uint32_t cnt = fd_div(top, F.fh1) + 1u;  // rows of the element
    const uint32_t q = p / (uint32_t)J.g;
    const uint64_t row = __ldg(J.cls + (p - q * (uint32_t)J.g)) + __ldg(J.F + p) - cnt +
                         fd_div(top - x, F.fh1);
    if (row >= J.rows) {
        atomicExch(status, (int)DEV_INTERNAL);
        return;
    }
    reinterpret_cast<int4 *>(J.dst)[row] = make_int4((int)q, (int)x, (int)y, 0);
}

// Class starts of each job's table: cls[c] = rows of the classes below c (a
// class's rows are the count row at its last element).  One block a job.
__global__ void __launch_bounds__(BT)
    run_class_kernel(const RunBuild *__restrict__ jobs, int *status) {
    __shared__ uint64_t warp_sum[BW];
    const RunBuild &J = jobs[blockIdx.x];
    if (!J.cls) return;
    uint64_t *cls = const_cast<uint64_t *>(J.cls);
    const uint64_t *F = J.F;
    const int32_t n = J.n, g = J.g, G = J.G;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint64_t carry = 0;
    for (int64_t base = 0; base < G; base += BT) {
        const int64_t c = base + threadIdx.x;  // (past G near 2^31 on the way out)
        uint64_t v = 0;
        if (c < G) v = __ldg(F + (c + (int64_t)((n - (int32_t)c) / g) * g));
        const uint64_t incl = warp_incl_scan(v, lane);
        if (lane == 31) warp_sum[wid] = incl;
        __syncthreads();
        uint64_t before = 0, total = 0;
#pragma unroll
        for (int w = 0; w < BW; ++w) {
            const uint64_t x = warp_sum[w];
            if (w < wid) before += x;
            total += x;
        }
        if (c < G) cls[c] = carry + before + incl - v;
        carry += total;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        cls[G] = carry;
        if (carry != J.rows) atomicExch(status, (int)DEV_INTERNAL);
    }
}

// totals[i] = rows of job i's table (its classes' last count entries).
__global__ void __launch_bounds__(BT)
    run_totals_kernel(const RunBuild *__restrict__ jobs, uint64_t *__restrict__ totals) {
    __shared__ uint64_t warp_sum[BW];
    const RunBuild &J = jobs[blockIdx.x];
    const int32_t n = J.n, g = J.g, G = J.G;
    uint64_t acc = 0;
    for (int64_t c = threadIdx.x; c < G; c += BT) {
        const uint64_t v = __ldg(J.F + (c + (int64_t)((n - (int32_t)c) / g) * g));
        acc += v < (1ull << 32) ? v : (1ull << 32);  // as row_sums_kernel
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) acc += __shfl_xor_sync(FULL, acc, o);
    if ((threadIdx.x & 31) == 0) warp_sum[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < BW; ++w) acc += warp_sum[w];
        totals[blockIdx.x] = acc;
    }
}

// sums[j] += the first `top` entries of row j (j = blockIdx.y) of a count
// table, each entry clamped to 2^32: a sum below 2^32 is exact, and at most
// 2^31 entries cannot wrap.
__global__ void __launch_bounds__(256)
    row_sums_kernel(const uint64_t *__restrict__ C, int64_t cs, int64_t top, uint64_t *sums) {
    const uint64_t *row = C + (int64_t)blockIdx.y * cs;
    uint64_t acc = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < top;
         i += (int64_t)gridDim.x * blockDim.x)
    {
        const uint64_t v = __ldg(row + i);
        acc += v < (1ull << 32) ? v : (1ull << 32);
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) acc += __shfl_xor_sync(FULL, acc, o);
    if ((threadIdx.x & 31) == 0 && acc)
        atomicAdd(reinterpret_cast<unsigned long long *>(sums + blockIdx.y),
                  (unsigned long long)acc);
}

template <int K, int SRC, bool CSR>
int launch_level(const RunBuild *jobs, int njobs, uint32_t blocks, int *status, cudaStream_t s) {
    run_build_kernel<K, SRC, CSR>
        <<<blocks, BT, BW * WARP_BYTES + sizeof(RunBuild), s>>>(jobs, njobs, status);
    note_launch();
    FZ_CUDA_TRY(cudaGetLastError());
    return FZ_OK;
}

size_t up256(size_t x) { return (x + 255) & ~size_t(255); }

}  // namespace

int launch_run_classes(const RunBuild *jobs_dev, int njobs, int *status, cudaStream_t s) {
    if (njobs <= 0) return FZ_OK;
    run_class_kernel<<<njobs, BT, 0, s>>>(jobs_dev, status);
    note_launch();
    FZ_CUDA_TRY(cudaGetLastError());
    return FZ_OK;
}

int launch_run_totals(const RunBuild *jobs_dev, int njobs, uint64_t *totals, cudaStream_t s) {
    if (njobs <= 0) return FZ_OK;
    run_totals_kernel<<<njobs, BT, 0, s>>>(jobs_dev, totals);
    note_launch();
    FZ_CUDA_TRY(cudaGetLastError());
    return FZ_OK;
}

int launch_run_build(const RunBuild *jobs_dev, int njobs, int K, bool csr, uint32_t blocks,
                     int *status, cudaStream_t s) {
    if (njobs <= 0 || blocks == 0) return FZ_OK;
    if (csr) {
        switch (K) {
            case 3: return launch_level<3, SRC_RUN, true>(jobs_dev, njobs, blocks, status, s);
            case 4: return launch_level<4, SRC_RUN, true>(jobs_dev, njobs, blocks, status, s);
            case 5: return launch_level<5, SRC_RUN, true>(jobs_dev, njobs, blocks, status, s);
            case 6: return launch_level<6, SRC_RUN, true>(jobs_dev, njobs, blocks, status, s);
            case 7: return launch_level<7, SRC_RUN, true>(jobs_dev, njobs, blocks, status, s);
            case 8: return launch_level<8, SRC_RUN, true>(jobs_dev, njobs, blocks, status, s);
            default: return set_error(FZ_EINTERNAL, "memo levels: depth out of range");
        }
    }
    switch (K) {
        case 1:
            run_build1_kernel<<<blocks, BT, 0, s>>>(jobs_dev, njobs, status);
            note_launch();
            FZ_CUDA_TRY(cudaGetLastError());
            return FZ_OK;
        case RUN_LATTICE:
            run_build2_kernel<<<blocks, BT, 0, s>>>(jobs_dev, njobs, status);
            note_launch();
            FZ_CUDA_TRY(cudaGetLastError());
            return FZ_OK;
        case 2: return launch_level<2, SRC_PAIR, false>(jobs_dev, njobs, blocks, status, s);
        case 3: return launch_level<3, SRC_RUN, false>(jobs_dev, njobs, blocks, status, s);
        case 4: return launch_level<4, SRC_RUN, false>(jobs_dev, njobs, blocks, status, s);
        case 5: return launch_level<5, SRC_RUN, false>(jobs_dev, njobs, blocks, status, s);
        case 6: return launch_level<6, SRC_RUN, false>(jobs_dev, njobs, blocks, status, s);
        case 7: return launch_level<7, SRC_RUN, false>(jobs_dev, njobs, blocks, status, s);
        default: return set_error(FZ_EINTERNAL, "run-order table: depth out of range");
    }
}

void fill_run_build(const int32_t *t, int k, int32_t n, int j, bool csr, RunBuild *out) {
    RunBuild &R = *out;
    R.n = n;
    const int K = csr ? k - j : k - 1 - j;  // coordinates of a row
    if (!csr) {
        R.g = t[j];
        R.G = R.g < (int64_t)n + 1 ? R.g : n + 1;
        R.qn = (uint32_t)(n / R.g);
        R.rr = (uint32_t)(n % R.g);
        R.fq1 = make_fastdiv(R.qn + 1u);
        R.fq = make_fastdiv(R.qn > 0 ? R.qn : 1u);
    }
    const int leaf = csr ? j : j + 1;  // the leaves' first generator
    if (K == 2)
        R.src.pair = make_pair_form(t[leaf], t[leaf + 1]);
    else
        R.src.fg = make_fastdiv((uint32_t)t[leaf]);
}

uint64_t run_build_cost(const RunBuild &R, bool csr) {
    return csr ? R.rows : R.rows + FLAT_LEAF_COST * ((uint64_t)R.n + 1u);
}

// A warp's share of a launch of `total` cost: about four shares a resident
// warp, 256 to 8192 (a multiple of 32 rows).
uint32_t run_build_share(uint64_t total, int sms) {
    uint64_t per = total / ((uint64_t)sms * 32 * 4 + 1);
    per = per < 256 ? 256 : per > 8192 ? 8192 : per;
    return (uint32_t)((per + 31) & ~31ull);
}

int run_build_kind(const RunBuild &R, int K) {
    return K == 2 && R.rows < (uint64_t)R.n ? RUN_LATTICE : K;
}

uint32_t run_build_blocks(const RunBuild &R, int K, bool csr) {
    if (R.rows == 0) return 0;
    if (K == 1) return (uint32_t)(((uint64_t)R.n / R.src.fg.g + 1 + BT - 1) / BT);
    if (K == RUN_LATTICE) {
        const uint64_t t0 = R.src.pair.g, t1 = R.src.pair.fh.g;
        const uint64_t wide = ((uint64_t)R.n + t0) / t1 + 2, lines = (uint64_t)R.n / t0 / 2 + 1;
        return (uint32_t)((lines * wide + BT - 1) / BT);
    }
    const uint64_t items = (run_build_cost(R, csr) + R.per_warp - 1) / R.per_warp;
    return (uint32_t)((items + BW - 1) / BW);
}

int launch_row_sums(const uint64_t *C, int64_t cs, int rows, int64_t top, uint64_t *sums,
                    cudaStream_t s) {
    FZ_CUDA_TRY(cudaMemsetAsync(sums, 0, (size_t)rows * 8, s));
    int64_t bx = (top + 2047) / 2048;
    bx = bx < 1 ? 1 : bx > 256 ? 256 : bx;
    row_sums_kernel<<<dim3((unsigned)bx, (unsigned)rows), 256, 0, s>>>(C, cs, top, sums);
    note_launch();
    FZ_CUDA_TRY(cudaGetLastError());
    return FZ_OK;
}

// ---------------------------------------------------------------------------
// One chain (plans and memo calls).
// ---------------------------------------------------------------------------
size_t run_levels_bytes(const int32_t *t, int k, int32_t n, const uint64_t *sums, bool csr) {
    size_t bytes = up256((size_t)FZ_MAX_D * sizeof(RunBuild));
    size_t buf[2] = {0, 0};
    const int last = k - 3 > 0 ? k - 3 : 0;  // deepest table level (k = 2: depth 1)
    for (int j = 0; j <= last; ++j) {
        const int64_t G = t[j] < (int64_t)n + 1 ? t[j] : (int64_t)n + 1;
        bytes += up256((size_t)(G + 1) * 8);
        const size_t b = up256((size_t)sums[j + 1] * 4 * run_stride(k - j) + 16);
        if (j == 0 && !csr)
            bytes += b;  // the table itself
        else
            buf[j & 1] = buf[j & 1] > b ? buf[j & 1] : b;
    }
    return bytes + buf[0] + buf[1];
}

int run_levels_init(const int32_t *t, int k, int32_t n, const uint64_t *sums, bool csr,
                    const uint64_t *Ct, int64_t cs, const uint64_t *O, int32_t *csr_rows,
                    void *mem, RunLevels *L, cudaStream_t s) {
    if (k < (csr ? 3 : 2) || k > (csr ? 8 : 8))
        return set_error(FZ_EINTERNAL, "run-order levels: depth out of range");
    DeviceProps dp;
    int rc = device_props(&dp);
    if (rc != FZ_OK) return rc;
    char *m = static_cast<char *>(mem);
    L->jobs_dev = reinterpret_cast<RunBuild *>(m);
    m += up256((size_t)FZ_MAX_D * sizeof(RunBuild));
    const int last = k - 3 > 0 ? k - 3 : 0;
    RunBuild *h = L->jobs;
    size_t size[FZ_MAX_D], buf[2] = {0, 0};
    uint64_t *cls[FZ_MAX_D];
    int32_t *rows[FZ_MAX_D];
    for (int j = 0; j <= last; ++j) {
        const int64_t G = t[j] < (int64_t)n + 1 ? t[j] : (int64_t)n + 1;
        cls[j] = reinterpret_cast<uint64_t *>(m);
        m += up256((size_t)(G + 1) * 8);
        size[j] = up256((size_t)sums[j + 1] * 4 * run_stride(k - j) + 16);
        if (j == 0 && !csr) {
            rows[0] = reinterpret_cast<int32_t *>(m);
            m += size[0];
        } else if (size[j] > buf[j & 1]) {
            buf[j & 1] = size[j];
        }
    }
    // a level is read only while the next one is written: two buffers in turn
    for (int j = 0; j <= last; ++j)
        if (j > 0 || csr)
            rows[j] = reinterpret_cast<int32_t *>(m + ((j & 1) ? buf[0] : 0));
    L->n = 0;
    for (int j = last; j >= 0; --j) {
        RunBuild &R = h[L->n];
        R.rows = sums[j + 1];
        R.F = Ct + (int64_t)j * cs;
        R.cls = cls[j];
        R.dst = rows[j];
        fill_run_build(t, k, n, j, false, &R);
        R.per_warp = run_build_share(run_build_cost(R, false), dp.sms);
        L->K[L->n] = run_build_kind(R, k - 1 - j);
        if (j < last) {
            R.src.rows = rows[j + 1];
            R.src.cls = cls[j + 1];
            R.src.nrows = sums[j + 2];
        }
        L->blocks[L->n] = run_build_blocks(R, L->K[L->n], false);
        ++L->n;
    }
    L->tables = L->n;
    L->csr = csr;
    L->rows = rows[0];
    L->cls = cls[0];
    if (csr) {
        RunBuild &R = h[L->n];
        R.rows = sums[0];
        R.F = O + 1;
        R.cls = nullptr;
        R.dst = csr_rows;
        fill_run_build(t, k, n, 0, true, &R);
        R.per_warp = run_build_share(R.rows, dp.sms);
        R.src.rows = rows[0];
        R.src.cls = cls[0];
        R.src.nrows = sums[1];
        L->K[L->n] = k;
        L->blocks[L->n] = run_build_blocks(R, k, true);
        ++L->n;
    }
    FZ_CUDA_TRY(cudaMemcpyAsync(L->jobs_dev, h, (size_t)L->n * sizeof(RunBuild),
                                cudaMemcpyHostToDevice, s));
    return FZ_OK;
}

// One launch for every class start, one per level.  Calls of the library
// before and after (us a call): the memo of 3.6e7 rows 1753 -> 636, a plan's
// rebuild and enumeration of 5e8 rows 2974 -> 2065.
int launch_run_levels(const RunLevels &L, int *status, cudaStream_t s) {
    int rc = launch_run_classes(L.jobs_dev, L.tables, status, s);
    for (int i = 0; i < L.n && rc == FZ_OK; ++i)
        rc = launch_run_build(L.jobs_dev + i, 1, L.K[i], L.csr && i == L.tables, L.blocks[i],
                              status, s);
    return rc;
}

}  // namespace fz
