// fz_walk.cuh -- device pieces shared by the enumeration (fz_enum.cu), the
// run-order tables and the memo build (fz_runs.cu): invariant division, the
// staged row writer and the flat leaf walk.
#pragma once

#include "fz_internal.cuh"

namespace fz {

// ---------------------------------------------------------------------------
// Staged rows.  A warp assembles rows in a shared-memory ring of two halves
// of B rows and sends every full half to global memory with one bulk (TMA)
// store, or with plain stores when the output is not 16-byte aligned (or is
// host memory reached over the host link).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void flush_words(int32_t *gdst, bool aligned, const int32_t *src,
                                            uint32_t words, int lane, uint64_t pol) {
    if (aligned) {
        const uint32_t bytes = words * 4u;
        const uint32_t bulk = bytes & ~15u;
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0 && bulk) {
            bulk_store(gdst, src, bulk, pol);
            bulk_commit();
        }
        const uint32_t rem_words = (bytes - bulk) >> 2;
        if ((uint32_t)lane < rem_words) gdst[(bulk >> 2) + lane] = src[(bulk >> 2) + lane];
    } else {
        // plain stores (unaligned output, or host memory over the host link):
        // 16-byte vectors when both sides allow it
        __syncwarp();
        uint32_t w0 = 0;
        if ((((uintptr_t)gdst | (uintptr_t)src) & 15u) == 0) {
            const uint32_t nv = words >> 2;
            const int4 *s4 = reinterpret_cast<const int4 *>(src);
            int4 *g4 = reinterpret_cast<int4 *>(gdst);
            for (uint32_t v = lane; v < nv; v += 32) g4[v] = s4[v];
            w0 = nv << 2;
        }
        for (uint32_t w = w0 + lane; w < words; w += 32) gdst[w] = src[w];
        __syncwarp();
    }
}

// One row of DS words to shared memory, in the widest stores its alignment
// allows (row starts are multiples of DS words from a 128-byte boundary).
// DS = 8: lanes 4-7 of each eight store their upper half first, so the eight
// 16-byte stores of a phase fall on different banks.
template <int DS>
__device__ __forceinline__ void store_row(int32_t *dst, const int (&w)[DS], int lane) {
    if constexpr (DS == 8) {
        const bool hi = (lane & 4) != 0;
        const int4 lo4 = make_int4(w[0], w[1], w[2], w[3]), hi4 = make_int4(w[4], w[5], w[6], w[7]);
        int4 *d4 = reinterpret_cast<int4 *>(dst);
        d4[hi ? 1 : 0] = hi ? hi4 : lo4;
        d4[hi ? 0 : 1] = hi ? lo4 : hi4;
    } else if constexpr (DS % 4 == 0) {
#pragma unroll
        for (int c = 0; c < DS; c += 4)
            *reinterpret_cast<int4 *>(dst + c) = make_int4(w[c], w[c + 1], w[c + 2], w[c + 3]);
    } else if constexpr (DS % 2 == 0) {
#pragma unroll
        for (int c = 0; c < DS; c += 2)
            *reinterpret_cast<int2 *>(dst + c) = make_int2(w[c], w[c + 1]);
    } else {
#pragma unroll
        for (int c = 0; c < DS; ++c) dst[c] = w[c];
    }
}

// Words between the rows of a run-order table whose rows hold W words (the
// quotient and W - 1 coordinates): whole 16-byte vectors, or 24 bytes for 5
// and 6 words (a memo of 3.6e7 rows copied from rows of 32 bytes was bound by
// L2: 197 us, 171 us with 24).
__host__ __device__ constexpr int run_stride(int W) {
    return W == 5 || W == 6 ? 6 : (W + 3) & ~3;
}
template <int SS>
__device__ __forceinline__ void load_run_row(const int32_t *p, int (&x)[SS]) {
    if constexpr (SS % 4 == 0) {
#pragma unroll
        for (int v = 0; v < SS / 4; ++v) {
            const int4 y = __ldg(reinterpret_cast<const int4 *>(p) + v);
            x[4 * v] = y.x;
            x[4 * v + 1] = y.y;
            x[4 * v + 2] = y.z;
            x[4 * v + 3] = y.w;
        }
    } else {
#pragma unroll
        for (int v = 0; v < SS / 2; ++v) {
            const int2 y = __ldg(reinterpret_cast<const int2 *>(p) + v);
            x[2 * v] = y.x;
            x[2 * v + 1] = y.y;
        }
    }
}

// Where the rows of a leaf (an element p) come from.
//   SRC_RUN:  the run-order table of (gen; tail): the rows of Z(p, (gen,
//             tail)) are the contiguous range [cls[p mod gen], + count) of
//             `rows`, each row (quotient, tail words), and the coordinate of
//             gen is p div gen - quotient.
//   SRC_PAIR: the closed form of the last two generators; nothing is read.
//   SRC_RANK: batches only, the pair's rows found by rank (rank_rows).
enum : int { SRC_RUN = 0, SRC_PAIR = 1, SRC_RANK = 2 };
struct LeafSource {
    const int32_t *rows;
    const uint64_t *cls;
    uint64_t nrows;
    FastDiv fg;
    PairForm pair;
};

// One table (or memo in element order) to be written by run_build_kernel
// (fz_runs.cu).  Jobs of a launch own consecutive block ranges from blk0 on.
struct RunBuild {
    LeafSource src;       // depth 1: src.fg holds the tail's one generator
    const uint64_t *F;    // row ends: element p of class c ends at cls[c] + F[p]
    const uint64_t *cls;  // class starts of this table (G + 1), null in element order
    int32_t *dst;
    uint64_t rows;
    int32_t n;            // elements 0..n
    int32_t g, G;         // class generator, G = min(g, n + 1)
    uint32_t qn, rr;      // n div g, n mod g
    uint32_t per_warp;    // a warp's share: rows (element order) or cost (tables)
    uint32_t blk0;
    FastDiv fq1, fq;      // division by qn + 1 and qn
};

// The levels of one chain (fz_runs.cu): tables[, the memo in element order].
struct RunLevels {
    RunBuild *jobs_dev = nullptr;
    // source of the copy to jobs_dev, which need not have been read when the
    // call that enqueued it returns: stays until the stream is synchronised
    RunBuild jobs[FZ_MAX_D] = {};
    int n = 0, tables = 0;
    bool csr = false;
    int K[FZ_MAX_D] = {};
    uint32_t blocks[FZ_MAX_D] = {};
    int32_t *rows = nullptr;       // the last table: rows and class starts
    uint64_t *cls = nullptr;
};

// Cost of a leaf of the flat walk in rows (work-balanced slicing): 32 leaves
// take about as many instructions as 100 rows.
constexpr uint64_t FLAT_LEAF_COST = 4;

// Deepest memo the levels build (rows of a table: quotient and coordinates).
constexpr int RUN_MAX_K = 7;   // run-order tables
constexpr int CSR_MAX_K = 8;   // memos in element order (from depth 3 on)

// True if the flat walk has a kernel (fz_flat.cu) for tuples of width d with
// leaves of np prefix words.
constexpr bool flat_serves(int d, int np, int src) {
    if (d < 3 || d > 9) return false;
    if (src == SRC_PAIR) return np == d - 2;
    return np >= 1 && np <= 3 && d - 1 - np >= 1 && d - 1 - np <= RUN_MAX_K;
}

// sums[j] (device) = sum over r < top of row j of C, exact when below 2^32.
int launch_row_sums(const uint64_t *C, int64_t cs, int rows, int64_t top, uint64_t *sums,
                    cudaStream_t s);
// Chain over the generators t_0..t_{k-1} and elements 0..n: the run-order
// table keyed by t_0 of the rows of Z(p, (t_1..)) (csr false, 2 <= k <= 8), or the
// memo Z(p, (t_0..)) in element order (csr true, 3 <= k <= 8; O: its
// offsets, csr_rows: its rows).  sums[j] = rows of all Z(p, (t_j..)), p <= n,
// below 2^32 from j = 1 on; Ct: count table rows 0..k of t.  `mem` has
// run_levels_bytes bytes and holds tables, scratch and jobs.
size_t run_levels_bytes(const int32_t *t, int k, int32_t n, const uint64_t *sums, bool csr);
int run_levels_init(const int32_t *t, int k, int32_t n, const uint64_t *sums, bool csr,
                    const uint64_t *Ct, int64_t cs, const uint64_t *O, int32_t *csr_rows,
                    void *mem, RunLevels *L, cudaStream_t s);
int launch_run_levels(const RunLevels &L, int *status, cudaStream_t s);
// The pieces, for many chains at once (batches).
void fill_run_build(const int32_t *t, int k, int32_t n, int j, bool csr, RunBuild *out);
uint64_t run_build_cost(const RunBuild &R, bool csr);
uint32_t run_build_share(uint64_t total, int sms);
// How a table of depth K is built: K, or RUN_LATTICE for depth 2 with fewer
// rows than elements (rows and n set).
constexpr int RUN_LATTICE = -2;
int run_build_kind(const RunBuild &R, int K);
uint32_t run_build_blocks(const RunBuild &R, int K, bool csr);
int launch_run_totals(const RunBuild *jobs_dev, int njobs, uint64_t *totals, cudaStream_t s);
int launch_run_classes(const RunBuild *jobs_dev, int njobs, int *status, cudaStream_t s);
int launch_run_build(const RunBuild *jobs_dev, int njobs, int K, bool csr, uint32_t blocks,
                     int *status, cudaStream_t s);

// Descriptors of a warp's 32 leaves, as 16-byte vectors [DV][32].
template <int NP, int SRC>
__host__ __device__ constexpr int leaf_vecs() {
    return ((SRC == SRC_RUN ? 2 : 3) + NP + 3) / 4;
}
template <int NP, int SRC>
__host__ __device__ constexpr int leaf_bytes() {
    return leaf_vecs<NP, SRC>() * 32 * 16;
}
// Rows per ring half when a warp has `bytes` of shared memory for both its
// leaf descriptors and its ring of DS-word rows.
template <int NP, int SRC, int DS>
__host__ __device__ constexpr uint32_t flat_half_rows(int bytes) {
    const int b = (bytes - ((SRC == SRC_RUN ? 2 : 3) + NP + 3) / 4 * 512) / (8 * DS) / 32 * 32;
    return b < 32 ? 32u : (uint32_t)b;
}

// ---------------------------------------------------------------------------
// The flat leaf walk.  The output of an enumeration, of a run-order table and
// of a memo in element order are all the concatenation, over a sequence of
// leaves (elements p with a few prefix words), of rows copied from a
// LeafSource.  A warp writes rows [row0, row0 + left) of such an output:
// lane l holds leaf f + l of the sequence and reads its cumulative row end
// from a count row, so 32 leaves cost one round of loads whatever they hold;
// their descriptors go to shared memory (empty leaves dropped), and rounds of
// 32 RPL output rows then find their leaves by counting the leaf ends that
// lie inside the round (one ballot and one OR-reduction of end bits).  So a
// leaf of a few rows costs no round of its own, and a long leaf's rounds are
// plain copies.  The table rows of the next round are loaded before this
// round's rows are stored.
//
// What bounds it: instruction issue while leaves are short (a copy with one
// leaf a warp at a time needed about 12 warp instructions a row where leaves
// hold a row or two), the output's bandwidth when they are long.
//
// Walk: leaf(p, end) gives lane's element and cumulative row end and returns
// false past the last leaf (a suffix of the lanes), word(c) its prefix words;
// next() moves every lane 32 leaves on.  `base` is the row at which
// leaf 0 starts (same origin as the ends) and `skip` its rows already behind.
// Returns false, with the status recorded, if the tables disagree.
// ---------------------------------------------------------------------------
//
// Sink: src(), out(), aligned() and status() of the rows written.  Parameters
// kept in shared memory are read through a Sink (and a Walk) that hides their
// address from the compiler at every use: hoisted into registers they cost
// the kernel its 64 (spills of 100 to 300 bytes a thread that miss the small
// L1 left beside 4 blocks' shared memory: 2.0 TB/s written instead of 4).
template <int NP, int W, int DS, int SRC, class Walk, class Sink>
__device__ __forceinline__ bool flat_rows(Walk &wk, uint64_t base, uint32_t skip, const Sink &K,
                                          uint64_t row0, uint32_t left, int4 *desc,
                                          int32_t *ring, uint32_t B, uint64_t pol, int lane) {
    static_assert(NP + W <= DS, "row words");
    constexpr int RPL = SRC == SRC_PAIR || W <= 4 ? 2 : 1;  // rows a lane per round
    constexpr int DV = leaf_vecs<NP, SRC>();
    constexpr int SS = SRC == SRC_RUN ? run_stride(W) : 4;
    constexpr uint32_t RR = 32u * RPL;
    const uint32_t le = 0xffffffffu >> (31 - lane);
    uint32_t hpos = 0, half = 0, nfull = 0;
    bool ok = true;

    struct Frag {
        int x[RPL][SRC == SRC_RUN ? SS : 1];
        int l[RPL];
    };

    // lane's leaf of the next batch: its row end and where its rows start are
    // loaded together, before the rounds of the batch in hand
    uint32_t p = 0, qt = 0;
    uint64_t nE = 0, nsrc = 0;
    bool have = false;
    auto load_leaf = [&] {
        have = wk.leaf(p, nE);
        if constexpr (SRC == SRC_RUN) {
            if (have) {
                const LeafSource &S = K.src();
                qt = fd_div(p, S.fg);
                nsrc = __ldg(S.cls + (p - qt * S.fg.g));
            }
        }
    };
    load_leaf();
    while (left > 0) {
        // ---- 32 leaves
        uint64_t E = nE;
        const bool live = have;
        const int nlive = __popc(__ballot_sync(FULL, live));
        if (nlive == 0) {  // past the last leaf with rows still owed
            if (lane == 0) atomicExch(K.status(), (int)DEV_INTERNAL);
            ok = false;
            break;
        }
        const uint64_t Elast = shfl_u64(E, nlive - 1);
        if (!live) E = Elast;
        uint64_t Eprev = __shfl_up_sync(FULL, E, 1);
        if (lane == 0) Eprev = base;
        const uint64_t size = E - Eprev;
        const uint32_t e = E - base < 0xffffffffull ? (uint32_t)(E - base) : 0xffffffffu;
        const uint32_t s = Eprev - base < 0xffffffffull ? (uint32_t)(Eprev - base) : 0xffffffffu;
        const uint32_t e_all = __shfl_sync(FULL, e, 31);
        // the end of this batch's rows (skip may lie a row past leaf 0)
        const uint32_t q_end = e_all <= skip ? skip : e_all - skip < left ? e_all : skip + left;
        // leaves with rows in the window, in order
        const bool used = live && e > s && e > skip && s < q_end;
        const uint32_t rank = __popc(__ballot_sync(FULL, used) & (le >> 1));
        bool bad = E < Eprev;
        __syncwarp();  // the previous batch's descriptors have been read
        if (used) {
            int d[DV * 4];
#pragma unroll
            for (int c = 0; c < DV * 4; ++c) d[c] = 0;
            constexpr int H = SRC == SRC_RUN ? 2 : 3;
            if constexpr (SRC == SRC_RUN) {
                bad = bad || nsrc + size > K.src().nrows;  // bounds guard: in the table
                d[0] = (int)((uint32_t)nsrc - s);
                d[1] = (int)qt;
            } else {
                const LeafSource &S = K.src();
                const uint32_t at = pair_form_top(S.pair, p);
                d[0] = (int)s;
                d[1] = (int)at;
                d[2] = (int)fd_div(p - at * S.pair.g, S.pair.fh);
            }
#pragma unroll
            for (int c = 0; c < NP; ++c) d[H + c] = wk.word(c);
#pragma unroll
            for (int v = 0; v < DV; ++v)
                desc[v * 32 + rank] = make_int4(d[4 * v], d[4 * v + 1], d[4 * v + 2], d[4 * v + 3]);
        }
        if (__any_sync(FULL, bad)) {
            if (lane == 0) atomicExch(K.status(), (int)DEV_INTERNAL);
            ok = false;
            break;
        }
        __syncwarp();
        const uint32_t rows = q_end - skip;
        if (left > rows) {
            wk.next();
            load_leaf();
        }

        // ---- rounds
        auto fetch = [&](Frag &F, uint32_t q0, uint32_t cnt) {
#pragma unroll
            for (int u = 0; u < RPL; ++u) {
                const uint32_t qh = q0 + 32u * u;
                const uint32_t done = __popc(__ballot_sync(FULL, used && e <= qh));
                const uint32_t b = e - qh;
                const unsigned bits =
                    __reduce_or_sync(FULL, used && b - 1u < 31u ? 1u << b : 0u);
                F.l[u] = (int)(done + __popc(bits & le));
                if constexpr (SRC == SRC_RUN) {
                    if ((uint32_t)lane + 32u * u < cnt) {
                        const uint32_t row =
                            reinterpret_cast<const uint32_t *>(desc + F.l[u])[0] + qh + lane;
                        load_run_row<SS>(K.src().rows + (size_t)row * SS, F.x[u]);
                    }
                }
            }
        };
        auto emit = [&](const Frag &F, uint32_t q0, uint32_t cnt) {
            if (hpos == 0 && nfull >= 2) {
                // re-entering a half: the bulk store issued from it two
                // flushes ago must have finished reading it
                if (lane == 0) bulk_wait_read<1>();
                __syncwarp();
            }
            int32_t *dst = ring + (size_t)(half * B + hpos + lane) * DS;
#pragma unroll
            for (int u = 0; u < RPL; ++u) {
                if ((uint32_t)lane + 32u * u < cnt) {
                    int d[DV * 4];
#pragma unroll
                    for (int v = 0; v < DV; ++v) {
                        const int4 x = desc[v * 32 + F.l[u]];
                        d[4 * v] = x.x;
                        d[4 * v + 1] = x.y;
                        d[4 * v + 2] = x.z;
                        d[4 * v + 3] = x.w;
                    }
                    constexpr int H = SRC == SRC_RUN ? 2 : 3;
                    int w[DS];
#pragma unroll
                    for (int c = 0; c < DS; ++c) w[c] = 0;
#pragma unroll
                    for (int c = 0; c < NP; ++c) w[c] = d[H + c];
                    if constexpr (SRC == SRC_RUN) {
                        w[NP] = d[1] - F.x[u][0];
#pragma unroll
                        for (int c = 1; c < W; ++c) w[NP + c] = F.x[u][c];
                    } else {
                        const uint32_t o = q0 + 32u * u + lane - (uint32_t)d[0];
                        w[NP] = d[1] - (int)(o * K.src().pair.h1);
                        w[NP + 1] = d[2] + (int)(o * K.src().pair.g1);
                    }
                    store_row<DS>(dst + u * 32 * DS, w, lane);
                }
            }
            hpos += cnt;
            if (hpos == B) {
                flush_words(K.out() + (row0 + (uint64_t)nfull * B) * DS, K.aligned(),
                            ring + (size_t)half * B * DS, B * DS, lane, pol);
                ++nfull;
                half ^= 1u;
                hpos = 0;
            }
        };
        // rows of the round at q0 with `at` rows already in the ring half
        // (rounds never cross a half)
        auto rows_at = [&](uint32_t q0, uint32_t at) {
            uint32_t c = q_end - q0;
            if (c > RR) c = RR;
            return c < B - at ? c : B - at;
        };
        uint32_t q0 = skip;
        if (q0 < q_end) {
            if constexpr (SRC == SRC_RUN) {
                Frag x, y;
                uint32_t c0 = rows_at(q0, hpos);
                fetch(x, q0, c0);
                for (;;) {
                    uint32_t c1 = 0;
                    if (q0 + c0 < q_end) {
                        c1 = rows_at(q0 + c0, hpos + c0 == B ? 0u : hpos + c0);
                        fetch(y, q0 + c0, c1);
                    }
                    emit(x, q0, c0);
                    q0 += c0;
                    if (c1 == 0) break;
                    c0 = 0;
                    if (q0 + c1 < q_end) {
                        c0 = rows_at(q0 + c1, hpos + c1 == B ? 0u : hpos + c1);
                        fetch(x, q0 + c1, c0);
                    }
                    emit(y, q0, c1);
                    q0 += c1;
                    if (c0 == 0) break;
                }
            } else {
                Frag x;
                while (q0 < q_end) {
                    const uint32_t c = rows_at(q0, hpos);
                    fetch(x, q0, c);
                    emit(x, q0, c);
                    q0 += c;
                }
            }
        }
        left -= rows;
        skip = skip > e_all ? skip - e_all : 0u;
        base = Elast;
    }
    if (hpos > 0)
        flush_words(K.out() + (row0 + (uint64_t)nfull * B) * DS, K.aligned(),
                    ring + (size_t)half * B * DS, hpos * DS, lane, pol);
    if (lane == 0) bulk_wait_read_all();
    __syncwarp();
    return ok;
}

// Largest u in [0, n) with f(u) <= R (f non-decreasing, f(0) <= R), searched
// 32 probes at a time by a warp; *val = f(u).
template <class Fn>
__device__ __forceinline__ uint32_t warp_last_le(uint32_t n, uint64_t R, int lane, uint64_t *val,
                                                 Fn f) {
    uint32_t lo = 0, hi = n;  // f(lo) <= R; f(hi) > R or hi == n
    uint64_t flo = f(0u);
    while (hi - lo > 1) {
        const uint32_t step = (hi - lo + 31) >> 5;
        const uint64_t u = (uint64_t)lo + (uint64_t)(lane + 1) * step;
        bool okp = false;
        uint64_t fu = 0;
        if (u < hi) {
            fu = f((uint32_t)u);
            okp = fu <= R;
        }
        const int cnt = __popc(__ballot_sync(FULL, okp));
        const uint64_t fsel = shfl_u64(fu, cnt > 0 ? cnt - 1 : 0);
        if (cnt > 0) {
            flo = fsel;
            lo += (uint32_t)cnt * step;
        }
        if (lo + step < hi) hi = lo + step;
    }
    *val = flo;
    return lo;
}

}  // namespace fz
