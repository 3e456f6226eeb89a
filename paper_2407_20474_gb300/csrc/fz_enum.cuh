// fz_enum.cuh -- parameters of an enumeration launch, rank and cost searches
// and the items of work-balanced slicing, shared by the enumeration kernels
// (fz_enum.cu, fz_flat.cu).
#pragma once

#include "fz_walk.cuh"

namespace fz {

constexpr int ENUM_WARPS = 8;
constexpr int ENUM_THREADS = ENUM_WARPS * 32;
constexpr int RING_BYTES_PER_WARP = 6 * 1024;  // two halves; 4 CTAs of 8 warps per SM
constexpr uint32_t CAP32 = 0xffffffffu;

constexpr int FLAT_MAX_NP = 7;  // longest prefix of the flat walk

struct EnumParams {
    const uint64_t *C;     // count table rows 0..d, stride cs
    int64_t cs;
    const uint64_t *O;     // memo CSR offsets (top + 1), or null
    const int32_t *memo;   // memo rows, K int32 each, or null
    uint64_t memo_rows;    // rows in memo (bounds guard)
    int32_t *out;          // row 0 = rank rank_begin
    int *status;
    unsigned long long *slice_counter;
    uint64_t rank_begin;   // absolute rank of out row 0
    uint64_t nrows;        // rows to write
    uint64_t slice_rows;   // S (multiple of 4), used when RT is null
    uint64_t nslices;
    const uint64_t *RT;    // candidates table rows 0..lam_r (stride cs), or null
    int by_cost;           // items by cost (see EnumLaunch)
    int whole;             // all rows of the set are asked for
    uint64_t W;            // cost of one unit of walk work (a prefix of length lam_r), in rows
    uint64_t slice_cost;   // cost units per work item when RT is set
    int lam_r;             // one past the leaf coordinate (RT[lam_r] = 1)
    int n, d, K, top;
    int lam_m;             // coordinate whose children are memo leaves (d-K-1), or -1
    int lam_w;             // coordinate whose children are walk leaves (d-2)
    int half_rows;         // B: rows per ring half (multiple of 32)
    int aligned;           // out is 16-byte aligned
    int ctas_per_sm;       // occupancy cap of the launch (0 = none)
    int dense_min;         // memo batches with >= dense_min rows per leaf go leaf by leaf
    const int4 *run_memo;  // full memo in run order (k <= 3), or null
    const uint64_t *cls_beg;
    int g[FZ_MAX_D];
    FastDiv fdg[FLAT_MAX_NP];  // division by g_0, g_1, ... (the flat walk)
    // Where the rows of a leaf come from: the run-order table (run_memo and
    // cls_beg, its generator g_{d-K-1}) or the closed form of the last two
    // generators.
    LeafSource leaf;
    // Walk leaves as a progression: the candidates a_{d-2} = v of remainder r
    // with g_{d-1} | r - v g_{d-2} are v = v* (mod h1), along which a_{d-1}
    // grows by g1 (leaf.pair).  0: candidate by candidate.
    int progression;
    // Pair memo: a full memo of depth 2 kept as a formula, no table.  Memo
    // leaf p (remainder at depth d-2) holds Z(p, (g_{d-2}, g_{d-1})): row o
    // is a_{d-2} = a_top - o h1, a_{d-1} = (p - a_{d-2} g_{d-2}) / g_{d-1}.
    int pair_memo;
    int flat_np;           // > 0: the flat walk, leaves are prefixes of this length
    int flat_src;          // SRC_RUN, SRC_PAIR or (batches) SRC_RANK
};

struct WarpPath {
    int a[FZ_MAX_D];      // a_0..a_{lam-1}
    int r[FZ_MAX_D + 1];  // r[0] = n, r[c+1] = r[c] - a[c] g[c]
};

enum LeafType : int { T_NONE = 0, T_MEMO = 1, T_WALK = 2, T_INTERNAL = 3 };

// Largest u in [0, umax] with F(u) <= R, F(u) = C[c][rem - (umax + 1 - u) g_c]
// (rows in the children with a_c > umax - u), searched 32 probes at a time.
// Returns the child a_c = umax - u holding relative rank R and the rows
// before it.  Requires R < C[c][rem].
__device__ __forceinline__ void find_child(const EnumParams &P, int c, int rem, uint64_t R,
                                           int lane, int &v_out, uint64_t &before_out) {
    const uint32_t g = (uint32_t)P.g[c];
    const uint32_t umax = (uint32_t)rem / g;
    const uint64_t *row = P.C + (long long)c * P.cs + rem;
    const uint32_t u = warp_last_le(umax + 1u, R, lane, &before_out, [&](uint32_t x) {
        return x == 0 ? 0ull : __ldg(row - (int64_t)((umax + 1u - x) * g));
    });
    v_out = (int)(umax - u);
}

// find_child by one thread: the child a_j = v of a node with remainder rem that
// holds relative rank R, i.e. the least v with at most R rows in the children
// above it, C[j][rem - (v + 1) g] <= R; *before = those rows.  Gallops from v0.
__device__ __forceinline__ uint32_t thread_child_from(const uint64_t *row, uint32_t rem,
                                                      uint32_t g, uint32_t vmax, uint64_t R,
                                                      uint32_t v0, uint64_t *before) {
    auto above = [&](uint32_t v) {
        return v >= vmax ? 0ull : __ldg(row + (rem - (v + 1u) * g));
    };
    // lo: above(lo) > R (or -1); hi: above(hi) <= R
    int64_t lo, hi;
    uint64_t ahi = above(v0);
    int64_t st = 1;
    if (ahi <= R) {
        hi = v0;
        for (;; st *= 2) {
            lo = hi - st;
            if (lo < 0) {
                lo = -1;
                break;
            }
            const uint64_t t = above((uint32_t)lo);
            if (t > R) break;
            hi = lo;
            ahi = t;
        }
    } else {
        lo = v0;
        for (;; st *= 2) {
            hi = lo + st;
            if (hi > (int64_t)vmax) hi = vmax;
            ahi = above((uint32_t)hi);
            if (ahi <= R) break;
            lo = hi;
        }
    }
    while (hi - lo > 1) {
        const int64_t mid = (lo + hi) >> 1;
        const uint64_t t = above((uint32_t)mid);
        if (t <= R) {
            hi = mid;
            ahi = t;
        } else {
            lo = mid;
        }
    }
    *before = ahi;
    return (uint32_t)hi;
}

// The same from an estimate: the rows above grow about as the `power`-th power
// of the count row's index (all: rows under the node).
__device__ __forceinline__ uint32_t thread_child(const uint64_t *row, uint32_t rem, uint32_t g,
                                                 uint32_t vmax, uint64_t R, uint64_t all,
                                                 int power, uint64_t *before) {
    const float f = __log2f((float)R + 0.5f) - __log2f((float)all);
    const float x = (float)rem * exp2f(f / (float)power);
    uint32_t v = x < (float)rem ? (uint32_t)(((float)rem - x) / (float)g) : 0u;
    return thread_child_from(row, rem, g, vmax, R, v < vmax ? v : vmax, before);
}

// Walk state of one warp (warp-uniform).
struct RunState {
    int lam;          // coordinate of the current run of sibling leaves
    int inwalk;       // inside the subtree of a memo-level child with p >= top
    long long vcur;   // next candidate value of a_lam (descending)
    uint64_t base;    // rows in the siblings before vcur
};

// Choose the first live child at depths c_from..c_to-1 (path stored by lane 0).
__device__ __forceinline__ void descend(const EnumParams &P, WarpPath *wp, int c_from,
                                        int c_to, int lane) {
    int rem = wp->r[c_from];
    for (int c = c_from; c < c_to; ++c) {
        int v = rem / P.g[c];
        // usually the largest child is live (one load); else search
        if (__ldg(P.C + (long long)(c + 1) * P.cs + (rem - v * P.g[c])) == 0ull) {
            uint64_t before;
            find_child(P, c, rem, 0ull, lane, v, before);
        }
        rem -= v * P.g[c];
        if (lane == 0) {
            wp->a[c] = v;
            wp->r[c + 1] = rem;
        }
    }
    __syncwarp();
}

// Position the warp on the leaf holding absolute rank R.  Returns the offset
// of R inside that leaf.  Sets *ok = false if the table is inconsistent.
__device__ inline uint64_t unrank_to_leaf(const EnumParams &P, WarpPath *wp, uint64_t R, int lane,
                                   RunState &st, bool *ok) {
    int rem = P.n;
    if (lane == 0) wp->r[0] = rem;
    int inwalk = 0;
    const bool memo = P.lam_m >= 0;
    *ok = true;
    for (int c = 0; c < P.d; ++c) {
        const int runlev = (memo && !inwalk) ? P.lam_m : P.lam_w;
        const uint64_t total = __ldg(P.C + (long long)c * P.cs + rem);
        if (R >= total) {
            *ok = false;
            break;
        }
        int v;
        uint64_t before;
        find_child(P, c, rem, R, lane, v, before);
        R -= before;
        const int p = rem - v * P.g[c];
        if (c == runlev) {
            if (memo && !inwalk && p >= P.top && P.lam_m < P.lam_w) {
                // memo-level child beyond the memo: walk its subtree
                if (lane == 0) {
                    wp->a[c] = v;
                    wp->r[c + 1] = p;
                }
                rem = p;
                inwalk = 1;
                continue;
            }
            st.lam = c;
            st.inwalk = inwalk;
            st.vcur = v;
            st.base = before;
            __syncwarp();
            return R;
        }
        if (lane == 0) {
            wp->a[c] = v;
            wp->r[c + 1] = p;
        }
        rem = p;
    }
    __syncwarp();
    *ok = false;
    return 0;
}

// Move to the next run after the current one is exhausted.  Returns false at
// the end of the stream.
__device__ inline bool advance(const EnumParams &P, WarpPath *wp, int lane, RunState &st) {
    const bool memo = P.lam_m >= 0;
    for (int j = st.lam - 1; j >= 0; --j) {
        const int rem = wp->r[j];
        const int aj = wp->a[j];
        const uint64_t *row = P.C + (long long)j * P.cs;
        const uint64_t R = __ldg(row + (rem - aj * P.g[j]));  // rows in children >= aj
        const uint64_t total = __ldg(row + rem);
        if (R >= total) continue;
        // usually the next smaller value is live (one load); else search
        int v = aj - 1;
        if (__ldg(P.C + (long long)(j + 1) * P.cs + (rem - v * P.g[j])) == 0ull) {
            uint64_t before;
            find_child(P, j, rem, R, lane, v, before);
        }
        const int p = rem - v * P.g[j];
        if (lane == 0) {
            wp->a[j] = v;
            wp->r[j + 1] = p;
        }
        __syncwarp();
        int nw;
        if (memo && j < P.lam_m)
            nw = 0;
        else if (memo)
            nw = 1;  // at or below the memo level: inside a walked subtree
        else
            nw = 0;
        const int newlam = (memo && !nw) ? P.lam_m : P.lam_w;
        descend(P, wp, j + 1, newlam, lane);
        st.lam = newlam;
        st.inwalk = nw;
        st.vcur = wp->r[newlam] / P.g[newlam];
        st.base = 0;
        return true;
    }
    return false;
}

// ---------------------------------------------------------------------------
// Work-balanced slicing.  The cost of a subtree is its rows plus W for every
// unit of walk work in it -- a leaf candidate, a walk run or a run-order run,
// i.e. a prefix of length lam_r the walk evaluates, live or not (balance_level
// picks lam_r and W); RT[j][x] counts those prefixes (RT[lam_r] = 1, and row j
// is row j+1 strided-summed with stride g_j, like the count table; a memo
// leaf above level lam_r is clamped to one unit), so the cost of the
// children a_j >= v of a node is
// C[j][x] + W RT[j][x] with x = rem - v g_j.  Work items are equal cost ranges, located by the same
// 32-probe search as ranks, then snapped to ranks that are multiples of 32
// from rank_begin: 32 rows are 128 d bytes, so every bulk store of a slice
// starts on a 128-byte line when the output is 128-byte aligned.
// ---------------------------------------------------------------------------
// A memo leaf above the counted level (a partial memo of depth K > 2 whose
// runs table counts walk runs): the node at depth j is one unit of cost.
__device__ __forceinline__ bool is_memo_unit(const EnumParams &P, int j, int rem) {
    return P.lam_m >= 0 && j == P.lam_m + 1 && j < P.lam_r && rem < P.top;
}

__device__ __forceinline__ uint64_t cost_at(const EnumParams &P, int j, long long idx) {
    if (idx < 0) return 0ull;
    return __ldg(P.C + (long long)j * P.cs + idx) + P.W * __ldg(P.RT + (long long)j * P.cs + idx);
}

// Rank of the first row whose cumulative cost reaches `target` (clamped to
// the total row count).
__device__ inline uint64_t cost_to_rank(const EnumParams &P, uint64_t target, int lane) {
    int rem = P.n;
    uint64_t rank = 0;
    if (target >= cost_at(P, 0, rem)) return __ldg(P.C + rem);
    int lev = P.lam_r;
    for (int j = 0; j < P.lam_r; ++j) {
        if (is_memo_unit(P, j, rem)) {
            lev = j;
            break;
        }
        const long long g = P.g[j];
        const long long umax = rem / g;
        const long long base = (long long)rem - (umax + 1) * g;
        long long lo = 0, hi = umax + 1;
        uint64_t flo = 0;
        while (hi - lo > 1) {
            const long long step = (hi - lo + 31) >> 5;
            const long long u = lo + (long long)(lane + 1) * step;
            bool ok = false;
            uint64_t fu = 0;
            if (u < hi) {
                fu = cost_at(P, j, base + u * g);
                ok = fu <= target;
            }
            const int cnt = __popc(__ballot_sync(FULL, ok));
            const uint64_t fsel = shfl_u64(fu, cnt > 0 ? cnt - 1 : 0);
            if (cnt > 0) {
                flo = fsel;
                lo += (long long)cnt * step;
            }
            const long long nh = lo + step;
            if (nh < hi) hi = nh;
        }
        const long long idx = base + lo * g;
        rank += idx >= 0 ? __ldg(P.C + (long long)j * P.cs + idx) : 0ull;
        target -= flo;
        rem = (int)(rem - (umax - lo) * g);
    }
    const uint64_t rows = __ldg(P.C + (long long)lev * P.cs + rem);
    const uint64_t t = target > P.W ? target - P.W : 0ull;
    return rank + (t < rows ? t : rows);
}

// Cumulative cost of everything before rank R.
__device__ inline uint64_t rank_to_cost(const EnumParams &P, uint64_t R, int lane) {
    int rem = P.n;
    if (R >= __ldg(P.C + rem)) return cost_at(P, 0, rem);
    uint64_t cost = 0;
    for (int j = 0; j < P.lam_r; ++j) {
        if (is_memo_unit(P, j, rem)) break;
        int v;
        uint64_t before;
        find_child(P, j, rem, R, lane, v, before);
        cost += before + P.W * (rem - (long long)(v + 1) * P.g[j] >= 0
                                    ? __ldg(P.RT + (long long)j * P.cs +
                                            (rem - (long long)(v + 1) * P.g[j]))
                                    : 0ull);
        R -= before;
        rem -= v * P.g[j];
    }
    return cost + P.W + R;
}

// Rows [row0, row1) (relative to out) of work item s.  With a candidates
// table the items are cost ranges of [cost_lo, cost_hi) snapped to multiples
// of 32 rows: the first four fifths of the cost in items of slice_cost, the
// rest in items of an eighth of that, so the warps that take the last items
// finish close together.  Otherwise equal-row ranges.  Returns 0 when s is
// past the last item, 1 when the item is empty, 2 otherwise.
__device__ __forceinline__ int item_rows(const EnumParams &P, uint64_t s, uint64_t cost_lo,
                                         uint64_t cost_hi, int lane, uint64_t &row0,
                                         uint64_t &row1) {
    if (P.RT) {
        const uint64_t sc = P.slice_cost;
        const uint64_t n1 = (cost_hi - cost_lo) / sc * 4 / 5;  // large items
        const uint64_t sc_t = sc / 8 > 64 ? sc / 8 : 64;
        uint64_t c0, c1;
        if (s < n1) {
            c0 = cost_lo + s * sc;
            c1 = c0 + sc;
        } else {
            const uint64_t t = s - n1;
            const uint64_t base = cost_lo + n1 * sc;
            if (t >= (cost_hi - base + sc_t - 1) / sc_t) return 0;
            c0 = base + t * sc_t;
            c1 = c0 + sc_t;
        }
        if (c0 >= cost_hi) return 0;
        row0 = 0;
        if (s > 0) {
            const uint64_t r = cost_to_rank(P, c0, lane);
            row0 = r > P.rank_begin ? ((r - P.rank_begin) & ~31ull) : 0ull;
            if (row0 > P.nrows) row0 = P.nrows;
        }
        row1 = P.nrows;
        if (c1 < cost_hi) {
            const uint64_t r = cost_to_rank(P, c1, lane);
            row1 = r > P.rank_begin ? ((r - P.rank_begin) & ~31ull) : 0ull;
            if (row1 > P.nrows) row1 = P.nrows;
        }
        return row1 > row0 ? 2 : 1;
    }
    if (s >= P.nslices) return 0;
    row0 = s * P.slice_rows;
    row1 = row0 + P.slice_rows < P.nrows ? row0 + P.slice_rows : P.nrows;
    return 2;
}

__device__ __forceinline__ void flush_rows(const EnumParams &P, const int32_t *src,
                                           uint64_t out_row, uint32_t nrows, int d, int lane,
                                           uint64_t pol) {
    flush_words(P.out + out_row * (uint64_t)d, P.aligned, src, nrows * (uint32_t)d, lane, pol);
}

// Parameters of a launch as a walk and a sink read them: in constant memory
// (a kernel parameter), or in the warp's shared memory, whose address is
// hidden at every use so that nothing is kept in registers between uses.
struct ConstParams {
    const EnumParams &p;
    __device__ __forceinline__ const EnumParams &operator()() const { return p; }
};
extern __shared__ __align__(128) unsigned char enum_smem[];
struct SharedParams {
    uint32_t off;  // from the start of the block's dynamic shared memory
    __device__ __forceinline__ const EnumParams &operator()() const {
        uint32_t o = off;
        asm volatile("" : "+r"(o));
        return *reinterpret_cast<const EnumParams *>(enum_smem + o);
    }
};
template <class PA>
struct EnumSink {
    PA params;
    __device__ __forceinline__ const LeafSource &src() const { return params().leaf; }
    __device__ __forceinline__ int32_t *out() const { return params().out; }
    __device__ __forceinline__ bool aligned() const { return params().aligned != 0; }
    __device__ __forceinline__ int *status() const { return params().status; }
};

// The flat walk's leaves of an enumeration: the prefixes (a_0..a_{NP-1}) in
// descending order, each lane at its own, 32 apart from one batch to the
// next.  Row ends are absolute ranks: the rows of the greater prefixes of
// every level (pb, read again when the parent changes) plus the count row of
// the last prefix coordinate.
template <int NP, class PA>
struct PrefixWalk {
    PA params;
    int a[NP], r[NP];  // r[j]: remainder before a_j
    uint64_t pb = 0;
    bool dead = false;
    __device__ __forceinline__ explicit PrefixWalk(const PA &pa) : params(pa) {}

    __device__ __forceinline__ void parents() {
        const EnumParams &P = params();
        pb = 0;
#pragma unroll
        for (int j = 0; j < NP - 1; ++j) {
            const int idx = r[j + 1] - P.g[j];  // r[j] - (a[j] + 1) g_j
            if (idx >= 0) pb += __ldg(P.C + (int64_t)j * P.cs + idx);
        }
    }
    __device__ __forceinline__ void step(int s) {
        if (dead) return;
        int x = a[NP - 1] - s;
        if (x < 0) {
            if constexpr (NP == 1) {
                dead = true;
                return;
            } else {
                const EnumParams &P = params();
                do {
                    const int owe = -x - 1;  // prefixes past the next parent's first
                    // the next parent: decrement its deepest positive
                    // coordinate, reset the ones after it to their maxima
                    int jj = -1;
#pragma unroll
                    for (int j = 0; j < NP - 1; ++j)
                        if (a[j] > 0) jj = j;
                    if (jj < 0) {
                        dead = true;
                        return;
                    }
#pragma unroll
                    for (int j = 0; j < NP - 1; ++j) {
                        if (j == jj)
                            a[j] -= 1;
                        else if (j > jj)
                            a[j] = (int)fd_div((uint32_t)r[j], P.fdg[j]);
                        if (j >= jj) r[j + 1] = r[j] - a[j] * P.g[j];
                    }
                    x = (int)fd_div((uint32_t)r[NP - 1], P.fdg[NP - 1]) - owe;
                } while (x < 0);
                parents();
            }
        }
        a[NP - 1] = x;
    }
    __device__ __forceinline__ int word(int c) const { return a[c]; }
    __device__ __forceinline__ bool leaf(uint32_t &p, uint64_t &E) const {
        if (dead) return false;
        const EnumParams &P = params();
        p = (uint32_t)(r[NP - 1] - a[NP - 1] * P.g[NP - 1]);
        E = pb + __ldg(P.C + (int64_t)(NP - 1) * P.cs + p);
        return true;
    }
    __device__ __forceinline__ void next() { step(32); }
};

// Rows [row0, row1) of an enumeration by the flat walk.  `mem`: the warp's
// shared memory (leaf descriptors, then a ring of two halves of B rows).
template <int D, int NP, int SRC, class PA>
__device__ __forceinline__ bool flat_slice(const PA &pa, unsigned char *mem, uint32_t B,
                                           uint64_t row0, uint64_t row1, uint64_t pol, int lane) {
    const EnumParams &P = pa();
    const uint64_t R = P.rank_begin + row0;
    PrefixWalk<NP, PA> wk(pa);
    uint64_t off = R;
    int rem = P.n;
#pragma unroll
    for (int j = 0; j < NP; ++j) {
        uint64_t before;
        wk.r[j] = rem;
        find_child(P, j, rem, off, lane, wk.a[j], before);
        off -= before;
        rem -= wk.a[j] * P.g[j];
    }
    wk.parents();
    wk.step(lane);
    int4 *desc = reinterpret_cast<int4 *>(mem);
    int32_t *ring = reinterpret_cast<int32_t *>(mem + leaf_bytes<NP, SRC>());
    return flat_rows<NP, D - NP, D, SRC>(wk, R - off, (uint32_t)off, EnumSink<PA>{pa}, row0,
                                         (uint32_t)(row1 - row0), desc, ring, B, pol, lane);
}

// The flat walk's costs: the candidates table's row NP - 1 is x / g + 1, computed.
template <int NP>
__device__ __forceinline__ uint64_t flat_total_cost(const EnumParams &P) {
    const uint64_t runs =
        NP == 1 ? (uint64_t)fd_div((uint32_t)P.n, P.fdg[0]) + 1ull : __ldg(P.RT + P.n);
    return __ldg(P.C + P.n) + P.W * runs;
}

// Ranks at which the cumulative costs t0 <= t1 are reached (cost_to_rank for a
// candidates table counted at level NP), both searches' loads in flight
// together.
template <int NP>
__device__ __forceinline__ void flat_cost_to_ranks(const EnumParams &P, uint64_t t0, uint64_t t1,
                                                   int lane, uint64_t &rank0, uint64_t &rank1) {
    uint64_t tgt[2] = {t0, t1}, rank[2] = {0, 0}, rows[2] = {0, 0};
    uint32_t rem[2] = {(uint32_t)P.n, (uint32_t)P.n};
#pragma unroll
    for (int j = 0; j < NP; ++j) {
        const uint32_t g = (uint32_t)P.g[j];
        const uint64_t *C = P.C + (int64_t)j * P.cs;
        const uint64_t *T = j < NP - 1 ? P.RT + (int64_t)j * P.cs : nullptr;
        uint32_t lo[2] = {0, 0}, hi[2], um[2];
        uint64_t flo[2] = {0, 0}, clo[2] = {0, 0};
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            um[k] = fd_div(rem[k], P.fdg[j]);
            hi[k] = um[k] + 1u;
        }
        while (hi[0] - lo[0] > 1u || hi[1] - lo[1] > 1u) {
            uint64_t cu[2] = {0, 0}, fu[2] = {0, 0};
            uint32_t step[2];
            bool in[2];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                step[k] = (hi[k] - lo[k] + 31) >> 5;
                const uint64_t u = (uint64_t)lo[k] + (uint64_t)(lane + 1) * step[k];
                in[k] = u < hi[k];
                if (in[k]) {
                    const uint32_t x = rem[k] - (um[k] + 1u - (uint32_t)u) * g;
                    cu[k] = __ldg(C + x);
                    fu[k] = j < NP - 1 ? __ldg(T + x) : (uint64_t)fd_div(x, P.fdg[j]) + 1ull;
                }
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                fu[k] = cu[k] + P.W * fu[k];
                const int cnt = __popc(__ballot_sync(FULL, in[k] && fu[k] <= tgt[k]));
                const int src = cnt > 0 ? cnt - 1 : 0;
                const uint64_t fs = shfl_u64(fu[k], src), cs = shfl_u64(cu[k], src);
                if (hi[k] - lo[k] > 1u) {
                    if (cnt > 0) {
                        flo[k] = fs;
                        clo[k] = cs;
                        lo[k] += (uint32_t)cnt * step[k];
                    }
                    if (lo[k] + step[k] < hi[k]) hi[k] = lo[k] + step[k];
                }
            }
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            rank[k] += clo[k];
            tgt[k] -= flo[k];
            // the leaf's rows: the count row there less the children above it
            if (j == NP - 1) rows[k] = __ldg(C + (rem[k] - (um[k] - lo[k]) * g)) - clo[k];
            rem[k] -= (um[k] - lo[k]) * g;
        }
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const uint64_t t = tgt[k] > P.W ? tgt[k] - P.W : 0ull;
        rank[k] += t < rows[k] ? t : rows[k];
    }
    rank0 = rank[0];
    rank1 = rank[1];
}

// ---------------------------------------------------------------------------
// Many instances.  Work items (instance, slice) are numbered consecutively,
// instance i owning items [item0[i], item0[i+1]); a launch covers the
// instances [first, last) -- those of one shape, or all the general kernel
// takes -- and its warps take items from an atomic counter, copying the
// instance's parameters into their own shared-memory slot when it changes.
// ---------------------------------------------------------------------------
struct BatchEnumParams {
    const EnumParams *inst;   // per-instance parameters; `out` holds a byte offset
    int32_t *out_base;        // output base the offsets are added to
    const uint64_t *item0;    // prefix of work items over all instances
    int first, last;
    uint64_t item_lo, item_hi;  // items of this launch
    unsigned long long *item_counter;
    int chained;              // launched to overlap the launch before it
};

// Instance of `item`, its parameters in *ep.  By 32 probes at a time, or
// (HALVING, the general kernel, whose items are long) one: the wide search
// there costs the walk's loops 28 more bytes of spills a thread (512 partial
// memos, 1.1e7 rows: 8.5 ms against 8.1).
template <bool HALVING = false>
__device__ __forceinline__ uint64_t batch_locate(const BatchEnumParams &BP, EnumParams *ep,
                                                 int &cur, uint64_t item, int lane) {
    uint64_t start;
    int id = BP.first;
    if constexpr (HALVING) {
        for (int hi = BP.last; hi - id > 1;) {  // item0[id] <= item < item0[hi]
            const int mid = (id + hi) >> 1;
            if (__ldg(BP.item0 + mid) <= item)
                id = mid;
            else
                hi = mid;
        }
        start = __ldg(BP.item0 + id);
    } else {
        id += (int)warp_last_le((uint32_t)(BP.last - BP.first), item, lane, &start,
                                [&](uint32_t u) { return __ldg(BP.item0 + BP.first + u); });
    }
    if (id != cur) {
        const uint32_t *src = reinterpret_cast<const uint32_t *>(BP.inst + id);
        uint32_t *dst = reinterpret_cast<uint32_t *>(ep);
        __syncwarp();
        for (int w = lane; w < (int)(sizeof(EnumParams) / 4); w += 32) dst[w] = __ldg(src + w);
        __syncwarp();
        if (lane == 0) {
            int32_t *o = reinterpret_cast<int32_t *>(reinterpret_cast<char *>(BP.out_base) +
                                                     reinterpret_cast<uintptr_t>(ep->out));
            ep->out = o;
            ep->aligned = ((uintptr_t)o & 15u) == 0;
        }
        __syncwarp();
        cur = id;
    }
    return item - start;
}

// fz_flat.cu
int launch_enum_flat(const EnumParams &P, int warp_bytes, cudaStream_t s, int sms);
// The rank walk: sets whose prefixes of d - 2 coordinates are mostly empty.
bool rank_walk_serves(int d);
int launch_rank_walk(const EnumParams &P, int warp_bytes, cudaStream_t s, int sms);
int launch_flat_batch(const BatchEnumParams &BP, int d, int np, int src, cudaStream_t s, int sms,
                      int ctas_per_sm);
// fz_enum.cu: grid and launch of a persistent enumeration kernel.
constexpr int ENUM_MAX_SMEM = 200 * 1024;
// Blocks an SM takes when `fit` do.
inline int blocks_for(int fit, int ctas_per_sm) {
    if (ctas_per_sm > 0 && ctas_per_sm < fit) fit = ctas_per_sm;
    return fit < 1 ? 1 : fit;
}
// Batches: three blocks of the flat walk's kernels fill an SM's registers, so a
// cap that is to leave room takes one less than fit.
inline int batch_blocks_for(int fit, int ctas_per_sm) {
    return blocks_for(leaves_room(ctas_per_sm) ? fit - 1 : fit, ctas_per_sm);
}
// A launch of ENUM_THREADS threads a block.  Under a cap the SM is asked for
// all its shared memory, so that other kernels' blocks find some; chained: it
// may start while the launch before it drains.
template <typename Kern, typename... Args>
int launch_capped(Kern kern, unsigned grid, size_t smem, cudaStream_t s, int ctas_per_sm,
                  bool chained, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(ENUM_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    cfg.attrs = attr;
    if (chained) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (leaves_room(ctas_per_sm)) {
        attr[cfg.numAttrs].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
        attr[cfg.numAttrs++].val.sharedMemCarveout = cudaSharedmemCarveoutMaxShared;
    }
    FZ_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, args...));
    note_launch();
    return FZ_OK;
}
template <typename Kern, typename... Args>
int launch_enum_grid(Kern kern, const EnumParams &P, size_t smem, cudaStream_t s, int sms,
                     DeviceOnce &attr_set, Args... args) {
    if (smem > (size_t)ENUM_MAX_SMEM) return set_error(FZ_EINTERNAL, "enumerate: ring too large");
    int dev = 0;
    FZ_CUDA_TRY(cudaGetDevice(&dev));
    if (!attr_set.is_set(dev)) {
        FZ_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         ENUM_MAX_SMEM));
        attr_set.set(dev);
    }
    int per_sm = 0;
    FZ_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, ENUM_THREADS, smem));
    uint64_t want = (P.nslices + ENUM_WARPS - 1) / ENUM_WARPS;
    uint64_t grid = (uint64_t)blocks_for(per_sm, P.ctas_per_sm) * sms;
    if (want < grid) grid = want;
    if (grid < 1) grid = 1;
    FZ_CUDA_TRY(cudaMemsetAsync(P.slice_counter, 0, sizeof(unsigned long long), s));
    return launch_capped(kern, (unsigned)grid, smem, s, P.ctas_per_sm, false, P, args...);
}

}  // namespace fz
