// fz_enum.cu -- lexicographic enumeration of Z(n, g) with low-dimension
// tabulation (Section 3.1), sliced by exact ranks.
//
// The output list (descending lexicographic order) is the depth-first walk of
// the tree whose depth-c nodes are prefixes (a_0..a_{c-1}) with remainder
// rem = n - phi(prefix) >= 0; the children of a node are a_c = floor(rem/g_c)
// down to 0 (the order in which the next-candidate step of Algorithm 3.1
// visits them).  The subtree of the child a_c = v holds C[c+1][rem - v g_c]
// rows, and the rows of all children with a_c >= v number C[c][rem - v g_c]
// (count table, fz_count.cu), so any rank is located by searching one table
// row per level.
//
// Leaves ("blocks"), as in the dynamic next-candidate step:
//  * memo leaf: a prefix of length L = d - K whose remainder p is < top;
//    its rows are Memo[p] = Z(p, (g_L..g_{d-1})) with the prefix prepended
//    (the block copy of Section 3.1; the walk then continues from
//    (prefix, 0, ..., 0), the observation of Section 3.1);
//  * walk leaf: a prefix of length d - 1 (reached when no memo applies);
//    its one row, if g_{d-1} divides p, is the candidate of Algorithm 3.1's
//    ordinary step with a_d = p / g_d.
//
// Work split: each warp takes slices of S consecutive ranks (an atomic
// counter hands them out), finds the leaf holding its first rank by table
// search (this replaces the paper's splitWork with exact bounds), and walks
// from there.  A run of sibling leaves is processed 32 at a time: every lane
// evaluates one candidate, the table gives each lane its cumulative row end
// directly, and lanes then fill rows: each lane finds the leaf of its row by
// a 5-step shuffle search.  Rows are assembled in a per-warp shared-memory
// ring of two halves and each full half is written to HBM with one bulk
// (TMA) store, so the stream is written with 16-byte aligned, fully
// coalesced transactions while the warp generates the next half.
#include <algorithm>
#include <cstring>
#include <map>

#include <cstdlib>

#include "fz_enum.cuh"

namespace fz {

// 4-byte global -> shared copy that does not hold a register (cp.async).
// No memory clobber: the source (memo) is read-only, the destination word is
// touched by nothing else until cp.async.wait_group (which has the clobber),
// and volatile keeps issue order with the commit and the wait.
__device__ __forceinline__ void cp_async4(int32_t *sdst, const int32_t *gsrc) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(sdst)), "l"(gsrc));
}
__device__ __forceinline__ void cp_async_commit() {
    asm volatile("cp.async.commit_group;");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Rounds a completed ring half waits before its bulk store, so that the
// cp.async copies of its last rows have landed without stalling the warp.
constexpr int FLUSH_LAG = 2;

// One work item: rows [row0, row1) of the output (relative to P.out),
// produced by unranking row0 and walking from there.  D > 0: tuple width known
// at compile time; D == 0: width P.d (at most FZ_MAX_D).  LAMF >= 0: every run
// is a memo run at coordinate LAMF (full memo, k = D-1-LAMF) fixed at compile
// time; LAMF < 0: generic (runtime run level, walk leaves).  Returns false if
// a device-side consistency check failed (status already recorded).  DMAX:
// with D == 0, the largest width the call serves (shorter row loops and
// prefix arrays for narrow tuples).
template <int D, int LAMF, int DMAX = FZ_MAX_D>
__device__ __forceinline__ bool enum_slice(const EnumParams &P, WarpPath *wp, int32_t *ring,
                                           uint32_t B, uint64_t row0, uint64_t row1,
                                           uint64_t pol, int lane) {
    constexpr int DM = D > 0 ? D : DMAX;
    const int d = D > 0 ? D : P.d;
    constexpr int KF = LAMF >= 0 ? D - 1 - LAMF : 0;
    uint32_t rows_left = (uint32_t)(row1 - row0);

    RunState st;
    bool ok;
    uint64_t skip = unrank_to_leaf(P, wp, P.rank_begin + row0, lane, st, &ok);
    if (!ok) {
        if (lane == 0) atomicExch(P.status, (int)DEV_INTERNAL);
        return false;
    }

    // ring: rows go to half `half` at position hpos; `nfull` halves of
    // this slice are complete; a completed half is flushed FLUSH_LAG
    // rounds later (pend_rounds counts them).
    uint32_t hpos = 0, half = 0, nfull = 0, pend_rounds = 0;
    bool pend = false;

    int pre[DM];
#pragma unroll
    for (int c = 0; c < DM; ++c) pre[c] = (c < st.lam) ? wp->a[c] : 0;

    // ring bookkeeping after a round of cnt rows (both paths)
    auto after_round = [&](uint32_t cnt) {
        cp_async_commit();
        hpos += cnt;
        if (pend && ++pend_rounds >= (uint32_t)FLUSH_LAG) {
            cp_async_wait<FLUSH_LAG>();
            flush_rows(P, ring + (size_t)(half ^ 1u) * B * d,
                          row0 + (uint64_t)(nfull - 1) * B, B, d, lane, pol);
            pend = false;
        }
        if (hpos == B) {
            if (pend) {  // (only if a half holds fewer than FLUSH_LAG rounds)
                cp_async_wait<0>();
                flush_rows(P, ring + (size_t)(half ^ 1u) * B * d,
                              row0 + (uint64_t)(nfull - 1) * B, B, d, lane, pol);
            }
            pend = true;
            pend_rounds = 0;
            ++nfull;
            half ^= 1u;
            hpos = 0;
        }
    };
    auto before_round = [&]() {
        if (hpos == 0 && nfull >= 2) {
            // re-entering a half: its bulk store (the most recent bulk
            // group) must have finished reading it
            if (lane == 0) bulk_wait_read_all();
            __syncwarp();
        }
    };
    while (rows_left > 0) {
        const int lam = LAMF >= 0 ? LAMF : st.lam;
        const int rem = wp->r[lam];
        const int glam = P.g[lam];
        const bool memo_run =
            LAMF >= 0 ? true : ((P.lam_m >= 0) && !st.inwalk && lam == P.lam_m);
        if (LAMF < 0 && !memo_run && lam == P.lam_w && P.progression) {
            // A run of walk leaves (the ordinary step at the last two
            // coordinates): only the candidates a_{d-2} = v whose remainder
            // g_{d-1} divides hold a row, and they form a progression, so
            // rows are produced directly -- v from the largest valid value
            // <= st.vcur down by h1, a_{d-1} up by g1 -- with no candidate
            // that holds no row evaluated.
            long long vtop = -1;
            if (rem % (int)P.leaf.pair.fe.g == 0) {
                const long long h1 = (int)P.leaf.pair.h1;
                const long long vstar = (long long)((rem / (int)P.leaf.pair.fe.g) % h1) * (int)P.leaf.pair.inv % h1;
                if (st.vcur >= vstar) vtop = st.vcur - (st.vcur - vstar) % h1;
            }
            const uint32_t nrun = vtop >= 0 ? (uint32_t)(vtop / (int)P.leaf.pair.h1) + 1u : 0u;
            const int wtop =
                vtop >= 0 ? (int)(((long long)rem - vtop * glam) / P.g[d - 1]) : 0;
            uint64_t qe = skip + rows_left;
            if (qe > nrun) qe = nrun;
            const uint32_t q_end = (uint32_t)qe;
            for (uint32_t q0 = (uint32_t)skip; q0 < q_end;) {
                uint32_t cnt = q_end - q0;
                if (cnt > 32u) cnt = 32u;
                if (cnt > B - hpos) cnt = B - hpos;
                before_round();
                if ((uint32_t)lane < cnt) {
                    const int q = (int)(q0 + lane);
                    int32_t *dst = ring + (size_t)(half * B + hpos + lane) * d;
#pragma unroll
                    for (int c = 0; c < DM; ++c) {
                        if (c >= d - 2) break;
                        dst[c] = pre[c];
                    }
                    dst[d - 2] = (int)(vtop - (long long)q * (int)P.leaf.pair.h1);
                    dst[d - 1] = wtop + q * (int)P.leaf.pair.g1;
                }
                q0 += cnt;
                after_round(cnt);
            }
            const uint32_t emitted = q_end > (uint32_t)skip ? q_end - (uint32_t)skip : 0u;
            rows_left -= emitted;
            if (rows_left == 0) break;
            skip = 0;
            st.vcur = -1;
            if (!advance(P, wp, lane, st)) {
                if (lane == 0) atomicExch(P.status, (int)DEV_INTERNAL);
                ok = false;
                break;
            }
#pragma unroll
            for (int c = 0; c < DM; ++c) pre[c] = (c < st.lam) ? wp->a[c] : 0;
            continue;
        }
        const long long vl = st.vcur - lane;
        const bool valid = vl >= 0;
        int p = 0;
        uint64_t incl = 0;
        int type = T_NONE;
        // a run of walk leaves: candidate v is valid iff g_{d-1} divides the
        // remainder (the ordinary step's test); row ends by counting, no table
        const bool walk_run = LAMF < 0 && !memo_run && lam == P.lam_w;
        uint32_t wq = 0;
        bool wvalid = false;
        if (valid) {
            p = (int)((long long)rem - vl * glam);
            if (p < 0 || p > P.n) {  // cannot happen for 0 <= vl <= rem / glam
                atomicExch(P.status, (int)DEV_INTERNAL);
                p = 0;
            }
            if (walk_run) {
                wq = fd_div((uint32_t)p, P.leaf.pair.fh);
                wvalid = (uint32_t)p - wq * P.leaf.pair.fh.g == 0u;
            } else {
                incl = __ldg(P.C + (long long)lam * P.cs + p);
            }
            if (memo_run && (LAMF >= 0 || p < P.top))
                type = T_MEMO;
            else if (lam == P.lam_w)
                type = T_WALK;
            else
                type = T_INTERNAL;
        }
        if (walk_run) {
            const unsigned vm = __ballot_sync(FULL, wvalid);
            incl = st.base + (uint64_t)__popc(vm & (0xffffffffu >> (31 - lane)));
        }
        uint64_t prev = __shfl_up_sync(FULL, incl, 1);
        if (lane == 0) prev = st.base;
        const uint64_t size = valid ? incl - prev : 0ull;
        const unsigned im = __ballot_sync(FULL, type == T_INTERNAL && size > 0);
        const int first_int = im ? __ffs(im) - 1 : 32;
        const int nvalid = st.vcur + 1 < 32 ? (int)(st.vcur + 1) : 32;
        const int consumed = first_int < nvalid ? first_int : nvalid;
        const uint64_t last_incl = consumed > 0 ? shfl_u64(incl, consumed - 1) : st.base;
        const uint64_t batch_rows = last_incl - st.base;
        uint32_t E32 = CAP32, X32 = 0;
        if (lane < consumed) {
            const uint64_t e = incl - st.base;
            E32 = e < (uint64_t)CAP32 ? (uint32_t)e : CAP32;
            if (type == T_MEMO)
                X32 = (LAMF < 0 && P.pair_memo) ? pair_form_top(P.leaf.pair, (uint32_t)p) : (uint32_t)__ldg(P.O + p);
            else if (type == T_WALK)
                X32 = walk_run ? wq : fd_div((uint32_t)p, P.leaf.pair.fh);
        }
        uint64_t q_end64 = skip + rows_left;
        if (q_end64 > batch_rows) q_end64 = batch_rows;
        const uint32_t q_begin = (uint32_t)skip;
        const uint32_t q_end = (uint32_t)q_end64;
        // Dense batches of memo leaves: rounds follow the leaves, so every
        // lane of a round copies a row of the same leaf (no per-row search).
        const bool all_memo = __all_sync(FULL, lane >= consumed || type == T_MEMO);
        const bool dense = memo_run && all_memo && consumed > 0 &&
                           batch_rows >= (uint64_t)P.dense_min * (uint64_t)consumed;
        if (dense && q_end > q_begin) {
            const int lfirst = __popc(__ballot_sync(FULL, E32 <= q_begin));
            for (int j = lfirst; j < consumed; ++j) {
                const uint32_t ej = __shfl_sync(FULL, E32, j);
                uint32_t sj = __shfl_sync(FULL, E32, j > 0 ? j - 1 : 0);
                if (j == 0) sj = 0;
                const uint32_t lo = sj > q_begin ? sj : q_begin;
                const uint32_t hi = ej < q_end ? ej : q_end;
                if (lo < hi) {
                    const uint32_t xj = __shfl_sync(FULL, X32, j);
                    const int pj = __shfl_sync(FULL, p, j);
                    const int vj = (int)(st.vcur - j);
                    const bool pair = LAMF < 0 && P.pair_memo;
                    if (!pair && (uint64_t)xj + (hi - sj) > P.memo_rows) {  // bounds guard
                        if (lane == 0) atomicExch(P.status, (int)DEV_INTERNAL);
                        break;
                    }
                    const int kk = LAMF >= 0 ? KF : P.K;
                    const int32_t *mbase = pair ? P.memo : P.memo + (size_t)xj * (size_t)kk;
                    for (uint32_t q0 = lo; q0 < hi;) {
                        uint32_t cnt = hi - q0;
                        if (cnt > 32u) cnt = 32u;
                        if (cnt > B - hpos) cnt = B - hpos;
                        before_round();
                        if ((uint32_t)lane < cnt) {
                            int32_t *dst = ring + (size_t)(half * B + hpos + lane) * d;
                            const int32_t *mrow =
                                pair ? mbase : mbase + (size_t)(q0 + lane - sj) * (size_t)kk;
                            if (pair) {
                                // pair memo: the row from the progression
                                const int o = (int)(q0 + lane - sj);
                                const int av = (int)xj - o * (int)P.leaf.pair.h1;
#pragma unroll
                                for (int c = 0; c < DM; ++c) {
                                    if (c >= lam) break;
                                    dst[c] = pre[c];
                                }
                                dst[lam] = vj;
                                dst[lam + 1] = av;
                                dst[lam + 2] = (int)fd_div(
                                    (uint32_t)(pj - av * P.g[d - 2]), P.leaf.pair.fh);
                            } else if constexpr (LAMF >= 0) {
#pragma unroll
                                for (int c = 0; c < LAMF; ++c) dst[c] = pre[c];
                                dst[LAMF] = vj;
#pragma unroll
                                for (int c = 0; c < KF; ++c)
                                    cp_async4(dst + LAMF + 1 + c, mrow + c);
                            } else {
#pragma unroll
                                for (int c = 0; c < DM; ++c) {
                                    if (c >= d)
                                        break;
                                    if (c < lam)
                                        dst[c] = pre[c];
                                    else if (c == lam)
                                        dst[c] = vj;
                                    else
                                        cp_async4(dst + c, mrow + (c - lam - 1));
                                }
                            }
                        }
                        q0 += cnt;
                        after_round(cnt);
                    }
                }
                if (ej >= q_end) break;
            }
        } else {
        for (uint32_t q0 = q_begin; q0 < q_end;) {
            uint32_t cnt = q_end - q0;
            if (cnt > 32u) cnt = 32u;
            if (cnt > B - hpos) cnt = B - hpos;  // rounds never cross a half boundary
            before_round();
            const bool act = (uint32_t)lane < cnt;
            const uint32_t q_last = q0 + cnt - 1;
            const uint32_t q = act ? q0 + lane : q_last;  // idle lanes map a row of the round
            // owning leaf of row q: l = number of leaves ending at or before q
            const int lcur = __popc(__ballot_sync(FULL, E32 <= q0));
            const int nb = __popc(__ballot_sync(FULL, E32 > q0 && E32 <= q_last));
            int l = lcur;
            if (nb <= 3) {
                for (int t = 0; t < nb; ++t) {
                    const uint32_t e = __shfl_sync(FULL, E32, lcur + t);
                    if (e <= q) ++l;
                }
            } else {
                l = 0;
#pragma unroll
                for (int sft = 16; sft >= 1; sft >>= 1) {
                    const uint32_t e = __shfl_sync(FULL, E32, l + sft - 1);
                    if (e <= q) l += sft;
                }
            }
            uint32_t eprev = __shfl_sync(FULL, E32, l > 0 ? l - 1 : 0);
            if (l == 0) eprev = 0;
            const uint32_t o = q - eprev;
            const int pl = __shfl_sync(FULL, p, l);
            const uint32_t xl = __shfl_sync(FULL, X32, l);
            const int vrow = (int)(st.vcur - l);
            bool mleaf = memo_run && (LAMF >= 0 || pl < P.top);
            const bool pair = LAMF < 0 && P.pair_memo && mleaf;
            if (act && mleaf && !pair && (uint64_t)xl + o >= P.memo_rows) {  // bounds guard
                atomicExch(P.status, (int)DEV_INTERNAL);
                mleaf = false;
            }
            if (act) {
                int32_t *dst = ring + (size_t)(half * B + hpos + lane) * d;
                if constexpr (LAMF >= 0) {
#pragma unroll
                    for (int c = 0; c < LAMF; ++c) dst[c] = pre[c];
                    dst[LAMF] = vrow;
                    const int32_t *mrow = P.memo + (size_t)(xl + o) * (size_t)KF;
                    if (mleaf) {
#pragma unroll
                        for (int c = 0; c < KF; ++c) cp_async4(dst + LAMF + 1 + c, mrow + c);
                    } else {
#pragma unroll
                        for (int c = 0; c < KF; ++c) dst[LAMF + 1 + c] = 0;
                    }
                } else if (pair) {
                    // pair memo: the row from the progression
                    const int av = (int)xl - (int)o * (int)P.leaf.pair.h1;
#pragma unroll
                    for (int c = 0; c < DM; ++c) {
                        if (c >= lam) break;
                        dst[c] = pre[c];
                    }
                    dst[lam] = vrow;
                    dst[lam + 1] = av;
                    dst[lam + 2] = (int)fd_div((uint32_t)(pl - av * P.g[d - 2]), P.leaf.pair.fh);
                } else {
                    const int32_t *mrow =
                        mleaf ? P.memo + (size_t)(xl + o) * (size_t)P.K : nullptr;
#pragma unroll
                    for (int c = 0; c < DM; ++c) {
                        if (c >= d)
                            break;
                        if (c < lam)
                            dst[c] = pre[c];
                        else if (c == lam)
                            dst[c] = vrow;
                        else if (mleaf)
                            cp_async4(dst + c, mrow + (c - lam - 1));
                        else
                            dst[c] = (int)xl;
                    }
                }
            }
            q0 += cnt;
            after_round(cnt);
        }
        }
        const uint32_t emitted = q_end > q_begin ? q_end - q_begin : 0u;
        rows_left -= emitted;
        if (rows_left == 0) break;
        skip = 0;
        if (first_int < nvalid) {
            // the next child is a memo-level prefix beyond the memo: walk it
            const int ve = (int)(st.vcur - first_int);
            const int pe = rem - ve * glam;
            if (lane == 0) {
                wp->a[lam] = ve;
                wp->r[lam + 1] = pe;
            }
            __syncwarp();
            descend(P, wp, lam + 1, P.lam_w, lane);
            st.lam = P.lam_w;
            st.inwalk = 1;
            st.vcur = wp->r[P.lam_w] / P.g[P.lam_w];
            st.base = 0;
        } else {
            st.base = last_incl;
            st.vcur -= consumed;
            if (st.vcur < 0 && !advance(P, wp, lane, st)) {
                if (lane == 0) atomicExch(P.status, (int)DEV_INTERNAL);
                ok = false;
                break;
            }
        }
#pragma unroll
        for (int c = 0; c < DM; ++c) pre[c] = (c < st.lam) ? wp->a[c] : 0;
    }
    cp_async_wait<0>();
    if (pend)
        flush_rows(P, ring + (size_t)(half ^ 1u) * B * d,
                      row0 + (uint64_t)(nfull - 1) * B, B, d, lane, pol);
    if (hpos > 0)
        flush_rows(P, ring + (size_t)half * B * d, row0 + (uint64_t)nfull * B, hpos, d,
                      lane, pol);
    if (lane == 0) bulk_wait_read_all();
    __syncwarp();
    return ok;
}

// Rows are handed out as work items (equal-cost ranges when the runs table
// is present, else equal-row ranges) from an atomic counter.
template <int D, int LAMF>
__global__ void __launch_bounds__(ENUM_THREADS, 4)
    fz_enum_kernel(const __grid_constant__ EnumParams P) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31;
    const int wid = threadIdx.x >> 5;
    const uint32_t B = (uint32_t)P.half_rows;
    int32_t *ring = reinterpret_cast<int32_t *>(smem_raw) + (size_t)wid * 2 * B * D;
    WarpPath *wp =
        reinterpret_cast<WarpPath *>(smem_raw + (size_t)ENUM_WARPS * 2 * B * D * 4) + wid;
    const uint64_t pol = policy_evict_first();

    // cost range of the requested ranks (work-balanced slicing)
    uint64_t cost_lo = 0, cost_hi = 0;
    if (P.RT) {
        cost_lo = rank_to_cost(P, P.rank_begin, lane);
        cost_hi = rank_to_cost(P, P.rank_begin + P.nrows, lane);
    }
    for (;;) {
        unsigned long long s = 0;
        if (lane == 0) s = atomicAdd(P.slice_counter, 1ull);
        s = __shfl_sync(FULL, s, 0);
        uint64_t row0 = 0, row1 = 0;  // relative to out
        const int it = item_rows(P, s, cost_lo, cost_hi, lane, row0, row1);
        if (it == 0) break;
        if (it == 1) continue;
        if (!enum_slice<D, LAMF>(P, wp, ring, B, row0, row1, pol, lane)) break;
    }
    cp_async_wait<0>();
    if (lane == 0) bulk_wait_all();
    __syncwarp();
}

// ---------------------------------------------------------------------------
// Full memo of depth K <= 3 in run order.  The walk covers the leading LAMF
// coordinates only: for a prefix (a_0..a_{LAMF-1}) with remainder r, the
// rows of its whole subtree -- every a_LAMF from r div g down to 0, each with
// Memo[r - a_LAMF g] -- are the contiguous run-memo range
// [cls_beg[r mod g], + C[LAMF][r]) with a_LAMF = r div g - (first word).  A
// round is then one 16-byte load and one row store per lane.
// ---------------------------------------------------------------------------
template <int D, int LAMF, int K>
__device__ __forceinline__ void run_store_row(int32_t *dst, const int (&a)[LAMF > 0 ? LAMF : 1],
                                              int vmax, int4 m) {
    int32_t w[D];
#pragma unroll
    for (int c = 0; c < LAMF; ++c) w[c] = a[c];
    w[LAMF] = vmax - m.x;
    if constexpr (K >= 1) w[LAMF + 1] = m.y;
    if constexpr (K >= 2) w[LAMF + 2] = m.z;
    if constexpr (K >= 3) w[LAMF + 3] = m.w;
    if constexpr (D % 2 == 0) {  // row starts are 8-byte aligned: 8-byte stores
#pragma unroll
        for (int c = 0; c < D; c += 2)
            *reinterpret_cast<int2 *>(dst + c) = make_int2(w[c], w[c + 1]);
    } else {
#pragma unroll
        for (int c = 0; c < D; ++c) dst[c] = w[c];
    }
}

template <int D, int LAMF, int K>
__device__ __forceinline__ bool runs_slice(const EnumParams &P, int32_t *ring, uint32_t B,
                                           uint64_t row0, uint64_t row1, uint64_t pol,
                                           int lane) {
    // unrank the first row: the prefix, its remainder and the offset in its run
    int a[LAMF > 0 ? LAMF : 1];
    int r[LAMF + 1];
    uint64_t R = P.rank_begin + row0;
    r[0] = P.n;
    a[0] = 0;
#pragma unroll
    for (int j = 0; j < LAMF; ++j) {
        int v;
        uint64_t before;
        find_child(P, j, r[j], R, lane, v, before);
        a[j] = v;
        R -= before;
        r[j + 1] = r[j] - v * P.g[j];
    }
    uint64_t off = R;
    uint64_t left = row1 - row0;
    uint32_t hpos = 0, half = 0, nfull = 0;
    const int glam = P.g[LAMF];
    bool ok = true;
    for (;;) {
        const int rem = r[LAMF];
        const uint64_t run_rows = __ldg(P.C + (long long)LAMF * P.cs + rem);
        if (off < run_rows) {
            const int vmax = rem / glam;
            const int cls = rem - vmax * glam;
            const uint64_t src64 = __ldg(P.cls_beg + cls) + off;
            uint64_t take64 = run_rows - off;
            if (take64 > left) take64 = left;
            if (src64 + take64 > P.memo_rows) {  // bounds guard: the run lies in the memo
                if (lane == 0) atomicExch(P.status, (int)DEV_INTERNAL);
                ok = false;
                break;
            }
            left -= take64;
            // the run lies in the memo (< 2^30 rows): 32-bit row indices
            uint32_t src = (uint32_t)src64, take = (uint32_t)take64;
            // Rounds of up to 64 rows (never across a ring half); lane l
            // stores rows l and l + 32 of a round.  The memo rows of the next
            // round are loaded before this round's rows are stored.  The loop
            // is unrolled twice so the two register sets swap roles without
            // moves.
            uint32_t c0 = take < 64u ? take : 64u;
            if (c0 > B - hpos) c0 = B - hpos;
            int4 x0 = make_int4(0, 0, 0, 0), x1 = x0, y0 = x0, y1 = x0;
            {
                const int4 *ms = P.run_memo + src;
                if ((uint32_t)lane < c0) x0 = __ldg(ms + lane);
                if ((uint32_t)lane + 32u < c0) x1 = __ldg(ms + 32 + lane);
            }
            auto round = [&](const int4 &cur0, const int4 &cur1, int4 &nxt0, int4 &nxt1) {
                const uint32_t hp1 = hpos + c0 == B ? 0u : hpos + c0;
                const uint32_t t1 = take - c0;
                uint32_t c1 = t1 < 64u ? t1 : 64u;
                if (c1 > B - hp1) c1 = B - hp1;
                const int4 *ns = P.run_memo + (src + c0);
                if ((uint32_t)lane < c1) nxt0 = __ldg(ns + lane);
                if ((uint32_t)lane + 32u < c1) nxt1 = __ldg(ns + 32 + lane);
                if (hpos == 0 && nfull >= 2) {
                    // re-entering a half: the bulk store issued from it two
                    // flushes ago must have finished reading it
                    if (lane == 0) bulk_wait_read<1>();
                    __syncwarp();
                }
                int32_t *dst = ring + (size_t)(half * B + hpos + lane) * D;
                if ((uint32_t)lane < c0) run_store_row<D, LAMF, K>(dst, a, vmax, cur0);
                if ((uint32_t)lane + 32u < c0)
                    run_store_row<D, LAMF, K>(dst + 32 * D, a, vmax, cur1);
                if (hp1 == 0) {
                    flush_rows(P, ring + (size_t)half * B * D, row0 + (uint64_t)nfull * B, B, D,
                               lane, pol);
                    ++nfull;
                    half ^= 1u;
                }
                hpos = hp1;
                src += c0;
                take = t1;
                c0 = c1;
            };
            for (;;) {
                round(x0, x1, y0, y1);
                if (take == 0) break;
                round(y0, y1, x0, x1);
                if (take == 0) break;
            }
            if (left == 0) break;
        }
        off = 0;
        // the next prefix in descending order: decrement the deepest positive
        // coordinate, reset the ones after it to their maxima
        int jj = -1;
#pragma unroll
        for (int j = 0; j < LAMF; ++j)
            if (a[j] > 0) jj = j;
        if (jj < 0) {  // past the last prefix with rows still owed
            if (lane == 0) atomicExch(P.status, (int)DEV_INTERNAL);
            ok = false;
            break;
        }
#pragma unroll
        for (int j = 0; j < LAMF; ++j) {
            if (j == jj) {
                a[j] -= 1;
                r[j + 1] = r[j] - a[j] * P.g[j];
            } else if (j > jj) {
                a[j] = r[j] / P.g[j];
                r[j + 1] = r[j] - a[j] * P.g[j];
            }
        }
    }
    if (hpos > 0)
        flush_rows(P, ring + (size_t)half * B * D, row0 + (uint64_t)nfull * B, hpos, D, lane,
                   pol);
    if (lane == 0) bulk_wait_read_all();
    __syncwarp();
    return ok;
}

// Work items from an atomic counter: equal-cost ranges when the plan has a
// candidates table counted at level LAMF (each walked prefix costs W rows, so
// the items at the start of the order, where prefixes hold few rows each, are
// short), else equal-row ranges.
template <int D, int LAMF, int K>
__global__ void __launch_bounds__(ENUM_THREADS, 4)
    fz_enum_runs_kernel(const __grid_constant__ EnumParams P) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31;
    const int wid = threadIdx.x >> 5;
    const uint32_t B = (uint32_t)P.half_rows;
    int32_t *ring = reinterpret_cast<int32_t *>(smem_raw) + (size_t)wid * 2 * B * D;
    const uint64_t pol = policy_evict_first();
    uint64_t cost_lo = 0, cost_hi = 0;
    if (P.RT) {
        cost_lo = rank_to_cost(P, P.rank_begin, lane);
        cost_hi = rank_to_cost(P, P.rank_begin + P.nrows, lane);
    }
    for (;;) {
        unsigned long long s = 0;
        if (lane == 0) s = atomicAdd(P.slice_counter, 1ull);
        s = __shfl_sync(FULL, s, 0);
        uint64_t row0 = 0, row1 = 0;
        const int it = item_rows(P, s, cost_lo, cost_hi, lane, row0, row1);
        if (it == 0) break;
        if (it == 1) continue;
        if (!runs_slice<D, LAMF, K>(P, ring, B, row0, row1, pol, lane)) break;
    }
    if (lane == 0) bulk_wait_all();
    __syncwarp();
}

// The run-order copy with the tuple width D <= 8 and the memo depth
// 1 <= K <= 3 read at run time (batches): the rounds of runs_slice, with the
// prefix a_0..a_{LAMF-1} (LAMF = D - K - 1 <= 6) kept in registers through
// loops unrolled to their maxima and guarded by the run-time bounds.
constexpr int RT_LAMF_MAX = 6;

__device__ __forceinline__ void run_store_row_rt(int32_t *dst, const int (&a)[RT_LAMF_MAX], int D,
                                                 int LAMF, int vmax, int4 m) {
    int w[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const int t = c - LAMF;
        int v = c < RT_LAMF_MAX ? a[c] : 0;
        if (t == 0)
            v = vmax - m.x;
        else if (t == 1)
            v = m.y;
        else if (t == 2)
            v = m.z;
        else if (t == 3)
            v = m.w;
        w[c] = v;
    }
    if ((D & 3) == 0) {  // row starts 16-byte aligned
#pragma unroll
        for (int c = 0; c < 8; c += 4)
            if (c < D)
                *reinterpret_cast<int4 *>(dst + c) = make_int4(w[c], w[c + 1], w[c + 2], w[c + 3]);
    } else if ((D & 1) == 0) {  // 8-byte aligned
#pragma unroll
        for (int c = 0; c < 8; c += 2)
            if (c < D) *reinterpret_cast<int2 *>(dst + c) = make_int2(w[c], w[c + 1]);
    } else {
#pragma unroll
        for (int c = 0; c < 8; ++c)
            if (c < D) dst[c] = w[c];
    }
}

__device__ __noinline__ bool runs_slice_rt(const EnumParams &P, int32_t *ring, uint32_t B,
                                           uint64_t row0, uint64_t row1, uint64_t pol,
                                           int lane) {
    const int D = P.d;
    const int LAMF = P.d - P.K - 1;
    if (LAMF < 1 || D > 8 || P.K < 1 || P.K > 3) {  // shapes the host never sends here
        if (lane == 0) atomicExch(P.status, (int)DEV_INTERNAL);
        return false;
    }
    // unrank the first row: the prefix, its remainder and the offset in its run
    int a[RT_LAMF_MAX];
#pragma unroll
    for (int c = 0; c < RT_LAMF_MAX; ++c) a[c] = 0;
    uint64_t R = P.rank_begin + row0;
    int rem = P.n;
#pragma unroll 1
    for (int j = 0; j < LAMF; ++j) {
        int v;
        uint64_t before;
        find_child(P, j, rem, R, lane, v, before);
        R -= before;
        rem -= v * P.g[j];
#pragma unroll
        for (int c = 0; c < RT_LAMF_MAX; ++c)
            if (c == j) a[c] = v;
    }
    uint64_t off = R;
    uint64_t left = row1 - row0;
    uint32_t hpos = 0, half = 0, nfull = 0;
    const int glam = P.g[LAMF];
    bool ok = true;
    for (;;) {
        const uint64_t run_rows = __ldg(P.C + (long long)LAMF * P.cs + rem);
        if (off < run_rows) {
            const int vmax = rem / glam;
            const int cls = rem - vmax * glam;
            const uint64_t src64 = __ldg(P.cls_beg + cls) + off;
            uint64_t take64 = run_rows - off;
            if (take64 > left) take64 = left;
            if (src64 + take64 > P.memo_rows) {  // bounds guard: the run lies in the memo
                if (lane == 0) atomicExch(P.status, (int)DEV_INTERNAL);
                ok = false;
                break;
            }
            left -= take64;
            uint32_t src = (uint32_t)src64, take = (uint32_t)take64;
            uint32_t c0 = take < 64u ? take : 64u;
            if (c0 > B - hpos) c0 = B - hpos;
            int4 x0 = make_int4(0, 0, 0, 0), x1 = x0, y0 = x0, y1 = x0;
            {
                const int4 *ms = P.run_memo + src;
                if ((uint32_t)lane < c0) x0 = __ldg(ms + lane);
                if ((uint32_t)lane + 32u < c0) x1 = __ldg(ms + 32 + lane);
            }
            auto round = [&](const int4 &cur0, const int4 &cur1, int4 &nxt0, int4 &nxt1) {
                const uint32_t hp1 = hpos + c0 == B ? 0u : hpos + c0;
                const uint32_t t1 = take - c0;
                uint32_t c1 = t1 < 64u ? t1 : 64u;
                if (c1 > B - hp1) c1 = B - hp1;
                const int4 *ns = P.run_memo + (src + c0);
                if ((uint32_t)lane < c1) nxt0 = __ldg(ns + lane);
                if ((uint32_t)lane + 32u < c1) nxt1 = __ldg(ns + 32 + lane);
                if (hpos == 0 && nfull >= 2) {
                    if (lane == 0) bulk_wait_read<1>();
                    __syncwarp();
                }
                int32_t *dst = ring + (size_t)(half * B + hpos + lane) * D;
                if ((uint32_t)lane < c0) run_store_row_rt(dst, a, D, LAMF, vmax, cur0);
                if ((uint32_t)lane + 32u < c0) run_store_row_rt(dst + 32 * D, a, D, LAMF, vmax, cur1);
                if (hp1 == 0) {
                    flush_rows(P, ring + (size_t)half * B * D, row0 + (uint64_t)nfull * B, B, D,
                               lane, pol);
                    ++nfull;
                    half ^= 1u;
                }
                hpos = hp1;
                src += c0;
                take = t1;
                c0 = c1;
            };
            for (;;) {
                round(x0, x1, y0, y1);
                if (take == 0) break;
                round(y0, y1, x0, x1);
                if (take == 0) break;
            }
            if (left == 0) break;
        }
        off = 0;
        // the next prefix in descending order: decrement the deepest positive
        // coordinate, reset the ones after it to their maxima (the remainder
        // is carried forward from r_0 = n)
        int jj = -1;
#pragma unroll
        for (int j = 0; j < RT_LAMF_MAX; ++j)
            if (j < LAMF && a[j] > 0) jj = j;
        if (jj < 0) {
            if (lane == 0) atomicExch(P.status, (int)DEV_INTERNAL);
            ok = false;
            break;
        }
        int rr = P.n;
#pragma unroll
        for (int j = 0; j < RT_LAMF_MAX; ++j) {
            if (j < LAMF) {
                if (j == jj)
                    a[j] -= 1;
                else if (j > jj)
                    a[j] = rr / P.g[j];
                rr -= a[j] * P.g[j];
            }
        }
        rem = rr;
    }
    if (hpos > 0)
        flush_rows(P, ring + (size_t)half * B * D, row0 + (uint64_t)nfull * B, hpos, D, lane,
                   pol);
    if (lane == 0) bulk_wait_read_all();
    __syncwarp();
    return ok;
}

// ---------------------------------------------------------------------------
// Batches: the instances the flat walk has no kernel for (partial memos,
// memos in element order, widths above 8, single blocks), any mix of widths in
// one persistent launch with the tuple width read at run time.
// ---------------------------------------------------------------------------
constexpr size_t BATCH_RING_BYTES = RING_BYTES_PER_WARP;

__global__ void __launch_bounds__(ENUM_THREADS, 4)
    fz_enum_batch_kernel(const __grid_constant__ BatchEnumParams BP) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31;
    const int wid = threadIdx.x >> 5;
    int32_t *ring = reinterpret_cast<int32_t *>(smem_raw + (size_t)wid * BATCH_RING_BYTES);
    EnumParams *ep =
        reinterpret_cast<EnumParams *>(smem_raw + (size_t)ENUM_WARPS * BATCH_RING_BYTES) + wid;
    WarpPath *wp = reinterpret_cast<WarpPath *>(smem_raw + (size_t)ENUM_WARPS * BATCH_RING_BYTES +
                                                ENUM_WARPS * sizeof(EnumParams)) +
                   wid;
    const uint64_t pol = policy_evict_first();
    int cur = -1;
    for (;;) {
        unsigned long long item = 0;
        if (lane == 0) item = BP.item_lo + atomicAdd(BP.item_counter, 1ull);
        item = __shfl_sync(FULL, item, 0);
        if (item >= BP.item_hi) break;
        const uint64_t s = batch_locate<true>(BP, ep, cur, item, lane);
        const EnumParams &P = *ep;
        uint64_t row0, row1;
        if (P.RT) {
            const uint64_t cost_hi = cost_at(P, 0, P.n);
            const uint64_t c0 = s * P.slice_cost;
            if (c0 >= cost_hi) continue;
            const uint64_t c1 = c0 + P.slice_cost;
            row0 = 0;
            if (s > 0) {
                row0 = cost_to_rank(P, c0, lane) & ~31ull;
                if (row0 > P.nrows) row0 = P.nrows;
            }
            row1 = P.nrows;
            if (c1 < cost_hi) {
                row1 = cost_to_rank(P, c1, lane) & ~31ull;
                if (row1 > P.nrows) row1 = P.nrows;
            }
        } else {
            row0 = s * P.slice_rows;
            row1 = row0 + P.slice_rows < P.nrows ? row0 + P.slice_rows : P.nrows;
        }
        if (row1 <= row0) continue;
        if (P.d == 1 || (P.K == P.d && P.top > P.n)) {
            // a single block: d == 1 or the output is Memo[n] itself
            if (P.d == 1) {
                if (lane == 0 && row0 == 0) P.out[0] = P.n / P.g[0];
            } else {
                const uint64_t src0 = (__ldg(P.O + P.n) + row0) * (uint64_t)P.d;
                for (uint64_t w = lane; w < (row1 - row0) * (uint64_t)P.d; w += 32)
                    P.out[row0 * (uint64_t)P.d + w] = __ldg(P.memo + src0 + w);
            }
            continue;
        }
        // full memos in run order take the run copy, the rest one walk for
        // every width up to 8 (row loops unrolled to 8), the 16-wide one beyond
        bool ok;
        if (P.run_memo)
            ok = runs_slice_rt(P, ring, (uint32_t)P.half_rows, row0, row1, pol, lane);
        else if (P.d <= 8)
            ok = enum_slice<0, -1, 8>(P, wp, ring, (uint32_t)P.half_rows, row0, row1, pol, lane);
        else
            ok = enum_slice<0, -1>(P, wp, ring, (uint32_t)P.half_rows, row0, row1, pol, lane);
        if (!ok) break;
    }
    cp_async_wait<0>();
    if (lane == 0) bulk_wait_all();
    __syncwarp();
}

// Tuples of given ranks, a thread per rank.  Each leading coordinate is a
// search in one count row: the rows of the children a_j >= v number
// C[j][rem - v g_j], which grows about as the (d - 1 - j)-th power of its
// index, so the search starts at that power's estimate and gallops from it
// (two to four dependent loads a coordinate where a binary search over 300 to
// 600 children takes 9).  With the memo in run order the coordinates from
// d - K - 1 on are one table row; otherwise the searches go down to a_{d-2}.
// Rows are staged in shared memory and written coalesced.
//
// Bound by the latency of the dependent loads, all of them random: a million
// ranks of a width-6 set of 1e8 rows with a depth-3 table took 418 us with a
// warp per rank and 32-probe searches, 33 us with a thread per rank.
constexpr int UNRANK_THREADS = 256;

template <int D>
__global__ void __launch_bounds__(UNRANK_THREADS)
    fz_unrank_kernel(const __grid_constant__ EnumParams P, const uint64_t *ranks, uint64_t m) {
    __shared__ int32_t stage[UNRANK_THREADS * D];
    const int lane = threadIdx.x & 31;
    int32_t *mine = stage + (size_t)(threadIdx.x & ~31) * D;
    const int levels = P.run_memo ? D - P.K - 1 : D - 1;
    const uint64_t total = __ldg(P.C + P.n);
    const uint64_t stride = (uint64_t)gridDim.x * UNRANK_THREADS;
    for (uint64_t base = (uint64_t)blockIdx.x * UNRANK_THREADS + (threadIdx.x & ~31); base < m;
         base += stride) {
        const uint64_t i = base + lane;
        if (i < m) {
            uint64_t R = __ldg(ranks + i);
            bool good = R < total;
            int a[D];
#pragma unroll
            for (int c = 0; c < D; ++c) a[c] = 0;
            uint32_t rem = (uint32_t)P.n;
            uint64_t all = total;  // rows under the current prefix
#pragma unroll
            for (int j = 0; j < D - 1; ++j) {
                if (j >= levels || !good) break;
                const uint32_t g = (uint32_t)P.g[j];
                const uint64_t *row = P.C + (int64_t)j * P.cs;
                const uint32_t vmax = rem / g;
                uint64_t ahi;
                const uint32_t hi = thread_child(row, rem, g, vmax, R, all, D - 1 - j, &ahi);
                a[j] = (int)hi;
                R -= ahi;
                rem -= hi * g;
                all = j + 1 < levels ? __ldg(row + P.cs + rem) : 0ull;
                good = j + 1 >= levels || R < all;
            }
            if (P.run_memo) {
                const uint32_t gl = P.leaf.fg.g, q = fd_div(rem, P.leaf.fg);
                const uint64_t at = good ? __ldg(P.cls_beg + (rem - q * gl)) + R : 0ull;
                good = good && at < P.memo_rows;  // bounds guard
                if (good) {
                    const int32_t *t = reinterpret_cast<const int32_t *>(P.run_memo) +
                                       (size_t)at * run_stride(P.K + 1);
#pragma unroll
                    for (int c = 0; c < D; ++c)
                        if (c == levels)
                            a[c] = (int)q - __ldg(t);
                        else if (c > levels)
                            a[c] = __ldg(t + (c - levels));
                }
            } else {
                a[D - 1] = (int)fd_div(rem, P.leaf.pair.fh);
                good = good && (uint32_t)a[D - 1] * P.leaf.pair.fh.g == rem;
            }
            if (!good) atomicExch(P.status, (int)DEV_INTERNAL);
#pragma unroll
            for (int c = 0; c < D; ++c) mine[lane * D + c] = good ? a[c] : -1;
        }
        __syncwarp();
        const uint64_t left = (m - base) * D;
        const uint32_t words = left < 32u * D ? (uint32_t)left : 32u * D;
        for (uint32_t w = lane; w < words; w += 32) P.out[base * D + w] = mine[w];
        __syncwarp();
    }
}

// The same for few ranks, a warp per rank: the 32-probe searches take two rounds
// of independent loads a coordinate where a thread's gallop takes three to
// five dependent ones, and a rank does not wait for the longest gallop of
// 32.  A memo in element order ends the searches where it applies, too.
constexpr int UNRANK_WARP_THREADS = 64;

template <int D>
__global__ void __launch_bounds__(UNRANK_WARP_THREADS)
    fz_unrank_warp_kernel(const __grid_constant__ EnumParams P, const uint64_t *ranks, uint64_t m) {
    constexpr int WARPS = UNRANK_WARP_THREADS / 32;
    const int lane = threadIdx.x & 31;
    const int levels = P.run_memo ? D - P.K - 1 : D - 1;
    const uint64_t total = __ldg(P.C + P.n);
    for (uint64_t i = (uint64_t)blockIdx.x * WARPS + (threadIdx.x >> 5); i < m;
         i += (uint64_t)gridDim.x * WARPS) {
        uint64_t R = __ldg(ranks + i);
        bool good = R < total, leaf = false;
        int rem = P.n, word = 0;  // word: a_lane
        for (int j = 0; j < levels; ++j) {
            int v;
            uint64_t before;
            find_child(P, j, rem, R, lane, v, before);
            if (lane == j) word = v;
            R -= before;
            rem -= v * P.g[j];
            leaf = j == P.lam_m && rem < P.top && !P.run_memo;
            if (leaf) break;
            if (j + 1 < levels) good = good && R < __ldg(P.C + (int64_t)(j + 1) * P.cs + rem);
        }
        if (leaf) {
            const uint64_t at = __ldg(P.O + rem) + R;
            good = good && at < P.memo_rows;  // bounds guard
            if (good && lane > P.lam_m && lane < D)
                word = __ldg(P.memo + (size_t)at * P.K + (lane - P.lam_m - 1));
        } else if (P.run_memo) {
            const uint32_t q = fd_div((uint32_t)rem, P.leaf.fg);
            const uint64_t at = __ldg(P.cls_beg + ((uint32_t)rem - q * P.leaf.fg.g)) + R;
            good = good && at < P.memo_rows;  // bounds guard
            if (good && lane >= levels && lane < D) {
                const int x = __ldg(reinterpret_cast<const int32_t *>(P.run_memo) +
                                    (size_t)at * run_stride(P.K + 1) + (lane - levels));
                word = lane == levels ? (int)q - x : x;
            }
        } else {
            const uint32_t q = fd_div((uint32_t)rem, P.leaf.pair.fh);
            good = good && q * P.leaf.pair.fh.g == (uint32_t)rem;
            if (lane == D - 1) word = (int)q;
        }
        if (lane < D) P.out[i * D + lane] = good ? word : -1;
        if (!good && lane == 0) atomicExch(P.status, (int)DEV_INTERNAL);
    }
}

// Whole output taken from one place: d == 1 (one candidate) or k == d (the
// output is Memo[n] itself).  mode 1: copy memo rows; mode 2: single row.
__global__ void fz_direct_kernel(const EnumParams P, int mode) {
    const uint64_t tid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint64_t nt = (uint64_t)gridDim.x * blockDim.x;
    if (mode == 1) {
        const uint64_t src0 = (__ldg(P.O + P.n) + P.rank_begin) * (uint64_t)P.d;
        const uint64_t words = P.nrows * (uint64_t)P.d;
        if (src0 + words > P.memo_rows * (uint64_t)P.d) {  // bounds guard
            if (tid == 0) atomicExch(P.status, (int)DEV_INTERNAL);
            return;
        }
        for (uint64_t w = tid; w < words; w += nt) P.out[w] = __ldg(P.memo + src0 + w);
    } else if (tid == 0 && P.nrows > 0) {
        P.out[0] = P.n / P.g[0];
    }
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
static int half_rows_for(int d, int ring_bytes = RING_BYTES_PER_WARP) {
    int b = ring_bytes / (8 * d);
    b = (b / 32) * 32;
    return b < 32 ? 32 : b;
}

// Ring bytes per warp for an occupancy cap: fewer resident warps get larger
// rings, so the bytes in flight per SM stay about the same.  A cap leaves 52 KB
// of an SM's 228 and a quarter of its registers: one block of any kernel of a
// rebuild (run_build_kernel has 45 KB; with rings of 192 KB together it waited
// for the end of the enumeration).
// FZ_ENUM_RING_KB overrides (tuning only).
static int ring_bytes_for(int ctas_per_sm) {
    static const int forced = [] {
        const char *e = getenv("FZ_ENUM_RING_KB");
        const int kb = e ? atoi(e) : 0;
        return (kb >= 4 && kb <= 24) ? kb * 1024 : 0;
    }();
    if (forced) return forced;
    if (!leaves_room(ctas_per_sm)) return RING_BYTES_PER_WARP;
    const int b = (176 * 1024) / (ctas_per_sm * ENUM_WARPS);
    return b > 16 * 1024 ? 16 * 1024 : (b / 1024) * 1024;
}

template <typename Kern>
static int launch_enum_kernel(Kern kern, const EnumParams &P, int D, cudaStream_t s, int sms,
                              DeviceOnce &attr_set) {
    return launch_enum_grid(kern, P,
                            (size_t)ENUM_WARPS * 2 * P.half_rows * D * 4 +
                                (size_t)ENUM_WARPS * sizeof(WarpPath),
                            s, sms, attr_set);
}

template <int D, int LAMF>
static int launch_enum_dl(const EnumParams &P, cudaStream_t s, int sms) {
    static DeviceOnce attr_set;
    return launch_enum_kernel(fz_enum_kernel<D, LAMF>, P, D, s, sms, attr_set);
}

template <int D, int LAMF, int K>
static int launch_enum_runs(const EnumParams &P, cudaStream_t s, int sms) {
    static DeviceOnce attr_set;
    return launch_enum_kernel(fz_enum_runs_kernel<D, LAMF, K>, P, D, s, sms, attr_set);
}

// Shapes the flat walk has no kernel for.  Full memo of depth 2, 3 or 4: every
// run is a memo run at a fixed coordinate; use the compile-time
// specialisation.  Otherwise generic.
template <int D>
static int launch_enum_d(const EnumParams &P, cudaStream_t s, int sms) {
    const bool full = P.lam_m >= 0 && P.top > P.n;
    const int K = P.K;
    if (full && P.run_memo && P.cls_beg) {
        if constexpr (D >= 2 && !flat_serves(D, D - 2, SRC_RUN))
            if (K == 1) return launch_enum_runs<D, D - 2, 1>(P, s, sms);
        if constexpr (D >= 3 && !flat_serves(D, D - 3, SRC_RUN))
            if (K == 2) return launch_enum_runs<D, D - 3, 2>(P, s, sms);
        if constexpr (D >= 4 && !flat_serves(D, D - 4, SRC_RUN))
            if (K == 3) return launch_enum_runs<D, D - 4, 3>(P, s, sms);
    }
    if (full && K == 2 && D >= 3) return launch_enum_dl<D, (D >= 3 ? D - 3 : 0)>(P, s, sms);
    if (full && K == 3 && D >= 4) return launch_enum_dl<D, (D >= 4 ? D - 4 : 0)>(P, s, sms);
    if (full && K == 4 && D >= 5) return launch_enum_dl<D, (D >= 5 ? D - 5 : 0)>(P, s, sms);
    return launch_enum_dl<D, -1>(P, s, sms);
}

// Up to how many ranks a warp takes each (us a launch by warps / by threads of
// a width-6 set at 1000, 6000, 8000, 12000 ranks: with a depth-3 table 3.8 /
// 5.8, 5.2 / 6.1, 5.8 / 6.1, 7.7 / 6.1; searched to the end 6.5 / 14.7, 8.2 /
// 14.7, 10.1 / 14.8, 14.1 / 14.8; width 4 with a depth-2 table 3.3 / 4.4, 4.4 /
// 4.4, 4.9 / 4.3).
constexpr uint64_t UNRANK_WARP_RUN = 6144, UNRANK_WARP_MAX = 8192;

template <int D>
static int launch_unrank_d(const EnumParams &P, const uint64_t *ranks, uint64_t m,
                           cudaStream_t s) {
    if (m <= (P.run_memo ? UNRANK_WARP_RUN : UNRANK_WARP_MAX)) {
        constexpr int WARPS = UNRANK_WARP_THREADS / 32;
        fz_unrank_warp_kernel<D>
            <<<(unsigned)((m + WARPS - 1) / WARPS), UNRANK_WARP_THREADS, 0, s>>>(P, ranks, m);
        note_launch();
        FZ_CUDA_TRY(cudaGetLastError());
        return FZ_OK;
    }
    uint64_t blocks = (m + UNRANK_THREADS - 1) / UNRANK_THREADS;
    if (blocks > 65536) blocks = 65536;
    fz_unrank_kernel<D><<<(unsigned)blocks, UNRANK_THREADS, 0, s>>>(P, ranks, m);
    note_launch();
    FZ_CUDA_TRY(cudaGetLastError());
    return FZ_OK;
}

// FZ_WALK_PROGRESSION=0 evaluates walk leaves candidate by candidate as the
// ordinary step does (tuning and testing only).
bool walk_progression_enabled() {
    static const bool on = [] {
        const char *e = getenv("FZ_WALK_PROGRESSION");
        return !(e && e[0] == '0');
    }();
    return on;
}

// Rows per leaf from which a batch of memo leaves is copied leaf by leaf:
// 16 for plans, 64 for batches (a 4096-instance batch of widths 3..8:
// 11.8 ms at 16, 11.3 at 64 and 256, 11.6 never leaf by leaf, 12.3 at 4).
// FZ_ENUM_DENSE_MIN overrides both (tuning only).
static int dense_min_for(bool batch) {
    static const int forced = [] {
        const char *e = getenv("FZ_ENUM_DENSE_MIN");
        const int v = e ? atoi(e) : -1;
        return v >= 0 ? v : -1;
    }();
    if (forced >= 0) return forced;
    return batch ? 64 : 16;
}

static EnumParams make_params(const EnumLaunch &L) {
    EnumParams P{};
    P.C = L.C;
    P.cs = L.cs;
    P.O = L.O;
    P.memo = L.memo;
    P.memo_rows = L.memo_rows;
    P.ctas_per_sm = L.ctas_per_sm;
    P.dense_min = dense_min_for(false);
    P.RT = L.RT;
    P.W = L.W;
    P.lam_r = L.lam_r;
    P.status = L.status;
    P.slice_counter = L.slice_counter;
    P.n = L.n;
    P.d = L.d;
    P.K = L.K;
    P.top = L.top;
    for (int i = 0; i < L.d; ++i) P.g[i] = L.g[i];
    P.pair_memo = L.pair_memo && L.K == 2 && L.d >= 3 && L.top > L.n;
    P.leaf = LeafSource{};
    if (L.d >= 2) {
        P.leaf.pair = make_pair_form(L.g[L.d - 2], L.g[L.d - 1]);
        P.progression = walk_progression_enabled() || P.pair_memo;
    } else {
        P.leaf.pair.fh = make_fastdiv((uint32_t)L.g[0]);
    }
    const bool memo = L.K >= 1 && L.K <= L.d - 1 && L.top > 0;
    P.lam_m = memo ? L.d - L.K - 1 : -1;
    P.lam_w = L.d - 2;
    if (!memo) {
        P.K = 0;
        P.top = 0;
    }
    // the run-order memo serves full memos
    const bool runs = memo && L.top > L.n && L.run_memo && L.cls_beg;
    P.run_memo = runs ? L.run_memo : nullptr;
    P.cls_beg = runs ? L.cls_beg : nullptr;
    for (int j = 0; j < FLAT_MAX_NP && j < L.d; ++j) P.fdg[j] = make_fastdiv((uint32_t)L.g[j]);
    if (runs) {
        P.leaf.rows = reinterpret_cast<const int32_t *>(L.run_memo);
        P.leaf.cls = L.cls_beg;
        P.leaf.nrows = L.memo_rows;
        P.leaf.fg = make_fastdiv((uint32_t)L.g[L.d - L.K - 1]);
        P.flat_np = L.d - L.K - 1;
        P.flat_src = SRC_RUN;
    } else if (P.pair_memo || (!memo && P.progression)) {
        // no memo table: leaves are the prefixes above the last two generators
        P.flat_np = L.d - 2;
        P.flat_src = SRC_PAIR;
    }
    if (!flat_serves(L.d, P.flat_np, P.flat_src)) P.flat_np = 0;
    P.by_cost = L.by_cost && (!P.flat_np || P.lam_r == P.flat_np);
    // the run walk's candidates are the prefixes of its LAMF = d - K - 1
    // leading coordinates; a table counted at another level cannot balance it
    if (runs && P.lam_r != L.d - L.K - 1) P.RT = nullptr;
    return P;
}

#define FZ_DISPATCH_D(d, FN, ...)                 \
    switch (d) {                                  \
        case 2: return FN<2>(__VA_ARGS__);        \
        case 3: return FN<3>(__VA_ARGS__);        \
        case 4: return FN<4>(__VA_ARGS__);        \
        case 5: return FN<5>(__VA_ARGS__);        \
        case 6: return FN<6>(__VA_ARGS__);        \
        case 7: return FN<7>(__VA_ARGS__);        \
        case 8: return FN<8>(__VA_ARGS__);        \
        case 9: return FN<9>(__VA_ARGS__);        \
        case 10: return FN<10>(__VA_ARGS__);      \
        case 11: return FN<11>(__VA_ARGS__);      \
        case 12: return FN<12>(__VA_ARGS__);      \
        case 13: return FN<13>(__VA_ARGS__);      \
        case 14: return FN<14>(__VA_ARGS__);      \
        case 15: return FN<15>(__VA_ARGS__);      \
        case 16: return FN<16>(__VA_ARGS__);      \
        default: return set_error(FZ_EINVAL, "d out of range"); \
    }

// More than `least` prefixes a row: by rank.  The flat walk visits every prefix
// (12 us a million), the rank walk searches every row (41 us a million; 1e7
// rows of width 6 under 8.6e7 prefixes: 1054 against 409 us): 3 for one set.
// In a batch the searches of many sets miss L2 (4096 sets of 1e2..1e6 rows:
// 4557 us without, 4672 with 3, 4557 with 10; 96 sets of 1e2..1e4 rows 218,
// 210, 209): 10.
static bool by_rank(const EnumLaunch &L, const EnumParams &P, uint64_t least) {
    return P.flat_np > 0 && P.flat_src == SRC_PAIR && rank_walk_serves(L.d) && L.RT &&
           prefixes_exceed(L.total_cost, L.total_rows, L.W, least);
}

// Enumerate ranks [rank_begin, rank_begin + nrows) into out.  Asynchronous.
int launch_enumerate(const EnumLaunch &L, uint64_t rank_begin, uint64_t nrows, int32_t *out,
                     uint64_t slice_rows, cudaStream_t s) {
    if (nrows == 0) return FZ_OK;
    if (!out || !L.C || !L.status || !L.slice_counter ||
        (L.K >= 1 && L.top > 0 && !L.run_memo &&
         (!L.O || (L.memo_rows > 0 && !L.memo))))
        return set_error(FZ_EINTERNAL, "enumerate: missing device buffer");
    EnumParams P = make_params(L);
    P.out = out;
    P.rank_begin = rank_begin;
    P.nrows = nrows;
    P.aligned = ((uintptr_t)out & 15u) == 0 && !L.plain_stores;
    P.whole = rank_begin == 0 && L.total_rows == nrows;
    if (L.d == 1 || (L.K == L.d && L.top > L.n)) {
        const int mode = (L.d == 1 && !(L.K == 1 && L.top > L.n)) ? 2 : 1;
        uint64_t words = nrows * (uint64_t)L.d;
        uint64_t blocks = (words + 255) / 256;
        if (blocks > 4096) blocks = 4096;
        if (blocks < 1) blocks = 1;
        fz_direct_kernel<<<(unsigned)blocks, 256, 0, s>>>(P, mode);
        note_launch();
        FZ_CUDA_TRY(cudaGetLastError());
        return FZ_OK;
    }
    DeviceProps dp;
    int rc = device_props(&dp);
    if (rc != FZ_OK) return rc;
    if (slice_rows < 4) slice_rows = 4;
    slice_rows = (slice_rows + 3) & ~3ull;
    P.slice_rows = slice_rows;
    P.nslices = (nrows + slice_rows - 1) / slice_rows;
    if (P.RT) {
        // equal-cost work items; about as many as equal-row items would be
        const uint64_t cost = L.total_cost ? L.total_cost : 1;
        const uint64_t rows = L.total_rows ? L.total_rows : 1;
        const double per_row = (double)cost / (double)rows;
        uint64_t sc = (uint64_t)((double)slice_rows * per_row);
        P.slice_cost = sc < 64 ? 64 : sc;
    }
    if (by_rank(L, P, 3)) return launch_rank_walk(P, ring_bytes_for(L.ctas_per_sm), s, dp.sms);
    if (P.flat_np > 0) return launch_enum_flat(P, ring_bytes_for(L.ctas_per_sm), s, dp.sms);
    P.half_rows = half_rows_for(L.d, ring_bytes_for(L.ctas_per_sm));
    FZ_DISPATCH_D(L.d, launch_enum_d, P, s, dp.sms);
}

int launch_unrank(const EnumLaunch &L, const uint64_t *ranks, uint64_t m, int32_t *out,
                  cudaStream_t s) {
    if (m == 0) return FZ_OK;
    if (!out || !ranks || !L.C || !L.status || (L.K >= 1 && L.top > 0 && !L.O && !L.run_memo))
        return set_error(FZ_EINTERNAL, "unrank: missing device buffer");
    EnumParams P = make_params(L);
    P.out = out;
    if (L.d == 1 || (L.K == L.d && L.top > L.n))
        return set_error(FZ_EINVAL, "unrank: d == 1 or k == d has a single block; use enumerate");
    FZ_DISPATCH_D(L.d, launch_unrank_d, P, ranks, m, s);
}

size_t enum_params_bytes() { return sizeof(EnumParams); }

// EnumParams of one batch instance (host-side image, copied to the device).
// (its work items: batch_items)
void fill_batch_params(const EnumLaunch &L, int32_t *out, uint64_t count, void *dst) {
    EnumParams P = make_params(L);
    P.dense_min = dense_min_for(true);
    P.out = out;
    P.rank_begin = 0;
    P.nrows = count;
    P.aligned = ((uintptr_t)out & 15u) == 0;
    P.half_rows = half_rows_for(L.d);
    if (L.d > BATCH_FLAT_MAX_D) P.flat_np = 0;
    if (by_rank(L, P, 10)) P.flat_src = SRC_RANK;
    memcpy(dst, &P, sizeof(P));
}

uint32_t enum_params_shape(const void *image) {
    EnumParams P;
    memcpy(&P, image, sizeof(P));
    return P.flat_np ? (uint32_t)(P.d << 8 | P.flat_np << 2 | P.flat_src) : 0u;
}

void batch_order(const unsigned char *images, size_t pb, const uint64_t *cost, int count,
                 std::vector<int> *order, std::vector<BatchGroup> *groups) {
    std::vector<uint32_t> shape((size_t)count);
    std::map<uint32_t, uint64_t> total;
    for (int i = 0; i < count; ++i) {
        shape[(size_t)i] = enum_params_shape(images + (size_t)i * pb);
        total[shape[(size_t)i]] += cost[i];
    }
    order->resize((size_t)count);
    for (int i = 0; i < count; ++i) (*order)[(size_t)i] = i;
    // The general kernel last: it is not one of the overlapped launches.  Its
    // instances by code path (run copy, walk up to width 8, wider walk) and
    // width, so that warps of an SM run the same code and share tables (512
    // partial memos of widths 4..8: 11.2 ms in the caller's order, 8.5 so).
    std::vector<int> path((size_t)count, 0);
    for (int i = 0; i < count; ++i) {
        EnumParams P;
        memcpy(&P, images + (size_t)i * pb, sizeof(P));
        if (!shape[(size_t)i]) path[(size_t)i] = (P.run_memo ? 0 : P.d <= 8 ? 32 : 64) + P.d;
    }
    std::stable_sort(order->begin(), order->end(), [&](int x, int y) {
        const uint32_t a = shape[(size_t)x], b = shape[(size_t)y];
        if (a == b) return path[(size_t)x] < path[(size_t)y];
        if (!a || !b) return !b;
        return total[a] != total[b] ? total[a] > total[b] : a < b;
    });
    groups->clear();
    for (int p = 0; p < count; ++p) {
        const uint32_t k = shape[(size_t)(*order)[(size_t)p]];
        if (groups->empty() || groups->back().shape != k)
            groups->push_back({k, p, p, 0, 0});
        groups->back().last = p + 1;
    }
}

// Work items: 1/8 of a resident warp's share of the whole call, 512 to 2048 of
// cost.  Small items keep the instances being written at any time few, so
// that their tables stay in L2 (4096 instances of 1e2..1e6 rows, 4.3e8 in
// all: 4.5 ms with items of 15400, 3.5 with 7700, 3.2 with 3900, 3.0 with
// 1900), although an item starts with a dozen dependent loads (about 10 us).
// The general kernel's items (a prefix costs it 16 or 64, and it is not one of
// the overlapped launches): 1/8 of a warp's share of its own instances, 4096
// at least (the same 512 partial memos: 14.5 ms with the items above).
void batch_items(unsigned char *params, size_t pb, const uint64_t *cost, const int *order,
                 std::vector<BatchGroup> *groups, int sms, uint64_t *item0) {
    // by rank a row costs about four rows of the flat walk, a prefix nothing
    auto cost_of = [&](int p) {
        EnumParams P;
        memcpy(&P, params + (size_t)p * pb, sizeof(P));
        return P.flat_src == SRC_RANK ? 4 * P.nrows : cost[order[p]];
    };
    uint64_t total = 0, general = 0;
    for (const BatchGroup &G : *groups)
        for (int p = G.first; p < G.last; ++p) (G.shape ? total : general) += cost_of(p);
    uint64_t flat_target = total / ((uint64_t)sms * 24 * 8 + 1);
    flat_target = flat_target < 512 ? 512 : flat_target > 2048 ? 2048 : flat_target;
    uint64_t general_target = general / ((uint64_t)sms * 16 * 8 + 1);
    general_target = general_target < 4096 ? 4096 : general_target;
    item0[0] = 0;
    for (BatchGroup &G : *groups) {
        const uint64_t target = G.shape ? flat_target : general_target;
        G.item_lo = item0[G.first];
        for (int p = G.first; p < G.last; ++p) {
            EnumParams P;
            memcpy(&P, params + (size_t)p * pb, sizeof(P));
            const uint64_t c = cost_of(p);
            const uint64_t items = P.nrows == 0 || c == 0 ? 0 : (c + target - 1) / target;
            if (items) {
                P.slice_cost = (c + items - 1) / items;
                P.slice_rows = (P.nrows + items - 1) / items;
                if (P.slice_cost < 64) P.slice_cost = 64;
                P.slice_rows = P.slice_rows < 4 ? 4 : (P.slice_rows + 3) & ~3ull;
                memcpy(params + (size_t)p * pb, &P, sizeof(P));
            }
            item0[p + 1] = item0[p] + items;
        }
        G.item_hi = item0[G.last];
    }
}

int launch_enumerate_batch(const void *params_dev, const uint64_t *item0_dev,
                           const BatchGroup *groups, int ngroups, unsigned long long *counters,
                           int32_t *out_base, cudaStream_t s, int ctas_per_sm) {
    if (ngroups <= 0) return FZ_OK;
    if (ngroups > BATCH_MAX_GROUPS) return set_error(FZ_EINTERNAL, "batch: too many groups");
    DeviceProps dp;
    int rc = device_props(&dp);
    if (rc != FZ_OK) return rc;
    FZ_CUDA_TRY(cudaMemsetAsync(counters, 0, (size_t)ngroups * sizeof(unsigned long long), s));
    bool chained = false;
    for (int i = 0; i < ngroups; ++i) {
        const BatchGroup &G = groups[i];
        // no launch for instances without rows; the next one is chained only
        // to a kernel that was launched
        if (G.item_hi == G.item_lo) continue;
        BatchEnumParams BP;
        BP.inst = static_cast<const EnumParams *>(params_dev);
        BP.out_base = out_base;
        BP.item0 = item0_dev;
        BP.first = G.first;
        BP.last = G.last;
        BP.item_lo = G.item_lo;
        BP.item_hi = G.item_hi;
        BP.item_counter = counters + i;
        BP.chained = chained ? 1 : 0;
        if (G.shape) {
            rc = launch_flat_batch(BP, (int)(G.shape >> 8), (int)(G.shape >> 2 & 63),
                                   (int)(G.shape & 3), s, dp.sms, ctas_per_sm);
            if (rc != FZ_OK) return rc;
            chained = true;
            continue;
        }
        chained = false;
        const size_t smem = (size_t)ENUM_WARPS *
                            (BATCH_RING_BYTES + sizeof(EnumParams) + sizeof(WarpPath));
        static DeviceOnce attr_set;
        if (!attr_set.is_set(dp.device)) {
            FZ_CUDA_TRY(cudaFuncSetAttribute(
                fz_enum_batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            attr_set.set(dp.device);
        }
        int per_sm = 0;
        FZ_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fz_enum_batch_kernel,
                                                                  ENUM_THREADS, smem));
        uint64_t grid = (uint64_t)batch_blocks_for(per_sm, ctas_per_sm) * dp.sms;
        const uint64_t want = (G.item_hi - G.item_lo + ENUM_WARPS - 1) / ENUM_WARPS;
        if (want < grid) grid = want;
        rc = launch_capped(fz_enum_batch_kernel, (unsigned)grid, smem, s, ctas_per_sm, false, BP);
        if (rc != FZ_OK) return rc;
    }
    return FZ_OK;
}

uint64_t default_slice_rows(uint64_t nrows, int sms) {
    // about 2.5 items a resident warp, between 128 and 24576 rows: an item
    // starts with a dozen dependent loads, long ones leave a tail and write
    // too far apart (kernel us at 1024 / 4096 / 16384 / 65536 rows an item:
    // 5e8 rows of width 6 2660 / 1914 / 1830 / 2456, 1e8 558 / 401 / 516 / -,
    // 1.4e7 of width 9 128 / 152 / 314 / -)
    uint64_t s = nrows * 2 / ((uint64_t)sms * 4 * ENUM_WARPS * 5);
    const uint64_t least = nrows / 64 < 128 ? 128 : nrows / 64 > 512 ? 512 : nrows / 64;
    if (s < least) s = least;
    if (s > 24576) s = 24576;
    return (s + 31) & ~31ull;
}

}  // namespace fz
