// fz_flat.cu -- enumeration by the flat walk (fz_walk.cuh): leaves are the
// prefixes (a_0..a_{NP-1}), 32 of them evaluated at a time, their rows copied
// from the memo in run order (SRC_RUN, NP = d - K - 1) or computed from the
// closed form of the last two generators (SRC_PAIR, NP = d - 2: no memo).
//
// Measured on one GB300 (us, kernel under ncu): width 9, 1.4e7 rows, 148 with
// the depth-5 table (43 rows a leaf) against 376 for the leaf walk over a
// depth-4 memo with 4-byte copies; width 6, 1e7 rows without a memo (8.6e7
// prefixes, most of them empty), 1054 against 7445 for a warp per walk run;
// width 6, 5e8 rows (3300 rows a leaf), 6.7 TB/s written, as the subtree-run
// copy.
#include "fz_enum.cuh"

namespace fz {

namespace {

// Work items from an atomic counter: four fifths of the cost in items of
// slice_cost, the rest in items of an eighth of that (a quarter of short ones),
// so that the warps finish close together.
template <int D, int NP, int SRC>
__global__ void __launch_bounds__(ENUM_THREADS, 4)
    fz_enum_flat_kernel(const __grid_constant__ EnumParams P, int warp_bytes) {
    const int lane = threadIdx.x & 31;
    const int wid = threadIdx.x >> 5;
    unsigned char *mem = enum_smem + (size_t)wid * warp_bytes;
    const uint64_t pol = policy_evict_first();
    uint64_t cost_lo = 0, cost_hi = 0;
    if (P.by_cost) {
        cost_hi = flat_total_cost<NP>(P);
        if (!P.whole) {
            cost_lo = rank_to_cost(P, P.rank_begin, lane);
            cost_hi = rank_to_cost(P, P.rank_begin + P.nrows, lane);
        }
    }
    const uint64_t sc = P.slice_cost, part = sc >= 8192 ? sc / 8 : sc / 4;
    const uint64_t sct = part > 64 ? part : 64;
    const uint64_t n1 = P.by_cost ? (cost_hi - cost_lo) / sc * 4 / 5 : 0;
    unsigned long long next = 0;
    if (lane == 0) next = atomicAdd(P.slice_counter, 1ull);
    for (;;) {
        const uint64_t s = __shfl_sync(FULL, next, 0);
        if (lane == 0) next = atomicAdd(P.slice_counter, 1ull);  // read after this item
        uint64_t row0 = 0, row1 = P.nrows;
        if (P.by_cost) {
            const uint64_t c0 = s < n1 ? cost_lo + s * sc : cost_lo + n1 * sc + (s - n1) * sct;
            const uint64_t c1 = c0 + (s < n1 ? sc : sct);
            if (c0 >= cost_hi) break;
            if (s > 0 || c1 < cost_hi) {
                uint64_t r0, r1;
                flat_cost_to_ranks<NP>(P, c0, c1 < cost_hi ? c1 : c0, lane, r0, r1);
                auto place = [&](uint64_t r) {
                    r = r > P.rank_begin ? (r - P.rank_begin) & ~31ull : 0ull;
                    return r < P.nrows ? r : P.nrows;
                };
                if (s > 0) row0 = place(r0);
                if (c1 < cost_hi) row1 = place(r1);
            }
        } else {
            if (s >= P.nslices) break;
            row0 = s * P.slice_rows;
            if (row0 + P.slice_rows < P.nrows) row1 = row0 + P.slice_rows;
        }
        if (row1 <= row0) continue;
        if (!flat_slice<D, NP, SRC>(ConstParams{P}, mem, (uint32_t)P.half_rows, row0, row1, pol,
                                    lane))
            break;
    }
    if (lane == 0) bulk_wait_all();
    __syncwarp();
}

template <int D, int NP, int SRC>
int launch_one(EnumParams P, int warp_bytes, cudaStream_t s, int sms) {
    static DeviceOnce attr_set;
    P.half_rows = (int)flat_half_rows<NP, SRC, D>(warp_bytes);
    const int need = leaf_bytes<NP, SRC>() + 2 * P.half_rows * D * 4;
    const int bytes = (need > warp_bytes ? need : warp_bytes + 127) & ~127;
    auto kern = fz_enum_flat_kernel<D, NP, SRC>;
    return launch_enum_grid(kern, P, (size_t)ENUM_WARPS * bytes, s, sms, attr_set, bytes);
}

// ---------------------------------------------------------------------------
// The rank walk: no memo, and most prefixes of d - 2 coordinates empty (a
// width-6 set of 1e7 rows has 8.6e7 of them).  Instead of visiting them, a
// lane goes from its row to the row 32 ranks on: each coordinate whose
// subtree ends before that rank is searched again in its count row, from the
// value it had (or, under a new parent, from the power-law estimate), so
// lanes of a warp follow consecutive rows and mostly share the upper
// coordinates' loads.  The last two coordinates are the pair's closed form.
// The cost is per row, so items are equal row ranges.
//
// Bound by the latency of the searches' dependent loads.  The case above: 1054
// us by the flat walk, 409 by the rank walk.
// ---------------------------------------------------------------------------
// Rows [row0, row0 + rows) of the set.  Returns false if the tables disagree.
template <int D, class PA>
__device__ __forceinline__ bool rank_rows(const PA &params, int32_t *ring, uint32_t B,
                                          uint64_t row0, uint32_t rows, uint64_t pol, int lane) {
    constexpr int NP = D - 2;
    bool ok = true;
    // a[j], remainders, and the ranks where the subtree of (a_0..a_{j-1})
    // begins and that of (a_0..a_j) ends
    uint32_t a[NP], r[NP + 1];
    uint64_t beg[NP + 1], end[NP];
    r[0] = (uint32_t)params().n;
    beg[0] = 0;
#pragma unroll
    for (int j = 0; j < NP; ++j) {
        a[j] = 0;
        end[j] = 0;
    }
    uint32_t at = 0, b0 = 0, hpos = 0, half = 0, nfull = 0;
    for (uint32_t q = 0; q < rows;) {
        uint32_t cnt = rows - q;
        if (cnt > 32u) cnt = 32u;
        if (cnt > B - hpos) cnt = B - hpos;
        const bool act = (uint32_t)lane < cnt;
        const uint64_t R = params().rank_begin + row0 + q + lane;
        if (act && R >= end[NP - 1]) {
            bool fresh = false;  // the parent changed
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                if (!fresh && R < end[j]) continue;
                const uint32_t g = (uint32_t)params().g[j];
                const uint64_t *row = params().C + (int64_t)j * params().cs;
                const uint32_t vmax = fd_div(r[j], params().fdg[j]);
                const bool again = !fresh && end[j] > 0;  // same parent, a later child
                const uint64_t all = again ? 0ull : __ldg(row + r[j]);
                uint64_t before;
                if (again)
                    a[j] = thread_child_from(row, r[j], g, vmax, R - beg[j],
                                             a[j] > 0 ? a[j] - 1u : 0u, &before);
                else
                    a[j] = thread_child(row, r[j], g, vmax, R - beg[j], all, D - 1 - j, &before);
                r[j + 1] = r[j] - a[j] * g;
                end[j] = beg[j] + __ldg(row + r[j + 1]);
                beg[j + 1] = beg[j] + before;
                fresh = true;
            }
            at = pair_form_top(params().leaf.pair, r[NP]);
            b0 = fd_div(r[NP] - at * params().leaf.pair.g, params().leaf.pair.fh);
            if (R >= end[NP - 1]) ok = false;  // the tables disagree
        }
        if (hpos == 0 && nfull >= 2) {
            if (lane == 0) bulk_wait_read<1>();
            __syncwarp();
        }
        if (act) {
            const uint32_t o = (uint32_t)(R - beg[NP]);
            int w[D];
#pragma unroll
            for (int j = 0; j < NP; ++j) w[j] = (int)a[j];
            w[NP] = (int)(at - o * params().leaf.pair.h1);
            w[NP + 1] = (int)(b0 + o * params().leaf.pair.g1);
            store_row<D>(ring + (size_t)(half * B + hpos + lane) * D, w, lane);
        }
        q += cnt;
        hpos += cnt;
        if (hpos == B) {
            flush_words(params().out + (row0 + (uint64_t)nfull * B) * D, params().aligned != 0,
                        ring + (size_t)half * B * D, B * D, lane, pol);
            ++nfull;
            half ^= 1u;
            hpos = 0;
        }
    }
    if (hpos > 0)
        flush_words(params().out + (row0 + (uint64_t)nfull * B) * D, params().aligned != 0,
                    ring + (size_t)half * B * D, hpos * D, lane, pol);
    if (lane == 0) bulk_wait_read_all();
    ok = __all_sync(FULL, ok);
    if (!ok && lane == 0) atomicExch(params().status, (int)DEV_INTERNAL);
    return ok;
}

template <int D>
__global__ void __launch_bounds__(ENUM_THREADS, 4)
    fz_enum_rank_kernel(const __grid_constant__ EnumParams P, int warp_bytes) {
    const int lane = threadIdx.x & 31;
    const int wid = threadIdx.x >> 5;
    int32_t *ring = reinterpret_cast<int32_t *>(enum_smem + (size_t)wid * warp_bytes);
    const uint64_t pol = policy_evict_first();
    for (;;) {
        unsigned long long s = 0;
        if (lane == 0) s = atomicAdd(P.slice_counter, 1ull);
        s = __shfl_sync(FULL, s, 0);
        if (s >= P.nslices) break;
        const uint64_t row0 = s * P.slice_rows;
        const uint64_t rest = P.nrows - row0;
        const uint32_t rows = rest < P.slice_rows ? (uint32_t)rest : (uint32_t)P.slice_rows;
        if (!rank_rows<D>(ConstParams{P}, ring, (uint32_t)P.half_rows, row0, rows, pol, lane)) break;
    }
    if (lane == 0) bulk_wait_all();
    __syncwarp();
}

template <int D>
int launch_rank_d(EnumParams P, int warp_bytes, cudaStream_t s, int sms) {
    static DeviceOnce attr_set;
    uint32_t b = (uint32_t)(warp_bytes / (8 * D)) / 32 * 32;
    P.half_rows = (int)(b < 32 ? 32 : b);
    const int bytes = (2 * P.half_rows * D * 4 + 127) & ~127;
    // an item starts with a full search: 256 to 2048 rows, about eight a warp
    uint64_t rows = P.nrows / ((uint64_t)sms * 32 * 8 + 1);
    rows = rows < 256 ? 256 : rows > 2048 ? 2048 : rows;
    if (P.slice_rows < rows) rows = P.slice_rows;
    P.slice_rows = (rows + 31) & ~31ull;
    P.nslices = (P.nrows + P.slice_rows - 1) / P.slice_rows;
    return launch_enum_grid(fz_enum_rank_kernel<D>, P, (size_t)ENUM_WARPS * bytes, s, sms, attr_set,
                            bytes);
}

// The flat or rank walk of a batch's instances of one shape.  A launch may start while
// the one before it drains (chained): it reads nothing that one writes, and
// waits for its completion only before it ends, so the last launch's end is
// the end of all.  Three blocks an SM: at 64 registers the loops spill (see
// flat_rows), 4 blocks of them are no faster.
template <int D, int NP, int SRC>
__global__ void __launch_bounds__(ENUM_THREADS, 3)
    fz_flat_batch_kernel(const __grid_constant__ BatchEnumParams BP) {
    const int lane = threadIdx.x & 31;
    const int wid = threadIdx.x >> 5;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    constexpr bool RANK = SRC == SRC_RANK;
    unsigned char *mem = enum_smem + (size_t)wid * RING_BYTES_PER_WARP;
    const SharedParams params{(uint32_t)(ENUM_WARPS * RING_BYTES_PER_WARP + wid * sizeof(EnumParams))};
    EnumParams *ep = reinterpret_cast<EnumParams *>(enum_smem + params.off);
    constexpr uint32_t B = RANK ? RING_BYTES_PER_WARP / (8 * D) / 32 * 32
                                : flat_half_rows<NP, SRC, D>(RING_BYTES_PER_WARP);
    static_assert((RANK ? 0 : leaf_bytes<NP, SRC>()) + 2 * (int)B * D * 4 <= RING_BYTES_PER_WARP,
                  "ring");
    const uint64_t pol = policy_evict_first();
    int cur = -1;
    unsigned long long next = 0;
    if (lane == 0) next = atomicAdd(BP.item_counter, 1ull);
    for (;;) {
        const uint64_t item = BP.item_lo + __shfl_sync(FULL, next, 0);
        if (item >= BP.item_hi) break;
        if (lane == 0) next = atomicAdd(BP.item_counter, 1ull);  // read after this item
        const uint64_t s = batch_locate(BP, ep, cur, item, lane);
        const EnumParams &P = params();
        uint64_t row0, row1;
        if (!RANK && P.by_cost) {
            const uint64_t cost_hi = flat_total_cost<NP>(P);
            const uint64_t c0 = s * P.slice_cost, c1 = c0 + P.slice_cost;
            if (c0 >= cost_hi) continue;
            row0 = 0;
            row1 = P.nrows;
            if (s > 0 || c1 < cost_hi) {
                uint64_t r0, r1;
                flat_cost_to_ranks<NP>(P, c0, c1 < cost_hi ? c1 : c0, lane, r0, r1);
                if (s > 0) row0 = r0 & ~31ull;
                if (c1 < cost_hi) row1 = r1 & ~31ull;
                if (row0 > P.nrows) row0 = P.nrows;
                if (row1 > P.nrows) row1 = P.nrows;
            }
        } else {
            row0 = s * P.slice_rows;
            row1 = row0 + P.slice_rows < P.nrows ? row0 + P.slice_rows : P.nrows;
        }
        if (row1 <= row0) continue;
        if constexpr (RANK) {
            if (!rank_rows<D>(params, reinterpret_cast<int32_t *>(mem), B, row0,
                              (uint32_t)(row1 - row0), pol, lane))
                break;
        } else {
            if (!flat_slice<D, NP, SRC>(params, mem, B, row0, row1, pol, lane)) break;
        }
    }
    if (lane == 0) bulk_wait_all();
    __syncwarp();
    if (BP.chained) asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <int D, int NP, int SRC>
int launch_batch_one(const BatchEnumParams &BP, cudaStream_t s, int sms, int ctas_per_sm) {
    auto kern = fz_flat_batch_kernel<D, NP, SRC>;
    constexpr size_t smem = (size_t)ENUM_WARPS * (RING_BYTES_PER_WARP + sizeof(EnumParams));
    static DeviceOnce attr_set;
    static int occupancy[64];
    int dev = 0;
    FZ_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return set_error(FZ_EINVAL, "device ordinal out of range");
    if (!attr_set.is_set(dev)) {
        FZ_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem));
        FZ_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occupancy[dev], kern,
                                                                  ENUM_THREADS, smem));
        attr_set.set(dev);
    }
    uint64_t grid = (uint64_t)batch_blocks_for(occupancy[dev], ctas_per_sm) * sms;
    const uint64_t want = (BP.item_hi - BP.item_lo + ENUM_WARPS - 1) / ENUM_WARPS;
    if (want < grid) grid = want;
    return launch_capped(kern, (unsigned)grid, smem, s, ctas_per_sm, BP.chained != 0, BP);
}

template <int D>
int launch_batch_d(const BatchEnumParams &BP, int np, int src, cudaStream_t s, int sms, int cap) {
    if (src == SRC_PAIR) return launch_batch_one<D, D - 2, SRC_PAIR>(BP, s, sms, cap);
    if constexpr (D >= 4 && D <= 7)
        if (src == SRC_RANK) return launch_batch_one<D, D - 2, SRC_RANK>(BP, s, sms, cap);
    if (src != SRC_RUN) return set_error(FZ_EINTERNAL, "flat walk: no kernel for this shape");
    if (np == 1) return launch_batch_one<D, 1, SRC_RUN>(BP, s, sms, cap);
    if constexpr (D >= 4)
        if (np == 2) return launch_batch_one<D, 2, SRC_RUN>(BP, s, sms, cap);
    if constexpr (D >= 5)
        if (np == 3) return launch_batch_one<D, 3, SRC_RUN>(BP, s, sms, cap);
    return set_error(FZ_EINTERNAL, "flat walk: no kernel for this shape");
}

template <int D>
int launch_d(const EnumParams &P, int warp_bytes, cudaStream_t s, int sms) {
    if (P.flat_src == SRC_PAIR) {
        if constexpr (D >= 3) return launch_one<D, D - 2, SRC_PAIR>(P, warp_bytes, s, sms);
    } else {
        // K = D - 1 - NP between 1 and RUN_MAX_K
        if constexpr (D >= 3 && D - 2 <= RUN_MAX_K)
            if (P.flat_np == 1) return launch_one<D, 1, SRC_RUN>(P, warp_bytes, s, sms);
        if constexpr (D >= 4)
            if (P.flat_np == 2) return launch_one<D, 2, SRC_RUN>(P, warp_bytes, s, sms);
        if constexpr (D >= 5)
            if (P.flat_np == 3) return launch_one<D, 3, SRC_RUN>(P, warp_bytes, s, sms);
    }
    return set_error(FZ_EINTERNAL, "flat walk: no kernel for this shape");
}

}  // namespace

int launch_enum_flat(const EnumParams &P, int warp_bytes, cudaStream_t s, int sms) {
    switch (P.d) {
        case 3: return launch_d<3>(P, warp_bytes, s, sms);
        case 4: return launch_d<4>(P, warp_bytes, s, sms);
        case 5: return launch_d<5>(P, warp_bytes, s, sms);
        case 6: return launch_d<6>(P, warp_bytes, s, sms);
        case 7: return launch_d<7>(P, warp_bytes, s, sms);
        case 8: return launch_d<8>(P, warp_bytes, s, sms);
        case 9: return launch_d<9>(P, warp_bytes, s, sms);
        default: return set_error(FZ_EINTERNAL, "flat walk: no kernel for this shape");
    }
}

int launch_flat_batch(const BatchEnumParams &BP, int d, int np, int src, cudaStream_t s, int sms,
                      int ctas_per_sm) {
    switch (d) {
        case 3: return launch_batch_d<3>(BP, np, src, s, sms, ctas_per_sm);
        case 4: return launch_batch_d<4>(BP, np, src, s, sms, ctas_per_sm);
        case 5: return launch_batch_d<5>(BP, np, src, s, sms, ctas_per_sm);
        case 6: return launch_batch_d<6>(BP, np, src, s, sms, ctas_per_sm);
        case 7: return launch_batch_d<7>(BP, np, src, s, sms, ctas_per_sm);
        case 8: return launch_batch_d<8>(BP, np, src, s, sms, ctas_per_sm);
        default: return set_error(FZ_EINTERNAL, "flat walk: no kernel for this shape");
    }
}

bool rank_walk_serves(int d) { return d >= 4 && d <= 7; }

int launch_rank_walk(const EnumParams &P, int warp_bytes, cudaStream_t s, int sms) {
    switch (P.d) {
        case 4: return launch_rank_d<4>(P, warp_bytes, s, sms);
        case 5: return launch_rank_d<5>(P, warp_bytes, s, sms);
        case 6: return launch_rank_d<6>(P, warp_bytes, s, sms);
        case 7: return launch_rank_d<7>(P, warp_bytes, s, sms);
        default: return set_error(FZ_EINTERNAL, "rank walk: no kernel for this width");
    }
}

}  // namespace fz
