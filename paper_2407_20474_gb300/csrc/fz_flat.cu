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

// Work items from an atomic counter, as in the other enumeration kernels.
template <int D, int NP, int SRC>
__global__ void __launch_bounds__(ENUM_THREADS, 4)
    fz_enum_flat_kernel(const __grid_constant__ EnumParams P, int warp_bytes) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31;
    const int wid = threadIdx.x >> 5;
    unsigned char *mem = smem_raw + (size_t)wid * warp_bytes;
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
        if (!flat_slice<D, NP, SRC>(P, mem, (uint32_t)P.half_rows, row0, row1, pol, lane)) break;
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

bool flat_serves(int d, int np, int src) {
    if (d < 3 || d > 9) return false;
    if (src == SRC_PAIR) return np == d - 2;
    return np >= 1 && np <= 3 && d - 1 - np >= 1 && d - 1 - np <= RUN_MAX_K;
}

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

}  // namespace fz
