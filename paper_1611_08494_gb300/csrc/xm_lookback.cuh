// xm_lookback.cuh -- the decoupled look-back of single-pass kernels (prefix
// sums, the radix sort, the index build): tiles take ids in launch order,
// publish their own sum, and add up the sums of the tiles before them until
// one with an inclusive prefix. Every wait has a poll limit.
#pragma once

#include "xm_internal.cuh"

namespace xm {

// Status word of a tile: flag in the top two bits, sum (or inclusive
// prefix) below.
constexpr uint64_t kStAgg = 1ull << 62;   // tile's own sum is available
constexpr uint64_t kStInc = 2ull << 62;   // inclusive prefix is available
constexpr uint64_t kStMask = (1ull << 62) - 1;
constexpr int kSpinLimit = 1 << 22;      // polls before a look-back gives up (~1-2 s)

// Settings of the look-backs (xm_debug_lookback): poll budget, and the tile
// that withholds its status words (-1: none).
struct Lookback {
    int spin_limit, silent_tile;
};
Lookback lookback_settings();

__device__ __forceinline__ uint64_t ld_relaxed(const uint64_t* p) {
    uint64_t v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_relaxed(uint64_t* p, uint64_t v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Sum of the tiles before `tile`, whose own sum is `all`; called by one whole
// warp, the result is in every lane. 32 predecessors' words are read per
// step. A look-back that runs out of polls sets kErrTimeout in *err and
// returns what it has (no more than the true sum).
__device__ __forceinline__ int64_t lookback_warp(uint64_t* status, int64_t tile, int64_t all,
                                                 int spin_limit, bool silent, int32_t* err) {
    const int lane = threadIdx.x & 31;
    uint64_t* my = status + tile;
    if (tile == 0) {
        if (lane == 0 && !silent) st_relaxed(my, kStInc | (uint64_t)all);
        return 0;
    }
    if (lane == 0 && !silent) st_relaxed(my, kStAgg | (uint64_t)all);
    int64_t prefix = 0;
    int64_t top = tile - 1;  // lane j reads tile top - j (before tile 0: an inclusive 0)
    int spins = 0;
    while (true) {
        const int64_t j = top - lane;
        const uint64_t w = j >= 0 ? ld_relaxed(status + j) : kStInc;
        const uint64_t flag = w & ~kStMask;
        const uint32_t inc = __ballot_sync(0xffffffffu, flag == kStInc);
        const uint32_t unready = __ballot_sync(0xffffffffu, flag == 0);
        const int first = inc ? __ffs(inc) - 1 : 31;  // words needed: lanes 0..first
        const uint32_t need = first == 31 ? 0xffffffffu : ((1u << (first + 1)) - 1u);
        if (unready & need) {
            if (++spins > spin_limit) {
                if (lane == 0) atomicOr(err, kErrTimeout);
                break;
            }
            __nanosleep(64);
            continue;
        }
        int64_t v = lane <= first ? (int64_t)(w & kStMask) : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        prefix += v;
        if (inc) break;
        top -= 32;
    }
    if (lane == 0 && !silent) st_relaxed(my, kStInc | (uint64_t)(prefix + all));
    return prefix;
}

}  // namespace xm
