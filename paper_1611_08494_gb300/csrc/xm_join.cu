// xm_join.cu -- the join types of paper §2.2 over a selected pair set.
//
// i) 1 and 2: the selected pairs; ii) 1 or 2: pairs, unmatched A rows and
// unmatched B rows; iii) all from 1 (2): pairs plus unmatched A (B) rows;
// iv) 1 not 2 (2 not 1): unmatched A (B) rows; v) 1 xor 2: unmatched A and
// unmatched B rows. A source is matched when it appears in the selected
// pairs. Row order: rows carrying an A source in ascending (a_row, b_row),
// then unmatched B rows in ascending b_row.
//
// Device steps of xm_join: a bitset of matched B rows (idempotent atomicOr, so
// the result is deterministic); one pass over the A sources that knows the
// unmatched ones before each and writes their rows, the best pairs or the
// pairs (many pairs for each source: a pass of their own, each as many places
// on as unmatched A rows come before it; many for a few: left to a pass over a
// list of them); one pass over the bitset that counts
// the unmatched B rows before each word by a chained prefix sum and writes
// them. xm_join_noalloc, which learns the row count before it writes, keeps
// rows per source and per word and their prefix sums in its scratch array.
#include <math.h>

#include <mutex>
#include <new>

#include "xm_lookback.cuh"

namespace xm {
namespace {

constexpr int kBlock = 256;

unsigned grid_for(int64_t n) { return (unsigned)((n + kBlock - 1) / kBlock); }

// Grid of a grid-stride kernel: enough blocks to fill the GPU, no more.
unsigned grid_cap(int64_t n) {
    const unsigned g = grid_for(n);
    return g < 8u * 152u ? g : 8u * 152u;
}

__global__ void k_mark_b(const int64_t* __restrict__ b_row, int64_t n, uint32_t* __restrict__ bits) {
    pdl_wait();
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int64_t b = b_row[i];
    if (b >= 0) atomicOr(&bits[b >> 5], 1u << (b & 31));
}

// Rows each A source contributes, and the number of unmatched A sources.
// (grid-stride; the unmatched A sources are summed per block, so the one
// counter takes an atomic per block, not per warp)
__global__ void k_rows_a(const int32_t* __restrict__ count, int64_t nA, int sel_all,
                         int with_pairs, int with_un_a, int32_t* __restrict__ rows,
                         unsigned long long* __restrict__ n_un_a) {
    pdl_wait();
    __shared__ unsigned long long block_un;
    if (threadIdx.x == 0) block_un = 0;
    __syncthreads();
    uint32_t un = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nA;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t c = count[i];
        const int32_t sel = sel_all ? c : (c > 0 ? 1 : 0);
        int32_t r = with_pairs ? sel : 0;
        if (sel == 0 && with_un_a) r = 1;
        rows[i] = r;
        un += c == 0;
    }
    un = __reduce_add_sync(0xffffffffu, un);
    if ((threadIdx.x & 31) == 0 && un) atomicAdd(&block_un, (unsigned long long)un);
    __syncthreads();
    if (threadIdx.x == 0 && block_un) atomicAdd(n_un_a, block_un);
}

__device__ __forceinline__ uint32_t word_valid(int64_t w, int64_t nB) {
    int64_t rem = nB - (w << 5);
    return rem >= 32 ? 0xFFFFFFFFu : ((1u << rem) - 1u);
}

__global__ void k_word_unmatched(const uint32_t* __restrict__ bits, int64_t nwords, int64_t nB,
                                 int32_t* __restrict__ wcount) {
    pdl_wait();
    int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= nwords) return;
    wcount[w] = __popc(~bits[w] & word_valid(w, nB));
}

// A-side join rows, one thread per A row.
__global__ void k_write_a(const int32_t* __restrict__ count, const int64_t* __restrict__ pair_off,
                          const int64_t* __restrict__ pb, const double* __restrict__ ps,
                          const int64_t* __restrict__ best_b, const double* __restrict__ best_s,
                          const int64_t* __restrict__ row_off, int64_t nA, int sel_all,
                          int with_pairs, int with_un_a, int64_t* __restrict__ oa,
                          int64_t* __restrict__ ob, double* __restrict__ os) {
    pdl_wait();
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nA) return;
    int32_t c = count[i];
    int64_t o = row_off[i];
    if (c > 0) {
        if (!with_pairs) return;
        if (sel_all) {
            int64_t p = pair_off[i];
            for (int32_t k = 0; k < c; k++) {
                oa[o + k] = i;
                ob[o + k] = pb[p + k];
                os[o + k] = ps[p + k];
            }
        } else {
            oa[o] = i;
            ob[o] = best_b[i];
            os[o] = best_s[i];
        }
    } else if (with_un_a) {
        oa[o] = i;
        ob[o] = -1;
        os[o] = NAN;
    }
}

// B-only rows after the A-side rows: base_ptr (device) holds their count.
__global__ void k_write_b(const uint32_t* __restrict__ bits, const int64_t* __restrict__ word_off,
                          int64_t nB, const int64_t* __restrict__ base_ptr, int64_t* __restrict__ oa,
                          int64_t* __restrict__ ob, double* __restrict__ os) {
    pdl_wait();
    int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= nB) return;
    const int64_t base = *base_ptr;
    int64_t w = j >> 5;
    uint32_t un = ~bits[w] & word_valid(w, nB);
    uint32_t bit = 1u << (j & 31);
    if (!(un & bit)) return;
    int64_t o = base + word_off[w] + __popc(un & (bit - 1u));
    oa[o] = -1;
    ob[o] = j;
    os[o] = NAN;
}

// ---- the passes of xm_join

constexpr int kRowsA = 4;  // A sources per thread: 128 in a row per warp
constexpr int kTileA = kRowsA * kBlock;
static_assert(kTileA == kCountTile, "the match counts unmatched sources per tile");
constexpr int kRowsWarp = 512;   // pairs that a warp writes for its 32 sources
constexpr int kRowsChunk = 4 * kBlock;  // pairs of a listed chunk

// Exclusive prefix of v over the block; *all: the block's sum.
__device__ __forceinline__ uint32_t block_prefix(uint32_t v, uint32_t* all) {
    __shared__ uint32_t warp_tot[kBlock / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    uint32_t before = incl - v, tot = 0;
#pragma unroll
    for (int w = 0; w < kBlock / 32; w++) {
        if (w < warp) before += warp_tot[w];
        tot += warp_tot[w];
    }
    *all = tot;
    return before;
}

struct JoinTile {
    unsigned int tile;
    long long prefix;
};

// Pairs that the A-side pass leaves: [p0, p0 + n) of the 32 sources from i0 on,
// before which `un` sources are unmatched, and of which those in `mask` are.
struct __align__(32) PairChunk {
    int64_t p0, un, i0;
    uint32_t mask;
    int32_t n;
};

// What the A-side pass reads and writes. counts: [0] A-side rows, [2]
// unmatched A sources.
struct JoinA {
    const int32_t* count;
    const int64_t* pair_off;
    const int64_t* pb;
    const double* ps;
    const int64_t* best_b;
    const double* best_s;
    int64_t nA, n_pairs;
    int32_t sel_all, with_pairs, with_un_a;
    int64_t a_off;
    const int64_t* zeros;  // unmatched A sources before each tile (NULL: chained)
    int32_t rows;          // this pass writes the "all" selection's pair rows
    int32_t* un_before;    // (nullable) unmatched A sources before each source
    PairChunk* chunks;
    unsigned int* n_chunks;
    int64_t* oa;
    int64_t* ob;
    double* os;
    int64_t* counts;
};

// One pass over the A sources: reads their member counts once and writes the
// rows of the unmatched ones, and the best pairs or (J.rows) the pairs of the
// "all" selection. The unmatched ones before a tile are known from the match
// of many sources, else they come from a chained prefix sum over tiles in
// launch order. A thread writes the pairs of its own sources while no source
// of the warp's 32 has more than kRowsThread, else (MANY: where the match may
// have counted such a source) the warp writes them a pair per lane, or lists
// them for k_join_long where the 32 have more than kRowsWarp. Bound by memory: pair rows and unmatched rows share sectors,
// so they are written together, and nothing is kept per source between passes.
// 0.50 ms for 5e7 sources, 3e7 pairs and 5.1e7 rows (2.8 GB, 5.6 TB/s) against
// 1.3 ms in a pass for the rows of each source, their prefix sum, a pass over
// the pairs and one over the sources.
template <bool MANY>
__global__ void __launch_bounds__(kBlock) k_join_a(JoinA J, uint64_t* status, unsigned int* counter,
                                                   Lookback lb, int32_t* err) {
    pdl_wait();
    __shared__ JoinTile S;
    if (!J.zeros) {
        if (threadIdx.x == 0) S.tile = atomicAdd(counter, 1u);
        __syncthreads();
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t tile = J.zeros ? blockIdx.x : S.tile, first = tile * kTileA;
    const int64_t i0 = first + warp * (32 * kRowsA) + lane;
    // (pair rows come before an unmatched one)
    const bool off = J.sel_all && J.with_pairs && (J.rows || J.with_un_a);
    int32_t c[kRowsA];
    uint32_t un_mask[kRowsA], mine = 0;  // (un_mask: of the warp's 32 sources)
    int64_t at[kRowsA];
#pragma unroll
    for (int k = 0; k < kRowsA; k++) {
        const int64_t i = i0 + 32 * k;
        c[k] = i < J.nA ? __ldcs(J.count + i) : -1;
        at[k] = off ? (i < J.nA ? __ldcs(J.pair_off + i) : INT64_MAX) : 0;
    }
#pragma unroll
    for (int k = 0; k < kRowsA; k++) {
        un_mask[k] = __ballot_sync(0xffffffffu, c[k] == 0);
        mine += __popc(un_mask[k]);
    }
    uint32_t all;
    uint32_t before = block_prefix(lane == 0 ? mine : 0u, &all);
    before = __shfl_sync(0xffffffffu, before, 0);  // (of the warp)
    if (threadIdx.x < 32) {
        const int64_t p = J.zeros ? J.zeros[tile]
                                  : lookback_warp(status, tile, (int64_t)all, lb.spin_limit,
                                                  tile == lb.silent_tile, err);
        if (threadIdx.x == 0) {
            S.prefix = p;
            if (first + kTileA >= J.nA) {
                const int64_t un = p + all;
                J.counts[2] = un;
                J.counts[0] = (J.with_pairs ? (J.sel_all ? J.n_pairs : J.nA - un) : 0) +
                              (J.with_un_a ? un : 0);
            }
        }
    }
    __syncthreads();
    const int64_t un_base = S.prefix;
#pragma unroll
    for (int k = 0; k < kRowsA; k++) {
        const int64_t i = i0 + 32 * k;
        const int64_t un = un_base + before + __popc(un_mask[k] & ((1u << lane) - 1u));
        before += __popc(un_mask[k]);
        if (c[k] == 0) {
            if (J.with_un_a) {
                const int64_t o = off ? at[k] + un : J.with_pairs ? i : un;
                J.oa[o] = i + J.a_off;
                J.ob[o] = -1;
                J.os[o] = NAN;
            }
        } else if (c[k] > 0 && J.with_pairs && !J.sel_all) {
            const int64_t o = J.with_un_a ? i : i - un;
            J.oa[o] = i + J.a_off;
            J.ob[o] = __ldg(J.best_b + i);
            J.os[o] = __ldg(J.best_s + i);
        }
        if (J.un_before && c[k] >= 0) J.un_before[i] = (int32_t)un;
        if (!J.rows) continue;
        if (!MANY || __reduce_max_sync(0xffffffffu, c[k]) <= kRowsThread) {
            const int64_t o = at[k] + (J.with_un_a ? un : 0);
#pragma unroll 1
            for (int32_t j = 0; j < c[k]; j++) {
                J.oa[o + j] = i + J.a_off;
                J.ob[o + j] = __ldg(J.pb + at[k] + j);
                J.os[o + j] = __ldg(J.ps + at[k] + j);
            }
            continue;
        }
        // the pairs of the warp's 32 sources, which are consecutive
        const int64_t p0 = __shfl_sync(0xffffffffu, at[k], 0);
        int64_t p1 = c[k] > 0 ? at[k] + c[k] : 0;
#pragma unroll
        for (int o = 16; o; o >>= 1) p1 = max(p1, __shfl_xor_sync(0xffffffffu, p1, o));
        if (p1 - p0 > kRowsWarp) {
            const int64_t un0 = __shfl_sync(0xffffffffu, un, 0);
            const uint32_t n = (uint32_t)((p1 - p0 + kRowsChunk - 1) / kRowsChunk);
            uint32_t base = 0;
            if (lane == 0) base = atomicAdd(J.n_chunks, n);
            base = __shfl_sync(0xffffffffu, base, 0);
            for (uint32_t j = lane; j < n; j += 32) {
                const int64_t q = p0 + (int64_t)j * kRowsChunk;
                J.chunks[base + j] = PairChunk{q, un0, i - lane, un_mask[k],
                                               (int32_t)min((int64_t)kRowsChunk, p1 - q)};
            }
            continue;
        }
        for (int64_t q = p0; q < p1; q += 32) {
            const int64_t p = q + lane;
            int l = 0;  // the last source whose pairs start at p or before
#pragma unroll
            for (int o = 16; o; o >>= 1)
                if (__shfl_sync(0xffffffffu, at[k], l + o) <= p) l += o;
            const int64_t u = __shfl_sync(0xffffffffu, un, l);
            if (p < p1) {
                const int64_t o = J.with_un_a ? p + u : p;
                J.oa[o] = i - lane + l + J.a_off;
                J.ob[o] = __ldcs(J.pb + p);
                J.os[o] = __ldcs(J.ps + p);
            }
        }
    }
}

// The pair rows of the listed chunks, a block each: 12 us for a region of 1e6
// members among 1e6 small ones, whose join takes 0.088 ms (26 ms with one warp
// for all the pairs of its 32 sources). Where no source has more than
// kRowsThread, no 32 of them have more than kRowsWarp: nothing is launched.
__global__ void __launch_bounds__(kBlock) k_join_long(JoinA J, const int64_t* __restrict__ pa) {
    pdl_wait();
    const unsigned int n = *J.n_chunks;
    for (unsigned int c = blockIdx.x; c < n; c += gridDim.x) {
        const PairChunk C = J.chunks[c];
        int64_t a[4], b[4];
        double v[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const int32_t j = k * kBlock + threadIdx.x;
            if (j < C.n) {
                a[k] = __ldcs(pa + C.p0 + j);
                b[k] = __ldcs(J.pb + C.p0 + j);
                v[k] = __ldcs(J.ps + C.p0 + j);
            }
        }
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const int32_t j = k * kBlock + threadIdx.x;
            if (j >= C.n) break;
            const uint32_t below = (1u << ((uint32_t)(a[k] - C.i0) & 31u)) - 1u;
            const int64_t o = C.p0 + j + (J.with_un_a ? C.un + __popc(C.mask & below) : 0);
            J.oa[o] = a[k] + J.a_off;
            J.ob[o] = b[k];
            J.os[o] = v[k];
        }
    }
}

// The pair rows of the "all" selection, four per thread: pair p of A source a
// goes to row p + un_before[a] (NULL: no unmatched A rows among them).
__global__ void __launch_bounds__(kBlock) k_join_pairs(
    const int64_t* __restrict__ pa, const int64_t* __restrict__ pb, const double* __restrict__ ps,
    int64_t n_pairs, const int32_t* __restrict__ un_before, int64_t a_off, int64_t* __restrict__ oa,
    int64_t* __restrict__ ob, double* __restrict__ os) {
    pdl_wait();
    const int64_t p0 = (int64_t)blockIdx.x * (4 * kBlock) + threadIdx.x;
    int64_t a[4], b[4];
    double v[4];
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const int64_t p = p0 + k * kBlock;
        if (p < n_pairs) {
            a[k] = __ldcs(pa + p);
            b[k] = __ldcs(pb + p);
            v[k] = __ldcs(ps + p);
        }
    }
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const int64_t p = p0 + k * kBlock;
        if (p >= n_pairs) break;
        const int64_t o = un_before ? p + __ldg(un_before + a[k]) : p;
        oa[o] = a[k] + a_off;
        ob[o] = b[k];
        os[o] = v[k];
    }
}

// Unmatched B rows: the bitset in tiles of a word per thread (8192 rows), in
// launch order, with a chained prefix sum; a tile's rows are listed in shared
// memory and leave as 16-byte stores from the A-side rows on (counts[0]).
// counts[1]: their number. Bound by the 24 bytes written per row: 0.65 ms for
// the 1.7e8 rows of an all-sky step (6.2 TB/s) against 1.0 ms with 8-byte
// stores, a thread per B row, after a pass and a prefix sum over the words.
__global__ void __launch_bounds__(kBlock) k_join_b(const uint32_t* __restrict__ bits, int64_t nwords,
                                                   int64_t nB, int64_t* counts, uint64_t* status,
                                                   unsigned int* counter, int64_t* __restrict__ oa,
                                                   int64_t* __restrict__ ob, double* __restrict__ os,
                                                   Lookback lb, int32_t* err) {
    pdl_wait();
    __shared__ JoinTile S;
    __shared__ uint16_t list[32 * kBlock];
    if (threadIdx.x == 0) S.tile = atomicAdd(counter, 1u);
    __syncthreads();
    const int64_t tile = S.tile, w = tile * kBlock + threadIdx.x;
    const uint32_t un = w < nwords ? ~bits[w] & word_valid(w, nB) : 0u;
    uint32_t all;
    const uint32_t at = block_prefix((uint32_t)__popc(un), &all);
    if (threadIdx.x < 32) {
        const int64_t p = lookback_warp(status, tile, (int64_t)all, lb.spin_limit,
                                        tile == lb.silent_tile, err);
        if (threadIdx.x == 0) {
            S.prefix = p;
            if ((tile + 1) * kBlock >= nwords) counts[1] = p + (int64_t)all;
        }
    }
    // lane l lists bit l of the warp's words, one word after the other
    const int lane = threadIdx.x & 31;
    const uint32_t below = (1u << lane) - 1u;
#pragma unroll 4
    for (int k = 0; k < 32; k++) {
        const uint32_t u = __shfl_sync(0xffffffffu, un, k), a = __shfl_sync(0xffffffffu, at, k);
        if ((u >> lane) & 1u)
            list[a + __popc(u & below)] = (uint16_t)(((threadIdx.x & ~31) + k) * 32 + lane);
    }
    __syncthreads();
    const int64_t row0 = tile * (32 * kBlock), o0 = counts[0] + S.prefix;
    const int n = (int)all;
    int head = (int)(o0 & 1);  // (16-byte stores start at even rows)
    if (head > n) head = n;
    const int pairs = (n - head) / 2;
    for (int k = threadIdx.x; k < pairs; k += kBlock) {
        const int e = head + 2 * k;
        const int64_t o = o0 + e;
        *reinterpret_cast<longlong2*>(ob + o) = make_longlong2(row0 + list[e], row0 + list[e + 1]);
        *reinterpret_cast<longlong2*>(oa + o) = make_longlong2(-1, -1);
        *reinterpret_cast<double2*>(os + o) = make_double2(NAN, NAN);
    }
    // the first row before them and the last one after
    const int e = threadIdx.x == 0 && head ? 0 : threadIdx.x == 1 && head + 2 * pairs < n ? n - 1 : -1;
    if (e >= 0) {
        ob[o0 + e] = row0 + list[e];
        oa[o0 + e] = -1;
        os[o0 + e] = NAN;
    }
}

// The number of unmatched B rows alone (counts[1]).
__global__ void __launch_bounds__(kBlock) k_count_b(const uint32_t* __restrict__ bits, int64_t nwords,
                                                    int64_t nB, unsigned long long* n_un) {
    pdl_wait();
    uint32_t un = 0;
    for (int64_t w = (int64_t)blockIdx.x * kBlock + threadIdx.x; w < nwords;
         w += (int64_t)gridDim.x * kBlock)
        un += __popc(~bits[w] & word_valid(w, nB));
    uint32_t all;
    block_prefix(un, &all);
    if (threadIdx.x == 0 && all) atomicAdd(n_un, (unsigned long long)all);
}

}  // namespace
}  // namespace xm

namespace xm {

// ------------------------------------------------ join without allocation
//
// Some callers cannot allocate device memory at the moment they need a join:
// a serving process or a framework whose caching allocator has reserved the
// whole GPU (a cudaMalloc would fail or fragment its pool), or a
// latency-critical loop that must not enter the driver's allocator.
// xm_join_noalloc gives them the join with no allocation at all: the caller
// passes the output arrays, and the scratch lives in one file-scope device
// array sized for results of at most kNoAllocMaxA A rows and kNoAllocMaxB B
// rows. Every GPU that loads the library holds that array (about 16 MB)
// until the process exits.

namespace {

constexpr int64_t kNoAllocMaxA = 1 << 20;  // A rows
constexpr int64_t kNoAllocMaxB = 1 << 23;  // B rows
constexpr int64_t kNoAllocWords = kNoAllocMaxB / 32;

struct JoinScratch {
    uint32_t bits[kNoAllocWords];      // matched B rows
    int32_t rows[kNoAllocMaxA];        // rows per A source
    int64_t row_off[kNoAllocMaxA];
    int32_t wcount[kNoAllocWords];     // unmatched B rows per word
    int64_t word_off[kNoAllocWords];
    int64_t ws_a[2 * (kNoAllocMaxA / 4096)];     // scan workspace (rows)
    int64_t ws_b[2 * (kNoAllocWords / 4096)];    // scan workspace (words)
    int64_t small[4];                  // totals, unmatched A count
};

static __device__ __align__(256) JoinScratch g_join_scratch;

// Device address of the scratch array, looked up once per device with that
// device current (the host-side symbol is not a device address); *dev_out
// is the current device. Thread-safe.
xm_status join_scratch(JoinScratch** out, int* dev_out) {
    static std::mutex mu;
    static JoinScratch* addr[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
    if (dev < 0 || dev >= 64) return set_error(XM_EUNSUPPORTED, "device %d", dev);
    std::lock_guard<std::mutex> g(mu);
    if (!addr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_join_scratch);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(join scratch)");
        addr[dev] = (JoinScratch*)p;
    }
    *out = addr[dev];
    *dev_out = dev;
    return XM_OK;
}

}  // namespace
}  // namespace xm

extern "C" xm_status xm_join_noalloc(const xm_result* R, int32_t selection, int32_t join_type,
                                     int64_t* a_row, int64_t* b_row, double* sep,
                                     int64_t capacity, int64_t* n_rows, void* stream) {
    using namespace xm;
    if (!n_rows) return set_error(XM_EINVAL, "xm_join_noalloc: n_rows is NULL");
    *n_rows = 0;
    if (!R) return set_error(XM_EINVAL, "xm_join_noalloc: NULL result");
    if (selection != XM_SEL_ALL && selection != XM_SEL_BEST)
        return set_error(XM_EINVAL, "xm_join_noalloc: selection must be ALL or BEST");
    if (!(R->selection & selection))
        return set_error(XM_EINVAL, "xm_join_noalloc: selection not computed by xm_match");
    if (join_type < XM_JOIN_AND || join_type > XM_JOIN_XOR)
        return set_error(XM_EINVAL, "xm_join_noalloc: bad join type %d", join_type);
    if (capacity < 0 || (capacity > 0 && (!a_row || !b_row || !sep)))
        return set_error(XM_EINVAL, "xm_join_noalloc: bad output arrays");
    const int64_t nA = R->n_a, nB = R->n_b;
    if (nA > kNoAllocMaxA || nB > kNoAllocMaxB)
        return set_error(XM_EOVERFLOW,
                         "xm_join_noalloc: the result has %lld A rows and %lld B rows; this entry "
                         "point takes at most %lld and %lld (use xm_join)",
                         (long long)nA, (long long)nB, (long long)kNoAllocMaxA,
                         (long long)kNoAllocMaxB);
    const bool with_pairs = join_type == XM_JOIN_AND || join_type == XM_JOIN_OR ||
                            join_type == XM_JOIN_ALL1 || join_type == XM_JOIN_ALL2;
    const bool with_un_a = join_type == XM_JOIN_OR || join_type == XM_JOIN_ALL1 ||
                           join_type == XM_JOIN_NOT1_2 || join_type == XM_JOIN_XOR;
    const bool with_un_b = join_type == XM_JOIN_OR || join_type == XM_JOIN_ALL2 ||
                           join_type == XM_JOIN_NOT2_1 || join_type == XM_JOIN_XOR;
    const int sel_all = selection == XM_SEL_ALL;
    const int64_t nwords = (nB + 31) / 32;
    cudaStream_t s = (cudaStream_t)stream;
    JoinScratch* S = nullptr;
    int dev = -1;
    xm_status st = join_scratch(&S, &dev);
    if (st != XM_OK) return st;
    // the scratch array is the current device's; the result's arrays live on
    // the device it was computed on
    if (dev != R->device)
        return set_error(XM_EINVAL, "xm_join_noalloc: the result belongs to device %d, current is %d",
                         R->device, dev);
    // the array keeps the previous call's contents: clear what starts at zero
    cudaError_t e = cudaMemsetAsync(S->bits, 0, (nwords > 0 ? nwords : 1) * sizeof(uint32_t), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(S->small, 0, sizeof(S->small), s);
    if (e != cudaSuccess) return cuda_fail(e, "xm_join_noalloc memset");
    if (sel_all) {
        if (R->n_pairs > 0) k_mark_b<<<grid_for(R->n_pairs), kBlock, 0, s>>>(R->b_row, R->n_pairs, S->bits);
    } else if (nA > 0) {
        k_mark_b<<<grid_for(nA), kBlock, 0, s>>>(R->best_b, nA, S->bits);
    }
    if (nA > 0)
        k_rows_a<<<grid_cap(nA), kBlock, 0, s>>>(R->count, nA, sel_all, (int)with_pairs,
                                                 (int)with_un_a, S->rows,
                                                 (unsigned long long*)&S->small[2]);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "xm_join_noalloc launch");
    st = exclusive_scan_i32_ws(S->rows, S->row_off, nA, &S->small[0], S->ws_a, s);
    if (st != XM_OK) return st;
    if (nwords > 0)
        k_word_unmatched<<<grid_for(nwords), kBlock, 0, s>>>(S->bits, nwords, nB, S->wcount);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "xm_join_noalloc launch");
    st = exclusive_scan_i32_ws(S->wcount, S->word_off, nwords, &S->small[1], S->ws_b, s);
    if (st != XM_OK) return st;
    int64_t h[4];
    e = cudaMemcpyAsync(h, S->small, sizeof(h), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(e, "xm_join_noalloc sync");
    const int64_t total_a = h[0], un_b = h[1];
    const int64_t n = total_a + (with_un_b ? un_b : 0);
    *n_rows = n;
    if (n > capacity)
        return set_error(XM_EOVERFLOW, "xm_join_noalloc: %lld rows do not fit the capacity %lld",
                         (long long)n, (long long)capacity);
    if (nA > 0)
        k_write_a<<<grid_for(nA), kBlock, 0, s>>>(R->count, R->pair_off, R->b_row, R->sep, R->best_b,
                                                 R->best_sep, S->row_off, nA, sel_all,
                                                 (int)with_pairs, (int)with_un_a, a_row, b_row, sep);
    if (with_un_b && nB > 0)
        k_write_b<<<grid_for(nB), kBlock, 0, s>>>(S->bits, S->word_off, nB, &S->small[0], a_row,
                                                 b_row, sep);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "xm_join_noalloc launch");
    return XM_OK;
}

using namespace xm;

// The rows' memory returns to the pool in the order of the stream they were
// written on, after whatever the caller queued there to read them.
static void free_rows(xm_rows* J) {
    if (!J) return;
    dev_free(J->a_row, J->stream);
    dev_free(J->pending, J->stream);
    delete J;
}

// Reads the counts of a join launched without synchronising (once).
static std::mutex g_rows_mu;

static xm_status resolve_rows(xm_rows* J) {
    std::lock_guard<std::mutex> g(g_rows_mu);
    if (!J->pending) return XM_OK;
    int64_t h[5];
    HostReads rd(J->stream);
    cudaError_t e = rd.add(h, J->pending, sizeof(h));
    if (e == cudaSuccess) e = rd.sync();
    if (e != cudaSuccess) return cuda_fail(e, "xm_rows_get sync");
    if ((int32_t)h[4] & kErrTimeout) return set_error(XM_ETIMEOUT, "xm_join: scan look-back timed out");
    J->n_unmatched_a = h[2];
    J->n_unmatched_b = h[1];
    J->n = h[0] + (J->with_un_b ? h[1] : 0);
    dev_free(J->pending, J->stream);
    J->pending = nullptr;
    return XM_OK;
}

// The rows of one join type over one selection of a result. ext_bits
// (nullable): the matched B rows of a catalogue 1 split over several results
// (the union of their selections), which then decides the unmatched B rows
// instead of this result's own pairs; a_off is added to every A row written;
// with_b: write the B-only rows (else only count them).
static xm_status join_impl(const xm_result* R, int32_t selection, int32_t join_type,
                           const uint32_t* ext_bits, int64_t a_off, bool with_b, void* stream,
                           xm_rows** out, const char* who) {
    if (!out) return set_error(XM_EINVAL, "%s: out is NULL", who);
    *out = nullptr;
    if (!R) return set_error(XM_EINVAL, "%s: NULL result", who);
    if (selection != XM_SEL_ALL && selection != XM_SEL_BEST)
        return set_error(XM_EINVAL, "%s: selection must be ALL or BEST", who);
    if (!(R->selection & selection))
        return set_error(XM_EINVAL, "%s: selection not computed by xm_match", who);
    if (join_type < XM_JOIN_AND || join_type > XM_JOIN_XOR)
        return set_error(XM_EINVAL, "%s: bad join type %d", who, join_type);
    if (a_off < 0) return set_error(XM_EINVAL, "%s: negative A row offset", who);
    const bool with_pairs = join_type == XM_JOIN_AND || join_type == XM_JOIN_OR ||
                            join_type == XM_JOIN_ALL1 || join_type == XM_JOIN_ALL2;
    const bool with_un_a = join_type == XM_JOIN_OR || join_type == XM_JOIN_ALL1 ||
                           join_type == XM_JOIN_NOT1_2 || join_type == XM_JOIN_XOR;
    const bool with_un_b = join_type == XM_JOIN_OR || join_type == XM_JOIN_ALL2 ||
                           join_type == XM_JOIN_NOT2_1 || join_type == XM_JOIN_XOR;
    const bool write_b = with_un_b && with_b;
    const int sel_all = selection == XM_SEL_ALL;
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t nA = R->n_a, nB = R->n_b;
    const int64_t nwords = (nB + 31) / 32;
    xm_rows* J = new (std::nothrow) xm_rows();
    if (!J) return set_error(XM_ENOMEM, "%s: host allocation", who);

    // The A-side pass writes the pair rows too where a source has few of them
    // (0.7 each, 2.5e7 sources: 0.29 ms, 0.53 in two passes); with more than
    // four for each source a pass of its own shares the pairs out evenly (8.4
    // each, 2e5 sources: 26 us in two passes, 48 to 70 in one).
    const bool pair_rows = sel_all && with_pairs && R->n_pairs > 0 && R->a_row;
    const bool apart = pair_rows && R->n_pairs > 4 * nA;
    // Where a few sources have very many, their pairs go to a list: room for
    // two chunks per kRowsChunk pairs, as the listed 32 have more than half.
    const bool many = pair_rows && !apart && (R->max_count == 0 || R->max_count > kRowsThread);
    const bool listed = many && R->n_pairs > kRowsWarp;
    static_assert(2 * kRowsWarp >= kRowsChunk, "chunks of the listed sources fit their list");
    const int64_t max_chunks = listed ? R->n_pairs / kRowsWarp : 0;
    // one work block: the chained sums' status words and tile counters and the
    // matched B rows (all of which start as zeros), then the unmatched A
    // sources before each one, where a pass of its own writes the pair rows, or
    // the list
    const int64_t tiles_a = (nA + kTileA - 1) / kTileA, tiles_b = (nwords + kBlock - 1) / kBlock;
    auto up = [](size_t b) { return (b + 255) & ~size_t(255); };
    const size_t o_bits = up((tiles_a + tiles_b + 2) * sizeof(uint64_t));
    const size_t zeroed = o_bits + (ext_bits ? 0 : up(nwords * sizeof(uint32_t)));
    unsigned char* work = (unsigned char*)dev_alloc(
        zeroed + (apart && with_un_a ? nA * sizeof(int32_t) : max_chunks * sizeof(PairChunk)), s);
    uint64_t* const status = (uint64_t*)work;
    unsigned int* const counter = work ? (unsigned int*)(status + tiles_a + tiles_b) : nullptr;
    uint32_t* const own_bits = ext_bits || !work ? nullptr : (uint32_t*)(work + o_bits);
    const uint32_t* bits = ext_bits ? ext_bits : own_bits;
    int32_t* const un_before = apart && with_un_a && work ? (int32_t*)(work + zeroed) : nullptr;
    PairChunk* const chunks = listed && work ? (PairChunk*)(work + zeroed) : nullptr;
    // counts read later by xm_rows_get: [0] A-side rows, [1] unmatched B,
    // [2] unmatched A, [4] error bits
    int64_t* small = (int64_t*)dev_alloc(5 * sizeof(int64_t), s);
    J->pending = small;
    J->stream = s;
    J->with_un_b = write_b;
    auto body = [&]() -> xm_status {
        if (!work || !small) return set_error(XM_ENOMEM, "%s: work buffers", who);
        cudaError_t e = cudaMemsetAsync(small, 0, 5 * sizeof(int64_t), s);
        if (e == cudaSuccess) e = cudaMemsetAsync(work, 0, zeroed, s);
        if (e != cudaSuccess) return cuda_fail(e, "memset");
        if (own_bits) {
            if (sel_all) {
                if (R->n_pairs > 0)
                    XM_LAUNCH("k_mark_b", grid_for(R->n_pairs), kBlock, 0, s, k_mark_b, R->b_row,
                              R->n_pairs, own_bits);
            } else if (nA > 0) {
                XM_LAUNCH("k_mark_b", grid_for(nA), kBlock, 0, s, k_mark_b, R->best_b, nA, own_bits);
            }
        }
        int32_t* err = (int32_t*)(small + 4);
        // rows are written at device-side offsets into room for the most
        // rows the join can have; the count is read by xm_rows_get
        const int64_t a_side = (with_pairs ? (sel_all ? R->n_pairs : nA) : 0) + (with_un_a ? nA : 0);
        const int64_t bound = a_side + (write_b ? nB : 0);
        int64_t nr = bound > 0 ? (bound + 1) & ~int64_t(1) : 2;  // (even: 16-byte stores)
        J->a_row = (int64_t*)dev_alloc(nr * (2 * sizeof(int64_t) + sizeof(double)), s);
        if (!J->a_row) return set_error(XM_ENOMEM, "%s: %lld rows", who, (long long)bound);
        J->b_row = J->a_row + nr;
        J->sep = (double*)(J->b_row + nr);
        const Lookback lb = lookback_settings();
        if (nA > 0) {
            const JoinA P{R->count, R->pair_off, R->b_row, R->sep, R->best_b, R->best_sep, nA,
                          R->n_pairs, sel_all, with_pairs, with_un_a, a_off, R->zeros,
                          pair_rows && !apart, un_before, chunks, counter + 2, J->a_row, J->b_row,
                          J->sep, small};
            if (many)
                XM_LAUNCH("k_join_a", (unsigned)tiles_a, kBlock, 0, s, k_join_a<true>, P, status,
                          counter, lb, err);
            else
                XM_LAUNCH("k_join_a", (unsigned)tiles_a, kBlock, 0, s, k_join_a<false>, P, status,
                          counter, lb, err);
            if (listed)
                XM_LAUNCH("k_join_long", (unsigned)(max_chunks < 4 * 152 ? max_chunks : 4 * 152),
                          kBlock, 0, s, k_join_long, P, R->a_row);
        }
        if (apart)
            XM_LAUNCH("k_join_pairs", grid_for((R->n_pairs + 3) / 4), kBlock, 0, s, k_join_pairs,
                      R->a_row, R->b_row, R->sep, R->n_pairs, un_before, a_off, J->a_row, J->b_row,
                      J->sep);
        if (write_b && nB > 0)
            XM_LAUNCH("k_join_b", (unsigned)tiles_b, kBlock, 0, s, k_join_b, bits, nwords, nB, small,
                      status + tiles_a, counter + 1, J->a_row, J->b_row, J->sep, lb, err);
        else if (nB > 0)
            XM_LAUNCH("k_count_b", grid_cap(nwords), kBlock, 0, s, k_count_b, bits, nwords, nB,
                      (unsigned long long*)small + 1);
        return XM_OK;
    };
    xm_status st = body();
    dev_free(work, s);
    if (st != XM_OK) {
        free_rows(J);  // (frees the counts too)
        return st;
    }
    *out = J;
    return XM_OK;
}

extern "C" xm_status xm_join(const xm_result* R, int32_t selection, int32_t join_type,
                             void* stream, xm_rows** out) {
    return join_impl(R, selection, join_type, nullptr, 0, true, stream, out, "xm_join");
}

extern "C" xm_status xm_result_mark_b(const xm_result* R, int32_t selection, uint32_t* bits,
                                      void* stream) {
    if (!R || !bits) return set_error(XM_EINVAL, "xm_result_mark_b: NULL argument");
    if (selection != XM_SEL_ALL && selection != XM_SEL_BEST)
        return set_error(XM_EINVAL, "xm_result_mark_b: selection must be ALL or BEST");
    if (!(R->selection & selection))
        return set_error(XM_EINVAL, "xm_result_mark_b: selection not computed by xm_match");
    cudaStream_t s = (cudaStream_t)stream;
    if (selection == XM_SEL_ALL) {
        if (R->n_pairs > 0)
            XM_LAUNCH("k_mark_b", grid_for(R->n_pairs), kBlock, 0, s, k_mark_b, R->b_row,
                      R->n_pairs, bits);
    } else if (R->n_a > 0) {
        XM_LAUNCH("k_mark_b", grid_for(R->n_a), kBlock, 0, s, k_mark_b, R->best_b, R->n_a, bits);
    }
    return XM_OK;
}

extern "C" xm_status xm_join_shard(const xm_result* R, int32_t selection, int32_t join_type,
                                   const uint32_t* b_matched, int64_t a_row_offset,
                                   int32_t with_b_rows, void* stream, xm_rows** out) {
    if (!b_matched) {
        if (out) *out = nullptr;
        return set_error(XM_EINVAL, "xm_join_shard: b_matched is NULL");
    }
    return join_impl(R, selection, join_type, b_matched, a_row_offset, with_b_rows != 0, stream,
                     out, "xm_join_shard");
}

extern "C" xm_status xm_rows_free(xm_rows* J) {
    free_rows(J);
    return XM_OK;
}

extern "C" xm_status xm_rows_get(const xm_rows* J, xm_rows_view* v) {
    if (!J || !v) return set_error(XM_EINVAL, "xm_rows_get: NULL argument");
    const xm_status st = resolve_rows(const_cast<xm_rows*>(J));
    if (st != XM_OK) return st;
    v->n = J->n;
    v->a_row = J->a_row;
    v->b_row = J->b_row;
    v->sep_arcsec = J->sep;
    v->n_unmatched_a = J->n_unmatched_a;
    v->n_unmatched_b = J->n_unmatched_b;
    return XM_OK;
}
