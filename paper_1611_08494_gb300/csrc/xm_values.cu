// xm_values.cu -- the Exact Value functional case (paper §2.1): A_i and B_j
// match when their key columns hold the same value. The result has the
// layout of a positional match (pairs in ascending A row then B row, member
// counts, the best pair = the lowest B row), so the joins of §2.2 apply
// unchanged.
//
//   k_val_key     keys to order-preserving unsigned codes (int64: sign bit
//                 flipped; float64: IEEE total order with -0 folded into +0;
//                 NaN -> all ones, above every number, never looked up), and
//                 the AND / OR of all B codes (bits that never differ need no
//                 sort pass); writes a 32-bit hash of each code and its row,
//                 packed in 64 bits
//   k_val_pack    the same with the codes' low bits, when they differ in no
//                 more than 32
//   radix sort    stable, so equal keys keep ascending B rows (xm_sort.cu), on
//                 the high half of the packed words: one array of 8 bytes a
//                 source. Equal keys form one run, shared under the hash with
//                 the few keys that collide, which B's keys tell apart
//   k_val_lut     a bucket table over the sorted words (one bucket per two
//                 to four keys; long runs of entries by k_val_runs)
//   k_val_probe   per A: the run of equal words, searched inside one bucket;
//                 count, best B row, and that row or the first match's place
//   prefix sum    pair offsets
//   k_val_emit    the pairs of each A row
#include <math.h>

#include <new>

#include "xm_internal.cuh"

namespace xm {
namespace {

constexpr int kBlock = 256;
constexpr uint64_t kNaNCode = ~0ull;

__device__ __forceinline__ uint64_t key_code(const void* keys, int64_t i, int32_t type) {
    if (type == XM_KEY_INT64) return (uint64_t)((const int64_t*)keys)[i] ^ 0x8000000000000000ull;
    double v = ((const double*)keys)[i];
    uint64_t u = (uint64_t)__double_as_longlong(v);
    if ((u & 0x7FFFFFFFFFFFFFFFull) > 0x7FF0000000000000ull) return kNaNCode;  // NaN
    if ((u << 1) == 0) u = 0;  // -0 is +0
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}

// 32-bit hash of a code (the finaliser of the SplitMix64 generator, Steele,
// Lea & Flood 2014, high half): equal codes hash equally, distinct ones
// collide with probability about 2^-32.
__device__ __forceinline__ uint64_t code_hash(uint64_t x) {
    x ^= x >> 30;
    x *= 0xbf58476d1ce4e5b9ull;
    x ^= x >> 27;
    x *= 0x94d049bb133111ebull;
    x ^= x >> 31;
    return x >> 32;
}

// Grid-stride over B (a few blocks per SM), so the AND / OR of all codes
// costs one pair of atomics per block.
__global__ void k_val_key(const void* __restrict__ keys, int64_t n, int32_t type,
                          uint64_t* __restrict__ packed, unsigned long long* __restrict__ and_or) {
    pdl_wait();
    __shared__ unsigned long long s_and, s_or;
    if (threadIdx.x == 0) {
        s_and = ~0ull;
        s_or = 0ull;
    }
    __syncthreads();
    uint64_t c_and = ~0ull, c_or = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t c = key_code(keys, i, type);
        packed[i] = code_hash(c) << 32 | (uint32_t)i;
        c_and &= c;
        c_or |= c;
    }
    for (int s = 16; s > 0; s >>= 1) {
        c_and &= __shfl_xor_sync(0xffffffffu, c_and, s);
        c_or |= __shfl_xor_sync(0xffffffffu, c_or, s);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAnd(&s_and, (unsigned long long)c_and);
        atomicOr(&s_or, (unsigned long long)c_or);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        atomicAnd(&and_or[0], s_and);
        atomicOr(&and_or[1], s_or);
    }
}

// The low bits of the codes instead of their hashes.
__global__ void k_val_pack(const void* __restrict__ keys, int64_t n, int32_t type, uint64_t mask,
                           uint64_t* __restrict__ packed) {
    pdl_wait();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) packed[i] = (key_code(keys, i, type) & mask) << 32 | (uint32_t)i;
}

// Bucket table over the sorted words (word = hash or low code bits, above the
// row): bucket = word >> shift, and lut[k] is the first sorted position whose
// bucket reaches k (lut[nb] = n). Codes share every bit outside mask with
// prefix (unhashed). Runs of entries longer than kRunInline go to a list
// filled by k_val_runs.
struct ValLut {
    uint64_t prefix, mask;  // common high bits, mask of the low end_bit bits
    uint32_t shift, nb;     // bucket shift, buckets
    uint32_t* lut;
};

struct ValRun {
    int64_t first;
    uint32_t count, value;
};

constexpr int64_t kRunInline = 32;

__device__ __forceinline__ uint32_t val_bucket(const ValLut& V, uint64_t packed) {
    return (uint32_t)(packed >> 32) >> V.shift;
}

__global__ void k_val_lut(const uint64_t* __restrict__ sorted, int64_t n, ValLut V,
                          ValRun* __restrict__ runs, unsigned long long* __restrict__ n_runs,
                          long long run_cap, int32_t* err) {
    pdl_wait();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int64_t b = val_bucket(V, sorted[i]);
    const int64_t pb = i == 0 ? -1 : (int64_t)val_bucket(V, sorted[i - 1]);
    auto run = [&](int64_t first, int64_t count, uint32_t value) {
        if (count <= 0) return;
        if (count <= kRunInline) {
            for (int64_t k = 0; k < count; k++) V.lut[first + k] = value;
        } else {
            const unsigned long long g = atomicAdd(n_runs, 1ull);
            if ((long long)g < run_cap) runs[g] = ValRun{first, (uint32_t)count, value};
            else atomicOr(err, kErrOverflow);
        }
    };
    run(pb + 1, b - pb, (uint32_t)i);
    if (i == n - 1) run(b + 1, (int64_t)V.nb - b, (uint32_t)n);
}

__global__ void k_val_runs(const ValRun* __restrict__ runs, const unsigned long long* n_runs,
                           long long run_cap, uint32_t* __restrict__ lut) {
    pdl_wait();
    const long long nr = min((long long)*n_runs, run_cap);
    for (long long r = blockIdx.x; r < nr; r += gridDim.x) {
        const ValRun R = runs[r];
        for (uint32_t k = threadIdx.x; k < R.count; k += blockDim.x) lut[R.first + k] = R.value;
    }
}

// First position in sorted[lo, hi) whose word is >= w (or > w when upper).
__device__ __forceinline__ int64_t bound(const uint64_t* __restrict__ sorted, int64_t lo, int64_t hi,
                                         uint32_t w, bool upper) {
    while (lo < hi) {
        const int64_t mid = lo + ((hi - lo) >> 1);
        const uint32_t v = (uint32_t)(__ldg(&sorted[mid]) >> 32);
        if (upper ? v <= w : v < w) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

constexpr int kProbeRun = 4;  // words of a bucket read at once

// Per A key the B rows of equal keys. Bound by the latency of dependent loads
// (bucket table, bucket, B's key under the hash), which many threads of few
// registers overlap. first: the only match's row, or the place of the first of
// several (k_val_emit then reads no list for most keys: 0.45 ms for 2.5e7
// against 0.81 when each went through its place to a row). 1.46 ms for 2.5e7
// keys among 1e8, and 0.55 for 3e6 keys with 20 matches each among 1e7; with four
// keys per thread 1.73 and 0.94, since a thread then walks four runs one after
// the other, and 1.93 and 1.22 with their walks side by side, whose registers
// halve the threads.
template <bool HASHED>
__global__ void __launch_bounds__(kBlock) k_val_probe(
    const void* __restrict__ a_keys, int64_t n_a, int32_t type, const uint64_t* __restrict__ sorted,
    const void* __restrict__ b_keys, int64_t n_b, ValLut V, int32_t* __restrict__ count,
    int64_t* __restrict__ first, int64_t* __restrict__ best_b, double* __restrict__ best_sep,
    int32_t* max_count) {
    pdl_wait();
    const int64_t i = (int64_t)blockIdx.x * kBlock + threadIdx.x;
    if (i >= n_a) return;
    const uint64_t c = key_code(a_keys, i, type);
    // (NaN never matches; the int64 maximum has the same code and does)
    const bool any = n_b > 0 && !(type == XM_KEY_FLOAT64 && c == kNaNCode) &&
                     (HASHED || (c & ~V.mask) == V.prefix);
    const uint32_t w = (uint32_t)(HASHED ? code_hash(c) : c & V.mask);
    uint32_t lo = any ? __ldg(&V.lut[w >> V.shift]) : 0;
    const uint32_t hi = any ? __ldg(&V.lut[(w >> V.shift) + 1]) : 0;
    if (hi - lo > 2 * kProbeRun) lo = (uint32_t)bound(sorted, lo, hi, w, false);
    uint64_t e[kProbeRun];
#pragma unroll
    for (int j = 0; j < kProbeRun; j++) e[j] = lo + j < hi ? __ldg(&sorted[lo + j]) : 0;
    int at = -1;  // the first word equal to w among those read, or -1
    uint32_t row = 0;
#pragma unroll
    for (int j = kProbeRun - 1; j >= 0; j--)
        if (lo + j < hi && (uint32_t)(e[j] >> 32) == w) {
            at = j;
            row = (uint32_t)e[j];
        }
    bool known = at >= 0;  // (the first word's key is compared before the walk)
    const bool eq = known && (!HASHED || key_code(b_keys, row, type) == c);
    uint32_t p = known ? lo + at : hi;  // the first word equal to w, or one past those below it
    if (!known && hi - lo > kProbeRun && (uint32_t)(e[kProbeRun - 1] >> 32) < w)
        p = (uint32_t)bound(sorted, lo + kProbeRun, hi, w, false);
    uint32_t m = 0, f = 0;
    int64_t best = -1;
    for (; p < hi; p++) {
        const uint32_t j = p - lo;
        uint64_t v = 0;
        if (j < kProbeRun) {
#pragma unroll
            for (int q = 0; q < kProbeRun; q++) v = q == j ? e[q] : v;
        } else {
            v = __ldg(&sorted[p]);
        }
        if ((uint32_t)(v >> 32) != w) break;
        const uint32_t r = (uint32_t)v;
        const bool match = known ? eq : !HASHED || key_code(b_keys, r, type) == c;
        known = false;
        if (!match) continue;
        if (m == 0) {
            best = r;
            f = p;
        }
        m++;
        if (!HASHED && p - f >= 2 * kProbeRun) {  // a long run of equal keys
            m = (uint32_t)bound(sorted, p, hi, w, true) - f;
            break;
        }
    }
    const int32_t c32 = (int32_t)m;  // (there are at most 2^31 - 1 rows)
    count[i] = c32;
    if (c32 > kRowsThread && c32 > *(volatile const int32_t*)max_count) atomicMax(max_count, c32);
    first[i] = m == 1 ? best : (int64_t)f;
    if (best_b) {
        best_b[i] = best;
        best_sep[i] = m > 0 ? 0.0 : NAN;
    }
}

template <bool HASHED>
__global__ void k_val_emit(const void* __restrict__ a_keys, int32_t type,
                           const int32_t* __restrict__ count, const int64_t* __restrict__ first,
                           const int64_t* __restrict__ pair_off, const uint64_t* __restrict__ sorted,
                           const void* __restrict__ b_keys, int64_t n_a, int64_t* __restrict__ pa,
                           int64_t* __restrict__ pb, double* __restrict__ ps) {
    pdl_wait();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_a) return;
    const int32_t c = count[i];
    if (c == 0) return;
    const int64_t o = pair_off[i], f = first[i];
    if (c == 1) {
        pa[o] = i;
        pb[o] = f;
        ps[o] = 0.0;
        return;
    }
    const uint64_t code = HASHED ? key_code(a_keys, i, type) : 0;
    int32_t k = 0;
    for (int64_t p = f; k < c; p++) {  // (the run holds all c matches)
        const uint32_t r = (uint32_t)sorted[p];
        if (HASHED && key_code(b_keys, r, type) != code) continue;
        pa[o + k] = i;
        pb[o + k] = r;
        ps[o + k] = 0.0;
        k++;
    }
}

unsigned grid_of(int64_t n) { return (unsigned)((n + kBlock - 1) / kBlock); }

int top_bit(uint64_t x) {
    int b = 0;
    while (x) { b++; x >>= 1; }
    return b;
}

}  // namespace
}  // namespace xm

using namespace xm;

extern "C" xm_status xm_match_values(const void* a_keys, int64_t n_a, const void* b_keys,
                                     int64_t n_b, int32_t key_type, int32_t on_device,
                                     int32_t selection, void* stream, xm_result** out) {
    if (!out) return set_error(XM_EINVAL, "xm_match_values: out is NULL");
    *out = nullptr;
    if (n_a < 0 || n_b < 0 || n_a > 2147483647LL || n_b > 2147483647LL ||
        (n_a > 0 && !a_keys) || (n_b > 0 && !b_keys))
        return set_error(XM_EINVAL, "xm_match_values: bad key columns");
    if (key_type != XM_KEY_INT64 && key_type != XM_KEY_FLOAT64)
        return set_error(XM_EINVAL, "xm_match_values: bad key type %d", key_type);
    if (selection < 1 || selection > 3)
        return set_error(XM_EINVAL, "xm_match_values: bad selection %d", selection);
    cudaStream_t s = (cudaStream_t)stream;
    xm_result* R = new (std::nothrow) xm_result();
    if (!R) return set_error(XM_ENOMEM, "xm_match_values: host allocation");
    R->stream = (cudaStream_t)stream;
    cudaGetDevice(&R->device);
    R->selection = selection;
    R->precision = XM_PREC_FP64;
    R->shape = -1;
    R->n_a = n_a;
    R->n_b = n_b;
    const int64_t na1 = n_a > 0 ? n_a : 1, nb1 = n_b > 0 ? n_b : 1;
    const bool want_best = (selection & XM_SEL_BEST) != 0;
    R->count = (int32_t*)dev_alloc(na1 * sizeof(int32_t), s);
    const int64_t sum_words = count_scan_words(n_a);
    R->pair_off = (int64_t*)dev_alloc((na1 + sum_words) * sizeof(int64_t), s);
    R->zeros = R->pair_off && sum_words ? R->pair_off + na1 : nullptr;
    if (want_best) {
        R->best_b = (int64_t*)dev_alloc(na1 * (sizeof(int64_t) + sizeof(double)), s);
        R->best_sep = R->best_b ? (double*)(R->best_b + na1) : nullptr;
    }
    // temporaries: host key copies, codes and rows (and sort scratch), first
    // positions, totals and the error word
    void* d_a = nullptr;
    void* d_b = nullptr;
    uint64_t* packed = (uint64_t*)dev_alloc(2 * nb1 * sizeof(uint64_t), s);
    int64_t* first = (int64_t*)dev_alloc(na1 * sizeof(int64_t), s);
    unsigned long long* small = (unsigned long long*)dev_alloc(5 * sizeof(unsigned long long), s);
    uint32_t* lut = nullptr;
    ValRun* runs = nullptr;
    auto body = [&]() -> xm_status {
        if (!R->count || !R->pair_off || (want_best && !R->best_b) || !packed || !first || !small)
            return set_error(XM_ENOMEM, "xm_match_values: work buffers");
        cudaError_t e;
        const void* ak = a_keys;
        const void* bk = b_keys;
        if (!on_device) {
            d_a = dev_alloc(na1 * 8, s);
            d_b = dev_alloc(nb1 * 8, s);
            if (!d_a || !d_b) return set_error(XM_ENOMEM, "xm_match_values: key copies");
            e = n_a ? cudaMemcpyAsync(d_a, a_keys, n_a * 8, cudaMemcpyHostToDevice, s) : cudaSuccess;
            if (e == cudaSuccess && n_b)
                e = cudaMemcpyAsync(d_b, b_keys, n_b * 8, cudaMemcpyHostToDevice, s);
            if (e != cudaSuccess) return cuda_fail(e, "xm_match_values: key copies");
            ak = d_a;
            bk = d_b;
        }
        // small: [0] AND of codes, [1] OR, [2] pair total, [3] error bits, [4]
        // largest count above kRowsThread
        const unsigned long long init[5] = {~0ull, 0ull, 0ull, 0ull, 0ull};
        e = cudaMemcpyAsync(small, init, sizeof(init), cudaMemcpyHostToDevice, s);
        if (e != cudaSuccess) return cuda_fail(e, "xm_match_values: init");
        int32_t* err = (int32_t*)(small + 3);
        if (n_b > 0) {
            const unsigned gk = grid_of(n_b) < 8 * 152 ? grid_of(n_b) : 8 * 152;
            XM_LAUNCH("k_val_key", gk, kBlock, 0, s, k_val_key, bk, n_b, key_type, packed, small);
        }
        unsigned long long h_ao[2] = {~0ull, 0ull};
        e = cudaMemcpyAsync(h_ao, small, sizeof(h_ao), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return cuda_fail(e, "xm_match_values sync");
        // bits where the codes differ: the sort covers only those, or the
        // 32 bits of the hash when there are more
        const int code_bits = top_bit(h_ao[0] ^ h_ao[1]);
        const bool hashed = code_bits > 32;
        const int end_bit = hashed ? 32 : code_bits;
        if (n_b > 0 && !hashed)
            XM_LAUNCH("k_val_pack", grid_of(n_b), kBlock, 0, s, k_val_pack, bk, n_b, key_type,
                      (1ull << end_bit) - 1, packed);
        if (n_b > 1 && end_bit > 0) {
            xm_status r = radix_sort_u64(packed, nullptr, packed + nb1, nullptr, n_b, 32, 32 + end_bit,
                                         err, s);
            if (r != XM_OK) return r;
        }
        // bucket table: about one bucket per 2-4 keys over the differing bits
        ValLut V{};
        V.mask = end_bit >= 64 ? ~0ull : ((1ull << end_bit) - 1);
        V.prefix = hashed ? 0ull : (h_ao[0] & ~V.mask);
        int lg = top_bit((uint64_t)nb1) - 2;
        lg = lg < 1 ? 1 : (lg > 28 ? 28 : lg);
        if (lg > end_bit) lg = end_bit > 0 ? end_bit : 0;
        V.shift = (uint32_t)(end_bit - lg);
        V.nb = 1u << lg;
        lut = (uint32_t*)dev_alloc(((size_t)V.nb + 1) * sizeof(uint32_t), s);
        const long long run_cap = (long long)(V.nb + 1) / (kRunInline + 1) + 16;
        runs = (ValRun*)dev_alloc(run_cap * sizeof(ValRun) + 16, s);
        if (!lut || !runs) return set_error(XM_ENOMEM, "xm_match_values: bucket table");
        V.lut = lut;
        unsigned long long* n_runs = (unsigned long long*)(runs + run_cap);
        e = cudaMemsetAsync(n_runs, 0, sizeof(unsigned long long), s);
        if (e != cudaSuccess) return cuda_fail(e, "xm_match_values: memset");
        if (n_b > 0) {
            XM_LAUNCH("k_val_lut", grid_of(n_b), kBlock, 0, s, k_val_lut, packed, n_b, V, runs,
                      n_runs, run_cap, err);
            XM_LAUNCH("k_val_runs", 4 * 152, kBlock, 0, s, k_val_runs, runs, n_runs, run_cap, lut);
        }
        const unsigned gp = grid_of(n_a);
        if (n_a > 0 && hashed)
            XM_LAUNCH("k_val_probe", gp, kBlock, 0, s, k_val_probe<true>, ak, n_a, key_type, packed, bk,
                      n_b, V, R->count, first, R->best_b, R->best_sep, (int32_t*)(small + 4));
        else if (n_a > 0)
            XM_LAUNCH("k_val_probe", gp, kBlock, 0, s, k_val_probe<false>, ak, n_a, key_type, packed, bk,
                      n_b, V, R->count, first, R->best_b, R->best_sep, (int32_t*)(small + 4));
        xm_status r = R->zeros ? count_scan(R->count, R->pair_off, n_a, (int64_t*)(small + 2), R->zeros, s)
                               : exclusive_scan_i32(R->count, R->pair_off, n_a, (int64_t*)(small + 2),
                                                    err, s);
        if (r != XM_OK) return r;
        unsigned long long h[3] = {0, 0, 0};
        e = cudaMemcpyAsync(h, small + 2, sizeof(h), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return cuda_fail(e, "xm_match_values sync");
        if ((int32_t)h[1] & kErrTimeout) return set_error(XM_ETIMEOUT, "xm_match_values: look-back timed out");
        if ((int32_t)h[1] & kErrOverflow) return set_error(XM_ECUDA, "xm_match_values: run list overflow");
        R->max_count = h[2] ? (int32_t)h[2] : kRowsThread;
        R->n_pairs = (selection & XM_SEL_ALL) ? (int64_t)h[0] : 0;
        if (selection & XM_SEL_ALL) {
            const int64_t np = R->n_pairs > 0 ? R->n_pairs : 1;
            R->a_row = (int64_t*)dev_alloc(np * (2 * sizeof(int64_t) + sizeof(double)), s);
            if (!R->a_row) return set_error(XM_ENOMEM, "xm_match_values: %lld pairs", (long long)R->n_pairs);
            R->b_row = R->a_row + np;
            R->sep = (double*)(R->b_row + np);
            if (n_a > 0 && hashed)
                XM_LAUNCH("k_val_emit", grid_of(n_a), kBlock, 0, s, k_val_emit<true>, ak, key_type,
                          R->count, first, R->pair_off, packed, bk, n_a, R->a_row, R->b_row, R->sep);
            else if (n_a > 0)
                XM_LAUNCH("k_val_emit", grid_of(n_a), kBlock, 0, s, k_val_emit<false>, ak, key_type,
                          R->count, first, R->pair_off, packed, bk, n_a, R->a_row, R->b_row, R->sep);
        }
        return XM_OK;
    };
    const xm_status st = body();
    dev_free(d_a, s);
    dev_free(d_b, s);
    dev_free(packed, s);
    dev_free(first, s);
    dev_free(small, s);
    dev_free(lut, s);
    dev_free(runs, s);
    if (st != XM_OK) {
        xm_result_free(R);
        return st;
    }
    *out = R;
    return XM_OK;
}
