// xm_index.cu -- the resident index of the second catalogue (paper §2.3).
//
// The paper files every source of the second catalogue under a sky cell so a
// source of the first catalogue need only look at nearby cells. Here the
// partition is a set of equal-height declination zones cut into RA buckets.
// Within a bucket the order of the sources is free, so the build is not a
// sort but a partition that ends in shared memory: it reads and writes a
// source's 16-byte record two or three times.
//   k_zone_geom    per zone: sin/cos of its centre, number and width of RA
//                  cells (once per device and zone count)
//   k_zone_count   sources of each zone
//   k_zone_bins    (large catalogues) first row of each zone; bins of
//                  consecutive zones holding a few hundredths of the rows
//   k_ingest_b     validity, fixed-point position, the record (float32
//                  offsets in its cell, RA key, row), exact position kept by
//                  row; records leave grouped by bin
//   k_unit_b       float64 unit vectors by row, for a float64 index
//   k_zone_parts   (large catalogues) zones of many sources cut into RA parts
//   k_cell_count   (large catalogues) sources of each cell: zone or part
//   k_cell_units   first row of each cell; units of consecutive cells that
//                  fit one block's shared memory
//   k_split        (large catalogues) records of a bin grouped by unit
//   k_place_b      per unit: RA buckets counted in shared memory, the zones'
//                  bucket tables and the records in bucket order written
//   k_place_giant  the same for the units of very many rows, a cluster each
// Up to some 4e5 sources the bins are the units themselves and the
// steps marked "large catalogues" are left out.
#include <cooperative_groups.h>
#include <math.h>
#include <string.h>

#include <mutex>
#include <new>
#include <vector>

#include "xm_lookback.cuh"
#include "xm_plan.cuh"

namespace xm {

namespace {

constexpr int kBlock = 256;

// Zones of more than kPartMin sources are cut into parts of half of kPartRows
// to kPartRows on average, so nearly every unit (xm_plan.cuh) fits the stage.
// (Unstaged, a block per zone reading its records twice from L2, the placing
// of 2e8 records took 2.3 ms in zones of 7400 and 4 to 5 ms in zones of 22000
// and more, whose records no longer stay in L2.)
constexpr uint32_t kPartMin = 896, kPartRows = 800;

// Three blocks of 384 threads an SM, 3072 records a tile. Bound by latency and
// instruction issue (all-sky index, 2e8 sources: ingest 2.90 ms, second split
// 2.20 ms, at 0.4 of the copy bandwidth by their 48 and 32 bytes a source); two
// blocks of 512 with 4096 records measured within 7 % of it.
constexpr int kSplitThreads = 384;
constexpr int kTileItems = 8;
constexpr int kTile = kSplitThreads * kTileItems;  // records of a tile
constexpr int kCursorStep = 8;   // cursors lie 32 bytes apart: on one cache line
                                 // they slowed each other down 5 to 10 times
constexpr int kCellSlots = 4096;  // cells of a bin counted in shared memory
constexpr int kCountChunk = 8;    // tiles a k_cell_count block takes
constexpr size_t kCountSmem = 220 * 1024;  // k_zone_count's counters at most

__global__ void k_zone_geom(int32_t nz, ZoneGeo* __restrict__ geo) {
    pdl_wait();
    const int32_t z = blockIdx.x * blockDim.x + threadIdx.x;
    if (z >= nz) return;
    const double h = kPi / nz;
    const double lo = -kHalfPi + z * h;
    const double hi = lo + h;
    double sin_c, cos_c;
    sincos(-kHalfPi + (z + 0.5) * h, &sin_c, &cos_c);
    // widest edge of the zone: its cells are at most h wide there
    const double cos_edge = (lo <= 0.0 && hi >= 0.0) ? 1.0 : cos(fmin(fabs(lo), fabs(hi)));
    double nb = ceil(kTwoPi * cos_edge / h);
    if (nb < 1) nb = 1;
    if (nb > 1073741824.0) nb = 1073741824.0;
    ZoneGeo Z;
    Z.sin_cf = (float)sin_c;
    Z.cos_cf = (float)cos_c;
    Z.binw_f = (float)(kTwoPi / nb);
    Z.nbins = (uint32_t)nb;
    geo[z] = Z;
}

__device__ __forceinline__ ZoneGeo load_geo(const ZoneGeo* p) {
    const uint4 u = __ldg(reinterpret_cast<const uint4*>(p));
    ZoneGeo Z;
    Z.sin_cf = __uint_as_float(u.x);
    Z.cos_cf = __uint_as_float(u.y);
    Z.binw_f = __uint_as_float(u.z);
    Z.nbins = u.w;
    return Z;
}

// What the ingest reads of a source's zone, in one load: the geometry, and
// above the RA cells (fewer than 2^21: zones are at least 1 arcsec high) the
// digit of the first split, a bin or a unit.
constexpr int kDigitShift = 21;
static_assert(kMaxUnits <= 1 << (32 - kDigitShift), "a digit fits above the RA cells");

__device__ __forceinline__ void write_zone_in(const ZoneGeo* geo, uint4* zin, int64_t z, uint32_t digit) {
    uint4 u = __ldg(reinterpret_cast<const uint4*>(geo + z));
    u.w |= digit << kDigitShift;
    zin[z] = u;
}

// A latitude the index accepts (the others count as 0 and fail the call). A
// source's zone depends on its latitude alone, valid longitude or not, so that
// the counts hold for every row.
__device__ __forceinline__ double lat_or_zero(double lat) {
    const uint64_t b = (uint64_t)__double_as_longlong(lat) & 0x7FFFFFFFFFFFFFFFull;
    return keep_or_zero(lat, b <= 0x4056800000000000ull);  // bits of 90.0
}

__device__ __forceinline__ bool build_failed(const int32_t* err) {
    return (*(const volatile int32_t*)err & kErrTimeout) != 0;
}

// Sources per zone. WIDE 0: counters in global memory (few sources, or more
// zones than shared memory holds counters for), one atomic for a warp whose
// sources share a zone; 1: a 32-bit counter per zone in shared memory; 2: 16-bit
// counters, two a word, folded into the global ones by the thread whose source
// takes one to 0x8000. A barrier every kFoldLoops loads bounds what is added
// before that thread's subtraction. On 2e8 sources in 27,000 zones the shared
// form takes 0.54 ms (0.24 by the 8 bytes it reads per source), global atomics
// 2.1 ms.
template <int WIDE>
__global__ void __launch_bounds__(kCountThreads) k_zone_count(const double* __restrict__ lat, int64_t n,
                                                     int32_t nz, uint32_t* __restrict__ zcnt) {
    pdl_wait();
    extern __shared__ uint32_t h[];
    if (WIDE) {
        for (int i = threadIdx.x; i < (WIDE == 1 ? nz : (nz + 1) / 2); i += blockDim.x) h[i] = 0;
        __syncthreads();
    }
    const int64_t step = (int64_t)gridDim.x * kCountThreads;
    int loads = 0;
    for (int64_t b0 = (int64_t)blockIdx.x * kCountThreads; b0 < n; b0 += kCountLoads * step) {
        const int64_t i0 = b0 + threadIdx.x;
        double la[kCountLoads];
#pragma unroll
        for (int k = 0; k < kCountLoads; k++) la[k] = i0 + k * step < n ? lat[i0 + k * step] : 0.0;
#pragma unroll
        for (int k = 0; k < kCountLoads; k++) {
            const int32_t z = zone_of_lat(lat_or_zero(la[k]), nz);
            if (WIDE == 0) {
                const bool on = i0 + k * step < n;
                if (__all_sync(0xffffffffu, on && z == __shfl_sync(0xffffffffu, z, 0))) {
                    if ((threadIdx.x & 31) == 0) atomicAdd(&zcnt[z], 32u);
                } else if (on) {
                    atomicAdd(&zcnt[z], 1u);
                }
                continue;
            }
            if (i0 + k * step >= n) break;
            if (WIDE == 1) {
                atomicAdd(&h[z], 1u);
            } else {
                const int sh = 16 * (z & 1);
                if (((atomicAdd(&h[z >> 1], 1u << sh) >> sh) & 0xFFFFu) == 0x7FFFu) {
                    atomicSub(&h[z >> 1], 0x8000u << sh);
                    atomicAdd(&zcnt[z], 0x8000u);
                }
            }
        }
        if (WIDE == 2 && ++loads % kFoldLoops == 0) __syncthreads();
    }
    if (!WIDE) return;
    __syncthreads();
    for (int z = threadIdx.x; z < nz; z += blockDim.x) {
        const uint32_t v = WIDE == 1 ? h[z] : (h[z >> 1] >> (16 * (z & 1))) & 0xFFFFu;
        if (v) atomicAdd(&zcnt[z], v);
    }
}

// ---- prefix sums over zones and cells (256 threads x 4 elements a tile)

constexpr int kPreItems = 4;
constexpr int kPreTile = kBlock * kPreItems;

struct PreTile {
    int64_t warp_tot[kBlock / 32];
    int64_t prefix;
    unsigned int tile;
};

__device__ __forceinline__ int64_t take_tile(PreTile& S, unsigned int* counter) {
    if (threadIdx.x == 0) S.tile = atomicAdd(counter, 1u);
    __syncthreads();
    return S.tile;
}

// Exclusive prefix of v[0] of this thread over the block (thread t holds
// elements 4t .. 4t + 3, v their values) and the block's total.
__device__ __forceinline__ int64_t block_prefix(PreTile& S, const int64_t* v, int64_t* all) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t sum = 0;
#pragma unroll
    for (int k = 0; k < kPreItems; k++) sum += v[k];
    int64_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) S.warp_tot[warp] = incl;
    __syncthreads();
    int64_t woff = 0, tot = 0;
#pragma unroll
    for (int w = 0; w < kBlock / 32; w++) {
        if (w < warp) woff += S.warp_tot[w];
        tot += S.warp_tot[w];
    }
    __syncthreads();
    *all = tot;
    return woff + incl - sum;
}

// The same over the whole grid.
__device__ __forceinline__ int64_t tile_prefix(PreTile& S, int64_t tile, const int64_t* v,
                                               uint64_t* status, Lookback lb, int32_t* err) {
    int64_t all;
    const int64_t mine = block_prefix(S, v, &all);
    if (threadIdx.x < 32) {
        const int64_t p = lookback_warp(status, tile, all, lb.spin_limit, tile == lb.silent_tile, err);
        if (threadIdx.x == 0) S.prefix = p;
    }
    __syncthreads();
    return S.prefix + mine;
}

// Calls f(i, lo, a, b, c) for every i of each lane's [lo, hi): a lane its own
// few, the whole warp those of a lane with many (a zone of thousands of parts
// kept one thread busy for 0.37 ms; dozens, as a lane each has in a dense
// catalogue, are faster its own). Called by whole warps.
template <typename F>
__device__ __forceinline__ void warp_fill(uint32_t lo, uint32_t hi, uint32_t a, uint32_t b, uint32_t c,
                                          F&& f) {
    constexpr uint32_t kFew = 128;
    const bool many = hi > lo && hi - lo > kFew;
    if (!many)
        for (uint32_t i = lo; i < hi; i++) f(i, lo, a, b, c);
    uint32_t todo = __ballot_sync(0xffffffffu, many);
    while (todo) {
        const int l = __ffs(todo) - 1;
        todo &= todo - 1;
        const uint32_t l0 = __shfl_sync(0xffffffffu, lo, l), l1 = __shfl_sync(0xffffffffu, hi, l);
        const uint32_t la = __shfl_sync(0xffffffffu, a, l), lb = __shfl_sync(0xffffffffu, b, l),
                       lc = __shfl_sync(0xffffffffu, c, l);
        for (uint32_t i = l0 + (threadIdx.x & 31); i < l1; i += 32) f(i, l0, la, lb, lc);
    }
}

// First row of each zone, and the bins of the first split (two splits):
// zones whose first rows share row >> kb, and whose numbers share
// z >> kBinZoneBits.
__global__ void __launch_bounds__(kBlock) k_zone_bins(
    const uint32_t* __restrict__ zcnt, int32_t nz, int64_t n, int kb,
    const ZoneGeo* __restrict__ geo, uint4* __restrict__ zin, uint32_t* __restrict__ bin_start, uint32_t* __restrict__ bin_zone, uint32_t* __restrict__ bcur,
    int32_t nbins, uint64_t* status, unsigned int* counter, Lookback lb, int32_t* err) {
    pdl_wait();
    __shared__ PreTile S;
    const int64_t tile = take_tile(S, counter);
    const int64_t z0 = tile * kPreTile + threadIdx.x * kPreItems;
    int64_t v[kPreItems];
#pragma unroll
    for (int k = 0; k < kPreItems; k++) v[k] = z0 + k < nz ? zcnt[z0 + k] : 0;
    int64_t start = tile_prefix(S, tile, v, status, lb, err);
    int64_t before = z0 > 0 && z0 < nz ? start - zcnt[z0 - 1] : 0;
#pragma unroll
    for (int k = 0; k < kPreItems; k++) {
        const int64_t z = z0 + k;
        if (z >= nz) break;
        const int32_t b = (int32_t)(start >> kb) + (int32_t)(z >> kBinZoneBits);
        const int32_t bp = z == 0 ? -1 : (int32_t)(before >> kb) + (int32_t)((z - 1) >> kBinZoneBits);
        write_zone_in(geo, zin, z, (uint32_t)b);
        for (int32_t i = bp + 1; i <= b && i < nbins; i++) {  // (ids before b without a zone: empty)
            bin_start[i] = (uint32_t)start;
            bin_zone[i] = (uint32_t)z;
            bcur[i * kCursorStep] = (uint32_t)start;
        }
        if (z == nz - 1)
            for (int32_t i = b + 1; i <= nbins; i++) {
                bin_start[i] = (uint32_t)n;
                if (i < nbins) bin_zone[i] = 0;
            }
        before = start;
        start += v[k];
    }
}

// What the ingest narrows: the range of the top 16 bits of the RA key, as
// maxima (of 65535 - key and of key) so that zeroed memory is the empty range.
struct KeyRange {
    uint32_t not_min, max;
};

// Zone z's cells: its parts are (key >> (16 + shift)) - p0, cell first + part.
struct __align__(16) ZoneCells {
    uint32_t first;  // first cell
    uint32_t parts;
    uint32_t p0;
    uint32_t shift;  // RA bits (of the top 16) below a part number
};

__device__ __forceinline__ ZoneCells load_cells(const ZoneCells* p) {
    const uint4 u = __ldg(reinterpret_cast<const uint4*>(p));
    return ZoneCells{u.x, u.y, u.z, u.w};
}

__device__ __forceinline__ uint32_t cell_of(const ZoneCells& Z, uint32_t ra_key) {
    return Z.first + ((ra_key >> kIndexRaShift) >> Z.shift) - Z.p0;
}

// Zones of many sources into RA parts; the last block lays out the tiles of
// the second split and the chunks of the cell count (those of the bins before
// it, per bin).
__global__ void __launch_bounds__(kBlock) k_zone_parts(
    const uint32_t* __restrict__ zcnt, int32_t nz, const KeyRange* range,
    ZoneCells* __restrict__ zcells, uint32_t* __restrict__ cell_zone,
    uint32_t* __restrict__ cell_split, uint32_t cells_cap, uint32_t* n_cells,
    const uint32_t* __restrict__ bin_start, int32_t nbins, uint32_t* __restrict__ bin_tile,
    uint32_t* __restrict__ bin_chunk,
    uint64_t* status, unsigned int* counter, Lookback lb, int32_t* err) {
    pdl_wait();
    if (build_failed(err)) return;
    __shared__ PreTile S;
    if (blockIdx.x == gridDim.x - 1) {  // (takes no tile)
        static_assert(kMaxBins <= kPreTile, "a thread holds kPreItems bins");
        for (int which = 0; which < 2; which++) {
            const uint32_t rows = which ? kCountChunk * kTile : kTile;
            uint32_t* out = which ? bin_chunk : bin_tile;
            int64_t v[kPreItems], all;
#pragma unroll
            for (int k = 0; k < kPreItems; k++) {
                const int b = threadIdx.x * kPreItems + k;
                v[k] = b < nbins ? (bin_start[b + 1] - bin_start[b] + rows - 1) / rows : 0;
            }
            int64_t run = block_prefix(S, v, &all);
#pragma unroll
            for (int k = 0; k < kPreItems; k++) {
                const int b = threadIdx.x * kPreItems + k;
                if (b < nbins) out[b] = (uint32_t)run;
                run += v[k];
            }
            if (threadIdx.x == 0) out[nbins] = (uint32_t)all;
        }
        return;
    }
    const int64_t tile = take_tile(S, counter);
    const int64_t z0 = tile * kPreTile + threadIdx.x * kPreItems;
    const uint32_t kmin = 65535u - range->not_min, kmax = range->max;
    const uint64_t width = kmax >= kmin ? kmax - kmin + 1 : 1;
    uint32_t sh[kPreItems];
    int64_t v[kPreItems];  // cells, and above bit 31 the unit boundaries of parts
#pragma unroll
    for (int k = 0; k < kPreItems; k++) {
        const uint32_t m = z0 + k < nz ? zcnt[z0 + k] : 0;
        uint32_t s = 16, parts = 1;
        if (m > kPartMin) {
            s = 0;
            while (s < 16 && ((uint64_t)m << (s + 1)) <= kPartRows * width) s++;
            parts = (kmax >> s) - (kmin >> s) + 1;
            if (parts == 1) s = 16;
        }
        sh[k] = s;
        v[k] = z0 + k < nz ? (int64_t)parts + (parts > 1 ? (int64_t)(parts + 1) << 31 : 0) : 0;
    }
    int64_t run = tile_prefix(S, tile, v, status, lb, err);
#pragma unroll
    for (int k = 0; k < kPreItems; k++) {
        const int64_t z = z0 + k;
        const uint32_t first = (uint32_t)(run & 0x7FFFFFFF), split = (uint32_t)(run >> 31);
        const uint32_t parts = (uint32_t)(v[k] & 0x7FFFFFFF);  // (0 past the zones)
        if (parts) zcells[z] = ZoneCells{first, parts, parts > 1 ? kmin >> sh[k] : 0, sh[k]};
        warp_fill(first, first + parts, (uint32_t)z, split, parts > 1,
                  [&](uint32_t c, uint32_t c0, uint32_t zc, uint32_t sp, uint32_t many) {
                      if (c >= cells_cap) return;
                      cell_zone[c] = zc;
                      // parts are units of their own: each part (marked in the
                      // top bit), and the zone after them, starts a unit
                      cell_split[c] = many ? (sp + (c - c0) + 1) | 0x80000000u : sp;
                  });
        run += v[k];
        if (z == nz - 1) *n_cells = min((uint32_t)(run & 0x7FFFFFFF), cells_cap);
    }
}

// First row of each cell and the units. A cell is a zone when cell_zone is
// NULL (the cells are then the zones, in order, and the ingest splits by unit:
// zin).
__global__ void __launch_bounds__(kBlock) k_cell_units(
    const uint32_t* __restrict__ cnt, uint32_t n_cells, const uint32_t* n_cells_dev,
    const uint32_t* __restrict__ cell_zone, const uint32_t* __restrict__ cell_split, int64_t n,
    const ZoneGeo* __restrict__ geo, uint4* __restrict__ zin, uint32_t* __restrict__ cell_start,
    uint32_t* __restrict__ cell_unit,
    uint4* __restrict__ unit, uint32_t* __restrict__ ucur, uint32_t unit_cap,
    uint32_t* n_units, uint64_t* status, unsigned int* counter, Lookback lb, int32_t* err) {
    pdl_wait();
    if (n_cells_dev) {
        if (build_failed(err)) return;
        n_cells = *n_cells_dev;
    }
    __shared__ PreTile S;
    // a cell's rows, and above bit 31 whether it begins a unit by its size
    // (a part does so anyway)
    auto sums = [&](int64_t c) {
        const uint32_t m = cnt[c];
        const bool wide = m > (1u << kUnitRowBits) && !(cell_split && cell_split[c] >> 31);
        return (int64_t)m | (wide ? 1ll << 31 : 0);
    };
    const int64_t tile = take_tile(S, counter);
    if (tile * kPreTile >= n_cells) return;
    const int64_t c0 = tile * kPreTile + threadIdx.x * kPreItems;
    int64_t v[kPreItems];
#pragma unroll
    for (int k = 0; k < kPreItems; k++) v[k] = c0 + k < n_cells ? sums(c0 + k) : 0;
    const int64_t before = tile_prefix(S, tile, v, status, lb, err);
    int64_t start = before & 0x7FFFFFFF, wide = before >> 31;
    // (first row of cell c, wide cells up to and with it)
    auto unit_of = [&](int64_t c, int64_t first_row, int64_t n_wide) {
        const uint32_t z = cell_zone ? cell_zone[c] : (uint32_t)c;
        return (first_row >> kUnitRowBits) + (z >> kUnitZoneBits) + n_wide +
               (cell_split ? cell_split[c] & 0x7FFFFFFFu : 0);
    };
    int64_t up = c0 > 0 && c0 < n_cells ? unit_of(c0 - 1, start - cnt[c0 - 1], wide) : -1;
#pragma unroll
    for (int k = 0; k < kPreItems; k++) {
        const int64_t c = c0 + k;
        const bool on = c < n_cells;
        uint32_t z = 0;
        int64_t u = up;
        if (on) {
            wide += v[k] >> 31;
            u = unit_of(c, start, wide);
            cell_start[c] = (uint32_t)start;
            cell_unit[c] = (uint32_t)u;
            if (zin) write_zone_in(geo, zin, c, (uint32_t)u);
            z = cell_zone ? cell_zone[c] : (uint32_t)c;
        }
        // (ids skipped, after a cell of many rows: empty units)
        warp_fill((uint32_t)(up + 1), (uint32_t)min(u + 1, (int64_t)unit_cap), (uint32_t)c, z,
                  (uint32_t)start, [&](uint32_t i, uint32_t, uint32_t uc, uint32_t uz, uint32_t us) {
                      unit[i] = make_uint4(uc, uz, us, 0);
                      ucur[(int64_t)i * kCursorStep] = us;
                  });
        if (on && c == (int64_t)n_cells - 1) {
            cell_start[n_cells] = (uint32_t)n;
            const int64_t nu = min(u + 1, (int64_t)unit_cap);
            unit[nu] = make_uint4(n_cells, 0, (uint32_t)n, 0);
            *n_units = (uint32_t)nu;
        }
        up = u;
        start += v[k] & 0x7FFFFFFF;
    }
}

// ---- records

// The float32 offsets (xi, eta) of a source in the tangent frame of its cell
// (zone centre line, RA cell centre), from its exact fixed-point position k.
__device__ __forceinline__ void cell_offsets(const PosKey& k, float h_f, const ZoneGeo& Z,
                                             float* xi, float* eta) {
    const uint32_t ra_key = (uint32_t)(k.key64 >> 32) & kRaKeyMask;
    const uint32_t bin = bin_of(ra_key, Z.nbins);
    const LatTerms L = lat_terms(h_f * k.zfrac, Z.sin_cf, Z.cos_cf);
    float sa, hav_a;
    sin_hav(Z.binw_f * cells_from_centre(k.key64, Z.nbins, bin), &sa, &hav_a);
    *xi = L.cd * sa;
    *eta = fmaf(L.cd * Z.sin_cf, hav_a, L.sdd);
}

// On their way records carry the low bits of their zone where a finished
// record has zeros: 8 bits in the low byte of the RA key, and between the two
// splits 3 more in the top exponent bits of the offsets (which are below 2 in
// size) and the sign of the row.
__device__ __forceinline__ uint4 tag_record(float xi, float eta, uint32_t ra24, uint32_t row,
                                            uint32_t z, bool wide) {
    uint4 r = make_uint4(__float_as_uint(xi), __float_as_uint(eta), ra24 | (z & 255u), row);
    if (wide) {
        r.x |= ((z >> 8) & 1u) << 30;
        r.y |= ((z >> 9) & 1u) << 30;
        r.w |= ((z >> 10) & 1u) << 31;
    }
    return r;
}

__device__ __forceinline__ uint32_t wide_tag(const uint4& r) {
    return (r.z & 255u) | ((r.x >> 30) & 1u) << 8 | ((r.y >> 30) & 1u) << 9 | (r.w >> 31) << 10;
}

__device__ __forceinline__ uint4 narrow_record(uint4 r) {
    r.x &= ~(1u << 30);
    r.y &= ~(1u << 30);
    r.w &= ~(1u << 31);
    return r;
}

// Shared memory of a tile that leaves grouped by digit: staged records, their
// digits, digit counts (then starts), and where each digit's run goes.
template <int ITEMS, int DIGITS>
struct SplitSmem {
    uint4 rec[kSplitThreads * ITEMS];
    uint32_t cnt[DIGITS];
    uint32_t to[DIGITS];
    uint16_t dig[kSplitThreads * ITEMS];
    uint32_t warp_tot[kSplitThreads / 32];
};
constexpr uint32_t kNoRecord = 0xFFFFFFFFu;

// The tile's records to memory, grouped by digit (dr: digit << 16 | rank of
// each record, or kNoRecord): ranks are those of the counting atomics (any
// order within a digit), a run of each digit is claimed from its cursor by
// one atomic, and consecutive threads then store consecutive records of a
// run. (Records waiting in shared memory instead of registers, for more
// blocks per SM, measured slower: the shared-memory pipe limits it.)
template <int ITEMS, int DIGITS>
__device__ __forceinline__ void split_tile(SplitSmem<ITEMS, DIGITS>& S, const uint4 (&r)[ITEMS],
                                           const uint32_t (&dr)[ITEMS], int nd, uint32_t* cursors,
                                           int64_t n, uint4* __restrict__ out) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __syncthreads();
    // digit starts within the tile: thread t sums digits [t * per, ...)
    const int per = (nd + kSplitThreads - 1) / kSplitThreads;
    uint32_t sum = 0;
    for (int k = 0; k < per; k++) {
        const int d = tid * per + k;
        if (d < nd) sum += S.cnt[d];
    }
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) S.warp_tot[warp] = incl;
    __syncthreads();
    uint32_t run = incl - sum, total = 0;
#pragma unroll
    for (int w = 0; w < kSplitThreads / 32; w++) {
        if (w < warp) run += S.warp_tot[w];
        total += S.warp_tot[w];
    }
    for (int k = 0; k < per; k++) {
        const int d = tid * per + k;
        if (d >= nd) break;
        const uint32_t c = S.cnt[d];
        S.cnt[d] = run;
        if (c) S.to[d] = atomicAdd(&cursors[(int64_t)d * kCursorStep], c) - run;
        run += c;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < ITEMS; k++) {
        if (dr[k] == kNoRecord) continue;
        const uint32_t p = S.cnt[dr[k] >> 16] + (dr[k] & 0xFFFFu);
        S.rec[p] = r[k];
        S.dig[p] = (uint16_t)(dr[k] >> 16);
    }
    __syncthreads();
    for (uint32_t p = tid; p < total; p += kSplitThreads) {
        const uint32_t g = S.to[S.dig[p]] + p;
        if (g < n) out[g] = S.rec[p];
    }
}

// Counts a record under its digit; digit << 16 | its rank there. (Lanes that
// all hold one digit, as in a catalogue stored by position, add it once.)
__device__ __forceinline__ uint32_t count_digit(uint32_t* cnt, int32_t d) {
    if (__all_sync(0xffffffffu, d == __shfl_sync(0xffffffffu, d, 0))) {
        if (d < 0) return kNoRecord;
        const int lane = threadIdx.x & 31;
        uint32_t base = 0;
        if (lane == 0) base = atomicAdd(&cnt[d], 32u);
        return (uint32_t)d << 16 | (__shfl_sync(0xffffffffu, base, 0) + lane);
    }
    return d < 0 ? kNoRecord : (uint32_t)d << 16 | atomicAdd(&cnt[d], 1u);
}

// Places for the warp's records in c[step * i], one atomic per distinct i: the
// first of the lane's run, and the record's rank in it. (2e6 atomics on one
// counter take 1.3 ms.)
__device__ __forceinline__ uint32_t claim_places(uint32_t* c, int step, uint32_t i, bool on,
                                                 uint32_t* rank) {
    const int lane = threadIdx.x & 31;
    const uint32_t peers = __match_any_sync(0xffffffffu, on ? i : 0xFFFFFFFFu);
    const int first = __ffs(peers) - 1;
    uint32_t base = 0;
    if (on && lane == first) base = atomicAdd(&c[(int64_t)i * step], (uint32_t)__popc(peers));
    *rank = (uint32_t)__popc(peers & ((1u << lane) - 1u));
    return __shfl_sync(0xffffffffu, base, first);
}

// Ingest of B: validity, longitude mod 360, the exact position kept by row,
// the record, and the records grouped by digit. WIDE: two splits (the digits
// are bins; wide tags; the key range narrowed); otherwise the digits are
// the units.
template <int ITEMS, bool WIDE, int DIGITS>
__global__ void __launch_bounds__(kSplitThreads, 3) k_ingest_b(
    const double* __restrict__ lon, const double* __restrict__ lat, int64_t n, int32_t nz,
    float h_f, const uint4* __restrict__ zin, int nd, uint32_t* cursors, uint4* __restrict__ out,
    double2* __restrict__ pos, KeyRange* range, int32_t* err) {
    pdl_wait();
    if (build_failed(err)) return;
    extern __shared__ __align__(16) unsigned char split_smem[];
    auto& S = *reinterpret_cast<SplitSmem<ITEMS, DIGITS>*>(split_smem);
    const int64_t base = (int64_t)blockIdx.x * (kSplitThreads * ITEMS) + threadIdx.x;
    // (the coordinates wait where the records will be)
    uint4 r[ITEMS];
#pragma unroll
    for (int k = 0; k < ITEMS; k++) {
        const int64_t i = base + k * kSplitThreads;
        if (i < n) {
            const int2 a = __ldcs(reinterpret_cast<const int2*>(lon) + i);
            const int2 b = __ldcs(reinterpret_cast<const int2*>(lat) + i);
            r[k] = make_uint4((uint32_t)a.x, (uint32_t)a.y, (uint32_t)b.x, (uint32_t)b.y);
        }
    }
    for (int d = threadIdx.x; d < nd; d += kSplitThreads) S.cnt[d] = 0;
    __syncthreads();
    uint32_t dr[ITEMS];
    uint32_t not_min = 0, kmax = 0;
    bool bad = false;
#pragma unroll
    for (int k = 0; k < ITEMS; k++) {
        const int64_t i = base + k * kSplitThreads;
        int32_t dig = -1;
        if (i < n) {
            const double lo = __hiloint2double((int)r[k].y, (int)r[k].x);
            const double la = __hiloint2double((int)r[k].w, (int)r[k].z);
            const bool ok = coord_ok(lo, la);
            bad |= !ok;
            const double lat_k = lat_or_zero(la);
            const double lon_k = lon_mod360(keep_or_zero(lo, ok));
            const PosKey key = pos_key(lon_k, lat_k, nz);
            const uint4 zu = __ldg(zin + key.z);
            dig = (int32_t)(zu.w >> kDigitShift);
            ZoneGeo Z;
            Z.sin_cf = __uint_as_float(zu.x);
            Z.cos_cf = __uint_as_float(zu.y);
            Z.binw_f = __uint_as_float(zu.z);
            Z.nbins = zu.w & ((1u << kDigitShift) - 1u);
            __stcs(&pos[i], make_double2(lon_k, lat_k));
            const uint32_t ra = (uint32_t)(key.key64 >> 32) & kRaKeyMask;
            if (WIDE) {
                not_min = max(not_min, 65535u - (ra >> kIndexRaShift));
                kmax = max(kmax, ra >> kIndexRaShift);
            }
            float xi, eta;
            cell_offsets(key, h_f, Z, &xi, &eta);
            r[k] = tag_record(xi, eta, ra, (uint32_t)i, (uint32_t)key.z, WIDE);
        }
        dr[k] = count_digit(S.cnt, dig);
    }
    if (bad) atomicOr(err, kErrCoord);
    if (WIDE) {  // (a stale read of the range costs one redundant atomic, never a miss)
        not_min = __reduce_max_sync(0xffffffffu, not_min);
        kmax = __reduce_max_sync(0xffffffffu, kmax);
        if ((threadIdx.x & 31) == 0) {
            const volatile KeyRange* v = range;
            if (not_min > v->not_min) atomicMax(&range->not_min, not_min);
            if (kmax > v->max) atomicMax(&range->max, kmax);
        }
    }
    split_tile<ITEMS, DIGITS>(S, r, dr, nd, cursors, n, out);
}

// Float64 unit vectors of B, by row, from the positions the ingest kept. (In
// the ingest the evaluation's registers would cost it warps; here the pass is
// bound by its integer instructions, 0.4 of the bandwidth by its 48 bytes a
// source.)
__global__ void __launch_bounds__(kBlock) k_unit_b(const double2* __restrict__ pos, int64_t n,
                                                   double2* __restrict__ p64, const int32_t* err) {
    pdl_wait();
    const int64_t i = (int64_t)blockIdx.x * kBlock + threadIdx.x;
    if (i >= n || build_failed(err)) return;
    const double2 q = __ldcs(pos + i);
    double x, y, z;
    unit64_turn(lon_turn(q.x), lat_turn(q.y), &x, &y, &z);
    __stcs(&p64[2 * i], make_double2(x, y));
    __stcs(&p64[2 * i + 1], make_double2(z, 0.0));
}

// Chunk t of the bins' chunks: its bin (the last whose first chunk is <= t).
__device__ __forceinline__ int bin_of_chunk(const uint32_t* __restrict__ bin_chunk, int nbins, uint32_t t) {
    int lo = 0, hi = nbins;  // bin_chunk[lo] <= t < bin_chunk[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(bin_chunk + mid) <= t) lo = mid;
        else hi = mid;
    }
    return lo;
}

// Sources per cell, a chunk of one bin's records per block, counted in shared
// memory (cells past what that holds: in global memory). The block also lists
// its tiles for the second split: first row, row after the bin, bin.
__global__ void __launch_bounds__(kSplitThreads) k_cell_count(
    const uint4* __restrict__ rec, const uint32_t* __restrict__ bin_start,
    const uint32_t* __restrict__ bin_chunk, int nbins, const uint32_t* __restrict__ bin_zone,
    const ZoneCells* __restrict__ zcells, const uint32_t* n_cells,
    uint32_t* __restrict__ ccnt, const uint32_t* __restrict__ bin_tile, uint4* __restrict__ tiles,
    const int32_t* err) {
    pdl_wait();
    if (build_failed(err) || blockIdx.x >= bin_chunk[nbins]) return;
    __shared__ uint32_t h[kCellSlots];
    for (int i = threadIdx.x; i < kCellSlots; i += kSplitThreads) h[i] = 0;
    __syncthreads();
    const int b = bin_of_chunk(bin_chunk, nbins, blockIdx.x);
    const uint32_t zhi = bin_zone[b] >> kBinZoneBits << kBinZoneBits;
    const uint32_t lo = bin_start[b] + (blockIdx.x - bin_chunk[b]) * (kCountChunk * kTile);
    const uint32_t hi = min(bin_start[b + 1], lo + kCountChunk * kTile);
    const uint32_t first = zcells[bin_zone[b]].first;  // of the bin's cells
    if (threadIdx.x < kCountChunk && lo + threadIdx.x * kTile < hi)
        tiles[bin_tile[b] + (blockIdx.x - bin_chunk[b]) * kCountChunk + threadIdx.x] =
            make_uint4(lo + threadIdx.x * kTile, bin_start[b + 1], (uint32_t)b, 0);
    for (uint32_t i0 = lo + threadIdx.x; i0 < hi; i0 += kSplitThreads * 4) {
        uint4 r[4];
#pragma unroll
        for (int k = 0; k < 4; k++)
            if (i0 + k * kSplitThreads < hi) r[k] = __ldg(rec + i0 + k * kSplitThreads);
#pragma unroll
        for (int k = 0; k < 4; k++) {
            if (i0 + k * kSplitThreads >= hi) break;
            const uint32_t c = cell_of(load_cells(zcells + (zhi + wide_tag(r[k]))), r[k].z);
            if (c - first < kCellSlots) atomicAdd(&h[c - first], 1u);
            else atomicAdd(&ccnt[c], 1u);
        }
    }
    __syncthreads();
    const uint32_t nc = *n_cells;
    for (int i = threadIdx.x; i < kCellSlots && first + i < nc; i += kSplitThreads)
        if (h[i]) atomicAdd(&ccnt[first + i], h[i]);
}

// The second split: a tile of one bin's records grouped by unit. (A bin of more
// units than a tile counts -- of a zone of about a million rows, or after a cell
// of as many -- claims the places of a warp's records at a time: in pieces of
// kMaxDigits units it took as long.)
__global__ void __launch_bounds__(kSplitThreads, 3) k_split(
    const uint4* __restrict__ rec, const uint4* __restrict__ tiles, const uint32_t* n_tiles, int nbins,
    const uint32_t* __restrict__ bin_zone, const ZoneCells* __restrict__ zcells,
    const uint32_t* __restrict__ cell_unit, const uint32_t* n_units, int64_t n, uint32_t* ucur,
    uint4* __restrict__ out, const int32_t* err) {
    pdl_wait();
    if (build_failed(err) || blockIdx.x >= *n_tiles) return;
    extern __shared__ __align__(16) unsigned char split_smem[];
    auto& S = *reinterpret_cast<SplitSmem<kTileItems, kMaxDigits>*>(split_smem);
    const int tid = threadIdx.x;
    const uint4 tile = __ldg(tiles + blockIdx.x);
    const uint32_t lo = tile.x, hi = tile.y;
    const int b = (int)tile.z;
    uint4 r[kTileItems];
#pragma unroll
    for (int k = 0; k < kTileItems; k++) {
        const uint32_t i = lo + tid + k * kSplitThreads;
        if (i < hi) r[k] = __ldcs(rec + i);
    }
    const uint32_t z0 = bin_zone[b], zhi = z0 >> kBinZoneBits << kBinZoneBits;
    // the bin's units (a unit lies in one bin): those from its first zone on
    // that come before the next bin's first zone (0: there is none)
    const uint32_t u0 = cell_unit[zcells[z0].first];
    const uint32_t z1 = b + 1 < nbins ? bin_zone[b + 1] : 0;
    const uint32_t nd = (z1 > z0 ? cell_unit[zcells[z1].first] : *n_units) - u0;
    if (nd > kMaxDigits) {
#pragma unroll
        for (int k = 0; k < kTileItems; k++) {
            const bool on = lo + tid + k * kSplitThreads < hi;
            uint32_t u = 0, rank;
            if (on) u = __ldg(cell_unit + cell_of(load_cells(zcells + (zhi + wide_tag(r[k]))), r[k].z));
            const uint32_t g = claim_places(ucur, kCursorStep, u, on, &rank) + rank;
            if (on && g < n) out[g] = narrow_record(r[k]);
        }
        return;
    }
    for (uint32_t d = tid; d < nd; d += kSplitThreads) S.cnt[d] = 0;
    __syncthreads();
    uint32_t dr[kTileItems];
#pragma unroll
    for (int k = 0; k < kTileItems; k++) {
        int32_t dig = -1;
        if (lo + tid + k * kSplitThreads < hi) {
            const ZoneCells Z = load_cells(zcells + (zhi + wide_tag(r[k])));
            dig = (int32_t)(__ldg(cell_unit + cell_of(Z, r[k].z)) - u0);
            r[k] = narrow_record(r[k]);
        }
        dr[k] = count_digit(S.cnt, dig);
    }
    split_tile<kTileItems, kMaxDigits>(S, r, dr, (int)nd, ucur + (int64_t)u0 * kCursorStep, n, out);
}

// ---- the zones' buckets

constexpr int kPlaceThreads = 128, kPlaceItems = 8;
constexpr uint32_t kPlaceCap = kPlaceThreads * kPlaceItems;  // records staged
constexpr uint32_t kPlaceCtr = 2 * kPlaceCap + 2 * kUnitZones;  // 16-bit bucket counters
constexpr uint32_t kBigCtr = kPlaceCtr / 2 + 4 * kPlaceCap;  // 32-bit ones, with the stage's room
constexpr int kPlaceBlocks = 8;  // per SM

struct PlaceSmem {
    uint4 stage[kPlaceCap];
    uint32_t ctr[kPlaceCtr / 2];  // two 16-bit counters a word (directly after the stage)
    uint32_t zmin[kUnitZones], zmax[kUnitZones];  // keys of each zone, top 16 bits
    uint32_t zkmin[kUnitZones], zshift[kUnitZones], zlb[kUnitZones + 1];
    uint32_t warp_tot[kPlaceThreads / 32];
};
// (a unit of several cells holds fewer than two windows' rows)
static_assert(kPlaceCap >= 2u << kUnitRowBits, "units of several cells fit the stage");

// What a build leaves for k_place_b.
struct PlaceArgs {
    const uint4* rec;            // grouped by unit
    const uint4* unit;           // first cell, its zone and its first row, of each unit
    const uint32_t* n_units;
    const uint32_t* cell_start;  // first row of each cell
    const uint32_t* cell_zone;   // NULL: cells are zones
    const ZoneCells* zcells;     // NULL: cells are zones
    const KeyRange* range;
    const ZoneGeo* geo;
    int32_t nz;
    int64_t n;
    BRec* out;
    uint32_t* lut;
    ZoneHot* zhot;
    const int32_t* err;
    // units of one cell of more than giant_rows rows: a list for k_place_giant
    uint32_t giant_rows;
    uint32_t* giants;
    uint32_t* n_giants;
};

// Buckets of a zone of m rows whose keys span [kmin, kmax] (top 16 bits in
// place): one to two per row, never finer than kIndexRaShift bits. With
// `aligned`, buckets begin at multiples of their width and are at most 2^most
// wide, so that the bounds of the zone's parts are bounds of buckets.
struct Buckets {
    uint32_t kmin, shift, last;
};

__device__ __forceinline__ Buckets buckets_of(uint32_t m, uint32_t kmin, uint32_t kmax, bool aligned,
                                              uint32_t most) {
    Buckets B{kmin, (uint32_t)kIndexRaShift, 0};
    if (m == 0 || kmax < kmin) {
        B.kmin = 0;
        return B;
    }
    const int lg = m > 1 ? 32 - __clz(m - 1) : 0;  // 2^lg >= m
    for (int s = kIndexRaShift;; s++) {
        const uint32_t lo = aligned ? kmin >> s << s : kmin;
        const uint32_t last = (kmax - lo) >> s;
        if (last < (1u << lg) || s >= (int)most) {
            B.kmin = lo;
            B.shift = (uint32_t)s;
            B.last = last;
            return B;
        }
    }
}

__device__ __forceinline__ void write_zone(const PlaceArgs& P, uint32_t z, uint32_t start,
                                           uint32_t rel, const Buckets& B) {
    const ZoneGeo Z = load_geo(P.geo + z);
    ZoneHot H;
    H.start = start;
    H.lut_rel = (int32_t)rel;
    H.lut_kmin = B.kmin;
    H.shift_last = B.shift | (B.last << 8);
    H.nbins = Z.nbins;
    H.sin_cf = Z.sin_cf;
    H.cos_cf = Z.cos_cf;
    H.binw_f = Z.binw_f;
    P.zhot[z] = H;
}

// Block-wide exclusive prefix of one value per thread.
template <int THREADS = kPlaceThreads>
__device__ __forceinline__ uint32_t block_offset(uint32_t sum, uint32_t* warp_tot) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    uint32_t run = incl - sum;
#pragma unroll
    for (int w = 0; w < THREADS / 32; w++)
        if (w < warp) run += warp_tot[w];
    return run;
}

// Inclusive prefix, plus `add`, of n 32-bit counters in place. GLOBAL: they
// lie in global memory, counted by atomics (read past L1).
template <bool GLOBAL, int THREADS>
__device__ __forceinline__ void scan_counters(uint32_t* c, uint32_t n, uint32_t add,
                                              uint32_t* warp_tot) {
    const uint32_t per = ((n + THREADS - 1) / THREADS) | 1u;
    const uint32_t lo = min(n, threadIdx.x * per), hi = min(n, lo + per);
    uint32_t sum = 0;
    for (uint32_t i = lo; i < hi; i++) sum += GLOBAL ? __ldcg(c + i) : c[i];
    uint32_t run = add + block_offset<THREADS>(sum, warp_tot);
    for (uint32_t i = lo; i < hi; i++) {
        run += GLOBAL ? __ldcg(c + i) : c[i];
        c[i] = run;
    }
    __syncthreads();
}

// Exclusive prefix of 16-bit counters, two in each of n words, in place (the
// total fits 16 bits). A thread takes an odd number of consecutive words: no
// bank conflicts.
__device__ __forceinline__ void scan_pairs(uint32_t* c, uint32_t n, uint32_t* warp_tot) {
    const uint32_t per = ((n + kPlaceThreads - 1) / kPlaceThreads) | 1u;
    const uint32_t lo = min(n, threadIdx.x * per), hi = min(n, lo + per);
    uint32_t sum = 0;
    for (uint32_t i = lo; i < hi; i++) sum += c[i];
    sum = (sum & 0xFFFFu) + (sum >> 16);
    uint32_t run = block_offset(sum, warp_tot);
    for (uint32_t i = lo; i < hi; i++) {
        const uint32_t v = c[i], a = run + (v & 0xFFFFu);
        c[i] = run | a << 16;
        run = a + (v >> 16);
    }
    __syncthreads();
}

__device__ __forceinline__ uint32_t clean(uint32_t key) { return key & kRaKeyMask; }

// Rows [s, e) of one cell counted by bucket into c, and moved to their buckets'
// places (c then the row after each bucket, at the end its first row), by the
// threads `tid` of `step` (whole warps). B: the zone's buckets, of which the
// cell holds those from b0 on. Cells of so many rows are mostly sources on one
// spot: a warp's sources in one bucket take one atomic; with FEW buckets, each
// group of them does (which costs more where they lie apart).
__device__ __forceinline__ uint32_t clean_bucket(uint32_t key, const Buckets& B, uint32_t b0) {
    return ((clean(key) - B.kmin) >> B.shift) - b0;
}

// The lanes with the same b, or the lane alone.
template <bool FEW>
__device__ __forceinline__ uint32_t bucket_peers(uint32_t b, uint32_t lane) {
    if (FEW) return __match_any_sync(0xffffffffu, b);
    return __all_sync(0xffffffffu, b == __shfl_sync(0xffffffffu, b, 0)) ? 0xffffffffu : 1u << lane;
}

template <bool FEW>
__device__ __forceinline__ void count_rows(const PlaceArgs& P, uint32_t s, uint32_t e, uint32_t tid,
                                           uint32_t step, const Buckets& B, uint32_t b0, uint32_t* c) {
    const uint32_t lane = tid & 31;
    for (uint32_t i0 = s + (tid - lane); i0 < e; i0 += step * 4) {
        uint32_t key[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const uint32_t i = i0 + lane + k * step;
            key[k] = i < e ? __ldg(&P.rec[i].z) : 0;
        }
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const bool on = i0 + lane + k * step < e;
            const uint32_t b = on ? clean_bucket(key[k], B, b0) : 0xFFFFFFFFu;
            const uint32_t peers = bucket_peers<FEW>(b, lane);
            if (on && (peers & ((1u << lane) - 1u)) == 0) atomicAdd(&c[b], (uint32_t)__popc(peers));
        }
    }
}

template <bool FEW>
__device__ __forceinline__ void move_rows(const PlaceArgs& P, uint32_t s, uint32_t e, uint32_t tid,
                                          uint32_t step, const Buckets& B, uint32_t b0, uint32_t* c) {
    const uint32_t lane = tid & 31;
    for (uint32_t i0 = s + (tid - lane); i0 < e; i0 += step * 4) {
        uint4 r[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const uint32_t i = i0 + lane + k * step;
            if (i < e) r[k] = __ldg(&P.rec[i]);
        }
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const bool on = i0 + lane + k * step < e;
            const uint32_t b = on ? clean_bucket(r[k].z, B, b0) : 0xFFFFFFFFu;
            const uint32_t peers = bucket_peers<FEW>(b, lane);
            const uint32_t below = __popc(peers & ((1u << lane) - 1u));
            uint32_t at = 0;
            if (on && below == 0) at = atomicSub(&c[b], (uint32_t)__popc(peers));
            at = __shfl_sync(0xffffffffu, at, __ffs(peers) - 1);
            r[k].z = clean(r[k].z);
            if (on) reinterpret_cast<uint4*>(P.out)[at - 1u - below] = r[k];
        }
    }
}

// Rows [s, e) of one cell, too many to stage (or of too many buckets), by a
// block. The cell holds buckets [b0, b1); `base` is the table place of b0.
// Buckets past the counters in shared memory are counted in the table itself.
__device__ __noinline__ void place_large(const PlaceArgs& P, PlaceSmem& S, uint32_t s, uint32_t e,
                            const Buckets& B, uint32_t b0, uint32_t b1, int64_t base) {
    const uint32_t nb = b1 - b0;
    uint32_t* const L = P.lut + base;
    uint32_t* const c = nb <= kBigCtr ? reinterpret_cast<uint32_t*>(S.stage) : L;
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < nb; i += kPlaceThreads) c[i] = 0;
    __syncthreads();
    count_rows<false>(P, s, e, threadIdx.x, kPlaceThreads, B, b0, c);
    __syncthreads();
    if (c != L) scan_counters<false, kPlaceThreads>(c, nb, s, S.warp_tot);  // c[b]: the row after bucket b
    else scan_counters<true, kPlaceThreads>(c, nb, s, S.warp_tot);
    move_rows<false>(P, s, e, threadIdx.x, kPlaceThreads, B, b0, c);
    __syncthreads();  // (c[b]: the first row of bucket b)
    if (c != L)
        for (uint32_t i = threadIdx.x; i < nb; i += kPlaceThreads) L[i] = c[i];
    __syncthreads();
}

// The buckets of part cell c0 of zone z0: nb of them from b0 on, their table
// from `base` on. `write`: the first part's thread writes the zone, the last
// one's the entry after the table (row e).
__device__ __forceinline__ void part_buckets(const PlaceArgs& P, const ZoneCells& Z, uint32_t c0,
                                             uint32_t z0, uint32_t e, uint32_t rel0, bool write,
                                             Buckets* B, uint32_t* b0, uint32_t* nb, int64_t* base) {
    const uint32_t zs = P.cell_start[Z.first];
    const uint32_t mz = P.cell_start[Z.first + Z.parts] - zs;
    *B = buckets_of(mz, (65535u - P.range->not_min) << 16, P.range->max << 16, true,
                    Z.shift + kIndexRaShift);
    const uint32_t p = c0 - Z.first;
    const uint32_t at = Z.p0 + p, sh = Z.shift + 16;
    *b0 = p == 0 ? 0 : ((at << sh) - B->kmin) >> B->shift;
    *nb = (p + 1 == Z.parts ? B->last + 1 : (((at + 1) << sh) - B->kmin) >> B->shift) - *b0;
    *base = 2 * (int64_t)zs + rel0 + *b0;
    if (write) {
        if (p == 0) write_zone(P, z0, zs, rel0, *B);
        if (p + 1 == Z.parts) P.lut[*base + *nb] = e;
    }
}

// Units, a block each: the records of consecutive zones, or of one part of a
// zone, into the order of their buckets, with the zones' bucket tables. A
// unit's records pass through registers and shared memory once: each takes a
// rank in its bucket by a shared-memory atomic, the buckets' counts become
// their first rows, the records go to their places in the stage, and table and
// stage leave in order. The tables of a unit's zones lie one after the other
// from 2 * (its first row) + 3 z + 2 c on, z its first zone and c its first
// cell: a zone of m rows has at most 2 m + 1 entries, or one per part and one
// more. Bound by latency and instruction issue: 3.0 ms on the all-sky index
// (2e8 rows), 0.22 ms on 1.2e7; 384 threads with units twice as large took
// 3.24 and 0.27 ms, 512 threads with four times as large 3.3 and 0.21 ms.
__global__ void __launch_bounds__(kPlaceThreads, kPlaceBlocks) k_place_b(PlaceArgs P) {
    pdl_wait();
    extern __shared__ __align__(16) unsigned char place_smem[];
    PlaceSmem& S = *reinterpret_cast<PlaceSmem*>(place_smem);
    if (build_failed(P.err)) {  // an index that holds nothing
        if (blockIdx.x == 0 && threadIdx.x < 2) P.lut[threadIdx.x] = 0;
        for (int64_t z = (int64_t)blockIdx.x * kPlaceThreads + threadIdx.x; z < P.nz;
             z += (int64_t)gridDim.x * kPlaceThreads)
            write_zone(P, (uint32_t)z, 0, 0, Buckets{0, 31, 0});
        return;
    }
    const uint32_t n_units = *P.n_units;
    const uint32_t tid = threadIdx.x;
    uint4 d{}, d1{};  // this unit's first cell, zone and row, and the next's
    if (blockIdx.x < n_units) {
        d = __ldg(P.unit + blockIdx.x);
        d1 = __ldg(P.unit + blockIdx.x + 1);
    }
    for (uint32_t u = blockIdx.x; u < n_units; u += gridDim.x) {
        const uint32_t c0 = d.x, z0 = d.y, s = d.z, c1 = d1.x, e = d1.z;
        if (u + gridDim.x < n_units) {
            d = __ldg(P.unit + u + gridDim.x);
            d1 = __ldg(P.unit + u + gridDim.x + 1);
        }
        if (c0 == c1) continue;  // an id without cells
        const uint32_t m = e - s, nzones = c1 - c0;
        if (m > P.giant_rows) {
            if (tid == 0) P.giants[atomicAdd(P.n_giants, 1u)] = u;
            continue;
        }
        bool large = m > kPlaceCap;
        uint4 r[kPlaceItems];
        if (!large) {
#pragma unroll
            for (int k = 0; k < kPlaceItems; k++) {
                if (k * kPlaceThreads >= m) break;
                const uint32_t i = tid + k * kPlaceThreads;
                if (i < m) r[k] = __ldcs(P.rec + s + i);
            }
        }
        ZoneCells Z{c0, 1, 0, 16};
        if (P.zcells) Z = load_cells(P.zcells + z0);
        const bool part = Z.parts > 1;
        const uint32_t rel0 = P.zcells ? 3 * z0 + 2 * Z.first : 5 * z0;
        uint32_t nb = 0;                        // counters, and table entries written
        int64_t base = 2 * (int64_t)s + rel0;   // place of the first
        Buckets B{};
        uint32_t b0 = 0;
        __syncthreads();  // (the last unit's stage and tables are out)
        if (part) {
            part_buckets(P, Z, c0, z0, e, rel0, tid == 0, &B, &b0, &nb, &base);
            large |= nb > kPlaceCtr;
            if (tid == 0) {
                S.zkmin[0] = B.kmin;
                S.zshift[0] = B.shift;
                S.zlb[0] = 0u - b0;
            }
        } else if (large) {  // one zone
            uint32_t kmin = 0xFFFFu, kmax = 0;
            for (uint32_t i = s + tid; i < e; i += kPlaceThreads) {
                const uint32_t key = __ldg(&P.rec[i].z) >> 16;
                kmin = min(kmin, key);
                kmax = max(kmax, key);
            }
            kmin = __reduce_min_sync(0xffffffffu, kmin);
            kmax = __reduce_max_sync(0xffffffffu, kmax);
            if (tid == 0) {
                S.zmin[0] = 0xFFFFu;
                S.zmax[0] = 0;
            }
            __syncthreads();
            if ((tid & 31) == 0) {
                atomicMin(&S.zmin[0], kmin);
                atomicMax(&S.zmax[0], kmax);
            }
            __syncthreads();
            B = buckets_of(m, S.zmin[0] << 16, S.zmax[0] << 16, false, 32);
            nb = B.last + 1;
            if (tid == 0) {
                write_zone(P, z0, s, rel0, B);
                P.lut[base + nb] = e;
            }
        }
        if (large) {
            place_large(P, S, s, e, B, b0, b0 + nb, base);
            continue;
        }
        if (!part) {
            if (tid < nzones) {
                S.zmin[tid] = 0xFFFFu;
                S.zmax[tid] = 0;
            }
            __syncthreads();
#pragma unroll
            for (int k = 0; k < kPlaceItems; k++) {
                if (k * kPlaceThreads >= m) break;
                if (tid + k * kPlaceThreads < m) {
                    const uint32_t l = (r[k].z - z0) & 255u, key = r[k].z >> 16;
                    if (key < S.zmin[l]) atomicMin(&S.zmin[l], key);
                    if (key > S.zmax[l]) atomicMax(&S.zmax[l], key);
                }
            }
            __syncthreads();
            // zone l's buckets, and its table's place among the unit's
            uint32_t zs = 0, entries = 0;
            if (tid < nzones) {
                zs = P.cell_start[c0 + tid];
                B = buckets_of(P.cell_start[c0 + tid + 1] - zs, S.zmin[tid] << 16, S.zmax[tid] << 16,
                               false, 32);
                entries = B.last + 2;
            }
            static_assert(kUnitZones <= kPlaceThreads, "a thread per zone");
            const uint32_t lb = block_offset(entries, S.warp_tot);
            if (tid < nzones) {
                S.zkmin[tid] = B.kmin;
                S.zshift[tid] = B.shift;
                S.zlb[tid] = lb;
                if (tid + 1 == nzones) S.zlb[nzones] = lb + entries;
                write_zone(P, z0 + tid, zs, rel0 + lb - 2 * (zs - s), B);
            }
            __syncthreads();
            nb = S.zlb[nzones];
        }
        for (uint32_t i = tid; i < (nb + 1) / 2; i += kPlaceThreads) S.ctr[i] = 0;
        __syncthreads();
        uint32_t at[kPlaceItems];  // the record's counter, its rank there above
#pragma unroll
        for (int k = 0; k < kPlaceItems; k++) {
            if (k * kPlaceThreads >= m) break;
            if (tid + k * kPlaceThreads < m) {
                const uint32_t l = (r[k].z - z0) & 255u;  // (0 in a part)
                r[k].z &= kRaKeyMask;
                const uint32_t c = S.zlb[l] + ((r[k].z - S.zkmin[l]) >> S.zshift[l]);
                const uint32_t sh = 16 * (c & 1u);
                at[k] = c | ((atomicAdd(&S.ctr[c >> 1], 1u << sh) >> sh) & 0xFFFFu) << 16;
            }
        }
        __syncthreads();
        scan_pairs(S.ctr, (nb + 1) / 2, S.warp_tot);
        const uint16_t* const first = reinterpret_cast<const uint16_t*>(S.ctr);
#pragma unroll
        for (int k = 0; k < kPlaceItems; k++) {
            if (k * kPlaceThreads >= m) break;
            if (tid + k * kPlaceThreads < m) S.stage[first[at[k] & 0xFFFFu] + (at[k] >> 16)] = r[k];
        }
        for (uint32_t i = tid; i < nb; i += kPlaceThreads) P.lut[base + i] = s + first[i];
        __syncthreads();
        for (uint32_t i = tid; i < m; i += kPlaceThreads)
            reinterpret_cast<uint4*>(P.out)[s + i] = S.stage[i];
    }
}

// The units of very many rows, which one block of k_place_b would hold up (a
// unit of 2e6 rows took it 5.8 ms): a cluster of eight blocks each, counting in
// the bucket table. Listed from kGiantRows rows on, some 50 us of a block's
// time, and a 2048th of the catalogue's, so that the list stays short; where
// one split makes the units, whose zones are not cut into parts and have up to
// 65536 buckets, from kGiantZone on (a zone of 11,000 rows takes a block 125 us,
// a cluster 23 with the rest). 0.17 to 0.22 ms for 2e6 rows on one point, 0.05
// for 5e5, 0.12 for 3e5 over one zone; a launch with an empty list costs a build
// 2 to 3 us, so none is made for kGiantRows rows or fewer.
constexpr uint32_t kGiantRows = 16384, kGiantZone = 4096;
constexpr int kGiantThreads = 1024, kGiantBlocks = 8;

__global__ void __cluster_dims__(kGiantBlocks, 1, 1) __launch_bounds__(kGiantThreads)
    k_place_giant(PlaceArgs P) {
    pdl_wait();
    const uint32_t n = *P.n_giants;
    if (n == 0 || build_failed(P.err)) return;  // (the whole cluster)
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const uint32_t rank = cluster.block_rank();
    constexpr uint32_t kStep = kGiantThreads * kGiantBlocks;
    const uint32_t tid = rank * kGiantThreads + threadIdx.x;
    __shared__ uint32_t kmin, kmax, total, warp_tot[kGiantThreads / 32];
    for (uint32_t g = blockIdx.x / kGiantBlocks; g < n; g += gridDim.x / kGiantBlocks) {
        const uint32_t u = P.giants[g];
        const uint4 d = __ldg(P.unit + u);
        const uint32_t c0 = d.x, z0 = d.y, s = d.z, e = __ldg(P.unit + u + 1).z;
        ZoneCells Z{c0, 1, 0, 16};
        if (P.zcells) Z = load_cells(P.zcells + z0);
        const uint32_t rel0 = P.zcells ? 3 * z0 + 2 * Z.first : 5 * z0;
        uint32_t b0 = 0, nb = 0;
        int64_t base = 2 * (int64_t)s + rel0;
        Buckets B{};
        if (Z.parts > 1) {
            part_buckets(P, Z, c0, z0, e, rel0, tid == 0, &B, &b0, &nb, &base);
        } else {  // one zone
            if (threadIdx.x == 0) {
                kmin = 0xFFFFu;
                kmax = 0;
            }
            __syncthreads();
            uint32_t lo = 0xFFFFu, hi = 0;
            for (uint32_t i = s + tid; i < e; i += kStep) {
                const uint32_t key = __ldg(&P.rec[i].z) >> 16;
                lo = min(lo, key);
                hi = max(hi, key);
            }
            lo = __reduce_min_sync(0xffffffffu, lo);
            hi = __reduce_max_sync(0xffffffffu, hi);
            if ((threadIdx.x & 31) == 0) {
                atomicMin(&kmin, lo);
                atomicMax(&kmax, hi);
            }
            cluster.sync();
            for (int k = 0; k < kGiantBlocks; k++) {
                lo = min(lo, *cluster.map_shared_rank(&kmin, k));
                hi = max(hi, *cluster.map_shared_rank(&kmax, k));
            }
            B = buckets_of(e - s, lo << 16, hi << 16, false, 32);
            nb = B.last + 1;
            if (tid == 0) {
                write_zone(P, z0, s, rel0, B);
                P.lut[base + nb] = e;
            }
        }
        uint32_t* const L = P.lut + base;
        for (uint32_t i = tid; i < nb; i += kStep) L[i] = 0;
        if (threadIdx.x == 0) total = 0;
        cluster.sync();
        count_rows<true>(P, s, e, tid, kStep, B, b0, L);
        cluster.sync();
        // each block's share of the buckets, after the sums of those before it
        const uint32_t share = (nb + kGiantBlocks - 1) / kGiantBlocks;
        const uint32_t l0 = min(nb, rank * share), l1 = min(nb, l0 + share);
        uint32_t sum = 0;
        for (uint32_t i = l0 + threadIdx.x; i < l1; i += kGiantThreads) sum += __ldcg(L + i);
        sum = __reduce_add_sync(0xffffffffu, sum);
        if ((threadIdx.x & 31) == 0) atomicAdd(&total, sum);
        cluster.sync();
        uint32_t before = s;
        for (uint32_t k = 0; k < rank; k++) before += *cluster.map_shared_rank(&total, k);
        scan_counters<true, kGiantThreads>(L + l0, l1 - l0, before, warp_tot);
        cluster.sync();
        move_rows<true>(P, s, e, tid, kStep, B, b0, L);
    }
    cluster.sync();  // (no block ends while another reads its shared memory)
}

// Zone geometry depends only on the zone count: it is computed once per
// (device, zone count) into a table kept for the life of the process (at most
// 64 of them; past that, into `own`, the caller's memory).
struct GeomCache {
    int device;
    int32_t nz;
    ZoneGeo* geo;
};

xm_status zone_geometry(int32_t nz, ZoneGeo* own, const ZoneGeo** out, cudaStream_t s) {
    static std::mutex mu;
    static std::vector<GeomCache> cache;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
    {
        std::lock_guard<std::mutex> g(mu);
        for (const GeomCache& c : cache)
            if (c.device == dev && c.nz == nz) {
                *out = c.geo;
                return XM_OK;
            }
        if (cache.size() < 64) {
            ZoneGeo* t = nullptr;
            if (cudaMalloc(&t, (size_t)nz * sizeof(ZoneGeo)) == cudaSuccess) {
                k_zone_geom<<<(unsigned)((nz + kBlock - 1) / kBlock), kBlock>>>(nz, t);
                if (cudaDeviceSynchronize() == cudaSuccess) {
                    cache.push_back(GeomCache{dev, nz, t});
                    *out = t;
                    return XM_OK;
                }
                cudaFree(t);
            }
            cudaGetLastError();
        }
    }
    XM_LAUNCH("k_zone_geom", (unsigned)((nz + kBlock - 1) / kBlock), kBlock, 0, s, k_zone_geom, nz, own);
    *out = own;
    return XM_OK;
}

// Shared-memory limits of the build's kernels, set once per device.
void prepare_build() {
    static std::mutex mu;
    static bool done[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> g(mu);
    if (dev < 0 || dev >= 64 || done[dev]) return;
    auto set = [](auto k, size_t bytes) {
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    };
    set(k_zone_count<1>, kCountSmem);
    set(k_zone_count<2>, kCountSmem);
    set(k_ingest_b<2, false, kMaxUnits>, sizeof(SplitSmem<2, kMaxUnits>));
    set(k_ingest_b<4, false, kMaxUnits>, sizeof(SplitSmem<4, kMaxUnits>));
    set(k_ingest_b<kTileItems, true, kMaxBins>, sizeof(SplitSmem<kTileItems, kMaxBins>));
    set(k_split, sizeof(SplitSmem<kTileItems, kMaxDigits>));
    set(k_place_b, sizeof(PlaceSmem));
    done[dev] = true;
}

// Slices of one allocation, each 256-byte aligned.
struct Slices {
    size_t bytes = 0;
    template <typename T>
    size_t add(int64_t count) {
        const size_t at = bytes;
        bytes += ((size_t)(count > 0 ? count : 1) * sizeof(T) + 255) & ~size_t(255);
        return at;
    }
};

}  // namespace

}  // namespace xm

using namespace xm;

extern "C" xm_status xm_build_index(const xm_columns* B, const xm_index_opts* opts, void* stream,
                                    xm_index** out) {
    if (!out) return set_error(XM_EINVAL, "xm_build_index: out is NULL");
    *out = nullptr;
    if (!B || B->n < 0 || B->n > 2147483647LL || (B->n > 0 && (!B->lon_deg || !B->lat_deg)))
        return set_error(XM_EINVAL, "xm_build_index: bad catalogue columns");
    if (B->frame != XM_FRAME_EQ && B->frame != XM_FRAME_GAL)
        return set_error(XM_EINVAL, "xm_build_index: bad frame %d", B->frame);
    double h_as = (opts && opts->zone_height_arcsec > 0) ? opts->zone_height_arcsec : 20.0;
    if (!(h_as >= 1.0 && h_as <= 36000.0))
        return set_error(XM_EINVAL, "xm_build_index: zone height %g arcsec outside [1, 36000]",
                         h_as);
    cudaStream_t s = (cudaStream_t)stream;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");

    const int64_t n = B->n;
    xm_index* X = new (std::nothrow) xm_index();
    if (!X) return set_error(XM_ENOMEM, "xm_build_index: host allocation");
    X->device = dev;
    X->stream = s;
    X->frame = B->frame;
    X->n = n;
    X->nz = (int32_t)ceil(648000.0 / h_as - 1e-9);  // equal zones of height <= requested
    X->h_arcsec = 648000.0 / X->nz;
    X->h = kPi / X->nz;
    const bool fp64 = opts && opts->build_fp64;
    const bool deferred = opts && opts->deferred_check;
    const int64_t nn = n > 0 ? n : 1;

    const BuildPlan plan = build_plan(n, X->nz);
    const bool two = plan.two;
    const int kb = plan.kb, nbins = plan.nbins;
    const int64_t cells_cap = plan.cells_cap, units_cap = plan.units_cap;

    xm_status st = XM_OK;
    // temporaries: one block, the part that starts as zeros first
    Slices W;
    const size_t o_zcnt = W.add<uint32_t>(X->nz);
    const size_t o_ccnt = W.add<uint32_t>(two ? cells_cap : 0);
    const int64_t pre_z = (X->nz + kPreTile - 1) / kPreTile;
    const int64_t pre_c = (cells_cap + kPreTile - 1) / kPreTile;
    const size_t o_status = W.add<uint64_t>(2 * pre_z + pre_c);
    const size_t o_small = W.add<uint32_t>(16);
    const size_t zeroed = W.bytes;
    const size_t o_geo = W.add<ZoneGeo>(X->nz);
    const size_t o_zin = W.add<uint4>(X->nz);
    const size_t o_tiles = W.add<uint4>(two ? n / kTile + nbins + 1 : 0);
    const size_t o_bin = W.add<uint32_t>(4 * (int64_t)(nbins + 1));
    const size_t o_bcur = W.add<uint32_t>((int64_t)(nbins + 1) * kCursorStep);
    const size_t o_zcells = W.add<ZoneCells>(two ? X->nz : 0);
    const size_t o_czone = W.add<uint32_t>(two ? 2 * cells_cap : 0);
    const size_t o_cstart = W.add<uint32_t>(cells_cap + 1);
    const size_t o_cunit = W.add<uint32_t>(cells_cap);
    const size_t o_unit = W.add<uint4>(units_cap + 1);
    const size_t o_ucur = W.add<uint32_t>(units_cap * kCursorStep);
    const size_t o_giants = W.add<uint32_t>(n / kGiantZone + 1);
    double *d_lon = nullptr, *d_lat = nullptr;
    unsigned char* work = nullptr;
    uint4* tmp = nullptr;
    int32_t* err = nullptr;
    int32_t h_err = 0;

    auto fail = [&](xm_status code) { st = code; };
    do {
        X->rec = (BRec*)dev_alloc(nn * sizeof(BRec), s);
        X->pos = (double2*)dev_alloc(nn * sizeof(double2), s);
        X->zhot = (ZoneHot*)dev_alloc(X->nz * sizeof(ZoneHot), s);
        if (!X->rec || !X->pos || !X->zhot) { fail(set_error(XM_ENOMEM, "index arrays")); break; }
        X->bytes = nn * (sizeof(BRec) + sizeof(double2)) + X->nz * sizeof(ZoneHot);
        if (fp64) {
            X->p64 = (double2*)dev_alloc(2 * nn * sizeof(double2), s);
            if (!X->p64) { fail(set_error(XM_ENOMEM, "index unit vectors")); break; }
            X->bytes += 2 * nn * sizeof(double2);
        }
        if (B->id) {
            X->id = (int64_t*)dev_alloc(nn * sizeof(int64_t), s);
            if (!X->id) { fail(set_error(XM_ENOMEM, "index ids")); break; }
            X->bytes += nn * sizeof(int64_t);
            if (n > 0) {
                e = cudaMemcpyAsync(X->id, B->id, n * sizeof(int64_t),
                                    B->on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, s);
                if (e != cudaSuccess) { fail(cuda_fail(e, "id copy")); break; }
            }
        }
        const double* lon = B->lon_deg;
        const double* lat = B->lat_deg;
        if (!B->on_device && n > 0) {
            d_lon = (double*)dev_alloc(2 * n * sizeof(double), s);
            if (!d_lon) { fail(set_error(XM_ENOMEM, "input copy")); break; }
            d_lat = d_lon + n;
            e = cudaMemcpyAsync(d_lon, B->lon_deg, n * sizeof(double), cudaMemcpyHostToDevice, s);
            if (e == cudaSuccess)
                e = cudaMemcpyAsync(d_lat, B->lat_deg, n * sizeof(double), cudaMemcpyHostToDevice, s);
            if (e != cudaSuccess) { fail(cuda_fail(e, "input copy")); break; }
            lon = d_lon;
            lat = d_lat;
        }
        work = (unsigned char*)dev_alloc(W.bytes, s);
        tmp = (uint4*)dev_alloc(nn * sizeof(uint4), s);
        err = (int32_t*)dev_alloc(sizeof(int32_t), s);
        // bucket tables: see k_place_b
        X->lut_n = 2 * n + 3 * (int64_t)X->nz + 2 * cells_cap + 16;
        X->lut = (uint32_t*)dev_alloc(X->lut_n * sizeof(uint32_t), s);
        if (!work || !tmp || !err || !X->lut) {
            fail(set_error(XM_ENOMEM, "index build buffers"));
            break;
        }
        X->bytes += X->lut_n * sizeof(uint32_t);
        e = cudaMemsetAsync(err, 0, sizeof(int32_t), s);
        if (e == cudaSuccess) e = cudaMemsetAsync(work, 0, zeroed, s);
        if (e != cudaSuccess) { fail(cuda_fail(e, "memset")); break; }

        auto body = [&]() -> xm_status {
            const IndexGeom G = X->geom();
            const int32_t nz = X->nz;
            const Lookback lb = lookback_settings();
            auto at32 = [&](size_t o) { return (uint32_t*)(work + o); };
            uint32_t* const zcnt = at32(o_zcnt);
            uint64_t* const status = (uint64_t*)(work + o_status);
            // [0..2] tile counters, [4] cells, [5] units,
            // [6..7] range of the RA keys, [8] units listed
            uint32_t* const small = at32(o_small);
            KeyRange* const range = (KeyRange*)(small + 6);
            uint32_t* const cstart = at32(o_cstart);
            uint32_t* const cunit = at32(o_cunit);
            uint4* const unit = (uint4*)(work + o_unit);
            uint32_t* const ucur = at32(o_ucur);
            uint4* const zin = (uint4*)(work + o_zin);
            uint4* const tile_list = (uint4*)(work + o_tiles);
            uint32_t* const bin_start = at32(o_bin);
            uint32_t* const bin_zone = bin_start + nbins + 1;
            uint32_t* const bin_tile = bin_zone + nbins + 1;
            uint32_t* const bin_chunk = bin_tile + nbins + 1;
            ZoneCells* const zcells = two ? (ZoneCells*)(work + o_zcells) : nullptr;
            uint32_t* const czone = two ? at32(o_czone) : nullptr;
            uint32_t* const csplit = two ? czone + cells_cap : nullptr;
            uint32_t* const ccnt = two ? at32(o_ccnt) : zcnt;
            prepare_build();
            const ZoneGeo* geo = nullptr;
            xm_status r = zone_geometry(nz, (ZoneGeo*)(work + o_geo), &geo, s);
            if (r != XM_OK) return r;

            // (counters in shared memory are worth their set-up from about 1e5 sources)
            const size_t wide1 = (size_t)nz * 4, wide2 = ((size_t)nz + 1) / 2 * 4;
            if (n >= (1 << 17) && wide1 <= kCountSmem) {
                XM_LAUNCH("k_zone_count", 152, kCountThreads, wide1, s, k_zone_count<1>, lat, n, nz, zcnt);
            } else if (n >= (1 << 17) && wide2 <= kCountSmem) {
                XM_LAUNCH("k_zone_count", 152, kCountThreads, wide2, s, k_zone_count<2>, lat, n, nz, zcnt);
            } else if (n > 0) {
                const int64_t g = (n + kCountThreads - 1) / kCountThreads;
                XM_LAUNCH("k_zone_count", (unsigned)(g < 8 * 152 ? g : 8 * 152), kCountThreads, 0, s,
                          k_zone_count<0>, lat, n, nz, zcnt);
            }
            const int64_t tiles = (n + kTile - 1) / kTile;
            if (!two) {
                XM_LAUNCH("k_cell_units", (unsigned)pre_c, kBlock, 0, s, k_cell_units, zcnt,
                          (uint32_t)nz, (const uint32_t*)nullptr, (const uint32_t*)nullptr,
                          (const uint32_t*)nullptr, n, geo, zin, cstart, cunit, unit, ucur,
                          (uint32_t)units_cap, small + 5, status, small, lb, err);
                // (few sources: smaller tiles, so that more blocks share them)
                auto ingest = [&](auto kernel, size_t smem, int64_t rows) -> xm_status {
                    XM_LAUNCH("k_ingest_b", (unsigned)((n + rows - 1) / rows), kSplitThreads, smem, s,
                              kernel, lon, lat, n, nz, G.h_f, zin, (int)units_cap, ucur, tmp,
                              X->pos, range, err);
                    return XM_OK;
                };
                if (n > 0 && n <= 152 * 2048)
                    r = ingest(k_ingest_b<2, false, kMaxUnits>, sizeof(SplitSmem<2, kMaxUnits>),
                               kSplitThreads * 2);
                else if (n > 0)
                    r = ingest(k_ingest_b<4, false, kMaxUnits>, sizeof(SplitSmem<4, kMaxUnits>),
                               kSplitThreads * 4);
                if (r != XM_OK) return r;
            } else {
                // (the records go to the index's own array and back: the last
                // step writes it from `tmp`)
                uint4* const rec0 = (uint4*)X->rec;
                XM_LAUNCH("k_zone_bins", (unsigned)pre_z, kBlock, 0, s, k_zone_bins, zcnt, nz, n, kb,
                          geo, zin, bin_start, bin_zone, at32(o_bcur), nbins, status, small, lb,
                          err);
                if (n > 0)
                    XM_LAUNCH("k_ingest_b", (unsigned)tiles, kSplitThreads,
                              sizeof(SplitSmem<kTileItems, kMaxBins>), s,
                              (k_ingest_b<kTileItems, true, kMaxBins>), lon, lat, n, nz, G.h_f, zin,
                              nbins, at32(o_bcur), rec0, X->pos,
                              range, err);
                XM_LAUNCH("k_zone_parts", (unsigned)pre_z + 1, kBlock, 0, s, k_zone_parts, zcnt, nz,
                          range, zcells, czone, csplit, (uint32_t)cells_cap, small + 4, bin_start,
                          nbins, bin_tile, bin_chunk, status + pre_z, small + 1, lb, err);
                if (n > 0)
                    XM_LAUNCH("k_cell_count", (unsigned)(tiles / kCountChunk + nbins + 1),
                              kSplitThreads, 0, s, k_cell_count, rec0, bin_start, bin_chunk, nbins,
                              bin_zone, zcells, small + 4, ccnt, bin_tile, tile_list, err);
                XM_LAUNCH("k_cell_units", (unsigned)pre_c, kBlock, 0, s, k_cell_units, ccnt, 0u,
                          small + 4, czone, csplit, n, geo, (uint4*)nullptr, cstart, cunit, unit, ucur,
                          (uint32_t)units_cap, small + 5, status + 2 * pre_z, small + 2, lb, err);
                if (n > 0)
                    XM_LAUNCH("k_split", (unsigned)(tiles + nbins), kSplitThreads,
                              sizeof(SplitSmem<kTileItems, kMaxDigits>), s, k_split, rec0, tile_list,
                              bin_tile + nbins, nbins, bin_zone, zcells, cunit, small + 5, n, ucur, tmp,
                              err);
            }
            if (X->p64 && n > 0)
                XM_LAUNCH("k_unit_b", (unsigned)((n + kBlock - 1) / kBlock), kBlock, 0, s, k_unit_b,
                          X->pos, n, X->p64, err);
            const uint32_t giant_rows = n <= kGiantRows ? (uint32_t)n  // (a launch saved: no list)
                                        : !two          ? kGiantZone
                                        : n >> 11 > kGiantRows ? (uint32_t)(n >> 11)
                                                               : kGiantRows;
            const PlaceArgs P{tmp, unit, small + 5, cstart, czone, zcells, range, geo, nz, n,
                              X->rec, X->lut, X->zhot, err, giant_rows, at32(o_giants), small + 8};
            XM_LAUNCH("k_place_b", (unsigned)(units_cap < kPlaceBlocks * 152 ? units_cap : kPlaceBlocks * 152),
                      kPlaceThreads, sizeof(PlaceSmem), s, k_place_b, P);
            if (n > giant_rows)
                XM_LAUNCH("k_place_giant", 152 / kGiantBlocks * kGiantBlocks, kGiantThreads, 0, s,
                          k_place_giant, P);
            return XM_OK;
        };
        st = body();
        if (st != XM_OK) break;
        if (deferred) {  // the error word stays with the index, read by its first match
            X->build_err = err;
            err = nullptr;
            break;
        }
        e = cudaMemcpyAsync(&h_err, err, sizeof(int32_t), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) { fail(cuda_fail(e, "xm_build_index sync")); break; }
        const xm_status bs = index_build_status(h_err);
        if (bs != XM_OK) { fail(bs); break; }
    } while (0);

    dev_free(d_lon, s);
    dev_free(work, s);
    dev_free(tmp, s);
    dev_free(err, s);
    if (st != XM_OK) {
        xm_index_free(X);
        return st;
    }
    *out = X;
    return XM_OK;
}

xm_status xm::index_build_status(int32_t bits) {
    if (bits & kErrCoord) return set_error(XM_EINVAL, "B: NaN/inf or |lat| > 90");
    if (bits & kErrTimeout) return set_error(XM_ETIMEOUT, "index build: look-back timed out");
    return XM_OK;
}

// The index's memory returns to the pool in the order of the stream it was
// built on, after whatever the caller queued there.
extern "C" xm_status xm_index_free(xm_index* X) {
    if (!X) return XM_OK;
    cudaStream_t s = X->stream;
    dev_free(X->rec, s);
    dev_free(X->pos, s);
    dev_free(X->p64, s);
    dev_free(X->id, s);
    dev_free(X->zhot, s);
    dev_free(X->lut, s);
    dev_free(X->build_err, s);
    delete X;
    return XM_OK;
}

extern "C" xm_status xm_index_info(const xm_index* X, int64_t* n, int64_t* zones,
                                   double* zone_height_arcsec, int64_t* device_bytes) {
    if (!X) return set_error(XM_EINVAL, "xm_index_info: NULL index");
    if (n) *n = X->n;
    if (zones) *zones = X->nz;
    if (zone_height_arcsec) *zone_height_arcsec = X->h_arcsec;
    if (device_bytes) *device_bytes = X->bytes;
    return XM_OK;
}
