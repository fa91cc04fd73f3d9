// pd_cm_mean.cu — the paper's common-mode estimator and its stacked stages.
//
// Section "Common Mode" and Fig. c: the pixels of a group whose value v is
// below the noise cut are counted (N0) and summed (S), and the group's common
// mode is S / max(N0, sqrt(G)) with G the group's pixel count; the sqrt(G)
// term keeps a group with few background pixels from being corrected by a
// noisy estimate.  The same section obtains row, column and block variants by
// summing over other groups, and section "Performance" stacks three
// common-mode stages.  Here:
//
//   PD_CM_MEAN           one stage over each unit (v = d = raw - pedestal)
//   PD_CM_MEAN_STACKED   unit, then each module row on d - cm_u, then each
//                        module column on (d - cm_u) - cm_r
//
// S is defined independently of the summation order, so that any grid gives
// the same bits: with M the largest |v| of the selected values and
// E = max(floor(log2 M), -60), each v is rounded to the grid 2^(E-38)
// (round to nearest even) as a 64-bit integer, the integers are added
// exactly, and the total is rounded once to binary32.  Values down to
// M * 2^-15 lie on the grid, so for detector data S is the exactly rounded
// sum.  Each group takes two passes over its pixels: count and largest
// magnitude, then the integer sum.
//
// The scaled values are rounded to integers by additions alone (kSplitHi):
// a 64-bit conversion per value was most of the second pass's work.
//
// Kernels (the third to fifth only for the stacked mode):
//   mean_units_block_kernel  one CTA per (frame, unit) for units of 8+ rows
//   mean_units_warp_kernel   one warp per (frame, unit) for shorter units
//   mean_rows_cols_kernel    rows and columns of one (frame, module) per CTA
//                            (even column counts; see there)
//   mean_rows_kernel         one warp per (frame, module, row)
//   mean_cols_kernel         one warp per (frame, module, 32 columns), one
//                            lane per column walking down the rows
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>

#include "pd_dev.cuh"
#include "pd_internal.cuh"

namespace pd {

namespace {

constexpr int kMeanThreads = 256;
constexpr int kMeanWarps = kMeanThreads / 32;

__device__ __forceinline__ bool selects(float v, float cut) {
    return v < cut && v > -INFINITY;
}

__device__ __forceinline__ uint32_t abs_bits(float v) { return __float_as_uint(v) & 0x7fffffffu; }

// 2^k as a float for -126 < k < 128
__device__ __forceinline__ float pow2f(int k) { return __uint_as_float((uint32_t)(127 + k) << 23); }

// grid exponent: the values are scaled by 2^k before rounding to integers
__device__ __forceinline__ int grid_k(uint32_t max_bits) {
    int e = (int)(max_bits >> 23) - 127;  // floor(log2 M); subnormal M gives -127
    if (e < -60) e = -60;
    return 38 - e;
}

// A value on the grid 2^(E-38) as an integer, by additions alone.  With y =
// v * 2^(38-E) (exact, |y| < 2^39), t = y + kSplitHi holds the multiple of
// 2^22 nearest to y in its low mantissa bits; the remainder y - (t - kSplitHi)
// is exact and at most 2^21, and u = remainder + kSplitLo holds it rounded to
// nearest even (2^22 is even, so a tie falls as it does for the whole y).
// The integer is split_hi(t) * 2^22 + split_lo(u).
constexpr float kSplitHi = 52776558133248.0f;  // 1.5 * 2^45
constexpr float kSplitLo = 12582912.0f;        // 1.5 * 2^23
constexpr int kSplitHiBits = 0x56400000, kSplitLoBits = 0x4b400000;

struct Acc {
    uint32_t n0 = 0, max_bits = 0;
    long long total = 0;

    __device__ __forceinline__ void first(float v, float cut) {
        if (selects(v, cut)) {
            n0++;
            max_bits = max(max_bits, abs_bits(v));
        }
    }
    __device__ __forceinline__ void second(float v, float cut, float scale) {
        const float x = selects(v, cut) ? v : 0.0f;
        const float t = __fmaf_rn(x, scale, kSplitHi);
        const float u = __fadd_rn(__fmaf_rn(x, scale, -__fsub_rn(t, kSplitHi)), kSplitLo);
        total += (long long)(__float_as_int(t) - kSplitHiBits) * (1ll << 22) +
                 (__float_as_int(u) - kSplitLoBits);
    }
};

__device__ __forceinline__ float mean_of(long long total, uint32_t n0, uint32_t max_bits,
                                         float guard) {
    float sum = 0.0f;
    if (n0 > 0 && max_bits != 0) sum = __fmul_rn(__ll2float_rn(total), pow2f(-grid_k(max_bits)));
    return __fdiv_rn(sum, fmaxf((float)n0, guard));
}

__device__ __forceinline__ long long warp_sum64(long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ float dark(const uint16_t* raw, const float* nped, size_t off) {
    return __fadd_rn(__uint2float_rn(raw[off]), nped[off]);
}

// A pixel's common-mode input: d, or in the paper's order d * inv_gain (NaN
// for masked pixels, which no selection takes).
__device__ __forceinline__ float cmv(bool ag, const uint16_t* raw, const float* nped,
                                     const float* ig, size_t off) {
    const float d = dark(raw, nped, off);
    return ag ? cm_input(true, d, ig[off]) : d;
}

// Offsets of frame f, unit u in the pixel arrays and its rectangle origin.
struct UnitAt {
    size_t raw_off, map_off;
};

__device__ __forceinline__ UnitAt unit_at(const ChainParams& p, uint32_t f, uint32_t u) {
    const uint32_t m = u / p.units_per_module, uu = u % p.units_per_module;
    const uint32_t r0 = (uu / p.units_per_row) * p.unit_rows;
    const uint32_t c0 = (uu % p.units_per_row) * p.unit_cols;
    const size_t map = (size_t)m * p.module_px + (size_t)r0 * p.cols + c0;
    return UnitAt{(size_t)f * p.frame_px + map, map};
}

// ---------------------------------------------------------------------------
// Stage 1.  The threads of a group (a CTA or a warp) walk the unit's pixels in
// raster order, V adjacent columns a step, four steps of loads in flight; the
// position advances with a carry instead of a division.  V = 2 needs even
// columns and unit widths (4- and 8-byte loads).  f(v) sees every pixel of the
// unit and, at the end, NaN in the place of pixels past it; after() runs every
// kSweepSteps V pixels.
constexpr int kSweepSteps = 4;
template <int V, bool AG, class F, class G>
__device__ __forceinline__ void sweep_unit(const ChainParams& p, const uint16_t* __restrict__ rw,
                                           const float* __restrict__ np_,
                                           const float* __restrict__ ig_, uint32_t t,
                                           uint32_t stride, F f, G after) {
    constexpr int U = kSweepSteps;
    const uint32_t W = p.unit_cols / V, n = p.unit_rows * W;
    const uint32_t dr = stride / W, dc = stride - dr * W;
    uint32_t c = t % W, off = t / W * p.cols + c * V;
    const uint32_t step = dr * p.cols + dc * V, carry = p.cols - p.unit_cols;
    const float nan = __int_as_float(0x7fc00000);
    for (uint32_t i = t; i < n; i += U * stride) {
        uint32_t x[U];
        float2 np[U], ig[U];
#pragma unroll
        for (int k = 0; k < U; k++) {
            x[k] = 0;
            np[k] = make_float2(nan, nan);
            ig[k] = make_float2(1.0f, 1.0f);
            if (i + k * stride < n) {
                if (V == 2) {
                    x[k] = __ldg(reinterpret_cast<const uint32_t*>(rw + off));
                    np[k] = __ldg(reinterpret_cast<const float2*>(np_ + off));
                    if (AG) ig[k] = __ldg(reinterpret_cast<const float2*>(ig_ + off));
                } else {
                    x[k] = __ldg(rw + off);
                    np[k].x = __ldg(np_ + off);
                    if (AG) ig[k].x = __ldg(ig_ + off);
                }
            }
            off += step;
            c += dc;
            if (c >= W) {
                c -= W;
                off += carry;
            }
        }
#pragma unroll
        for (int k = 0; k < U; k++) {
            const float2 d = __fadd2_rn(raw_pair(x[k]), np[k]);
            f(AG ? cm_input(true, d.x, ig[k].x) : d.x);
            if (V == 2) f(AG ? cm_input(true, d.y, ig[k].y) : d.y);
        }
        after();
    }
}

// One pass where the context's pedestals allow it (p.mean_frac = g >= 0): every
// selected d is then a whole number of 2^-g below 2^26 (kFixedBits) of them (see
// mean_frac_bits), a grid the definition's 2^(E-38) always divides, so the
// integers can be added without knowing M, and the unit is read once.
constexpr int kFixedBits = 26;
struct FixedAcc {
    uint32_t n0 = 0;
    int part = 0;         // of the kSweepSteps V <= 8 values between two flushes
    static_assert(((2ll * kSweepSteps) << kFixedBits) < (1ll << 31), "part in 32 bits");
    long long total = 0;
    __device__ __forceinline__ void add(float d, float cut, float scale) {
        const bool sel = d < cut;
        n0 += sel;
        part += __float2int_rn(sel ? __fmul_rn(d, scale) : 0.0f);
    }
    __device__ __forceinline__ void flush() {
        total += part;
        part = 0;
    }
};

__device__ __forceinline__ float fixed_mean_of(long long total, uint32_t n0, int g, float guard) {
    return __fdiv_rn(__fmul_rn(__ll2float_rn(total), pow2f(-g)), fmaxf((float)n0, guard));
}

// units of at least 8 rows: one CTA each
template <int V, bool AG, bool FIXED>
__global__ void __launch_bounds__(kMeanThreads)
    mean_units_block_kernel(ChainParams p, const uint16_t* __restrict__ raw,
                            float* __restrict__ cm) {
    __shared__ uint32_t s_n0, s_max;
    __shared__ unsigned long long s_total;
    const uint32_t f = blockIdx.x / p.units_per_frame, u = blockIdx.x % p.units_per_frame;
    const UnitAt at = unit_at(p, f, u);
    const uint16_t* rw = raw + at.raw_off;
    const float* np_ = p.nped + at.map_off;
    const float* ig_ = p.inv_gain + at.map_off;
    const int lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        s_n0 = 0;
        s_max = 0;
        s_total = 0;
    }
    __syncthreads();
    float* dst = cm + (size_t)f * cm_per_frame(p) + u;
    const float guard = __fsqrt_rn((float)p.unit_px);
    if (FIXED) {
        FixedAcc a;
        const float scale = pow2f(p.mean_frac);
        sweep_unit<V, false>(p, rw, np_, ig_, threadIdx.x, kMeanThreads,
                             [&](float v) { a.add(v, p.cm_cut, scale); }, [&] { a.flush(); });
        const uint32_t wn = __reduce_add_sync(0xffffffffu, a.n0);
        const long long wt = warp_sum64(a.total);
        if (lane == 0) {
            atomicAdd(&s_n0, wn);
            atomicAdd(&s_total, (unsigned long long)wt);
        }
        __syncthreads();
        if (threadIdx.x == 0) *dst = fixed_mean_of((long long)s_total, s_n0, p.mean_frac, guard);
        return;
    }
    Acc a;
    sweep_unit<V, AG>(p, rw, np_, ig_, threadIdx.x, kMeanThreads,
                      [&](float v) { a.first(v, p.cm_cut); }, [] {});
    const uint32_t wn = __reduce_add_sync(0xffffffffu, a.n0);
    const uint32_t wm = __reduce_max_sync(0xffffffffu, a.max_bits);
    if (lane == 0) {
        atomicAdd(&s_n0, wn);
        atomicMax(&s_max, wm);
    }
    __syncthreads();
    const uint32_t n0 = s_n0, mb = s_max;
    if (n0 > 0 && mb != 0) {
        const float scale = pow2f(grid_k(mb));
        sweep_unit<V, AG>(p, rw, np_, ig_, threadIdx.x, kMeanThreads,
                          [&](float v) { a.second(v, p.cm_cut, scale); }, [] {});
        const long long wt = warp_sum64(a.total);
        if (lane == 0) atomicAdd(&s_total, (unsigned long long)wt);
        __syncthreads();
    }
    if (threadIdx.x == 0) *dst = mean_of((long long)s_total, n0, mb, guard);
}

// units of fewer than 8 rows: one warp each
template <int V, bool AG, bool FIXED>
__global__ void __launch_bounds__(kMeanThreads)
    mean_units_warp_kernel(ChainParams p, const uint16_t* __restrict__ raw,
                           float* __restrict__ cm, uint32_t n_units) {
    const uint32_t item = blockIdx.x * kMeanWarps + (threadIdx.x >> 5);
    if (item >= n_units) return;  // whole warps leave together
    const int lane = threadIdx.x & 31;
    const uint32_t f = item / p.units_per_frame;
    const uint32_t u = item % p.units_per_frame;
    const UnitAt at = unit_at(p, f, u);
    const uint16_t* rw = raw + at.raw_off;
    const float* np_ = p.nped + at.map_off;
    const float* ig_ = p.inv_gain + at.map_off;
    float* dst = cm + (size_t)f * cm_per_frame(p) + u;
    const float guard = __fsqrt_rn((float)p.unit_px);
    if (FIXED) {
        FixedAcc a;
        const float scale = pow2f(p.mean_frac);
        sweep_unit<V, false>(p, rw, np_, ig_, lane, 32,
                             [&](float v) { a.add(v, p.cm_cut, scale); }, [&] { a.flush(); });
        const uint32_t n0 = __reduce_add_sync(0xffffffffu, a.n0);
        const long long total = warp_sum64(a.total);
        if (lane == 0) *dst = fixed_mean_of(total, n0, p.mean_frac, guard);
        return;
    }
    Acc a;
    sweep_unit<V, AG>(p, rw, np_, ig_, lane, 32, [&](float v) { a.first(v, p.cm_cut); }, [] {});
    const uint32_t n0 = __reduce_add_sync(0xffffffffu, a.n0);
    const uint32_t mb = __reduce_max_sync(0xffffffffu, a.max_bits);
    long long total = 0;
    if (n0 > 0 && mb != 0) {
        const float scale = pow2f(grid_k(mb));
        sweep_unit<V, AG>(p, rw, np_, ig_, lane, 32,
                          [&](float v) { a.second(v, p.cm_cut, scale); }, [] {});
        total = warp_sum64(a.total);
    }
    if (lane == 0) *dst = mean_of(total, n0, mb, guard);
}

// ---------------------------------------------------------------------------
// Stages 2 and 3 of one (frame, module) per CTA, for even columns and unit
// widths (two-column loads; at most 64 NP columns).  Warps take whole rows: a
// row's values stay in registers from its selection to its sum, and once its
// term is known the same registers give the columns' counts and largest
// magnitudes; a second walk over the rows adds the columns' sums.  Each pixel
// is read twice instead of four times, and the next row's loads are in flight
// while a row is summed.  Bound by issue (about 20 and 15 instructions a pixel
// in the two walks); 16 warps of 128 registers per SM keep a row of loads each
// in flight.  The whole stacked common mode of 64 frames of 32 x 185 x 388
// took 1036 us with a warp per row and a lane per column, each reading its
// pixels twice and rounding by 64-bit conversions, and takes 372 us.  Wider
// modules than 1000 columns, odd widths and the paper's order keep those
// kernels.
struct RowsColsSmem {
    float* cu;       // [units_per_module]
    float* cr;       // [rows]
    uint32_t* cmax;  // [cols] largest selected |v| of a column, as bits
    uint32_t* cn;    // [cols] selected values
    uint32_t* chi;   // [cols] sums of the two parts of the grid integers
    uint32_t* clo;
};

size_t rows_cols_smem_bytes(const ChainParams& p) {
    return ((size_t)p.units_per_module + p.rows + 4 * (size_t)p.cols) * 4;
}

// NP: column pairs a lane holds, one per 64 columns.  Up to seven, a row's loads,
// values and column sums fit 128 registers and two CTAs an SM; more take 148 to
// 254 and one CTA (none spills).
template <int NP>
__global__ void __launch_bounds__(kMeanThreads, NP <= 7 ? 2 : 1)
    mean_rows_cols_kernel(ChainParams p, const uint16_t* __restrict__ raw,
                          float* __restrict__ cm) {
    extern __shared__ uint32_t rc_smem[];
    RowsColsSmem S;
    S.cu = reinterpret_cast<float*>(rc_smem);
    S.cr = S.cu + p.units_per_module;
    S.cmax = reinterpret_cast<uint32_t*>(S.cr + p.rows);
    S.cn = S.cmax + p.cols;
    S.chi = S.cn + p.cols;
    S.clo = S.chi + p.cols;
    const uint32_t m = blockIdx.x % p.n_modules, f = blockIdx.x / p.n_modules;
    const size_t map = (size_t)m * p.module_px;
    const uint16_t* rw = raw + (size_t)f * p.frame_px + map;
    const float* np_ = p.nped + map;
    float* cmf = cm + (size_t)f * cm_per_frame(p);
    const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (uint32_t i = tid; i < p.units_per_module; i += kMeanThreads)
        S.cu[i] = -cmf[(size_t)m * p.units_per_module + i];
    for (uint32_t i = tid; i < 4 * p.cols; i += kMeanThreads) S.cmax[i] = 0;
    __syncthreads();

    const uint32_t pairs = p.cols / 2;
    const float cut = p.cm_cut;
    const float nan = __int_as_float(0x7fc00000);
    uint32_t uc[NP];  // unit column of the lane's pairs
#pragma unroll
    for (int j = 0; j < NP; j++) uc[j] = min(2 * (lane + 32 * j), p.cols - 1) / p.unit_cols;

    uint32_t x[NP];
    float2 np[NP];
    auto load = [&](uint32_t r) {
        const uint32_t base = r * p.cols + 2 * lane;
#pragma unroll
        for (int j = 0; j < NP; j++) {
            x[j] = 0;
            np[j] = make_float2(nan, nan);
            if (lane + 32 * j < pairs) {
                x[j] = __ldg(reinterpret_cast<const uint32_t*>(rw + base + 64 * j));
                np[j] = __ldg(reinterpret_cast<const float2*>(np_ + base + 64 * j));
            }
        }
    };
    // d - cm_u of the loaded row r
    auto values = [&](uint32_t r, float2 (&v)[NP]) {
        const float* cu = S.cu + (p.unit_rows == p.rows ? 0u : r / p.unit_rows * p.units_per_row);
#pragma unroll
        for (int j = 0; j < NP; j++) {
            const float c = cu[uc[j]];
            v[j] = __fadd2_rn(__fadd2_rn(raw_pair(x[j]), np[j]), make_float2(c, c));
        }
    };
    const float2 hi2 = make_float2(kSplitHi, kSplitHi), nhi2 = make_float2(-kSplitHi, -kSplitHi);
    const float2 lo2 = make_float2(kSplitLo, kSplitLo);
    const float2 neg1 = make_float2(-1.0f, -1.0f);

    // walk 1: the rows' terms, and the columns' counts and magnitudes
    {
        float2 cmx[NP];
        uint32_t cn[NP];  // counts of the pair's columns, 16 bits each
#pragma unroll
        for (int j = 0; j < NP; j++) {
            cmx[j] = make_float2(0.0f, 0.0f);
            cn[j] = 0;
        }
        if (warp < p.rows) load(warp);
        const float guard = __fsqrt_rn((float)p.cols);
        for (uint32_t r = warp; r < p.rows; r += kMeanWarps) {
            float2 v[NP];
            values(r, v);
            if (r + kMeanWarps < p.rows) load(r + kMeanWarps);
            uint32_t n0 = 0;
            float mx = 0.0f;
#pragma unroll
            for (int j = 0; j < NP; j++) {
                if (v[j].x < cut) {
                    n0++;
                    mx = fmaxf(mx, fabsf(v[j].x));
                }
                if (v[j].y < cut) {
                    n0++;
                    mx = fmaxf(mx, fabsf(v[j].y));
                }
            }
            n0 = __reduce_add_sync(0xffffffffu, n0);
            const uint32_t mb = __reduce_max_sync(0xffffffffu, __float_as_uint(mx));
            long long total = 0;
            if (mb != 0) {
                const float sc = pow2f(grid_k(mb));
                const float2 sc2 = make_float2(sc, sc);
                uint32_t hi = 0, lo = 0;
#pragma unroll
                for (int j = 0; j < NP; j++) {
                    const float2 y = make_float2(v[j].x < cut ? v[j].x : 0.0f,
                                                 v[j].y < cut ? v[j].y : 0.0f);
                    const float2 t = __ffma2_rn(y, sc2, hi2);
                    const float2 a = __fadd2_rn(t, nhi2);
                    const float2 u = __fadd2_rn(__ffma2_rn(y, sc2, __fmul2_rn(a, neg1)), lo2);
                    hi += __float_as_uint(t.x) + __float_as_uint(t.y);
                    lo += __float_as_uint(u.x) + __float_as_uint(u.y);
                }
                hi = __reduce_add_sync(0xffffffffu, hi - 2u * NP * (uint32_t)kSplitHiBits);
                lo = __reduce_add_sync(0xffffffffu, lo - 2u * NP * (uint32_t)kSplitLoBits);
                total = (long long)(int)hi * (1ll << 22) + (int)lo;
            }
            const float ncr = -mean_of(total, n0, mb, guard);
            if (lane == 0) S.cr[r] = ncr;
            const float2 ncr2 = make_float2(ncr, ncr);
#pragma unroll
            for (int j = 0; j < NP; j++) {
                const float2 w = __fadd2_rn(v[j], ncr2);
                if (w.x < cut) {
                    cn[j]++;
                    cmx[j].x = fmaxf(cmx[j].x, fabsf(w.x));
                }
                if (w.y < cut) {
                    cn[j] += 0x10000u;
                    cmx[j].y = fmaxf(cmx[j].y, fabsf(w.y));
                }
            }
        }
#pragma unroll
        for (int j = 0; j < NP; j++) {
            const uint32_t c = 2 * (lane + 32 * j);
            if (c < p.cols) {
                atomicMax(&S.cmax[c], __float_as_uint(cmx[j].x));
                atomicMax(&S.cmax[c + 1], __float_as_uint(cmx[j].y));
                atomicAdd(&S.cn[c], cn[j] & 0xFFFFu);
                atomicAdd(&S.cn[c + 1], cn[j] >> 16);
            }
        }
    }
    __syncthreads();

    // walk 2: the columns' sums
    {
        float2 sc[NP];
        uint32_t hi[2 * NP], lo[2 * NP];
#pragma unroll
        for (int j = 0; j < NP; j++) {
            const uint32_t c = 2 * (lane + 32 * j);
            sc[j] = make_float2(0.0f, 0.0f);  // a column without values adds nothing
            if (c < p.cols) {
                if (S.cmax[c]) sc[j].x = pow2f(grid_k(S.cmax[c]));
                if (S.cmax[c + 1]) sc[j].y = pow2f(grid_k(S.cmax[c + 1]));
            }
            hi[2 * j] = hi[2 * j + 1] = lo[2 * j] = lo[2 * j + 1] = 0;
        }
        if (warp < p.rows) load(warp);
        uint32_t n_rows = 0;
        for (uint32_t r = warp; r < p.rows; r += kMeanWarps, n_rows++) {
            float2 v[NP];
            values(r, v);
            if (r + kMeanWarps < p.rows) load(r + kMeanWarps);
            const float ncr = S.cr[r];
            const float2 ncr2 = make_float2(ncr, ncr);
#pragma unroll
            for (int j = 0; j < NP; j++) {
                const float2 w = __fadd2_rn(v[j], ncr2);
                const float2 y = make_float2(w.x < cut ? w.x : 0.0f, w.y < cut ? w.y : 0.0f);
                const float2 t = __ffma2_rn(y, sc[j], hi2);
                const float2 a = __fadd2_rn(t, nhi2);
                const float2 u = __fadd2_rn(__ffma2_rn(y, sc[j], __fmul2_rn(a, neg1)), lo2);
                hi[2 * j] += __float_as_uint(t.x);
                hi[2 * j + 1] += __float_as_uint(t.y);
                lo[2 * j] += __float_as_uint(u.x);
                lo[2 * j + 1] += __float_as_uint(u.y);
            }
        }
#pragma unroll
        for (int j = 0; j < NP; j++) {
            const uint32_t c = 2 * (lane + 32 * j);
            if (c < p.cols) {
                atomicAdd(&S.chi[c], hi[2 * j] - n_rows * (uint32_t)kSplitHiBits);
                atomicAdd(&S.chi[c + 1], hi[2 * j + 1] - n_rows * (uint32_t)kSplitHiBits);
                atomicAdd(&S.clo[c], lo[2 * j] - n_rows * (uint32_t)kSplitLoBits);
                atomicAdd(&S.clo[c + 1], lo[2 * j + 1] - n_rows * (uint32_t)kSplitLoBits);
            }
        }
    }
    __syncthreads();
    float* row_out = cmf + p.units_per_frame + (size_t)m * p.rows;
    for (uint32_t r = tid; r < p.rows; r += kMeanThreads) row_out[r] = -S.cr[r];
    float* col_out = cmf + p.units_per_frame + (size_t)p.n_modules * p.rows + (size_t)m * p.cols;
    const float guard = __fsqrt_rn((float)p.rows);
    for (uint32_t c = tid; c < p.cols; c += kMeanThreads)
        col_out[c] = mean_of((long long)(int)S.chi[c] * (1ll << 22) + (int)S.clo[c], S.cn[c],
                             S.cmax[c], guard);
}

// ---------------------------------------------------------------------------
// stage 2: one warp per (frame, module, row), on d - cm_u
__global__ void __launch_bounds__(kMeanThreads)
    mean_rows_kernel(ChainParams p, const uint16_t* __restrict__ raw, float* __restrict__ cm,
                     uint32_t n_rows) {
    const uint32_t item = blockIdx.x * kMeanWarps + (threadIdx.x >> 5);
    if (item >= n_rows) return;
    const int lane = threadIdx.x & 31;
    const uint32_t r = item % p.rows;
    const uint32_t fm = item / p.rows;
    const uint32_t m = fm % p.n_modules, f = fm / p.n_modules;
    const size_t map = (size_t)m * p.module_px + (size_t)r * p.cols;
    const uint16_t* rw = raw + (size_t)f * p.frame_px + map;
    const float* np_ = p.nped + map;
    const float* ig_ = p.inv_gain + map;
    const bool ag = cm_after_gain(p);
    const float* cmf = cm + (size_t)f * cm_per_frame(p);
    const float* cmu = cmf + (size_t)m * p.units_per_module + (r / p.unit_rows) * p.units_per_row;
    Acc a;
    for (uint32_t j = 0; j < p.units_per_row; j++) {
        const float cu = cmu[j];
        for (uint32_t c = j * p.unit_cols + lane; c < (j + 1) * p.unit_cols; c += 32)
            a.first(__fsub_rn(cmv(ag, rw, np_, ig_, c), cu), p.cm_cut);
    }
    const uint32_t n0 = __reduce_add_sync(0xffffffffu, a.n0);
    const uint32_t mb = __reduce_max_sync(0xffffffffu, a.max_bits);
    long long total = 0;
    if (n0 > 0 && mb != 0) {
        const float scale = pow2f(grid_k(mb));
        for (uint32_t j = 0; j < p.units_per_row; j++) {
            const float cu = cmu[j];
            for (uint32_t c = j * p.unit_cols + lane; c < (j + 1) * p.unit_cols; c += 32)
                a.second(__fsub_rn(cmv(ag, rw, np_, ig_, c), cu), p.cm_cut, scale);
        }
        total = warp_sum64(a.total);
    }
    if (lane == 0)
        cm[(size_t)f * cm_per_frame(p) + p.units_per_frame + (size_t)m * p.rows + r] =
            mean_of(total, n0, mb, __fsqrt_rn((float)p.cols));
}

// stage 3: one warp per (frame, module, block of 32 columns), one lane per
// column, on (d - cm_u) - cm_r
__global__ void __launch_bounds__(kMeanThreads)
    mean_cols_kernel(ChainParams p, const uint16_t* __restrict__ raw, float* __restrict__ cm,
                     uint32_t col_blocks, uint32_t n_items) {
    const uint32_t item = blockIdx.x * kMeanWarps + (threadIdx.x >> 5);
    if (item >= n_items) return;
    const int lane = threadIdx.x & 31;
    const uint32_t cb = item % col_blocks;
    const uint32_t fm = item / col_blocks;
    const uint32_t m = fm % p.n_modules, f = fm / p.n_modules;
    const uint32_t c = cb * 32 + lane;
    if (c >= p.cols) return;  // lanes stay independent from here on
    const size_t map = (size_t)m * p.module_px + c;
    const uint16_t* rw = raw + (size_t)f * p.frame_px + map;
    const float* np_ = p.nped + map;
    const float* ig_ = p.inv_gain + map;
    const bool ag = cm_after_gain(p);
    const float* cmf = cm + (size_t)f * cm_per_frame(p);
    const float* cmu = cmf + (size_t)m * p.units_per_module + c / p.unit_cols;
    const float* cmr = cmf + p.units_per_frame + (size_t)m * p.rows;
    const uint32_t unit_blocks = p.rows / p.unit_rows;
    Acc a;
    for (uint32_t b = 0; b < unit_blocks; b++) {
        const float cu = cmu[(size_t)b * p.units_per_row];
        for (uint32_t r = b * p.unit_rows; r < (b + 1) * p.unit_rows; r++)
            a.first(__fsub_rn(__fsub_rn(cmv(ag, rw, np_, ig_, (size_t)r * p.cols), cu), cmr[r]),
                    p.cm_cut);
    }
    if (a.n0 > 0 && a.max_bits != 0) {
        const float scale = pow2f(grid_k(a.max_bits));
        for (uint32_t b = 0; b < unit_blocks; b++) {
            const float cu = cmu[(size_t)b * p.units_per_row];
            for (uint32_t r = b * p.unit_rows; r < (b + 1) * p.unit_rows; r++)
                a.second(__fsub_rn(__fsub_rn(cmv(ag, rw, np_, ig_, (size_t)r * p.cols), cu), cmr[r]),
                         p.cm_cut, scale);
        }
    }
    cm[(size_t)f * cm_per_frame(p) + p.units_per_frame + (size_t)p.n_modules * p.rows +
       (size_t)m * p.cols + c] = mean_of(a.total, a.n0, a.max_bits, __fsqrt_rn((float)p.rows));
}

unsigned warps_grid(unsigned long long items) {
    return (unsigned)((items + kMeanWarps - 1) / kMeanWarps);
}

}  // namespace

namespace {
template <int V, bool AG, bool FIXED>
void launch_units(const ChainParams& p, const uint16_t* fr, float* cm, uint32_t units,
                  cudaStream_t s) {
    if (p.unit_rows >= kMeanWarps)
        mean_units_block_kernel<V, AG, FIXED><<<units, kMeanThreads, 0, s>>>(p, fr, cm);
    else
        mean_units_warp_kernel<V, AG, FIXED><<<warps_grid(units), kMeanThreads, 0, s>>>(p, fr, cm,
                                                                                       units);
}
template <int V>
void launch_units(const ChainParams& p, const uint16_t* fr, float* cm, uint32_t units,
                  cudaStream_t s) {
    if (cm_after_gain(p))
        launch_units<V, true, false>(p, fr, cm, units, s);
    else if (p.mean_frac >= 0)
        launch_units<V, false, true>(p, fr, cm, units, s);
    else
        launch_units<V, false, false>(p, fr, cm, units, s);
}

// The fused rows and columns apply: column pairs inside one unit, at most 16
// pairs a lane, the 32-bit parts of the sums (2^21 a value) of a row and of a
// column in range, values that stay finite (mean_frac >= 0 bounds the
// pedestals), and the tables in the default shared memory.
bool rows_cols_ok(const ChainParams& p) {
    return !cm_after_gain(p) && p.mean_frac >= 0 && p.cols % 2 == 0 && p.unit_cols % 2 == 0 &&
           p.cols <= 1000 && p.rows <= 1000 && rows_cols_smem_bytes(p) <= 48 * 1024;
}

void launch_rows_cols(const ChainParams& p, const uint16_t* fr, float* cm, uint32_t nf,
                      cudaStream_t s) {
    // an instance for every number of pairs, so that no lane sums pairs past the
    // row's end (the call of 60 frames of 4 x 400 rows, against instances for 3, 6,
    // 7, 12 and 16 pairs: 64 columns 73 -> 60 us, 256 149 -> 131, 512 313 -> 264)
    using Kernel = decltype(&mean_rows_cols_kernel<1>);
    constexpr Kernel by_groups[] = {
        mean_rows_cols_kernel<1>,  mean_rows_cols_kernel<2>,  mean_rows_cols_kernel<3>,
        mean_rows_cols_kernel<4>,  mean_rows_cols_kernel<5>,  mean_rows_cols_kernel<6>,
        mean_rows_cols_kernel<7>,  mean_rows_cols_kernel<8>,  mean_rows_cols_kernel<9>,
        mean_rows_cols_kernel<10>, mean_rows_cols_kernel<11>, mean_rows_cols_kernel<12>,
        mean_rows_cols_kernel<13>, mean_rows_cols_kernel<14>, mean_rows_cols_kernel<15>,
        mean_rows_cols_kernel<16>};
    const Kernel k = by_groups[(p.cols + 63) / 64 - 1];
    k<<<nf * p.n_modules, kMeanThreads, rows_cols_smem_bytes(p), s>>>(p, fr, cm);
}
}  // namespace

int mean_frac_bits(const ChainParams& p, const float* pedestal) {
    // g: the finest binary place of any pedestal.  A difference d = raw -
    // pedestal is then a whole number of 2^-g whether or not binary32 rounded
    // it, and the selected ones, between -max(pedestal) and the cut, stay
    // below 2^26 of them.  E <= 38 - g follows, so the grid of the
    // definition divides 2^-g.
    if (!(p.cm_cut > -1e6f && p.cm_cut < 1e6f)) return -1;
    int g = 0;
    float most = fabsf(p.cm_cut);
    for (size_t i = 0; i < p.frame_px; i++) {
        uint32_t bits;
        memcpy(&bits, pedestal + i, 4);
        bits &= 0x7fffffffu;
        if (bits == 0) continue;
        const float v = fabsf(pedestal[i]);
        if (!(v < 1e6f)) return -1;
        most = fmaxf(most, v);
        // v = mant * 2^(e - 150), mant with its trailing zeros
        const int e = (int)(bits >> 23);
        const uint32_t mant = (bits & 0x7fffffu) | (e ? 0x800000u : 0u);
        g = std::max(g, 150 - std::max(e, 1) - __builtin_ctz(mant));
        if (g > 24) return -1;
    }
    return ldexpf(most, g) < (float)(1 << kFixedBits) ? g : -1;
}

cudaError_t launch_cm_mean(const ChainParams& p, const uint16_t* raw, uint32_t n_frames,
                           float* cm, cudaStream_t stream) {
    if (n_frames == 0) return cudaSuccess;
    // frames in groups whose work items (units, module rows, column blocks)
    // stay below 2^31, so the kernels index them in 32 bits
    const uint64_t per_frame = std::max<uint64_t>(
        {(uint64_t)p.units_per_frame, (uint64_t)p.n_modules * p.rows,
         (uint64_t)p.n_modules * ((p.cols + 31) / 32), 1});
    const uint32_t group = (uint32_t)std::max<uint64_t>(1, ((1ull << 31) - 1) / per_frame);
    const uint32_t col_blocks = (p.cols + 31) / 32;
    for (uint32_t f0 = 0; f0 < n_frames; f0 += group) {
        const uint32_t nf = std::min(group, n_frames - f0);
        const uint16_t* fr = raw + (size_t)f0 * p.frame_px;
        float* cmf = cm + (size_t)f0 * cm_per_frame(p);
        const uint32_t units = nf * p.units_per_frame;
        if (p.cols % 2 == 0 && p.unit_cols % 2 == 0)
            launch_units<2>(p, fr, cmf, units, stream);
        else
            launch_units<1>(p, fr, cmf, units, stream);
        if (cm_kind(p) != PD_CM_MEAN_STACKED) continue;
        if (rows_cols_ok(p)) {
            launch_rows_cols(p, fr, cmf, nf, stream);
            continue;
        }
        const uint32_t rows = nf * p.n_modules * p.rows;
        mean_rows_kernel<<<warps_grid(rows), kMeanThreads, 0, stream>>>(p, fr, cmf, rows);
        const uint32_t cols = nf * p.n_modules * col_blocks;
        mean_cols_kernel<<<warps_grid(cols), kMeanThreads, 0, stream>>>(p, fr, cmf, col_blocks,
                                                                        cols);
    }
    return cudaGetLastError();
}

}  // namespace pd
