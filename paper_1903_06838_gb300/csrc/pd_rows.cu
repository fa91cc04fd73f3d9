// pd_rows.cu — common mode of one-row units (ASIC rows), one warp per unit.
//
// Section "Common Mode", Fig. c; the estimator is the lower median over d <
// cut.  Each lane holds up to sixteen pixels as 16-bit bin codes, two a
// register: code = clamp(8 min(raw, rcap) + K'_p, first, spare), the integer
// form of floor(8 (d - lo)) that the bank median uses (pd_lean.cuh), over a
// window of 1024 ADU below the cut.  Non-negative binary16 numbers order like
// their bit patterns, so one packed half-precision comparison and one packed
// addition count two pixels below a pivot, and a few such counts bracket the
// rank: from a first pivot near the median (the mean of medians of three), a
// step scaled by the rank still missing, then bisection, until at most
// kRowFew values are left.  Those are ranked by their binary32 d, so values
// that share a code, or lie below the window, need no case of their own.
//
// Bound by issue (78 % of the cycles).  The histogram form (cm_rows_kernel,
// pd_fast.cu) spent 804 warp instructions on a 384-pixel row: codes pixel by
// pixel, a shared histogram zeroed, filled and scanned for the bin, a second
// for the sub-bin; this one spends 567.  45 frames of 16 x 352 x 384 at 12 keV:
// 214 -> 157 us; 15 frames of 704 x 768: 23.7 -> 18.0 us.  The histogram form
// stays for units of several rows, odd sizes and pedestals the codes cannot
// hold.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

#include "pd_dev.cuh"
#include "pd_lean.cuh"

namespace pd {

namespace {

constexpr int kRowUnitWarps = 8;
constexpr uint32_t kRowFew = 16;  // values left when counting stops
constexpr uint32_t kRowMost = 32; // more of them share one code: radix select

struct RowShared {
    uint32_t hist[256];                    // the radix select's
    __align__(16) uint32_t few[kRowMost];  // order keys of the values left
};

__device__ __forceinline__ uint32_t min_u16x2(uint32_t a, uint32_t b) {
    uint32_t d;
    asm("min.u16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
__device__ __forceinline__ uint32_t max_u16x2(uint32_t a, uint32_t b) {
    uint32_t d;
    asm("max.u16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
__device__ __forceinline__ uint32_t med3_u16x2(uint32_t a, uint32_t b, uint32_t c) {
    return max_u16x2(min_u16x2(a, b), min_u16x2(max_u16x2(a, b), c));
}
__device__ __forceinline__ __half2 as_half2(uint32_t v) {
    return *reinterpret_cast<const __half2*>(&v);
}

// Codes below the pivot, over the warp.  The halves count up from 512, so
// that their sum is 1024 + count, whose low mantissa bits are the count.
template <int W>
__device__ __forceinline__ uint32_t count_below(const uint32_t (&code)[W], uint32_t pivot) {
    const __half2 pv = as_half2(pivot * 0x10001u);
    __half2 acc = __floats2half2_rn(512.0f, 512.0f);
#pragma unroll
    for (int j = 0; j < W; j++) acc = __hadd2(acc, __hlt2(as_half2(code[j]), pv));
    const __half sum = __hadd(__low2half(acc), __high2half(acc));
    return __reduce_add_sync(0xffffffffu, (uint32_t)__half_as_ushort(sum)) - 32u * 0x6400u;
}

// The element of rank k among the unit's values below the cut, by four passes
// of 8 bits over their order keys (more than kRowMost values of one code).
__device__ float row_radix(const uint16_t* rw, const float* np_, uint32_t npx,
                                        float cut, uint32_t k, uint32_t* hist) {
    const uint32_t lane = threadIdx.x & 31;
    uint32_t prefix = 0;
    for (int shift = 24; shift >= 0; shift -= 8) {
        __syncwarp();
        for (uint32_t i = lane; i < 256; i += 32) hist[i] = 0;
        __syncwarp();
        for (uint32_t i = lane; i < npx; i += 32) {
            const float d = __fadd_rn(__uint2float_rn(rw[i]), np_[i]);
            const uint32_t key = order_key(d);
            if (d < cut && (shift == 24 || key >> (shift + 8) == prefix))
                atomicAdd(&hist[(key >> shift) & 255u], 1u);
        }
        __syncwarp();
        uint32_t sum = 0;
        for (int j = 0; j < 8; j++) sum += hist[8 * lane + j];
        uint32_t incl = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= (uint32_t)o) incl += v;
        }
        // the lane whose bins hold the rank finds the digit and what is left
        uint32_t below = incl - sum, digit = 0;
        const bool mine = below <= k && k < incl;
        if (mine)
            for (; below + hist[8 * lane + digit] <= k; digit++) below += hist[8 * lane + digit];
        const int src = __ffs(__ballot_sync(0xffffffffu, mine)) - 1;
        prefix = prefix << 8 | __shfl_sync(0xffffffffu, 8 * lane + digit, src);
        k -= __shfl_sync(0xffffffffu, below, src);
    }
    return key_value(prefix);
}

// Unit `item` of the call's frames starts at word item * unit_cols (one-row
// units tile the frames in order).  NC: four-pixel chunks per lane, chunk
// lane + 32 c.  Warps take items persistently, the next item's words and
// offsets in flight while one is ranked.
template <int NC>
__global__ void __launch_bounds__(32 * kRowUnitWarps, 5)
    cm_row_codes_kernel(RowCodes rc, const uint16_t* __restrict__ raw,
                        const float* __restrict__ nped, float* __restrict__ cm,
                        uint32_t n_items, uint32_t units_per_frame, uint32_t npx,
                        uint32_t min_count, float cut, uint32_t* __restrict__ zero) {
    constexpr int W = 2 * NC;
    start_next_kernel();
    if (zero && blockIdx.x == 0 && threadIdx.x == 0) *zero = 0;
    __shared__ RowShared shared[kRowUnitWarps];
    RowShared& S = shared[threadIdx.x >> 5];
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t step = gridDim.x * kRowUnitWarps;
    uint32_t item = blockIdx.x * kRowUnitWarps + (threadIdx.x >> 5);
    if (item >= n_items) return;  // whole warps; no block barrier follows
    const uint32_t cap2 = rc.rcap * 0x10001u, first2 = rc.first * 0x10001u,
                   spare2 = rc.spare * 0x10001u;
    // lanes whose chunks all lie in the unit take part in the first pivot
    // (at least one: 128 (NC - 1) < npx)
    const uint32_t whole = min(npx / 4 - 32u * (NC - 1), 32u);
    constexpr uint32_t kMeds = W >= 6 ? 4 : 2;  // medians (or values) per lane in it
    const float per = 1.0f / (float)(kMeds * whole);

    uint2 x[NC], kk[NC];
    uint32_t u = item % units_per_frame;  // the item's unit in its frame
    const uint32_t ustep = step % units_per_frame;
    auto load = [&](uint32_t it, uint32_t unit) {
        const uint16_t* rw = raw + (size_t)it * npx;
        const uint16_t* km = rc.kmap + unit * npx;
#pragma unroll
        for (int c = 0; c < NC; c++) {
            const uint32_t px = 4 * (lane + 32 * c);
            if (px < npx) {
                x[c] = __ldg(reinterpret_cast<const uint2*>(rw + px));
                kk[c] = __ldg(reinterpret_cast<const uint2*>(km + px));
            }
        }
    };
    load(item, u);
    for (; item < n_items; item += step) {
        const float* np_ = nped + u * npx;
        const uint16_t* rw = raw + (size_t)item * npx;
        uint32_t code[W];
#pragma unroll
        for (int c = 0; c < NC; c++) {
            const bool in = 4 * (lane + 32 * c) < npx;
            const uint32_t a = (min_u16x2(x[c].x, cap2) << 3) + kk[c].x;
            const uint32_t b = (min_u16x2(x[c].y, cap2) << 3) + kk[c].y;
            code[2 * c] = in ? min_u16x2(max_u16x2(a, first2), spare2) : spare2;
            code[2 * c + 1] = in ? min_u16x2(max_u16x2(b, first2), spare2) : spare2;
        }
        u += ustep;
        if (u >= units_per_frame) u -= units_per_frame;
        if (item + step < n_items) load(item + step, u);

        const uint32_t n = count_below<W>(code, rc.spare);
        if (n == 0 || n < min_count) {
            if (lane == 0) cm[item] = 0.0f;
            continue;
        }
        const uint32_t k = (n - 1) / 2;
        uint32_t g;
        {
            uint32_t m;
            if constexpr (W >= 6) {
                const uint32_t a = med3_u16x2(code[0], code[1], code[2]);
                const uint32_t b = med3_u16x2(code[3], code[4], code[5]);
                m = (a & 0xFFFFu) + (a >> 16) + (b & 0xFFFFu) + (b >> 16);
            } else if constexpr (W == 4) {
                const uint32_t a = med3_u16x2(code[0], code[1], code[2]);
                m = (a & 0xFFFFu) + (a >> 16);
            } else {
                const uint32_t a = min_u16x2(code[0], code[1]);
                m = (a & 0xFFFFu) + (a >> 16);
            }
            m = __reduce_add_sync(0xffffffffu, lane < whole ? m : 0u);
            g = (uint32_t)((float)m * per);
        }
        // c(lo) <= k < c(hi), c(x) the codes below x
        uint32_t lo = rc.first, hi = rc.spare, c_lo = 0, c_hi = n;
        uint32_t pivot = min(max(g, lo + 1), hi - 1);
        // (steps double until the rank is bracketed; codes are below 2^15)
        uint32_t stride = 0;
        while (c_hi - c_lo > kRowFew && hi - lo > 1) {
            const uint32_t c = count_below<W>(code, pivot);
            const bool up = c <= k;
            if (up) {
                lo = pivot;
                c_lo = c;
            } else {
                hi = pivot;
                c_hi = c;
            }
            stride = max(2 * stride, 1 + (up ? k - c : c - k) / 4);
            const uint32_t next = up ? pivot + stride : pivot - min(pivot, stride);
            const bool open = lo == rc.first || hi == rc.spare;
            pivot = open && next > lo && next < hi ? next : (lo + hi) / 2;
        }
        const uint32_t left = c_hi - c_lo;
        if (left > kRowMost) {
            const float v = row_radix(rw, np_, npx, cut, k, S.hist);
            if (lane == 0) cm[item] = v;
            continue;
        }
        // the lane's pixels whose codes lie in [lo, hi), as a bit per pixel
        uint32_t mine = 0;
        const __half2 lo2 = as_half2(lo * 0x10001u), hi2 = as_half2(hi * 0x10001u);
#pragma unroll
        for (int j = 0; j < W; j++) {
            const uint32_t in = __hge2_mask(as_half2(code[j]), lo2) &
                                __hlt2_mask(as_half2(code[j]), hi2) & 0x00020001u;
            mine |= (in | in >> 16) << (2 * j);
        }
        mine &= (1u << (2 * W)) - 1u;
        S.few[lane] = 0xFFFFFFFFu;  // past the values left: above every key
        __syncwarp();
        uint32_t at = 0;
        while (true) {
            const uint32_t who = __ballot_sync(0xffffffffu, mine != 0);
            if (!who) break;
            if (mine) {
                const uint32_t b = __ffs(mine) - 1;  // pixel b % 4 of chunk lane + 32 (b / 4)
                mine &= mine - 1;
                const uint32_t px = 4 * (lane + 32 * (b >> 2)) + (b & 3u);
                const float d = __fadd_rn(__uint2float_rn(rw[px]), np_[px]);
                S.few[at + __popc(who & ((1u << lane) - 1u))] = order_key(d);
            }
            at += __popc(who);
        }
        __syncwarp();
        // rank k - c_lo of the values left, by counting
        const uint32_t rank = k - c_lo;
        const uint32_t key = S.few[lane];
        uint32_t less = 0, leq = 0;
        for (uint32_t q = 0; q < left; q += 4) {
            const uint4 o = *reinterpret_cast<const uint4*>(S.few + q);
            less += (o.x < key) + (o.y < key) + (o.z < key) + (o.w < key);
            leq += (o.x <= key) + (o.y <= key) + (o.z <= key) + (o.w <= key);
        }
        if (lane < left && less <= rank && rank < leq) cm[item] = key_value(key);
        __syncwarp();  // the keys are read before the next unit's replace them
    }
}

}  // namespace

bool build_row_codes(const ChainParams& p, const float* pedestal, std::vector<uint16_t>* kmap,
                     RowCodes* out) {
    // lanes read four pixels a load, so units start on four-pixel chunks
    if (p.unit_rows != 1 || p.unit_cols % 4 || p.unit_px > 512) return false;
    if (!(p.cm_cut > -1e6f && p.cm_cut < 1e6f)) return false;
    constexpr int kCodes = 8192;  // 1024 ADU below the cut
    CodeBase cb;
    if (!code_base(p, pedestal, kCodes, &cb)) return false;
    // codes stay below the bit pattern of binary16's infinity
    if (cb.bias + kCodes > 0x7BFF) return false;
    kmap->resize(p.frame_px);
    const uint32_t bias = (uint32_t)cb.bias;
    uint16_t* k = kmap->data();
    for (size_t i = 0; i < p.frame_px; i++) k[i] = (uint16_t)((uint32_t)cb.F[i] + bias);
    *out = RowCodes{nullptr, (uint32_t)cb.rcap, (uint32_t)cb.bias, (uint32_t)(cb.bias + kCodes)};
    return true;
}

cudaError_t launch_row_codes(const ChainParams& p, const RowCodes& rc, const uint16_t* raw,
                             uint32_t n_frames, float* cm, cudaStream_t stream, uint32_t* zero) {
    // (items indexed in 32 bits: frames in groups)
    const uint32_t group = std::max(1u, (1u << 30) / p.units_per_frame);
    for (uint32_t f0 = 0; f0 < n_frames; f0 += group) {
        const uint32_t items = std::min(group, n_frames - f0) * p.units_per_frame;
        const uint32_t grid = std::min((items + kRowUnitWarps - 1) / kRowUnitWarps,
                                       5u * (uint32_t)device_sm_count());
        const uint32_t nc = (p.unit_px + 127) / 128;
        auto k = nc == 1   ? cm_row_codes_kernel<1>
                 : nc == 2 ? cm_row_codes_kernel<2>
                 : nc == 3 ? cm_row_codes_kernel<3>
                           : cm_row_codes_kernel<4>;
        k<<<grid, 32 * kRowUnitWarps, 0, stream>>>(
            rc, raw + (size_t)f0 * p.frame_px, p.nped, cm + (size_t)f0 * p.units_per_frame, items,
            p.units_per_frame, p.unit_px, p.cm_min_count, p.cm_cut, f0 ? nullptr : zero);
    }
    return cudaGetLastError();
}

}  // namespace pd
