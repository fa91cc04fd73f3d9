// pd_matched.cu — charge summing with the paper's matched filters.
//
// Section "Photon Charge Summing" (Figs. d, e) and section "Photon Subpixel
// Resolution" (Fig. f).  With T = (s > 0) the signal mask and s the zeroed
// signal, each feature f of the bank has four 4 x 5 filters F0, F1, F1dx,
// F1dy and a threshold F1Nmin:
//     Size_f = T * F1     Droplet_f = s * F1     Overflow_f = T * F0
//     Mx_f = s * F1dx     My_f = s * F1dy
//     Valid_f = (Overflow_f == 0) and (Size_f >= F1Nmin_f)
// and a pixel's energy is the sum of its valid droplets in feature order,
// its centroid the sum of Mx_f / Droplet_f (My_f / Droplet_f) over the valid
// features whose droplet is not 0.  A filter tap (i, j) applied at (r, c)
// meets (r + i - 1, c + j - 2), zero outside the module (TF's "SAME"
// alignment of a 4 x 5 kernel); each sum runs over the taps row-major from
// 0.0f with products rounded once.
//
// The bank is compiled on the host into lists of the nonzero taps.  Skipping
// a zero tap is exact for finite signals (1 / gain overflows for gains below
// 2.9e-39 ADU/keV, where an infinite signal times 0 would be NaN): its term is
// +-0, and a sum that starts at +0.0f is never -0 (x + (-x) rounds to +0), so
// adding +-0 never changes it.  For the
// same reason a pixel whose 4 x 5 window holds no signal has every Size,
// Overflow and Droplet equal to 0, so its energy is 0 and it is skipped.
//
// matched_kernel: grid-stride over 16 x 64 tiles of (frame, module); the
// corrected signal of the tile and its halo (one row above, two below, two
// columns each side) goes to shared memory together with, per halo row and
// column, the 5-bit signal mask of the five columns around; four of those
// give a pixel's 20-bit window mask.  Pixels with a non-empty window
// evaluate the bank: Size is a popcount for features whose F1 taps are all
// 1, and Overflow == 0 a mask test for features whose F0 taps are all
// positive (a sum of positive terms is positive, and of ones is exact);
// other features, and the droplet and momenta of valid features, run over
// the tap lists (a bank of binary features reads its valid features from the
// table described below).  Hits are compacted with a warp ballot and one
// atomic per warp.
//
// matched_band_kernel: the same per pixel on full-width bands of module rows
// (single gain, raw - pedestal before the common mode), with the band
// stencil's four-pixel vector loads and packed correction.  The signal bits of
// the band go to a bitmap of 32 columns a word, and one thread per word finds
// the pixels that may be hits, 32 at a time: a hit has a valid feature with
// signal under its F1, so some tap of any F1 sees signal, and every tap that
// all features' F0 share (those with positive taps) sees none.  The valid
// features of these candidates come next (for a bank of binary features, from
// a table indexed by the window mask); the sums then run over a second list of
// the candidates with a valid feature, so that they keep every lane busy.
// (Every pixel whose window held any signal was a candidate before: a quarter
// of all at an occupancy of 0.5 %, each marked with up to eight shared atomics
// and looked up in the table; 64 frames of 32 x 185 x 388: 556 -> 399 us,
// with bands of 47 rows in place of 31, one list of taps for the three sums and
// the common mode of full-height units in registers.  64 registers, so that two
// CTAs fit an SM, and 88 to 96 bytes of spills.)
// That holds while a tile's candidates fit kMbCap: a 47 x 388 tile has some 630
// at an occupancy of 0.5 %, 1200 at 1 %, 2200 at 2 %.  Past it every own pixel of
// the tile is tested, which costs 3.5 times as much; the call of 64 frames, before
// and now: 0.2 % 696 -> 595 us, 1 % 1076 -> 667 (the longer list of any signal in
// the window overflowed there), 1.5 % 733, 2 % 2123 -> 2017, 5 % 2442 -> 2387.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <new>

#include "pd_dev.cuh"
#include "pd_fast.cuh"
#include "pd_internal.cuh"

namespace pd {

namespace {

constexpr int kTY = 16, kTX = 64, kThreads = 256;
constexpr int kHY = kTY + 3, kHX = kTX + 4;

__device__ __forceinline__ uint32_t hist_bin(float v, float neg_lo_s, float inv_w,
                                             uint32_t bins) {
    const float t = __fmaf_rn(v, inv_w, neg_lo_s);
    if (!(t >= 0.0f)) return 0;
    if (t >= (float)bins) return bins - 1;
    return (uint32_t)t;
}

// The bank at one pixel: w points at its window's tap (0, 0) in a shared
// tile (tap (i, j) at w[i * pitch + j], the pitch folded into the taps'
// offsets), win is its 20-bit signal mask.  valid_features gives the mask
// of the valid features; sum_features their energy E, centroid sums dx, dy
// and npix (the signal pixels under the first valid feature's F1), as
// described above.
__device__ __forceinline__ uint32_t valid_features(const MatchedBank& sb, const float* w,
                                                   uint32_t win, float thr) {
    if (sb.vtab) return sb.vtab[win];
    uint32_t valid = 0;
    for (uint32_t ft = 0; ft < sb.n_features; ft++) {
        bool clear;
        if (sb.f0_pos[ft]) {
            clear = (win & sb.m0[ft]) == 0;
        } else {
            float over = 0.0f;
            for (uint32_t k = sb.off0[ft]; k < sb.off0[ft + 1]; k++)
                if (w[sb.t0[k].at] > thr) over = __fadd_rn(over, sb.t0[k].v);
            clear = over == 0.0f;
        }
        if (!clear) continue;
        float size;
        if (sb.f1_unit[ft]) {
            size = (float)__popc(win & sb.m1[ft]);
        } else {
            size = 0.0f;
            for (uint32_t k = sb.off1[ft]; k < sb.off1[ft + 1]; k++)
                if (w[sb.t1[k].at] > thr) size = __fadd_rn(size, sb.t1[k].v);
        }
        if (size >= sb.nmin[ft]) valid |= 1u << ft;
    }
    return valid;
}

// (a tap of weight 0 in one of the three filters adds nothing to its sum)
__device__ __forceinline__ void sum_features(const MatchedBank& sb, const float* w,
                                             uint32_t valid, float thr, float& E, float& dx,
                                             float& dy, uint32_t& npix) {
    E = dx = dy = 0.0f;
    npix = 0;
    bool any = false;
    while (valid) {
        const uint32_t ft = (uint32_t)(__ffs(valid) - 1);
        valid &= valid - 1;
        float drop = 0.0f, mx = 0.0f, my = 0.0f;
        uint32_t under = 0;
        const uint32_t k1 = sb.offs[ft + 1];
#pragma unroll 4
        for (uint32_t k = sb.offs[ft]; k < k1; k++) {
            const MatchedSum t = sb.ts[k];
            const float e = w[t.at & 0xFFFFu];
            const float sv = e > thr ? e : 0.0f;
            if (t.v1 != 0.0f) {
                drop = __fadd_rn(drop, __fmul_rn(sv, t.v1));
                under += sv > 0.0f;
            }
            if (t.vx != 0.0f) mx = __fadd_rn(mx, __fmul_rn(sv, t.vx));
            if (t.vy != 0.0f) my = __fadd_rn(my, __fmul_rn(sv, t.vy));
        }
        if (!any) npix = under;
        any = true;
        E = __fadd_rn(E, drop);
        if (drop != 0.0f) {
            dx = __fadd_rn(dx, __fdiv_rn(mx, drop));
            dy = __fadd_rn(dy, __fdiv_rn(my, drop));
        }
    }
}

// Count, flags and record of a pixel whose bank gave energy E (E != 0);
// returns whether it is a hit (count >= 1) and adds E to the hit histogram.
__device__ __forceinline__ bool make_hit(const ChainParams& p, uint32_t* hhit, float E, float dx,
                                         float dy, uint32_t npix, int r, int c, uint32_t frame,
                                         size_t mod_base, pd_hit& h, uint32_t& n, uint32_t& pix) {
    atomicAdd(&hhit[hist_bin(E, p.hist_neg_lo_s, p.hist_inv_w, p.hist_bins)], 1u);
    const float qr = rintf(__fdiv_rn(E, p.photon_kev));
    uint16_t flags = 0;
    if (!(qr >= 0.0f)) {
        n = 0;
    } else if (qr > 255.0f) {
        n = 255;
        flags |= PD_HIT_SATURATED;
    } else {
        n = (uint32_t)qr;
    }
    if (n < 1) return false;
    const int R = (int)p.rows, C = (int)p.cols;
    if (r == 0 || c == 0 || r == R - 1 || c == C - 1) flags |= PD_HIT_EDGE;
    pix = (uint32_t)mod_base + (uint32_t)r * p.cols + (uint32_t)c;
    h.frame = frame;
    h.pixel = pix;
    h.energy_kev = E;
    h.dx = dx;
    h.dy = dy;
    h.count = (uint8_t)n;
    h.npix = (uint8_t)(npix > 255 ? 255 : npix);
    h.flags = flags;
    return true;
}

// Warp-aggregated emission: one atomic on the hit counter per warp.  wm:
// the warp's lanes (all of them must call).
__device__ __forceinline__ void emit_hits(const ChainParams& p, const CallOut& out, bool emit,
                                          const pd_hit& h, uint32_t n, uint32_t pix, int lane,
                                          unsigned wm = 0xffffffffu) {
    const uint32_t mask = __ballot_sync(wm, emit);
    if (mask) {
        uint32_t slot = 0;
        if (lane == __ffs(mask) - 1) slot = atomicAdd(out.n_hits, __popc(mask));
        slot = __shfl_sync(wm, slot, __ffs(mask) - 1);
        if (emit) {
            slot += __popc(mask & ((1u << lane) - 1u));
            atomicAdd(&p.count_map[pix], n);
            if (slot < out.hit_capacity) out.hits[slot] = h;
        }
    }
}

template <bool STACKED, bool MG>
__global__ void __launch_bounds__(kThreads)
    matched_kernel(ChainParams p, const MatchedBank* __restrict__ bank,
                   const uint16_t* __restrict__ raw, uint32_t frame_base, CallOut out,
                   uint32_t tiles_y, uint32_t tiles_x, unsigned long long n_tiles,
                   MultiGain mg) {
    extern __shared__ uint32_t hsm[];  // [2][hist_bins]
    __shared__ float tile[kHY][kHX];
    __shared__ uint8_t row5[kHY][kTX];  // signal bits of columns c-2 .. c+2
    __shared__ uint32_t s_ucol[kHX], s_urow[kHY];  // unit offsets of halo columns / rows
    __shared__ MatchedBank sb;
    uint32_t* hpix = hsm;
    uint32_t* hhit = hsm + p.hist_bins;
    for (uint32_t b = threadIdx.x; b < 2 * p.hist_bins; b += kThreads) hsm[b] = 0;
    {
        const uint32_t* src = reinterpret_cast<const uint32_t*>(bank);
        uint32_t* dst = reinterpret_cast<uint32_t*>(&sb);
        for (uint32_t k = threadIdx.x; k < sizeof(MatchedBank) / 4; k += kThreads) dst[k] = src[k];
    }
    __syncthreads();

    const int R = (int)p.rows, C = (int)p.cols;
    const int lane = threadIdx.x & 31;
    __shared__ uint32_t s_at[4];  // the tile's column, row, module and frame
    __shared__ uint32_t s_list[kTY * kTX];  // pixel j | window mask << 10
    __shared__ uint32_t s_nc;
    for (unsigned long long t = blockIdx.x; t < n_tiles; t += gridDim.x) {
        // one thread splits the tile index (64-bit divisions are long
        // instruction sequences; every thread doing them cost more than
        // the tile's pixels)
        if (threadIdx.x == 0) {
            unsigned long long q = t;
            s_at[0] = (uint32_t)(q % tiles_x);
            q /= tiles_x;
            s_at[1] = (uint32_t)(q % tiles_y);
            q /= tiles_y;
            s_at[2] = (uint32_t)(q % p.n_modules);
            s_at[3] = (uint32_t)(q / p.n_modules);
            s_nc = 0;
        }
        __syncthreads();
        const int tx = (int)s_at[0], ty = (int)s_at[1];
        const uint32_t m = s_at[2], f = s_at[3];
        const int r0 = ty * kTY, c0 = tx * kTX;
        const size_t mod_base = (size_t)m * p.module_px;
        const uint16_t* fr = raw + (size_t)f * p.frame_px + mod_base;
        const float* cmf = out.cm + (size_t)f * cm_per_frame(p) + (size_t)m * p.units_per_module;
        const float* cmr = out.cm + (size_t)f * cm_per_frame(p) + p.units_per_frame +
                           (size_t)m * p.rows;
        const float* cmc = out.cm + (size_t)f * cm_per_frame(p) + p.units_per_frame +
                           (size_t)p.n_modules * p.rows + (size_t)m * p.cols;

        // unit of each halo column and row (divisions per column and row, not
        // per pixel)
        for (int k = threadIdx.x; k < kHX + kHY; k += kThreads) {
            if (k < kHX) {
                const int c = c0 + k - 2;
                s_ucol[k] = c >= 0 && c < C ? (uint32_t)c / p.unit_cols : 0u;
            } else {
                const int r = r0 + (k - kHX) - 1;
                s_urow[k - kHX] = r >= 0 && r < R ? ((uint32_t)r / p.unit_rows) * p.units_per_row : 0u;
            }
        }
        __syncthreads();
        // 1. zeroed signal of the tile and its halo
        for (int j = threadIdx.x; j < kHY * kHX; j += kThreads) {
            const int hr = j / kHX, hc = j % kHX;
            const int r = r0 + hr - 1, c = c0 + hc - 2;
            float s = 0.0f;
            if (r >= 0 && r < R && c >= 0 && c < C) {
                const uint32_t off = (uint32_t)r * p.cols + (uint32_t)c;
                const float cm = cmf[s_urow[hr] + s_ucol[hc]];
                float e;
                if (MG) {
                    e = mg_energy(mg, p.frame_px, fr[off], mod_base + off, cm);
                } else {
                    const float d = __fsub_rn(__uint2float_rn(fr[off]), p.ped[mod_base + off]);
                    e = energy<STACKED>(cm_after_gain(p), d, p.inv_gain[mod_base + off], cm,
                                        STACKED ? cmr[r] : 0.0f, STACKED ? cmc[c] : 0.0f);
                }
                s = e > p.zero_thr ? e : 0.0f;
                if (hr >= 1 && hr <= kTY && hc >= 2 && hc < kTX + 2) {
                    atomicAdd(&hpix[hist_bin(e, p.hist_neg_lo_s, p.hist_inv_w, p.hist_bins)], 1u);
                    if (out.corrected)
                        out.corrected[(size_t)f * p.frame_px + mod_base + off] = e;
                }
            }
            tile[hr][hc] = s;
        }
        __syncthreads();
        for (int j = threadIdx.x; j < kHY * kTX; j += kThreads) {
            const int hr = j / kTX, ic = j % kTX;
            const float* row = &tile[hr][ic];
            row5[hr][ic] = (uint8_t)((row[0] > 0.0f) | (row[1] > 0.0f) << 1 |
                                     (row[2] > 0.0f) << 2 | (row[3] > 0.0f) << 3 |
                                     (row[4] > 0.0f) << 4);
        }
        __syncthreads();

        // 2. pixels whose window holds signal into a list (warp-aggregated),
        //    so that the bank runs with every lane busy
        for (int base = 0; base < kTY * kTX; base += kThreads) {
            const int j = base + threadIdx.x;
            const int ir = j / kTX, ic = j % kTX;
            const uint32_t win = (uint32_t)row5[ir][ic] | (uint32_t)row5[ir + 1][ic] << 5 |
                                 (uint32_t)row5[ir + 2][ic] << 10 |
                                 (uint32_t)row5[ir + 3][ic] << 15;
            const bool cand = r0 + ir < R && c0 + ic < C && win;
            const uint32_t bal = __ballot_sync(0xffffffffu, cand);
            if (bal) {
                const int lead = __ffs(bal) - 1;
                uint32_t at0 = 0;
                if (lane == lead) at0 = atomicAdd(&s_nc, (uint32_t)__popc(bal));
                at0 = __shfl_sync(0xffffffffu, at0, lead);
                if (cand) s_list[at0 + __popc(bal & ((1u << lane) - 1u))] = (uint32_t)j | win << 10;
            }
        }
        __syncthreads();
        const uint32_t n_cand = s_nc;

        // 3. the bank at the listed pixels
        for (uint32_t base = 0; base < n_cand; base += kThreads) {
            const uint32_t k = base + threadIdx.x;
            bool emit = false;
            pd_hit h;
            uint32_t n = 0, pix = 0;
            const uint32_t e_k = k < n_cand ? s_list[k] : 0u;
            const int j = (int)(e_k & 1023u);
            const uint32_t win = e_k >> 10;
            const int ir = j / kTX, ic = j % kTX;
            const int r = r0 + ir, c = c0 + ic;
            if (k < n_cand) {
                // window tap (i, j) is tile[ir + i][ic + j]
                const uint32_t valid = valid_features(sb, &tile[ir][ic], win, 0.0f);
                if (valid) {
                    float E, dx, dy;
                    uint32_t npix;
                    sum_features(sb, &tile[ir][ic], valid, 0.0f, E, dx, dy, npix);
                    if (E != 0.0f)
                        emit = make_hit(p, hhit, E, dx, dy, npix, r, c, frame_base + f, mod_base,
                                        h, n, pix);
                }
            }
            emit_hits(p, out, emit, h, n, pix, lane);
        }
        __syncthreads();
    }
    for (uint32_t b = threadIdx.x; b < p.hist_bins; b += kThreads) {
        if (hpix[b]) atomicAdd(&p.hist_pix[b], (unsigned long long)hpix[b]);
        if (hhit[b]) atomicAdd(&p.hist_hit[b], (unsigned long long)hhit[b]);
    }
}

// Candidates per band tile, and those with a valid feature (a larger count
// tests every own pixel).
constexpr uint32_t kMbCap = 2048, kMbValid = 1024;

// Words of a signal bitmap row: 32 real columns each, a zero word on both sides.
__host__ __device__ inline uint32_t sig_words(uint32_t cols) { return (cols + 31) / 32 + 2; }

// Shared memory of the band kernel for bands of rb rows: the s-tile of
// rb + 3 rows (one above, two below) at the given pitch, both histograms
// (plus a spare bin), the candidate list and the list of those with a valid
// feature, the negated common mode of every (tile row, unit column), the
// stacked row terms and the signal bitmaps of this tile and the next.
size_t band_smem(const ChainParams& p, uint32_t rb, uint32_t pitch) {
    const size_t nr = rb + 3;
    return 4 * (nr * pitch + 2 * (size_t)p.hist_bins + 4 + kMbCap + kMbValid + nr * p.units_per_row +
                nr + 2 * nr * sig_words(p.cols));
}

constexpr uint32_t kMaxTaps = PD_MAX_FEATURES * 20;

// Bands of rb rows of (frame, module): tile t is band t % n_bands of module
// (t / n_bands) % n_modules of frame t / (n_bands * n_modules).  COLBANK: the
// common-mode units span the module's full height, so a thread's four pixels
// take the same two values on every row of a tile, held in registers.
template <bool STACKED, bool COLBANK>
__global__ void __launch_bounds__(kBandThreads, 2)
    matched_band_kernel(ChainParams p, const MatchedBank* __restrict__ bank,
                        const uint16_t* __restrict__ raw, uint32_t frame_base, CallOut out,
                        BandConfig bc, unsigned long long n_tiles) {
    extern __shared__ __align__(16) uint32_t msm[];
    __shared__ MatchedBank sb;
    __shared__ uint32_t s_nc, s_nv;
    __shared__ uint32_t s_tap[40];  // candidate test: bitmap word offset << 8 | shift
    const uint32_t P = bc.pitch, NR = bc.rb + 3;
    float* stile = reinterpret_cast<float*>(msm);  // NR x P; real column c at 4 + c
    uint32_t* hpix = msm + NR * P;                 // hist_bins + spare
    uint32_t* hhit = hpix + p.hist_bins + 4;       // hist_bins
    uint32_t* list = hhit + p.hist_bins;           // kMbCap: row << 16 | column
    uint32_t* vlist = list + kMbCap;               // kMbValid: list index | valid << 24
    float* cmt = reinterpret_cast<float*>(vlist + kMbValid);  // NR x units_per_row
    float* crt = cmt + NR * p.units_per_row;                  // NR row terms
    // signal bitmaps of this tile and the next: bit c % 32 of word 1 + c / 32
    // of a tile row is the signal of real column c
    const uint32_t W = ((uint32_t)p.cols + 31) / 32, SW = W + 2;
    uint32_t* sig = reinterpret_cast<uint32_t*>(crt + NR);  // NR x SW, twice
    uint32_t* sig_next = sig + NR * SW;

    const uint32_t tid = threadIdx.x, nthr = blockDim.x;
    const int lane = tid & 31;
    const int R = (int)p.rows, C = (int)p.cols;
    const uint32_t TX = bc.tx, TY = bc.ty;
    const uint32_t tx = tid % TX, ty = tid / TX;
    const bool active = ty < TY;
    const int col = (int)(tx * 4);  // first column of this thread's chunk
    const uint32_t uca = (uint32_t)col / p.unit_cols;
    const uint32_t ucb = (uint32_t)(col + 3) / p.unit_cols;
    const int split = (int)(ucb * p.unit_cols) - col;  // pixels i >= split use ucb
    const int max_bits = (int)(kMagicBits + p.hist_bins - 1);

    for (uint32_t i = tid; i < NR * P; i += nthr) stile[i] = 0.0f;
    for (uint32_t i = tid; i < 2 * NR * SW; i += nthr) sig[i] = 0;
    for (uint32_t i = tid; i < 2 * p.hist_bins + 4; i += nthr) hpix[i] = 0;
    {
        const uint32_t* src = reinterpret_cast<const uint32_t*>(bank);
        uint32_t* dst = reinterpret_cast<uint32_t*>(&sb);
        for (uint32_t k = tid; k < sizeof(MatchedBank) / 4; k += nthr) dst[k] = src[k];
    }
    __syncthreads();
    // the candidate test's taps, those that must be clear first: tap (i, j)
    // of pixel x is bit x + j - 2 of tile row rl - 1 + i
    const uint32_t m_clear = sb.clear, m_some = sb.some;
    const int n_clear = __popc(m_clear), n_test = n_clear + __popc(m_some);
    if (tid < 40) {
        const uint32_t k = tid % 20, mask = tid < 20 ? m_clear : m_some;
        if (mask >> k & 1u) {
            const int at = (tid < 20 ? 0 : n_clear) + __popc(mask & ((1u << k) - 1u));
            const uint32_t i = k / 5;
            const int d = (int)(k % 5) - 2;
            // (counted from the word before the pixel's, in tile row rl - 1)
            s_tap[at] = (i * SW + (d < 0 ? 0u : 1u)) << 8 | (uint32_t)(d & 31);
        }
    }
    // tap offsets at this pitch
    for (uint32_t k = tid; k < 3 * kMaxTaps; k += nthr) {
        if (k < 2 * kMaxTaps) {
            MatchedTap& tp = k < kMaxTaps ? sb.t1[k] : sb.t0[k - kMaxTaps];
            tp.at = (uint16_t)(tp.i * P + tp.j);
        } else {
            uint32_t& at = sb.ts[k - 2 * kMaxTaps].at;
            const uint32_t q = at >> 16;
            at = (q / 5) * P + q % 5;
        }
    }

    // negated common mode of entry i (tile row, unit column) of tile tt; each
    // thread holds its entry of the next tile in a register
    const uint32_t ncmt = NR * p.units_per_row;
    auto tile_cm = [&](unsigned long long tt, uint32_t i) -> float {
        const unsigned long long fm = tt / bc.n_bands;
        const int r = (int)(tt - fm * bc.n_bands) * (int)bc.rb - 1 + (int)(i / p.units_per_row);
        if (r < 0 || r >= R) return 0.0f;
        const size_t fbase = (size_t)fm * p.units_per_module +
                             (STACKED ? (size_t)(fm / p.n_modules) *
                                            (cm_per_frame(p) - p.units_per_frame)
                                      : 0);
        return -out.cm[fbase + ((uint32_t)r / p.unit_rows) * p.units_per_row +
                       i % p.units_per_row];
    };
    // (COLBANK: the two values of this thread's chunk)
    auto chunk_cm = [&](const TileWalk& w) {
        const float* cmf = out.cm +
                           (size_t)w.f * (STACKED ? cm_per_frame(p) : p.units_per_frame) +
                           (size_t)w.m * p.units_per_module;
        return make_float2(-__ldcg(cmf + uca), -__ldcg(cmf + ucb));
    };
    // the common mode (this kernel may start while it ends, launch_matched)
    wait_previous_kernel();
    TileWalk walk(blockIdx.x, gridDim.x, bc.n_bands, p.n_modules);
    float cmv = 0.0f;
    float2 cm2 = make_float2(0.0f, 0.0f);
    if (COLBANK && active)
        cm2 = chunk_cm(walk);
    else if (!COLBANK && blockIdx.x < n_tiles && tid < ncmt)
        cmv = tile_cm(blockIdx.x, tid);

    // the last thread asks L2 for the raw rows (the halo row above, two
    // below) of the next tile now and of the tile after next once a tile is
    // done, so that their loads find them there
    const unsigned long long step = gridDim.x;
    const bool prefetcher = tid == nthr - 1;
    if (prefetcher && blockIdx.x + step < n_tiles) {
        TileWalk nx = walk;
        nx.next();
        prefetch_tile_rows(raw, nx, bc.rb, p.rows, p.cols, p.frame_px, 2);
    }
    for (unsigned long long t = blockIdx.x; t < n_tiles; t += gridDim.x, walk.next()) {
        const int band = (int)walk.band;
        const uint32_t m = walk.m, f = walk.f;
        const int r0 = band * (int)bc.rb;
        const int rows_here = min((int)bc.rb, R - r0);
        const size_t mod_base = (size_t)m * p.module_px;
        const uint16_t* fr = raw + (size_t)f * p.frame_px + mod_base;
        const float* npm = p.nped + mod_base;
        const float* gm = p.inv_gain + mod_base;

        if (!COLBANK) {
            if (tid < ncmt) cmt[tid] = cmv;
            for (uint32_t i = tid + nthr; i < ncmt; i += nthr) cmt[i] = tile_cm(t, i);
        }
        const float2 b01 = make_float2(split > 0 ? cm2.x : cm2.y, split > 1 ? cm2.x : cm2.y);
        const float2 b23 = make_float2(split > 2 ? cm2.x : cm2.y, split > 3 ? cm2.x : cm2.y);
        float ncc[4];
        if (STACKED) {
            const float* cmf = out.cm + (size_t)f * cm_per_frame(p) + p.units_per_frame;
            for (uint32_t i = tid; i < NR; i += nthr) {
                const int r = r0 - 1 + (int)i;
                crt[i] = r >= 0 && r < R ? -cmf[(size_t)m * p.rows + r] : 0.0f;
            }
#pragma unroll
            for (int i = 0; i < 4; i++)
                ncc[i] = active ? -cmf[(size_t)p.n_modules * p.rows + (size_t)m * p.cols + col + i]
                                : 0.0f;
        }
        if (tid == 0) s_nc = s_nv = 0;
        __syncthreads();

        // 1. energies and signal bits (zeroed where they are read) of rows r0-1 .. r0+rows_here+1, two
        //    register sets so that the next row's loads are in flight; halo
        //    rows are not histogrammed
        if (active) {
            const int nrows = rows_here + 3;
            struct Row {
                uint2 rw;
                float4 np, g;
            };
            auto inside = [&](int rl) { return r0 - 1 + rl >= 0 && r0 - 1 + rl < R; };
            auto load = [&](int rl, Row& x) {
                if (rl >= nrows || !inside(rl)) return;
                const uint32_t off = (uint32_t)(r0 - 1 + rl) * p.cols + (uint32_t)col;
                x.rw = __ldg(reinterpret_cast<const uint2*>(fr + off));
                x.np = __ldg(reinterpret_cast<const float4*>(npm + off));
                x.g = __ldg(reinterpret_cast<const float4*>(gm + off));
            };
            auto row = [&](const Row& x, int rl) {
                float* srow = stile + rl * P + 4 + col;
                if (!inside(rl)) {
                    *reinterpret_cast<float4*>(srow) = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    return;
                }
                const bool own = rl >= 1 && rl <= rows_here;
                const float2 d01 = __fadd2_rn(raw_pair(x.rw.x), make_float2(x.np.x, x.np.y));
                const float2 d23 = __fadd2_rn(raw_pair(x.rw.y), make_float2(x.np.z, x.np.w));
                float2 n01 = b01, n23 = b23;
                if (!COLBANK) {
                    const float ncma = cmt[rl * p.units_per_row + uca];
                    const float ncmb = cmt[rl * p.units_per_row + ucb];
                    n01 = make_float2(split > 0 ? ncma : ncmb, split > 1 ? ncma : ncmb);
                    n23 = make_float2(split > 2 ? ncma : ncmb, split > 3 ? ncma : ncmb);
                }
                float2 c01 = __fadd2_rn(d01, n01), c23 = __fadd2_rn(d23, n23);
                if (STACKED) {
                    const float ncr = crt[rl];
                    c01 = __fadd2_rn(__fadd2_rn(c01, make_float2(ncr, ncr)),
                                     make_float2(ncc[0], ncc[1]));
                    c23 = __fadd2_rn(__fadd2_rn(c23, make_float2(ncr, ncr)),
                                     make_float2(ncc[2], ncc[3]));
                }
                const float2 e01 = __fmul2_rn(c01, make_float2(x.g.x, x.g.y));
                const float2 e23 = __fmul2_rn(c23, make_float2(x.g.z, x.g.w));
                const float2 iw = make_float2(p.hist_inv_w, p.hist_inv_w);
                const float2 nl = make_float2(p.hist_neg_lo_s, p.hist_neg_lo_s);
                const float2 mgc = make_float2(kMagic, kMagic);
                const float2 u01 = __fadd2_rd(__ffma2_rn(e01, iw, nl), mgc);
                const float2 u23 = __fadd2_rd(__ffma2_rn(e23, iw, nl), mgc);
                if (own) {
                    auto count = [&](float u) {
                        const int b = min(max(__float_as_int(u), (int)kMagicBits), max_bits);
                        atomicAdd(&hpix[(uint32_t)b - kMagicBits], 1u);
                    };
                    count(u01.x);
                    count(u01.y);
                    count(u23.x);
                    count(u23.y);
                }
                const float e[4] = {e01.x, e01.y, e23.x, e23.y};
                uint32_t bits = 0;
#pragma unroll
                for (int i = 0; i < 4; i++) bits |= e[i] > p.zero_thr ? 1u << i : 0u;
                *reinterpret_cast<float4*>(srow) = make_float4(e[0], e[1], e[2], e[3]);
                if (bits) atomicOr(&sig[rl * SW + 1 + (col >> 5)], bits << (col & 31));
                if (own && out.corrected) {
                    const uint32_t off = (uint32_t)(r0 - 1 + rl) * p.cols + (uint32_t)col;
                    float* dst = out.corrected + (size_t)f * p.frame_px + mod_base + off;
                    *reinterpret_cast<float4*>(dst) = make_float4(e[0], e[1], e[2], e[3]);
                }
            };
            Row xa, xb;
            load((int)ty, xa);
            for (int rl = (int)ty; rl < nrows; rl += 2 * (int)TY) {
                load(rl + (int)TY, xb);
                row(xa, rl);
                if (rl + (int)TY >= nrows) break;
                load(rl + 2 * (int)TY, xa);
                row(xb, rl + (int)TY);
            }
        }
        // the next tile's common mode, in flight during the rest of this one
        if (t + gridDim.x < n_tiles) {
            if (COLBANK && active) {
                TileWalk nx = walk;
                nx.next();
                cm2 = chunk_cm(nx);
            } else if (!COLBANK && tid < ncmt) {
                cmv = tile_cm(t + gridDim.x, tid);
            }
        }
        __syncthreads();

        // 2. the candidates into a list (a warp scan and one shared atomic per
        //    warp reserve each thread's slots; list order is free), the next
        //    tile's bitmap cleared
        for (uint32_t i = tid; i < NR * SW; i += nthr) sig_next[i] = 0;
        const uint32_t n_words = (uint32_t)rows_here * W;
        for (uint32_t base = 0; base < n_words; base += nthr) {
            const uint32_t q = base + tid;
            uint32_t word = 0;
            int rl = 0, x0 = 0;
            if (q < n_words) {
                rl = 1 + (int)(q / W);
                x0 = 32 * (int)(q % W);
                const uint32_t* s0 = sig + (uint32_t)(rl - 1) * SW + q % W;
                auto tap = [&](int k) {
                    const uint32_t t = s_tap[k];
                    const uint32_t* a = s0 + (t >> 8);
                    return __funnelshift_r(a[0], a[1], t & 31u);
                };
                for (int k = n_clear; k < n_test; k++) word |= tap(k);
                uint32_t over = 0;
                for (int k = 0; k < n_clear; k++) over |= tap(k);
                word &= ~over;
                if (C - x0 < 32) word &= 0xFFFFFFFFu >> (32 - (C - x0));
            }
            const unsigned wm = warp_lanes();
            const uint32_t cnt = (uint32_t)__popc(word);
            uint32_t incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t v = __shfl_up_sync(wm, incl, o);
                if (lane >= o) incl += v;
            }
            const int wl = 31 - __clz((int)wm);
            const uint32_t tot = __shfl_sync(wm, incl, wl);
            uint32_t at0 = 0;
            if (lane == wl && tot) at0 = atomicAdd(&s_nc, tot);
            at0 = __shfl_sync(wm, at0, wl);
            uint32_t at = at0 + incl - cnt;
            while (word && at < kMbCap) {
                const int bit = __ffs(word) - 1;
                word &= word - 1;
                list[at++] = ((uint32_t)rl << 16) | (uint32_t)(x0 + bit);
            }
        }
        __syncthreads();

        // 3. the bank at the listed pixels (every own pixel if the list
        //    overflowed): first the valid features of each, then, for the
        //    few with some valid feature (a second list), the sums and the
        //    hit, so that the sums run with every lane on such a pixel
        const uint32_t n_list = s_nc;
        bool scan = n_list > kMbCap;
        uint32_t n_work = scan ? (uint32_t)rows_here * (uint32_t)C : n_list;
        // (row, column) of work item j, and its window mask: rows rl-1 ..
        // rl+2, columns c-2 .. c+2
        auto item_at = [&](uint32_t j, int& rl, int& c) {
            if (scan) {
                rl = 1 + (int)(j / (uint32_t)C);
                c = (int)(j % (uint32_t)C);
            } else {
                const uint32_t e = list[j];
                rl = (int)(e >> 16);
                c = (int)(e & 0xFFFFu);
            }
        };
        auto window = [&](int rl, int c) -> uint32_t {
            const uint32_t* w = sig + (uint32_t)(rl - 1) * SW + (uint32_t)(c + 30) / 32;
            uint32_t win = 0;
#pragma unroll
            for (int i = 0; i < 4; i++)
                win |= (__funnelshift_r(w[i * SW], w[i * SW + 1], (uint32_t)(c + 30) & 31u) & 0x1Fu)
                       << (5 * i);
            return win;
        };
        if (!scan) {
            for (uint32_t base = 0; base < n_work; base += nthr) {
                const uint32_t j = base + tid;
                uint32_t valid = 0;
                if (j < n_work) {
                    int rl, c;
                    item_at(j, rl, c);
                    const uint32_t win = window(rl, c);
                    if (win) valid = valid_features(sb, stile + (rl - 1) * P + c + 2, win,
                                                        p.zero_thr);
                }
                const unsigned wm = __activemask();
                const uint32_t bal = __ballot_sync(wm, valid != 0);
                if (bal) {
                    const int lead = __ffs(bal) - 1;
                    uint32_t at0 = 0;
                    if (lane == lead) at0 = atomicAdd(&s_nv, (uint32_t)__popc(bal));
                    at0 = __shfl_sync(wm, at0, lead);
                    const uint32_t at = at0 + __popc(bal & ((1u << lane) - 1u));
                    if (valid && at < kMbValid) vlist[at] = j | valid << 24;
                }
            }
            __syncthreads();
            if (s_nv > kMbValid) {
                scan = true;
                n_work = (uint32_t)rows_here * (uint32_t)C;
            }
        }
        if (!scan) {
            const uint32_t n_valid = s_nv;
            for (uint32_t base = 0; base < n_valid; base += nthr) {
                const uint32_t k = base + tid;
                bool emit = false;
                pd_hit h;
                uint32_t n = 0, pix = 0;
                if (k < n_valid) {
                    const uint32_t e = vlist[k];
                    int rl, c;
                    item_at(e & 0xFFFFFFu, rl, c);
                    float E, dx, dy;
                    uint32_t npix;
                    sum_features(sb, stile + (rl - 1) * P + c + 2, e >> 24, p.zero_thr, E, dx, dy,
                                 npix);
                    if (E != 0.0f)
                        emit = make_hit(p, hhit, E, dx, dy, npix, r0 - 1 + rl, c, frame_base + f,
                                        mod_base, h, n, pix);
                }
                emit_hits(p, out, emit, h, n, pix, lane, __activemask());
            }
        } else {
            for (uint32_t base = 0; base < n_work; base += nthr) {
                const uint32_t j = base + tid;
                bool emit = false;
                pd_hit h;
                uint32_t n = 0, pix = 0;
                if (j < n_work) {
                    int rl, c;
                    item_at(j, rl, c);
                    const uint32_t win = window(rl, c);
                    const float* w = stile + (rl - 1) * P + c + 2;
                    const uint32_t valid = win ? valid_features(sb, w, win, p.zero_thr) : 0u;
                    if (valid) {
                        float E, dx, dy;
                        uint32_t npix;
                        sum_features(sb, w, valid, p.zero_thr, E, dx, dy, npix);
                        if (E != 0.0f)
                            emit = make_hit(p, hhit, E, dx, dy, npix, r0 - 1 + rl, c,
                                            frame_base + f, mod_base, h, n, pix);
                    }
                }
                emit_hits(p, out, emit, h, n, pix, lane, __activemask());
            }
        }
        __syncthreads();
        {
            uint32_t* const other = sig;
            sig = sig_next;
            sig_next = other;
        }
        if (prefetcher && t + 2 * step < n_tiles) {
            TileWalk nx = walk;
            nx.next();
            nx.next();
            prefetch_tile_rows(raw, nx, bc.rb, p.rows, p.cols, p.frame_px, 2);
        }
    }
    for (uint32_t b = tid; b < p.hist_bins; b += nthr) {
        if (hpix[b]) atomicAdd(&p.hist_pix[b], (unsigned long long)hpix[b]);
        if (hhit[b]) atomicAdd(&p.hist_hit[b], (unsigned long long)hhit[b]);
    }
}

// Valid features of every window mask of an all-binary bank (no tap is
// read: the tests are mask tests and popcounts).
__global__ void vtab_kernel(const MatchedBank* __restrict__ bank, uint8_t* __restrict__ vtab) {
    const uint32_t win = blockIdx.x * blockDim.x + threadIdx.x;
    if (win >= (1u << 20)) return;
    uint32_t valid = 0;
    for (uint32_t ft = 0; ft < bank->n_features; ft++)
        if ((win & bank->m0[ft]) == 0 && (float)__popc(win & bank->m1[ft]) >= bank->nmin[ft])
            valid |= 1u << ft;
    vtab[win] = (uint8_t)valid;
}

// Nonzero taps of one 4 x 5 filter, row-major, appended to list.
void compile_taps(const float (*flt)[5], MatchedTap* list, uint32_t* n) {
    for (int i = 0; i < 4; i++)
        for (int j = 0; j < 5; j++)
            if (flt[i][j] != 0.0f) {
                list[*n].i = (uint8_t)i;
                list[*n].j = (uint8_t)j;
                list[*n].at = (uint16_t)(i * kHX + j);
                list[*n].v = flt[i][j];
                (*n)++;
            }
}

}  // namespace

bool compile_bank(const pd_filter_bank& b, MatchedBank* out) {
    if (b.n_features < 1 || b.n_features > PD_MAX_FEATURES) return false;
    MatchedBank mb{};
    mb.n_features = b.n_features;
    uint32_t n1 = 0, n0 = 0, ns = 0;
    for (uint32_t f = 0; f < b.n_features; f++) {
        if (isnan(b.f1_nmin[f])) return false;
        for (int i = 0; i < 4; i++)
            for (int j = 0; j < 5; j++)
                if (!isfinite(b.f0[f][i][j]) || !isfinite(b.f1[f][i][j]) ||
                    !isfinite(b.f1_dx[f][i][j]) || !isfinite(b.f1_dy[f][i][j]))
                    return false;
        mb.nmin[f] = b.f1_nmin[f];
        mb.off1[f] = (uint16_t)n1;
        mb.off0[f] = (uint16_t)n0;
        compile_taps(b.f1[f], mb.t1, &n1);
        compile_taps(b.f0[f], mb.t0, &n0);
        mb.f1_unit[f] = mb.f0_pos[f] = 1;
        for (int i = 0; i < 4; i++)
            for (int j = 0; j < 5; j++) {
                if (b.f1[f][i][j] != 0.0f) {
                    mb.m1[f] |= 1u << (5 * i + j);
                    if (b.f1[f][i][j] != 1.0f) mb.f1_unit[f] = 0;
                }
                if (b.f0[f][i][j] != 0.0f) {
                    mb.m0[f] |= 1u << (5 * i + j);
                    if (!(b.f0[f][i][j] > 0.0f)) mb.f0_pos[f] = 0;
                }
            }
        mb.offs[f] = (uint16_t)ns;
        for (int i = 0; i < 4; i++)
            for (int j = 0; j < 5; j++)
                if (b.f1[f][i][j] != 0.0f || b.f1_dx[f][i][j] != 0.0f || b.f1_dy[f][i][j] != 0.0f)
                    mb.ts[ns++] = MatchedSum{(uint32_t)(i * kHX + j) | (uint32_t)(5 * i + j) << 16,
                                             b.f1[f][i][j], b.f1_dx[f][i][j], b.f1_dy[f][i][j]};
    }
    mb.offs[b.n_features] = (uint16_t)ns;
    mb.all_binary = 1;
    for (uint32_t f = 0; f < b.n_features; f++)
        if (!mb.f1_unit[f] || !mb.f0_pos[f]) mb.all_binary = 0;
    mb.vtab = nullptr;
    mb.clear = (1u << 20) - 1u;
    mb.some = 0;
    for (uint32_t f = 0; f < b.n_features; f++) {
        mb.some |= mb.m1[f];
        mb.clear &= mb.f0_pos[f] ? mb.m0[f] : 0u;
    }
    mb.off1[b.n_features] = (uint16_t)n1;
    mb.off0[b.n_features] = (uint16_t)n0;
    *out = mb;
    return true;
}

cudaError_t build_vtab(const MatchedBank* bank_dev, uint8_t* vtab) {
    vtab_kernel<<<(1u << 20) / 256, 256>>>(bank_dev, vtab);
    cudaError_t e = cudaGetLastError();
    return e != cudaSuccess ? e : cudaDeviceSynchronize();
}

// dynamic shared memory of one of two CTAs per SM
constexpr size_t kBandSmem = (size_t)(228 * 1024) / 2 - sizeof(MatchedBank) - 2048;

// Band form of the matched stencil: single gain, raw - pedestal before the
// common mode, four-pixel chunks (as the band stencil's), and bands of at
// least one row within about 100 KB of shared memory.
static bool matched_band_config(const ChainParams& p, BandConfig* out) {
    if (cm_after_gain(p)) return false;
    BandConfig bc = make_band_config(p);
    if (!bc.ok || bc.vec != 4) return false;
    // the tallest band that two CTAs per SM hold, split evenly over the rows
    // (the halo is three rows a band)
    const size_t least = band_smem(p, 0, bc.pitch);
    if (least >= kBandSmem) return false;
    const size_t tallest = (kBandSmem - least) / (band_smem(p, 1, bc.pitch) - least);
    if (tallest == 0) return false;
    const uint32_t rb = (uint32_t)std::min<size_t>(tallest, p.rows);
    const uint32_t bands = (p.rows + rb - 1) / rb;
    bc.rb = (p.rows + bands - 1) / bands;
    bc.n_bands = (p.rows + bc.rb - 1) / bc.rb;
    *out = bc;
    return true;
}

static int matched_ctas_per_sm(const ChainParams& p, const BandConfig& bc) {
    const size_t per_cta = band_smem(p, bc.rb, bc.pitch) + sizeof(MatchedBank) + 1024;
    return (int)std::max<size_t>(1, std::min<size_t>((228 * 1024) / per_cta, 2));
}

static uint32_t band_rows_of(const ChainParams& p, const BandConfig& bc, uint32_t n_frames,
                             int sms) {
    return fit_band_rows(p.rows, bc.rb, bc.ty, (uint64_t)n_frames * p.n_modules,
                         (uint64_t)sms * matched_ctas_per_sm(p, bc));
}

uint32_t matched_call_rows(const ChainParams& p, uint32_t n_frames, int sms) {
    BandConfig bc;
    return matched_band_config(p, &bc) ? band_rows_of(p, bc, n_frames, sms) : 0;
}

static int g_attr_dev_mband = -1;

cudaError_t launch_matched(const ChainParams& p, const MatchedBank* bank_dev,
                           const uint16_t* raw, uint32_t n_frames, uint32_t frame_base,
                           const CallOut& out, cudaStream_t stream, const MultiGain* mg,
                           bool early) {
    BandConfig bc;
    if (!mg && matched_band_config(p, &bc)) {
        if (n_frames == 0) return cudaSuccess;
        bc.rb = band_rows_of(p, bc, n_frames, device_sm_count());
        bc.n_bands = (p.rows + bc.rb - 1) / bc.rb;
        const unsigned long long n_tiles =
            (unsigned long long)n_frames * p.n_modules * bc.n_bands;
        int dev = 0;
        cudaGetDevice(&dev);
        if (g_attr_dev_mband != dev) {
            for (auto k : {matched_band_kernel<false, false>, matched_band_kernel<false, true>,
                           matched_band_kernel<true, false>, matched_band_kernel<true, true>}) {
                cudaError_t e = cudaFuncSetAttribute(
                    k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBandSmem);
                if (e != cudaSuccess) return e;
            }
            g_attr_dev_mband = dev;
        }
        const size_t smem = band_smem(p, bc.rb, bc.pitch);
        unsigned long long grid =
            (unsigned long long)device_sm_count() * matched_ctas_per_sm(p, bc);
        if (grid > n_tiles) grid = n_tiles;
        const unsigned threads = bc.tx * bc.ty;
        const bool st = cm_kind(p) == PD_CM_MEAN_STACKED, col = p.unit_rows == p.rows;
        auto k = st ? (col ? matched_band_kernel<true, true> : matched_band_kernel<true, false>)
                    : (col ? matched_band_kernel<false, true> : matched_band_kernel<false, false>);
        // (early: as in launch_stencil_lean)
        cudaLaunchAttribute attr{};
        attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr.val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)grid);
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = stream;
        cfg.attrs = &attr;
        cfg.numAttrs = early && n_tiles <= kEarlyWaves * grid ? 1 : 0;
        return cudaLaunchKernelEx(&cfg, k, p, bank_dev, raw, frame_base, out, (const BandConfig)bc,
                                  n_tiles);
    }
    const uint32_t tiles_y = (p.rows + kTY - 1) / kTY;
    const uint32_t tiles_x = (p.cols + kTX - 1) / kTX;
    const unsigned long long n_tiles =
        (unsigned long long)n_frames * p.n_modules * tiles_y * tiles_x;
    if (n_tiles == 0) return cudaSuccess;
    const size_t smem = 2 * (size_t)p.hist_bins * sizeof(uint32_t);
    static bool attr_set = false;
    if (!attr_set) {
        for (auto k : {matched_kernel<false, false>, matched_kernel<true, false>,
                       matched_kernel<false, true>}) {
            cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)(2 * PD_MAX_HIST_BINS * sizeof(uint32_t)));
            if (e != cudaSuccess) return e;
        }
        attr_set = true;
    }
    unsigned long long grid = (unsigned long long)device_sm_count() * 4;
    if (grid > n_tiles) grid = n_tiles;
    const MultiGain m = mg ? *mg : MultiGain{};
    if (mg)
        matched_kernel<false, true><<<(unsigned)grid, kThreads, smem, stream>>>(
            p, bank_dev, raw, frame_base, out, tiles_y, tiles_x, n_tiles, m);
    else if (cm_kind(p) == PD_CM_MEAN_STACKED)
        matched_kernel<true, false><<<(unsigned)grid, kThreads, smem, stream>>>(
            p, bank_dev, raw, frame_base, out, tiles_y, tiles_x, n_tiles, m);
    else
        matched_kernel<false, false><<<(unsigned)grid, kThreads, smem, stream>>>(
            p, bank_dev, raw, frame_base, out, tiles_y, tiles_x, n_tiles, m);
    return cudaGetLastError();
}

}  // namespace pd
