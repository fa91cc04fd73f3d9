// pd_net_train.cu — forward, loss and backward of the learned network for a
// training batch, as three launches.
//
// The network (pd_net.cu) is a few hundred kilobytes of weights and half a
// megaflop per hit, so a step of 2048 hits is bound by launches and by the
// latency of its chain of layers, not by a rate: as one launch per layer
// (twenty kernels) it took 230 us, most of them waits for the layer before; now
// 48, the step kernel about 25 (tensor pipe 18 % active, issue 17 %).
// Here a CTA carries eight hits through every layer with their activations
// in shared memory:
//
//   prep_kernel    the weights as bf16 MMA fragments (a lane's registers of a
//                  16-deep step are one 16-byte load), and the gradients zero
//   step_kernel    conv1, conv2, FC3, heads, loss, and back to conv1; every
//                  weight gradient but W3's is summed in registers over the
//                  CTA's tiles and written to the CTA's slice once
//   finish_kernel  the sum of the slices, and W3's gradient, dz3^T h2 over
//                  128 hits a block
//
// (256 CTAs adding their 9,568 sums to the result atomically took 13 of the
// step kernel's 35 us.)  Each launch starts while the one before ends
// (programmatic dependent launch): step_kernel clears its shared memory
// during prep_kernel.  So the images are read by ordinary cached loads and not
// by the read-only path, whose memory has to stay as it is for the kernel's
// whole life.
//
// Eight hits are 200 (hit, position) rows, thirteen 16-row tiles, and one
// n-tile of FC3 and its transpose, where the weights are the 16-row operand;
// two CTAs share an SM, so that one's barriers and weight loads overlap the
// other's MMAs.  W3 (102 KB, twice per tile) comes from L2.
//
// Numerics: every contraction multiplies bf16-rounded operands and
// accumulates in float32; bias gradients, the loss and the masks are taken
// from the float32 values before rounding, except that an activation is
// positive for the mask if its bf16 value is (the same above 2^-134).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "pd_net_train.cuh"

namespace pd {
namespace nettrain {

namespace {

constexpr int NPOS = 25, C1 = 32, C2 = 32, NH = 64, NOUT = 7, K3 = NPOS * C2;
constexpr int OW1 = 0, OB1 = OW1 + C1 * 9, OW2 = OB1 + C1, OB2 = OW2 + C2 * 9 * C1,
              OW3 = OB2 + C2, OB3 = OW3 + NH * K3, OW4 = OB3 + NH, OB4 = OW4 + NOUT * NH,
              NPARAM = OB4 + NOUT;
// a CTA's slice of sums: the parameters before W3, those after it, the loss
constexpr int SL_TAIL = OW3, SL_LOSS = OW3 + NPARAM - OB3, SLICE = SL_LOSS + 1;
static_assert(SLICE % 4 == 0, "slices are read four floats at a time");

// fragment images (16-byte units: one lane's share of a 16-deep step)
constexpr int I_W3 = 0;                  // FC3, rows = outputs: [4][50][32]
constexpr int I_W3T = I_W3 + 4 * 50 * 32;   // its transpose, rows = inputs: [50][4][32]
constexpr int I_W2 = I_W3T + 50 * 4 * 32;   // conv2, columns = outputs: [18][2][32]
constexpr int I_W2T = I_W2 + 18 * 2 * 32;   // its transpose, columns = inputs
constexpr int I_W1 = I_W2T + 18 * 2 * 32;   // conv1, columns = outputs: [2][32]
constexpr int I_ALL = I_W1 + 2 * 32;

constexpr int HB = 8;               // hits per tile
constexpr int ROWS = HB * NPOS;     // 200 rows of a tile
constexpr int MT = (ROWS + 15) / 16;  // 13 16-row tiles
constexpr int PROWS = HB * 49;      // rows of the zero-bordered 7x7 grids
constexpr int ZROW = 13;            // a border row (zero) with rows +-8 inside the grids
constexpr int THREADS = 256;

// Row pitches, bytes: multiples of 16 that put eight consecutive rows in
// eight different 16-byte columns of the banks (ldmatrix without conflicts).
constexpr int AP = 80;              // 32 channels
constexpr int XP = 48;              // 16 taps
constexpr int HP = 1616;            // 800 FC3 inputs
constexpr int DP = 144;             // 64 FC3 outputs

constexpr int S_H1 = 0;                        // bf16 h1, padded grids
constexpr int S_DZ2 = S_H1 + PROWS * AP;       // bf16 dz2, padded grids
constexpr int S_XC = S_DZ2 + PROWS * AP;       // bf16 im2col of the patches
constexpr int S_DZ1 = S_XC + MT * 16 * XP;     // bf16 dz1, rows in order
constexpr int S_ZERO_END = S_DZ1 + MT * 16 * AP;  // (all of the above start at zero)
constexpr int S_H2 = S_ZERO_END;               // bf16 h2 [hit][800]
constexpr int S_RED = S_H2 + HB * HP;          // FC3 halves [2][64][8] float
constexpr int S_H3 = S_RED + 2 * NH * HB * 4;  // bf16-valued h3 [hit][65] float
constexpr int S_DZ3 = S_H3 + HB * 65 * 4;      // bf16 dz3 [hit][64]
constexpr int S_DOUT = S_DZ3 + HB * DP;        // dout [hit][8] float
constexpr int S_W4 = S_DOUT + HB * 8 * 4;      // bf16-valued W4 float
constexpr int S_X = S_W4 + NOUT * NH * 4;      // bf16 patches, padded grids
constexpr int S_ROW = S_X + PROWS * 2;         // byte offset of row i in the padded grids
constexpr int S_BYTES = S_ROW + MT * 16 * 4;
static_assert(S_H2 % 16 == 0 && S_DZ3 % 16 == 0 && S_RED % 16 == 0 && S_ROW % 4 == 0, "alignment");
static_assert(2 * (S_BYTES + 1024) <= 228 * 1024, "two CTAs per SM");

__device__ __forceinline__ uint32_t bf16_bits(float v) {
    const __nv_bfloat16 b = __float2bfloat16_rn(v);
    return *reinterpret_cast<const uint16_t*>(&b);
}
__device__ __forceinline__ float bf16_round(float v) {
    return __bfloat162float(__float2bfloat16_rn(v));
}
__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi) {
    const __nv_bfloat162 v = __float22bfloat162_rn(make_float2(lo, hi));
    return *reinterpret_cast<const uint32_t*>(&v);
}
// a bf16 bit pattern that is positive (h > 0)
__device__ __forceinline__ bool positive(uint32_t bits) {
    return (bits & 0x8000u) == 0 && (bits & 0x7FFFu) != 0 && (bits & 0x7FFFu) <= 0x7F80u;
}

__device__ __forceinline__ void mma16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                      uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, "
        "{%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
__device__ __forceinline__ void ldsm4t(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
__device__ __forceinline__ void ldsm2t(uint32_t addr, uint32_t (&r)[2]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];"
                 : "=r"(r[0]), "=r"(r[1])
                 : "r"(addr));
}
// the kernel before this one in the stream is complete, its writes visible
__device__ __forceinline__ void wait_previous() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
// the next kernel in the stream may start (and wait for this one's end)
__device__ __forceinline__ void start_next() { asm volatile("griddepcontrol.launch_dependents;"); }
// two neighbouring floats of the result (8-byte aligned), added atomically
__device__ __forceinline__ void add2(float* dst, float a, float b) {
    asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(dst), "f"(a), "f"(b) : "memory");
}

__device__ __forceinline__ int pad7(int p) { return (p / 5 + 1) * 7 + p % 5 + 1; }
// rows between a position and its neighbour at tap k in the padded grids
__host__ __device__ constexpr int tap_off(int k) { return (k / 3 - 1) * 7 + k % 3 - 1; }

// ---------------------------------------------------------------------------
// Fragments of mma.m16n8k16: lane (g = lane / 4, t = lane % 4) holds of A the
// elements (g, 2t..), (g + 8, 2t..), (g, 2t + 8..), (g + 8, 2t + 8..), of B
// (k = 2t.., n = g), (k = 2t + 8.., n = g); a B image unit holds two n-tiles.
__global__ void prep_kernel(const float* __restrict__ w, uint4* __restrict__ img,
                            float* __restrict__ gw3) {
    start_next();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < I_ALL) {
        const int lane = i & 31, g = lane >> 2, t = lane & 3;
        uint32_t q[4];
#pragma unroll
        for (int j = 0; j < 4; j++) {
            float v[2];
#pragma unroll
            for (int b = 0; b < 2; b++) {
                if (i < I_W2) {  // A fragments of W3 or its transpose
                    const bool tr = i >= I_W3T;
                    const int u = (i - (tr ? I_W3T : I_W3)) >> 5;
                    const int mt = tr ? u >> 2 : u / 50, ks = tr ? u & 3 : u % 50;
                    const int row = mt * 16 + g + (j & 1) * 8;
                    const int k = ks * 16 + 2 * t + (j >> 1) * 8 + b;
                    v[b] = w[OW3 + (tr ? k * K3 + row : row * K3 + k)];
                } else if (i < I_W1) {  // B fragments of W2 or its transpose
                    const bool tr = i >= I_W2T;
                    const int u = (i - (tr ? I_W2T : I_W2)) >> 5, ks = u >> 1, np = u & 1;
                    const int n = (2 * np + (j >> 1)) * 8 + g;
                    const int k = (ks & 1) * 16 + 2 * t + (j & 1) * 8 + b, tap = ks >> 1;
                    const int co = tr ? k : n, ci = tr ? n : k;
                    v[b] = w[OW2 + co * (9 * C1) + tap * C1 + ci];
                } else {  // B fragments of W1 (taps 9..15 are zero)
                    const int np = (i - I_W1) >> 5;
                    const int n = (2 * np + (j >> 1)) * 8 + g, k = 2 * t + (j & 1) * 8 + b;
                    v[b] = k < 9 ? w[OW1 + n * 9 + k] : 0.0f;
                }
            }
            q[j] = bf16_pair(v[0], v[1]);
        }
        img[i] = make_uint4(q[0], q[1], q[2], q[3]);
    }
    for (int k = i; k < NH * K3; k += gridDim.x * blockDim.x) gw3[k] = 0.0f;
}

// acc[m][n] = rows x weights of a 3x3 convolution over the padded grids at
// `grid` (shared address) for the 16-row tiles mt0 and mt0 + 8 (`two`); lane
// l holds row l % 16 of a tile.  SIGN -1: the transpose (rows against the
// taps' direction).
template <int SIGN>
__device__ __forceinline__ void conv_tiles(uint32_t grid, const uint4* __restrict__ img,
                                           const uint32_t* s_row, int mt0, bool two, int lane,
                                           float (&acc)[2][4][4]) {
#pragma unroll
    for (int a = 0; a < 2; a++)
#pragma unroll
        for (int b = 0; b < 4; b++)
#pragma unroll
            for (int c = 0; c < 4; c++) acc[a][b][c] = 0.0f;
    const uint32_t half = (uint32_t)(lane >> 4) * 16;
    const uint32_t r0 = grid + s_row[mt0 * 16 + (lane & 15)] + half;
    const uint32_t r1 = two ? grid + s_row[(mt0 + 8) * 16 + (lane & 15)] + half : r0;
#pragma unroll
    for (int ks = 0; ks < 18; ks++) {
        const uint4 b0 = __ldca(img + (ks * 2) * 32 + lane);
        const uint4 b1 = __ldca(img + (ks * 2 + 1) * 32 + lane);
        const int off = SIGN * tap_off(ks >> 1) * AP + (ks & 1) * 32;
        uint32_t a[4];
        ldsm4(r0 + off, a);
        mma16(acc[0][0], a[0], a[1], a[2], a[3], b0.x, b0.y);
        mma16(acc[0][1], a[0], a[1], a[2], a[3], b0.z, b0.w);
        mma16(acc[0][2], a[0], a[1], a[2], a[3], b1.x, b1.y);
        mma16(acc[0][3], a[0], a[1], a[2], a[3], b1.z, b1.w);
        if (two) {
            ldsm4(r1 + off, a);
            mma16(acc[1][0], a[0], a[1], a[2], a[3], b0.x, b0.y);
            mma16(acc[1][1], a[0], a[1], a[2], a[3], b0.z, b0.w);
            mma16(acc[1][2], a[0], a[1], a[2], a[3], b1.x, b1.y);
            mma16(acc[1][3], a[0], a[1], a[2], a[3], b1.z, b1.w);
        }
    }
}

__global__ void __launch_bounds__(THREADS, 2)
    step_kernel(const float* __restrict__ w, const uint4* __restrict__ img,
                const float* __restrict__ x, const uint8_t* __restrict__ counts,
                const float* __restrict__ tgt, const uint8_t* __restrict__ mask, int n, float nreg,
                float lam, uint16_t* __restrict__ h2_out, uint16_t* __restrict__ dz3_out,
                float* __restrict__ slices) {
    extern __shared__ __align__(128) uint8_t sm[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, tq = lane & 3;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(sm);
    float* s_red = reinterpret_cast<float*>(sm + S_RED);
    float* s_h3 = reinterpret_cast<float*>(sm + S_H3);
    float* s_dout = reinterpret_cast<float*>(sm + S_DOUT);
    float* s_w4 = reinterpret_cast<float*>(sm + S_W4);
    uint16_t* s_x = reinterpret_cast<uint16_t*>(sm + S_X);
    uint32_t* s_row = reinterpret_cast<uint32_t*>(sm + S_ROW);

    for (int i = tid; i < S_ZERO_END / 16; i += THREADS)
        reinterpret_cast<uint4*>(sm)[i] = make_uint4(0, 0, 0, 0);
    for (int i = tid; i < PROWS; i += THREADS) s_x[i] = 0;
    for (int i = tid; i < MT * 16; i += THREADS)
        s_row[i] = (i < ROWS ? (i / NPOS) * 49 + pad7(i % NPOS) : ZROW) * AP;
    for (int i = tid; i < NOUT * NH; i += THREADS) s_w4[i] = bf16_round(w[OW4 + i]);

    // sums over the CTA's tiles
    float gw2[9][4];                 // W2: 16 c_out x 8 c_in of every tap
    float gw1[4] = {0, 0, 0, 0};     // W1: 16 c_out x 8 taps, half of the rows
    float gb1[8], gb2[2] = {0, 0};   // biases: this lane's channels
    float gw4[2] = {0, 0}, gb4 = 0.0f, gb3[2] = {0, 0}, l_sum = 0.0f;
#pragma unroll
    for (int k = 0; k < 9; k++)
#pragma unroll
        for (int c = 0; c < 4; c++) gw2[k][c] = 0.0f;
#pragma unroll
    for (int c = 0; c < 8; c++) gb1[c] = 0.0f;

    wait_previous();  // the weight images
    const int n_tiles = (n + HB - 1) / HB;
    for (int t = blockIdx.x; t < n_tiles; t += gridDim.x) {
        const int hit0 = t * HB, nh = min(HB, n - hit0);
        __syncthreads();  // shared memory set up, or the previous tile done
        if (tid < ROWS) {
            const float v = tid < nh * NPOS ? x[(size_t)hit0 * NPOS + tid] : 0.0f;
            s_x[(tid / NPOS) * 49 + pad7(tid % NPOS)] = (uint16_t)bf16_bits(v);
        }
        __syncthreads();

        // im2col of the patches: nine taps a row
        if (tid < ROWS) {
            const uint16_t* c = s_x + (tid / NPOS) * 49 + pad7(tid % NPOS);
            auto two = [&](int k) {
                return (uint32_t)c[tap_off(k)] | (uint32_t)c[tap_off(k + 1)] << 16;
            };
            uint8_t* row = sm + S_XC + tid * XP;
            *reinterpret_cast<uint4*>(row) = make_uint4(two(0), two(2), two(4), two(6));
            *reinterpret_cast<uint32_t*>(row + 16) = c[tap_off(8)];
        }
        __syncthreads();

        // conv1: 16 taps deep
        {
            const uint4 b0 = __ldca(img + I_W1 + lane), b1 = __ldca(img + I_W1 + 32 + lane);
            for (int mt = warp; mt < MT; mt += 8) {
                uint32_t a[4];
                ldsm4(base + S_XC + (mt * 16 + (lane & 15)) * XP + (lane >> 4) * 16, a);
                float c[4][4] = {};
                mma16(c[0], a[0], a[1], a[2], a[3], b0.x, b0.y);
                mma16(c[1], a[0], a[1], a[2], a[3], b0.z, b0.w);
                mma16(c[2], a[0], a[1], a[2], a[3], b1.x, b1.y);
                mma16(c[3], a[0], a[1], a[2], a[3], b1.z, b1.w);
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const int row = mt * 16 + g + 8 * h;
                    if (row >= ROWS) continue;
                    uint8_t* dst = sm + S_H1 + s_row[row] + 4 * tq;
#pragma unroll
                    for (int nt = 0; nt < 4; nt++) {
                        const float* b = w + OB1 + nt * 8 + 2 * tq;
                        *reinterpret_cast<uint32_t*>(dst + nt * 16) =
                            bf16_pair(fmaxf(c[nt][2 * h] + __ldg(b), 0.0f),
                                      fmaxf(c[nt][2 * h + 1] + __ldg(b + 1), 0.0f));
                    }
                }
            }
        }
        __syncthreads();

        // conv2
        const bool two = warp + 8 < MT;
        {
            float acc[2][4][4];
            conv_tiles<1>(base + S_H1, img + I_W2, s_row, warp, two, lane, acc);
#pragma unroll
            for (int m = 0; m < 2; m++)
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const int row = (warp + 8 * m) * 16 + g + 8 * h;
                    if (row >= ROWS) continue;
                    const int hit = row / NPOS, pos = row - hit * NPOS;
                    uint8_t* dst = sm + S_H2 + hit * HP + pos * 64 + 4 * tq;
#pragma unroll
                    for (int nt = 0; nt < 4; nt++) {
                        const float* b = w + OB2 + nt * 8 + 2 * tq;
                        *reinterpret_cast<uint32_t*>(dst + nt * 16) =
                            bf16_pair(fmaxf(acc[m][nt][2 * h] + __ldg(b), 0.0f),
                                      fmaxf(acc[m][nt][2 * h + 1] + __ldg(b + 1), 0.0f));
                    }
                }
        }
        __syncthreads();

        // FC3 (rows = outputs, columns = hits): warp (mt, half of K)
        {
            const int mt = warp & 3, k0 = (warp >> 2) * 25;
            const uint4* wp = img + I_W3 + (mt * 50 + k0) * 32 + lane;
            const uint8_t* hb = sm + S_H2 + g * HP + k0 * 32 + 4 * tq;
            float c[4] = {0, 0, 0, 0}, d[4] = {0, 0, 0, 0};
#pragma unroll
            for (int part = 0; part < 3; part++) {  // nine loads in flight
                uint4 a[9];
#pragma unroll
                for (int s = 0; s < 9; s++)
                    if (part * 9 + s < 25) a[s] = __ldcg(wp + (part * 9 + s) * 32);
#pragma unroll
                for (int s = 0; s < 9; s++) {
                    const int ks = part * 9 + s;
                    if (ks >= 25) continue;
                    const uint32_t b0 = *reinterpret_cast<const uint32_t*>(hb + ks * 32);
                    const uint32_t b1 = *reinterpret_cast<const uint32_t*>(hb + ks * 32 + 16);
                    if (s & 1)
                        mma16(d, a[s].x, a[s].y, a[s].z, a[s].w, b0, b1);
                    else
                        mma16(c, a[s].x, a[s].y, a[s].z, a[s].w, b0, b1);
                }
            }
            float* r = s_red + (warp >> 2) * (NH * HB) + (mt * 16 + g) * HB + 2 * tq;
            *reinterpret_cast<float2*>(r) = make_float2(c[0] + d[0], c[1] + d[1]);
            *reinterpret_cast<float2*>(r + 8 * HB) = make_float2(c[2] + d[2], c[3] + d[3]);
            // h2 rows for W3's gradient
            for (int e = tid; e < nh * (K3 / 8); e += THREADS) {
                const int hit = e / (K3 / 8), q = e - hit * (K3 / 8);
                reinterpret_cast<uint4*>(h2_out + (size_t)(hit0 + hit) * K3)[q] =
                    *reinterpret_cast<const uint4*>(sm + S_H2 + hit * HP + q * 16);
            }
        }
        __syncthreads();

        // heads, loss, dout and dz3: one warp per hit, two hidden units a lane
        {
            const int hit = warp;
            const bool in = hit < nh;
            float hv[2], o[NOUT];
#pragma unroll
            for (int u = 0; u < 2; u++) {
                const int j = lane + 32 * u;
                hv[u] = fmaxf(s_red[j * HB + hit] + s_red[NH * HB + j * HB + hit] + w[OB3 + j],
                              0.0f);
                s_h3[hit * 65 + j] = bf16_round(hv[u]);
            }
#pragma unroll
            for (int k = 0; k < NOUT; k++) {
                float v = __fmaf_rn(bf16_round(hv[1]), s_w4[k * NH + lane + 32],
                                    bf16_round(hv[0]) * s_w4[k * NH + lane]);
#pragma unroll
                for (int b = 16; b; b >>= 1) v += __shfl_xor_sync(0xffffffffu, v, b);
                o[k] = v + w[OB4 + k];
            }
            float mx = o[0];
#pragma unroll
            for (int k = 1; k < 5; k++) mx = fmaxf(mx, o[k]);
            float e[5], s = 0.0f, dk[NOUT];
#pragma unroll
            for (int k = 0; k < 5; k++) {
                e[k] = expf(o[k] - mx);
                s += e[k];
            }
            const int cnt = in ? min((int)counts[hit0 + hit], 4) : 0;
            float l = 0.0f;
#pragma unroll
            for (int k = 0; k < 5; k++) {
                dk[k] = (e[k] / s - (k == cnt ? 1.0f : 0.0f)) / (float)n;
                if (k == cnt) l = -logf(e[k] / s) / (float)n;
            }
            const float mk = in && mask[hit0 + hit] ? 1.0f : 0.0f;
#pragma unroll
            for (int k = 0; k < 2; k++) {
                const float diff = in ? (o[5 + k] - tgt[(size_t)(hit0 + hit) * 2 + k]) * mk : 0.0f;
                dk[5 + k] = 2.0f * lam * diff / nreg;
                l += lam * diff * diff / nreg;
            }
            if (in) l_sum += l;
#pragma unroll
            for (int k = 0; k < NOUT; k++) {
                if (!in) dk[k] = 0.0f;
                if (lane == k) s_dout[hit * 8 + k] = dk[k];
                dk[k] = bf16_round(dk[k]);
            }
#pragma unroll
            for (int u = 0; u < 2; u++) {
                const int j = lane + 32 * u;
                float v = 0.0f;
#pragma unroll
                for (int k = 0; k < NOUT; k++) v = __fmaf_rn(dk[k], s_w4[k * NH + j], v);
                v = hv[u] > 0.0f ? v : 0.0f;
                gb3[u] += v;
                const uint16_t b = (uint16_t)bf16_bits(v);
                *reinterpret_cast<uint16_t*>(sm + S_DZ3 + hit * DP + j * 2) = b;
                if (in) dz3_out[(size_t)(hit0 + hit) * NH + j] = b;
            }
        }
        __syncthreads();

        // the heads' gradients, and dz2 = dz3 W3 where h2 > 0 (rows = FC3
        // inputs, columns = hits)
        {
#pragma unroll
            for (int u = 0; u < 2; u++) {
                const int q = tid + u * THREADS;
                if (q < NOUT * NH) {
                    const int k = q / NH, j = q - k * NH;
#pragma unroll
                    for (int h = 0; h < HB; h++)
                        gw4[u] = __fmaf_rn(bf16_round(s_dout[h * 8 + k]), s_h3[h * 65 + j], gw4[u]);
                }
            }
            if (tid < NOUT)
#pragma unroll
                for (int h = 0; h < HB; h++) gb4 += s_dout[h * 8 + tid];
            uint32_t b[4][2];
#pragma unroll
            for (int ks = 0; ks < 4; ks++) {
                const uint8_t* r = sm + S_DZ3 + g * DP + ks * 32 + 4 * tq;
                b[ks][0] = *reinterpret_cast<const uint32_t*>(r);
                b[ks][1] = *reinterpret_cast<const uint32_t*>(r + 16);
            }
            // (mt is even for even warps, so a lane's channels stay the same)
#pragma unroll
            for (int i = 0; i < 7; i++) {
                const int mt = warp + 8 * i;
                if (mt >= 50) break;
                const uint4* wp = img + I_W3T + mt * 4 * 32 + lane;
                float c[4] = {0, 0, 0, 0};
#pragma unroll
                for (int ks = 0; ks < 4; ks++) {
                    const uint4 a = __ldcg(wp + ks * 32);
                    mma16(c, a.x, a.y, a.z, a.w, b[ks][0], b[ks][1]);
                }
                const int pos = mt >> 1, ch = (mt & 1) * 16 + g;
                const uint32_t prow = (uint32_t)pad7(pos);
#pragma unroll
                for (int q = 0; q < 4; q++) {  // (row g + 8 (q / 2), hit 2 tq + q % 2)
                    const int hit = 2 * tq + (q & 1), cc = ch + 8 * (q >> 1);
                    const uint32_t h = *reinterpret_cast<const uint16_t*>(
                        sm + S_H2 + hit * HP + pos * 64 + cc * 2);
                    const float v = positive(h) ? c[q] : 0.0f;
                    gb2[q >> 1] += v;
                    *reinterpret_cast<uint16_t*>(sm + S_DZ2 + (hit * 49 + prow) * AP + cc * 2) =
                        (uint16_t)bf16_bits(v);
                }
            }
        }
        __syncthreads();

        // dz1 = conv2's transpose of dz2 where h1 > 0
        {
            float acc[2][4][4];
            conv_tiles<-1>(base + S_DZ2, img + I_W2T, s_row, warp, two, lane, acc);
#pragma unroll
            for (int m = 0; m < 2; m++)
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const int row = (warp + 8 * m) * 16 + g + 8 * h;
                    if (row >= ROWS) continue;
                    const uint8_t* act = sm + S_H1 + s_row[row] + 4 * tq;
                    uint8_t* dst = sm + S_DZ1 + row * AP + 4 * tq;
#pragma unroll
                    for (int nt = 0; nt < 4; nt++) {
                        const uint32_t a = *reinterpret_cast<const uint32_t*>(act + nt * 16);
                        const float v0 = positive(a & 0xFFFFu) ? acc[m][nt][2 * h] : 0.0f;
                        const float v1 = positive(a >> 16) ? acc[m][nt][2 * h + 1] : 0.0f;
                        gb1[2 * nt] += v0;
                        gb1[2 * nt + 1] += v1;
                        *reinterpret_cast<uint32_t*>(dst + nt * 16) = bf16_pair(v0, v1);
                    }
                }
        }
        // W2: dz2^T (c_out x rows) h1 (rows shifted by the tap x c_in); warp
        // (16 c_out, 8 c_in), all taps
        {
            const uint32_t a_ch = (uint32_t)((warp & 1) * 32 + ((lane >> 3) & 1) * 16);
            const uint32_t b_ch = (uint32_t)((warp >> 1) * 16);
            const int a_r = (lane & 7) + ((lane >> 4) << 3), b_r = lane & 15;
            const int hi = lane >> 4;  // which tap of a pair this lane addresses
            for (int ks = 0; ks < MT; ks++) {
                uint32_t a[4], b[4], b8[2];
                ldsm4t(base + S_DZ2 + s_row[ks * 16 + a_r] + a_ch, a);
                const uint32_t br = base + S_H1 + s_row[ks * 16 + b_r] + b_ch;
#pragma unroll
                for (int k = 0; k < 8; k += 2) {
                    ldsm4t(br + (hi ? tap_off(k + 1) : tap_off(k)) * AP, b);
                    mma16(gw2[k], a[0], a[1], a[2], a[3], b[0], b[1]);
                    mma16(gw2[k + 1], a[0], a[1], a[2], a[3], b[2], b[3]);
                }
                ldsm2t(br + tap_off(8) * AP, b8);
                mma16(gw2[8], a[0], a[1], a[2], a[3], b8[0], b8[1]);
            }
        }
        __syncthreads();

        // W1: dz1^T (c_out x rows) im2col (rows x taps); warp (16 c_out, 8
        // taps, every other step)
        {
            const uint32_t a_ch = (uint32_t)((warp & 1) * 32 + ((lane >> 3) & 1) * 16);
            const uint32_t b_ch = (uint32_t)(((warp >> 1) & 1) * 16);
            const int a_r = (lane & 7) + ((lane >> 4) << 3), b_r = lane & 15;
            for (int ks = warp >> 2; ks < MT; ks += 2) {
                uint32_t a[4], b[2];
                ldsm4t(base + S_DZ1 + (ks * 16 + a_r) * AP + a_ch, a);
                ldsm2t(base + S_XC + (ks * 16 + b_r) * XP + b_ch, b);
                mma16(gw1, a[0], a[1], a[2], a[3], b[0], b[1]);
            }
        }
    }

    // the CTA's sums into its slice: W2's straight from registers, the others
    // summed over the warps in shared memory first
    start_next();
    float* slice = slices + (size_t)blockIdx.x * SLICE;
    constexpr int F_B1 = 288, F_B2 = F_B1 + C1, F_TAIL = F_B2 + C2, F_ALL = F_TAIL + SLICE - SL_TAIL;
    static_assert(F_ALL <= 2 * NH * HB, "the small sums fit the FC3 halves");
    for (int i = tid; i < F_ALL; i += THREADS) s_red[i] = 0.0f;
    {
        const int co = (warp & 1) * 16 + g, ci = (warp >> 1) * 8 + 2 * tq;
        float* d = slice + OW2 + co * (9 * C1) + ci;
#pragma unroll
        for (int k = 0; k < 9; k++) {
            *reinterpret_cast<float2*>(d + k * C1) = make_float2(gw2[k][0], gw2[k][1]);
            *reinterpret_cast<float2*>(d + 8 * 9 * C1 + k * C1) = make_float2(gw2[k][2], gw2[k][3]);
        }
    }
    __syncthreads();
    {
        const int co = (warp & 1) * 16 + g, k = ((warp >> 1) & 1) * 8 + 2 * tq;
#pragma unroll
        for (int c = 0; c < 4; c++)
            if (k + (c & 1) < 9)
                atomicAdd(s_red + (co + 8 * (c >> 1)) * 9 + k + (c & 1), gw1[c]);
    }
#pragma unroll
    for (int c = 0; c < 8; c++) {
        float v = gb1[c];
#pragma unroll
        for (int b = 4; b < 32; b <<= 1) v += __shfl_xor_sync(0xffffffffu, v, b);
        if (g == 0) atomicAdd(s_red + F_B1 + (c >> 1) * 8 + 2 * tq + (c & 1), v);
    }
#pragma unroll
    for (int c = 0; c < 2; c++) {
        float v = gb2[c];
#pragma unroll
        for (int b = 1; b < 4; b <<= 1) v += __shfl_xor_sync(0xffffffffu, v, b);
        if (tq == 0) atomicAdd(s_red + F_B2 + (warp & 1) * 16 + g + 8 * c, v);
        atomicAdd(s_red + F_TAIL + lane + 32 * c, gb3[c]);
        const int q = tid + c * THREADS;
        if (q < NOUT * NH) s_red[F_TAIL + OW4 - OB3 + q] = gw4[c];
    }
    if (tid < NOUT) s_red[F_TAIL + OB4 - OB3 + tid] = gb4;
    if (lane == 0) atomicAdd(s_red + F_TAIL + SL_LOSS - SL_TAIL, l_sum);
    __syncthreads();
    for (int i = tid; i < F_ALL; i += THREADS) {
        const int at = i < F_B1 ? OW1 + i : i < F_B2 ? OB1 + i - F_B1
                     : i < F_TAIL ? OB2 + i - F_B2 : SL_TAIL + i - F_TAIL;
        slice[at] = s_red[i];
    }
}

// ---------------------------------------------------------------------------
// The first SUM_BLOCKS blocks sum 128 places of the slices each (a warp every
// eighth slice); the others add dz3^T h2 over 128 hits to 80 columns of
// gw3[64][800], both operands read transposed from their rows in shared memory.
constexpr int W3_HITS = 128, W3_COLS = 80, W3_HP = 176;
constexpr int SUM_BLOCKS = (SLICE / 4 + 31) / 32;

__device__ __forceinline__ void sum_slices(const float* __restrict__ slices, int n_slices,
                                           float* __restrict__ grads, float* __restrict__ loss,
                                           float4 (*part)[32]) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int q = blockIdx.x * 32 + lane;
    float4 a = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (q < SLICE / 4)
#pragma unroll 8
        for (int i = warp; i < n_slices; i += THREADS / 32) {
            const float4 v = __ldcg(reinterpret_cast<const float4*>(slices + (size_t)i * SLICE) + q);
            a.x += v.x;
            a.y += v.y;
            a.z += v.z;
            a.w += v.w;
        }
    part[warp][lane] = a;
    __syncthreads();
    if (threadIdx.x < 128) {
        const float* f = reinterpret_cast<const float*>(part) + threadIdx.x;
        float v = 0.0f;
#pragma unroll
        for (int k = 0; k < THREADS / 32; k++) v += f[k * 128];
        const int at = blockIdx.x * 128 + threadIdx.x;
        if (at < SL_TAIL)
            grads[at] = v;
        else if (at < SL_LOSS)
            grads[OB3 + at - SL_TAIL] = v;
        else if (at == SL_LOSS && loss)
            atomicAdd(loss, v);
    }
}

__global__ void __launch_bounds__(THREADS)
    finish_kernel(const float* __restrict__ slices, int n_slices, const uint16_t* __restrict__ dz3,
                  const uint16_t* __restrict__ h2, int n, float* __restrict__ grads,
                  float* __restrict__ loss) {
    __shared__ __align__(128) uint8_t sd[W3_HITS * DP];
    __shared__ __align__(128) uint8_t sh[W3_HITS * W3_HP];
    wait_previous();
    if (blockIdx.x < SUM_BLOCKS) {
        sum_slices(slices, n_slices, grads, loss, reinterpret_cast<float4 (*)[32]>(sd));
        return;
    }
    const int block = blockIdx.x - SUM_BLOCKS;
    float* gw3 = grads + OW3;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, tq = lane & 3;
    const int col0 = block % (K3 / W3_COLS) * W3_COLS, hit0 = block / (K3 / W3_COLS) * W3_HITS;
    const int nh = min(W3_HITS, n - hit0);
    const uint32_t sda = (uint32_t)__cvta_generic_to_shared(sd);
    const uint32_t sha = (uint32_t)__cvta_generic_to_shared(sh);
    auto copy = [](uint32_t dst, const uint16_t* src, bool in) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src),
                     "r"(in ? 16 : 0)
                     : "memory");
    };
    for (int e = tid; e < W3_HITS * 8; e += THREADS) {
        const int r = e >> 3, q = e & 7;
        copy(sda + r * DP + q * 16, dz3 + (size_t)(hit0 + min(r, nh - 1)) * NH + q * 8, r < nh);
    }
    for (int e = tid; e < W3_HITS * (W3_COLS / 8); e += THREADS) {
        const int r = e / (W3_COLS / 8), q = e - r * (W3_COLS / 8);
        copy(sha + r * W3_HP + q * 16, h2 + (size_t)(hit0 + min(r, nh - 1)) * K3 + col0 + q * 8,
             r < nh);
    }
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
    const int mt = warp & 3, n0 = (warp >> 2) * 5;
    const int a_r = (lane & 7) + ((lane >> 4) << 3), b_r = lane & 15;
    const uint32_t a_ch = (uint32_t)(mt * 32 + ((lane >> 3) & 1) * 16);
    const uint32_t b_ch = (uint32_t)(n0 * 16 + (lane >> 4) * 16);
    float c[5][4];
#pragma unroll
    for (int i = 0; i < 5; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) c[i][j] = 0.0f;
#pragma unroll
    for (int ks = 0; ks < W3_HITS / 16; ks++) {
        uint32_t a[4], b[4], b4[2];
        ldsm4t(sda + (ks * 16 + a_r) * DP + a_ch, a);
        const uint32_t br = sha + (ks * 16 + b_r) * W3_HP + b_ch;
#pragma unroll
        for (int i = 0; i < 4; i += 2) {
            ldsm4t(br + i * 16, b);
            mma16(c[i], a[0], a[1], a[2], a[3], b[0], b[1]);
            mma16(c[i + 1], a[0], a[1], a[2], a[3], b[2], b[3]);
        }
        ldsm2t(br + 64, b4);
        mma16(c[4], a[0], a[1], a[2], a[3], b4[0], b4[1]);
    }
    float* d = gw3 + (size_t)(mt * 16 + g) * K3 + col0 + n0 * 8 + 2 * tq;
#pragma unroll
    for (int i = 0; i < 5; i++) {
        add2(d + i * 8, c[i][0], c[i][1]);
        add2(d + 8 * K3 + i * 8, c[i][2], c[i][3]);
    }
}

}  // namespace

size_t image_bytes() { return (size_t)I_ALL * sizeof(uint4); }
size_t h2_bytes(uint32_t max_batch) { return (size_t)max_batch * K3 * 2; }
size_t dz3_bytes(uint32_t max_batch) { return (size_t)max_batch * NH * 2; }
static uint32_t max_slices(int sms) { return 2u * (uint32_t)sms; }  // the persistent CTAs
size_t slice_bytes(uint32_t max_batch, int sms) {
    return (size_t)std::min((max_batch - 1) / HB + 1, max_slices(sms)) * SLICE * sizeof(float);
}

cudaError_t gradients(const float* w, const float* x, const uint8_t* counts, const float* targets,
                      const uint8_t* mask, uint32_t n, float n_reg, float lambda, uint4* img,
                      uint16_t* h2, uint16_t* dz3, float* slices, float* grads,
                      float* loss, int sms, cudaStream_t s) {
    static int attr_dev = -1;  // the shared-memory opt-in, once per device
    int dev = 0;
    cudaGetDevice(&dev);
    if (attr_dev != dev) {
        const cudaError_t e = cudaFuncSetAttribute(
            step_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, S_BYTES);
        if (e != cudaSuccess) return e;
        attr_dev = dev;
    }
    prep_kernel<<<(I_ALL + 255) / 256, 256, 0, s>>>(w, img, grads + OW3);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute early{};
    early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    early.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.blockDim = dim3(THREADS);
    cfg.stream = s;
    cfg.attrs = &early;
    cfg.numAttrs = 1;
    const uint32_t grid = std::min((n - 1) / HB + 1, max_slices(sms));
    cfg.gridDim = dim3(grid);
    cfg.dynamicSmemBytes = S_BYTES;
    e = cudaLaunchKernelEx(&cfg, step_kernel, w, (const uint4*)img, x, counts, targets, mask, (int)n,
                           n_reg, lambda, h2, dz3, slices);
    if (e != cudaSuccess) return e;
    cfg.gridDim = dim3(SUM_BLOCKS + K3 / W3_COLS * ((n + W3_HITS - 1) / W3_HITS));
    cfg.dynamicSmemBytes = 0;
    return cudaLaunchKernelEx(&cfg, finish_kernel, (const float*)slices, (int)grid,
                              (const uint16_t*)dz3, (const uint16_t*)h2, (int)n, grads, loss);
}

}  // namespace nettrain
}  // namespace pd
