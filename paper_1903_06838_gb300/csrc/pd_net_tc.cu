// pd_net_tc.cu — inference of the learned count / offset network on the
// fifth-generation tensor cores: tcgen05.mma with bfloat16 operands staged in
// shared memory and float32 accumulators in tensor memory (TMEM).
//
// The network (conv3x3x32 -> conv3x3x32 -> FC64 -> 7 outputs on the 5x5
// neighbourhood of a seed) is the learned refinement the paper proposes as
// future work (abstract; sections "Methods", "Conclusions").  Numerics match
// the training path: every contraction multiplies bfloat16-rounded operands
// (weights, input patch, and the ReLU activations h1, h2, h3) and
// accumulates in float32; biases and ReLU are float32.
//
//   conv_kernel  conv1 and conv2 on tiles of 64 hits, one persistent CTA per
//                SM with specialised warps (below)
//   fc_kernel    FC3 on tiles of 128 hits and the 7 heads: a ring of bulk
//                copies of h2 against W3 resident in shared memory, the heads
//                (FC4) on the CUDA cores
//
// Operand layout: the canonical no-swizzle K-major form: 8-row x 16-byte core
// matrices, core matrix (r, k) of a tile with R rows at byte
// ((k / 8) * (R / 8) + r / 8) * 128; descriptors carry the distance of
// K-adjacent core matrices (leading) and of row-adjacent ones (stride).
// Every wait on an mbarrier is bounded; a timeout sets an error flag.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "pd_net_tc.cuh"

namespace pd {
namespace nettc {

namespace {

constexpr int NPOS = 25, C1 = 32, C2 = 32, NH = 64, NOUT = 7;
constexpr int K2 = 9 * C1;           // 288
constexpr int K3 = NPOS * C2;        // 800
constexpr int TB = 64;               // hits per conv tile
constexpr int TF = 128;              // hits per fc tile
constexpr uint32_t kWaitLimit = 1u << 22;

// weight offsets (floats) in the parameter vector, as the training path
constexpr int OW1 = 0, OB1 = OW1 + C1 * 9, OW2 = OB1 + C1, OB2 = OW2 + C2 * K2, OW3 = OB2 + C2,
              OB3 = OW3 + NH * K3, OW4 = OB3 + NH, OB4 = OW4 + NOUT * NH;

// bf16 operand images of the weights (bytes)
constexpr uint32_t W2_BYTES = 32 * K2 * 2, W3_BYTES = NH * K3 * 2;
constexpr uint32_t OFF_W2 = 0, OFF_W3 = OFF_W2 + W2_BYTES;
constexpr uint32_t W2_SLICE = 96 * 16 * 2;  // one tap row, 16 input channels

__host__ __device__ __forceinline__ uint32_t cm_off(uint32_t r, uint32_t k, uint32_t rows) {
    return ((k >> 3) * (rows >> 3) + (r >> 3)) * 128u + (r & 7u) * 16u + (k & 7u) * 2u;
}

__device__ __forceinline__ uint16_t bf16_bits(float v) {
    const __nv_bfloat16 b = __float2bfloat16_rn(v);
    return *reinterpret_cast<const uint16_t*>(&b);
}
__device__ __forceinline__ float bf16_round(float v) {
    return __bfloat162float(__float2bfloat16_rn(v));
}
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo & 0x3FFFFu) >> 4) << 16) |
           ((uint64_t)((sbo & 0x3FFFFu) >> 4) << 32) | ((uint64_t)1 << 46);
}
// kind::f16 instruction descriptor: f32 accumulate, bf16 A and B, both
// K-major, N >> 3 at bit 17, M >> 4 at bit 24
__device__ __forceinline__ uint32_t idesc_bf16(uint32_t m, uint32_t n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((n >> 3) << 17) | ((m >> 4) << 24);
}
// (volatile keeps tcgen05 operations in program order; shared-memory
// operands are published before the issue by fences and a barrier, so no
// memory clobber is needed and the issuing thread's table loads can run
// ahead)
__device__ __forceinline__ void mma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc,
                                    uint32_t acc) {
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.u32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc));
}
__device__ __forceinline__ void commit(uint64_t* bar) {
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
            smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ void fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
// Programmatic dependent launch: the kernel before this one in the stream is
// complete; the next one may start when every CTA has said so or is done.
__device__ __forceinline__ void wait_previous() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void start_next() { asm volatile("griddepcontrol.launch_dependents;"); }
// bounded wait for the phase with parity `par`; false on timeout
__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t par) {
    const uint32_t a = smem_u32(bar);
    for (uint32_t it = 0; it < kWaitLimit; it++) {
        uint32_t ok;
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            "selp.u32 %0, 1, 0, p;\n}"
            : "=r"(ok)
            : "r"(a), "r"(par)
            : "memory");
        if (ok) return true;
    }
    return false;
}
__device__ __forceinline__ void bar_init(uint64_t* bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tmem_alloc(uint32_t* dst, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(dst)),
                 "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_free(uint32_t taddr, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols)
                 : "memory");
}
// 32 columns of 16 TMEM lanes as four 16 x 8 blocks: of block k, lane (g, t)
// gets rows g (r[4k], r[4k + 1]) and g + 8, columns 2t, 2t + 1
__device__ __forceinline__ void tmem_ld16x32(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
        "%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() {
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// 32 consecutive columns of this warp's 32 TMEM lanes, one wait
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
        "%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
          "=r"(r[31])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// neighbour of position p at 3x3 offset k (k = 3 (dy + 1) + dx + 1), or -1
__device__ __forceinline__ int nb(int p, int k) {
    const int y = p / 5 + k / 3 - 1, x = p % 5 + k % 3 - 1;
    return (y >= 0 && y < 5 && x >= 0 && x < 5) ? y * 5 + x : -1;
}

// ---------------------------------------------------------------------------
// bf16 operand images, K-major core matrices, from the float32 parameters:
// of W2 one matrix per tap row ky and half of the input channels, its 96 rows
// (j, c_out) the taps kx = 2 - j, so that with an input column x as A they are
// the outputs at x - 1, x, x + 1; and W3 (64 x 800).
__global__ void prep_weights(const float* __restrict__ w, uint8_t* __restrict__ img) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < 32 * K2) {
        const int co = i / K2, k = i % K2, tap = k / C1, ci = k % C1;
        const int row = (2 - tap % 3) * 32 + co;
        *reinterpret_cast<uint16_t*>(img + OFF_W2 + (tap / 3 * 2 + ci / 16) * W2_SLICE +
                                     cm_off(row, ci % 16, 96)) = bf16_bits(w[OW2 + i]);
    }
    if (i < NH * K3) {
        const int r = i / K3, k = i % K3;
        *reinterpret_cast<uint16_t*>(img + OFF_W3 + cm_off(r, k, NH)) = bf16_bits(w[OW3 + i]);
    }
}

// ---------------------------------------------------------------------------
// conv1 + conv2 on tiles of 64 hits, h2 out as bf16 in the layout fc_kernel
// copies: per 128 hits [k / 8][hit][8 values].  One CTA of 512 threads per SM
// with specialised warps:
//   warps 0-7   conv1 as m16n8k16 MMAs (bf16 operands, float32 accumulation)
//               into one of two h1 stages: per position a 64-hit x 32-channel
//               K-major block (4 KB), 100 KB per stage
//   warps 8-10  lane 0 of warp 8 + b issues the conv2 MMAs of the output rows
//               that use TMEM buffer b (160 columns: 5 positions): an implicit
//               GEMM read in place.  A is an input position's block, B the
//               three taps of a tap row for 16 input channels (96 columns, the
//               outputs at x - 1, x, x + 1; 64 at the border), added at the
//               output columns' place in TMEM, so no tap outside the patch is
//               computed.  The issue of an MMA costs 25 to 50 cycles whatever
//               its size: 145 MMAs of up to 64 x 96 x 16 a tile in place of
//               338 of 64 x 32 x 16, one per tap, took the kernel from 82 us
//               per 65,536 hits to 52.
//   warps 12-15 the epilogue: TMEM -> bias, ReLU, bf16 -> h2 (warp 12 + q
//               reads TMEM lanes 32q..32q+15, where M = 64 puts rows
//               16q..16q+15, as 16-lane blocks: every lane holds two rows'
//               column pairs, and a store of the warp is 128 contiguous bytes)
// mbarriers hand the stages and TMEM buffers around (h1 full / empty, TMEM
// full / empty), so conv1 of the next tile, conv2 MMAs and the epilogue of
// earlier rows overlap.  Every wait is bounded; a timeout sets *err, stops
// every role, and the issuing lane waits (bounded) for its last commit
// before TMEM is freed.
constexpr int WS_PROD_WARPS = 8, WS_MMA_WARP0 = 8, WS_EPI_WARP0 = 12;
constexpr int WS_PROD = WS_PROD_WARPS * 32, WS_THREADS = 512;
constexpr uint32_t H1_STAGE = TB * NPOS * C1 * 2;  // 102 400 bytes
constexpr uint32_t WS_W2 = 0, WS_H1 = WS_W2 + W2_BYTES, WS_X = WS_H1 + 2 * H1_STAGE,
                   WS_SMEM = WS_X + TB * NPOS * 2;
constexpr uint32_t kConvTmemCols = 512;
constexpr int kRowCols = 5 * 32;  // TMEM columns of an output row
constexpr int kTBufs = 3;         // TMEM buffers
static_assert(WS_H1 % 128 == 0 && H1_STAGE % 128 == 0, "alignment");
static_assert(kTBufs * kRowCols <= (int)kConvTmemCols, "TMEM buffers");

__device__ __forceinline__ void bar_init_n(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
                 : "memory");
}
__device__ __forceinline__ void bar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void producers_sync() {
    asm volatile("bar.sync 1, %0;" ::"n"(WS_PROD) : "memory");
}

__global__ void __launch_bounds__(WS_THREADS, 1)
    conv_kernel(const float* __restrict__ x, int n, const float* __restrict__ w,
                const uint8_t* __restrict__ img, uint16_t* __restrict__ h2, int* err) {
    extern __shared__ __align__(1024) uint8_t sm[];
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_abort;
    __shared__ int s_prod_go;  // the producers' uniform decision for a tile
    __shared__ __align__(8) uint64_t s_h1_full[2], s_h1_empty[2], s_t_full[kTBufs],
        s_t_empty[kTBufs];
    __shared__ int s_nb[NPOS * 9];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    uint16_t* sx = reinterpret_cast<uint16_t*>(sm + WS_X);      // [64][25] bf16 patches
    const uint32_t w2_addr = smem_u32(sm + WS_W2), h1_addr = smem_u32(sm + WS_H1);

    if (warp == 0) tmem_alloc(&s_tmem, kConvTmemCols);
    if (tid == 0) {
        for (int b = 0; b < 2; b++) {
            bar_init_n(&s_h1_full[b], WS_PROD);
            bar_init_n(&s_h1_empty[b], kTBufs);  // one commit per issuing thread
        }
        for (int b = 0; b < kTBufs; b++) {
            bar_init_n(&s_t_full[b], 1);
            bar_init_n(&s_t_empty[b], 4);
        }
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int i = tid; i < NPOS * 9; i += blockDim.x) s_nb[i] = nb(i / 9, i % 9);
    // the weight images (which prep_weights may still write when this kernel
    // starts: not by the read-only path), and fc_kernel's reads of h2 from the
    // chunk before
    wait_previous();
    start_next();
    for (uint32_t i = tid; i < W2_BYTES / 16; i += blockDim.x)
        reinterpret_cast<uint4*>(sm + WS_W2)[i] =
            __ldcg(reinterpret_cast<const uint4*>(img + OFF_W2) + i);
    fence_async_smem();
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = s_tmem;
    const int n_tiles = (n + TB - 1) / TB;
    // bounded wait that also gives up once another role has aborted
    auto wait_or_abort = [&](uint64_t* bar, uint32_t parity) -> bool {
        const uint32_t a = smem_u32(bar);
        for (uint32_t it = 0; it < kWaitLimit; it++) {
            uint32_t ok;
            asm volatile(
                "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                "selp.u32 %0, 1, 0, p;\n}"
                : "=r"(ok)
                : "r"(a), "r"(parity)
                : "memory");
            if (ok) return true;
            if ((it & 255) == 255 && s_abort) return false;
        }
        s_abort = 1;
        return false;
    };

    if (warp < WS_PROD_WARPS) {
        // ---- conv1 producers ------------------------------------------------
        const int ptid = tid;
        // B fragments of W1 (bf16, K = taps) and the biases of this lane's
        // channel pairs, for n-blocks of 8 channels
        uint32_t bw[4][2];
        float bias[4][2];
        {
            const int g = lane >> 2, tq = lane & 3;
            auto w1b = [&](int ch, int k) -> uint32_t {
                return k < 9 ? (uint32_t)bf16_bits(w[OW1 + ch * 9 + k]) : 0u;
            };
#pragma unroll
            for (int nb = 0; nb < 4; nb++) {
                const int ch = nb * 8 + g;
                bw[nb][0] = w1b(ch, 2 * tq) | (w1b(ch, 2 * tq + 1) << 16);
                bw[nb][1] = w1b(ch, 2 * tq + 8) | (w1b(ch, 2 * tq + 9) << 16);
                bias[nb][0] = w[OB1 + nb * 8 + 2 * tq];
                bias[nb][1] = w[OB1 + nb * 8 + 2 * tq + 1];
            }
        }
        // a tile's patches are loaded into registers one tile ahead, so the
        // global loads run during the previous tile's conv1
        constexpr int XPER = (TB * NPOS + WS_PROD - 1) / WS_PROD;
        float xn[XPER];
        auto load_x = [&](int t) {
            const int hit0 = t * TB, nh = t < n_tiles ? min(TB, n - hit0) : 0;
#pragma unroll
            for (int u = 0; u < XPER; u++) {
                const int e = ptid + u * WS_PROD;
                xn[u] = (e < TB * NPOS && e / NPOS < nh) ? x[(size_t)hit0 * NPOS + e] : 0.0f;
            }
        };
        load_x(blockIdx.x);
        int i = 0;
        for (int t = blockIdx.x; t < n_tiles; t += gridDim.x, i++) {
            const int stage = i & 1;
            // one thread waits for the stage; every producer follows its
            // decision, so the named barriers below stay uniform
            if (ptid == 0)
                s_prod_go = wait_or_abort(&s_h1_empty[stage], ((i >> 1) & 1) ^ 1) && !s_abort;
            producers_sync();  // also: the previous tile's patches are no longer read
            if (!s_prod_go) break;
#pragma unroll
            for (int u = 0; u < XPER; u++) {
                const int e = ptid + u * WS_PROD;
                if (e < TB * NPOS) sx[e] = bf16_bits(xn[u]);
            }
            load_x(t + gridDim.x);
            producers_sync();
            uint8_t* h1 = sm + WS_H1 + stage * H1_STAGE;
            // conv1 as warp-level m16n8k16 MMAs: a 16-row block is 16 hits of
            // one position, K the 9 taps (7 zero columns), N 4 x 8 channels;
            // lane (g, t) gathers its A fragment from the patches: rows g and
            // g + 8, taps 2t, 2t + 1 and 2t + 8 (only t = 0 has tap 8)
            const int pwarp = warp, g = lane >> 2, tq = lane & 3;
            for (int rb = pwarp; rb < NPOS * (TB / 16); rb += WS_PROD_WARPS) {
                const int p = rb >> 2, h0 = (rb & 3) * 16;
                const int q0 = s_nb[p * 9 + 2 * tq], q1 = s_nb[p * 9 + 2 * tq + 1];
                const int q2 = tq == 0 ? s_nb[p * 9 + 8] : -1;
                const uint16_t* x0 = sx + (h0 + g) * NPOS;
                const uint16_t* x1 = x0 + 8 * NPOS;
                uint32_t a[4];
                a[0] = (q0 >= 0 ? (uint32_t)x0[q0] : 0u) | (q1 >= 0 ? (uint32_t)x0[q1] << 16 : 0u);
                a[1] = (q0 >= 0 ? (uint32_t)x1[q0] : 0u) | (q1 >= 0 ? (uint32_t)x1[q1] << 16 : 0u);
                a[2] = q2 >= 0 ? (uint32_t)x0[q2] : 0u;
                a[3] = q2 >= 0 ? (uint32_t)x1[q2] : 0u;
                uint8_t* blk = h1 + p * 4096;
#pragma unroll
                for (int nb = 0; nb < 4; nb++) {
                    float c[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                    asm volatile(
                        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, "
                        "{%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
                        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(bw[nb][0]),
                          "r"(bw[nb][1]));
                    const int ch = nb * 8 + 2 * tq;
                    const __nv_bfloat162 v0 = __float22bfloat162_rn(
                        make_float2(fmaxf(c[0] + bias[nb][0], 0.0f), fmaxf(c[1] + bias[nb][1], 0.0f)));
                    const __nv_bfloat162 v1 = __float22bfloat162_rn(
                        make_float2(fmaxf(c[2] + bias[nb][0], 0.0f), fmaxf(c[3] + bias[nb][1], 0.0f)));
                    *reinterpret_cast<__nv_bfloat162*>(blk + cm_off(h0 + g, ch, TB)) = v0;
                    *reinterpret_cast<__nv_bfloat162*>(blk + cm_off(h0 + g + 8, ch, TB)) = v1;
                }
            }
            fence_async_smem();  // h1 is read by the tensor cores
            bar_arrive(&s_h1_full[stage]);
        }
    } else if (warp < WS_EPI_WARP0) {
        // ---- conv2 MMA issue: lane 0 of warp 8 + b, TMEM buffer b -----------
        const int ib = warp - WS_MMA_WARP0;
        if (lane == 0 && ib < kTBufs) {
            const uint32_t id32 = idesc_bf16(64, 32), id64 = idesc_bf16(64, 64),
                           id96 = idesc_bf16(64, 96);
            const uint64_t b_desc0 = sdesc(w2_addr, 1536, 128);
            const uint32_t d0 = tmem + (uint32_t)(ib * kRowCols);
            int i = 0, gq = 0;  // local tile, global row sequence
            bool issued = false;
            uint32_t last_par = 0;
            for (int t = blockIdx.x; t < n_tiles; t += gridDim.x, i++) {
                const int stage = i & 1;
                if (!wait_or_abort(&s_h1_full[stage], (i >> 1) & 1)) break;
                fence_after();
                const uint64_t a_desc0 = sdesc(h1_addr + stage * H1_STAGE, 1024, 128);
                bool ok = true;
                for (int yo = 0; yo < 5; yo++, gq++) {
                    if (gq % kTBufs != ib) continue;  // another thread's buffer
                    if (!wait_or_abort(&s_t_empty[ib], ((gq / kTBufs) & 1) ^ 1)) {
                        ok = false;
                        break;
                    }
                    fence_after();
                    const int y0 = max(yo - 1, 0), y1 = min(yo + 1, 4);
                    for (int yi = y0; yi <= y1; yi++) {
                        // (descriptor addresses count 16 bytes; input column x
                        // in order, so that every output adds its taps in order)
                        const uint64_t ay = a_desc0 + (uint32_t)(yi * 5 * 256);
                        const uint64_t by = b_desc0 + (uint32_t)((yi - yo + 1) * 2 * (W2_SLICE >> 4));
#pragma unroll
                        for (int x = 0; x < 5; x++)
#pragma unroll
                            for (int kk = 0; kk < 2; kk++) {
                                const uint64_t a = ay + (uint32_t)(x * 256 + kk * 128);
                                const uint64_t b = by + (uint32_t)(kk * (W2_SLICE >> 4));
                                const bool fresh = yi == y0 && kk == 0;  // new columns
                                const uint32_t d = d0 + (x > 0 ? x - 1 : 0) * 32;
                                if (x == 0)
                                    mma(d, a, b + 32, id64, !fresh);
                                else if (x == 4)
                                    mma(d, a, b, id64, 1);
                                else if (fresh) {
                                    mma(d, a, b, id64, 1);
                                    mma(d + 64, a, b + 64, id32, 0);
                                } else
                                    mma(d, a, b, id96, 1);
                            }
                    }
                    commit(&s_t_full[ib]);
                    issued = true;
                    last_par = (gq / kTBufs) & 1;
                }
                if (!ok) break;
                commit(&s_h1_empty[stage]);  // stage free once these MMAs complete
            }
            if (s_abort) {
                atomicExch(err, 1);
                if (issued) wait_bar(&s_t_full[ib], last_par);  // bounded
            }
        }
        __syncwarp();
    } else if (warp >= WS_EPI_WARP0) {
        // ---- conv2 epilogue (warps 12-15, TMEM lane quadrant q) --------------
        const int q = warp - WS_EPI_WARP0, g = lane >> 2, tq = lane & 3;
        const uint32_t lane_base = (uint32_t)(q * 32) << 16;
        float2 b2[4];
#pragma unroll
        for (int k = 0; k < 4; k++)
            b2[k] = make_float2(w[OB2 + 8 * k + 2 * tq], w[OB2 + 8 * k + 2 * tq + 1]);
        int gq = 0;
        for (int t = blockIdx.x; t < n_tiles; t += gridDim.x) {
            // this lane's first value of the tile's first hit row
            uint8_t* dst0 = reinterpret_cast<uint8_t*>(h2) + (size_t)(t >> 1) * (TF * K3 * 2) +
                            ((t & 1) * TB + q * 16 + g) * 16 + tq * 4;
            bool ok = true;
            for (int yo = 0; yo < 5; yo++, gq++) {
                const int b = gq % kTBufs;
                // lane 0 waits and the warp follows it (tcgen05.ld is warp-wide)
                const int got = __shfl_sync(
                    0xffffffffu, lane == 0 ? (int)wait_or_abort(&s_t_full[b], (gq / kTBufs) & 1) : 0,
                    0);
                if (!got) {
                    ok = false;
                    break;
                }
                fence_after();
                const uint32_t src = tmem + lane_base + (uint32_t)(b * kRowCols);
                auto put = [&](const uint32_t (&r)[16], int x) {
                    uint8_t* dst = dst0 + (size_t)(yo * 5 + x) * (4 * TF * 16);
#pragma unroll
                    for (int k = 0; k < 4; k++)
#pragma unroll
                        for (int h = 0; h < 2; h++) {
                            const float2 z = __fadd2_rn(
                                make_float2(__uint_as_float(r[4 * k + 2 * h]),
                                            __uint_as_float(r[4 * k + 2 * h + 1])),
                                b2[k]);
                            const __nv_bfloat162 v =
                                __float22bfloat162_rn(make_float2(fmaxf(z.x, 0.0f), fmaxf(z.y, 0.0f)));
                            *reinterpret_cast<__nv_bfloat162*>(dst + k * (TF * 16) + h * 128) = v;
                        }
                };
                uint32_t r0[16], r1[16], r2[16];
                tmem_ld16x32(src, r0);
                tmem_ld16x32(src + 32, r1);
                tmem_ld16x32(src + 64, r2);
                tmem_ld_wait();
                put(r0, 0);
                put(r1, 1);
                put(r2, 2);
                tmem_ld16x32(src + 96, r0);
                tmem_ld16x32(src + 128, r1);
                tmem_ld_wait();
                fence_before();
                __syncwarp();
                if (lane == 0) bar_arrive(&s_t_empty[b]);
                put(r0, 3);
                put(r1, 4);
            }
            if (!ok) break;
        }
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (s_abort && tid == 0) atomicExch(err, 1);
    if (warp == 0) tmem_free(tmem, kConvTmemCols);
}

// ---------------------------------------------------------------------------
// FC3 + heads on tiles of 128 hits; one CTA of 384 threads per SM:
//   warp 0      lane 0 copies h2 in chunks of 80 inputs (20 KB, contiguous)
//               into a ring of six stages, as long as a stage is free: with
//               the MMAs' 4 us of work and 105 MB of h2 per 65,536 hits, the
//               copies are the bound and stay in flight across tiles
//   warp 1      lane 0 issues each chunk's five 128 x 64 x 16 MMAs into one of
//               two TMEM accumulators
//   warps 4-11  the epilogue, warps 4-7 of even and 8-11 of odd tiles: bias,
//               ReLU, bf16, the 7 heads of one hit a lane
// (One role for all threads, copying a chunk ahead with barriers between:
// 58 us per 65,536 hits; now 23 us.)
constexpr int FC_KCH = 80, FC_NCH = K3 / FC_KCH, FC_STAGES = 6, FC_THREADS = 384;
constexpr uint32_t FC_CHUNK = TF * FC_KCH * 2;
constexpr uint32_t FC_W3 = 0, FC_A = FC_W3 + W3_BYTES, FC_W4 = FC_A + FC_STAGES * FC_CHUNK,
                   FC_SMEM = FC_W4 + NH * 8 * 4;
static_assert(FC_A % 128 == 0 && FC_CHUNK % 128 == 0 && W3_BYTES % FC_CHUNK == 0, "alignment");

__device__ __forceinline__ void bulk_copy(uint32_t dst, const void* src, uint32_t bytes,
                                          uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
            "r"(dst),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ void expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}

__global__ void __launch_bounds__(FC_THREADS, 1)
    fc_kernel(const uint16_t* __restrict__ h2, int n, const float* __restrict__ w,
              const uint8_t* __restrict__ img, float* __restrict__ out, int* err) {
    extern __shared__ __align__(1024) uint8_t sm[];
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_abort;
    __shared__ __align__(8) uint64_t s_full[FC_STAGES], s_empty[FC_STAGES], s_w3, s_t_full[2],
        s_t_empty[2];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    float* s_w4 = reinterpret_cast<float*>(sm + FC_W4);  // [unit][8], bf16-valued
    const uint32_t w3_addr = smem_u32(sm + FC_W3), a_addr = smem_u32(sm + FC_A);

    start_next();
    if (warp == 0) tmem_alloc(&s_tmem, 128);
    if (tid == 0) {
        for (int b = 0; b < FC_STAGES; b++) {
            bar_init(&s_full[b]);
            bar_init(&s_empty[b]);
        }
        bar_init(&s_w3);
        for (int b = 0; b < 2; b++) {
            bar_init(&s_t_full[b]);
            bar_init_n(&s_t_empty[b], 4);
        }
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int i = tid; i < NH * 8; i += FC_THREADS)
        s_w4[i] = (i & 7) < NOUT ? bf16_round(w[OW4 + (i & 7) * NH + (i >> 3)]) : 0.0f;
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = s_tmem;
    const int n_tiles = (n + TF - 1) / TF;
    // bounded wait that also gives up once another role has aborted
    auto wait_or_abort = [&](uint64_t* bar, uint32_t parity) -> bool {
        const uint32_t a = smem_u32(bar);
        for (uint32_t it = 0; it < kWaitLimit; it++) {
            uint32_t ok;
            asm volatile(
                "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                "selp.u32 %0, 1, 0, p;\n}"
                : "=r"(ok)
                : "r"(a), "r"(parity)
                : "memory");
            if (ok) return true;
            if ((it & 255) == 255 && s_abort) return false;
        }
        s_abort = 1;
        return false;
    };

    if (warp == 0) {
        if (lane == 0) {
            // ---- copies: W3 once, then every tile's chunks ----------------------
            expect_tx(&s_w3, W3_BYTES);
            for (uint32_t o = 0; o < W3_BYTES; o += FC_CHUNK)
                bulk_copy(w3_addr + o, img + OFF_W3 + o, FC_CHUNK, &s_w3);
            wait_previous();  // h2 (W3's image was complete before conv_kernel went on)
            uint32_t c = 0;  // chunks issued
            for (int t = blockIdx.x; t < n_tiles && !s_abort; t += gridDim.x) {
                const uint8_t* src = reinterpret_cast<const uint8_t*>(h2) + (size_t)t * (TF * K3 * 2);
                for (int k = 0; k < FC_NCH; k++, c++) {
                    const uint32_t s = c % FC_STAGES;
                    if (!wait_or_abort(&s_empty[s], ((c / FC_STAGES) & 1) ^ 1)) break;
                    expect_tx(&s_full[s], FC_CHUNK);
                    bulk_copy(a_addr + s * FC_CHUNK, src + (size_t)k * FC_CHUNK, FC_CHUNK, &s_full[s]);
                }
            }
            if (s_abort) {  // the copies in flight write this CTA's memory (bounded)
                wait_bar(&s_w3, 0);
                for (uint32_t k = c > FC_STAGES ? c - FC_STAGES : 0; k < c; k++)
                    wait_bar(&s_full[k % FC_STAGES], (k / FC_STAGES) & 1);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {
            // ---- MMA issue -------------------------------------------------------
            const uint32_t id3 = idesc_bf16(128, NH);
            uint32_t c = 0;
            int i = 0;
            uint64_t* last = nullptr;
            uint32_t last_par = 0;
            bool ok = wait_or_abort(&s_w3, 0);
            for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x, i++) {
                const int b = i & 1;
                if (!(ok = wait_or_abort(&s_t_empty[b], ((i >> 1) & 1) ^ 1))) break;
                fence_after();
                for (int k = 0; k < FC_NCH; k++, c++) {
                    const uint32_t s = c % FC_STAGES;
                    if (!(ok = wait_or_abort(&s_full[s], (c / FC_STAGES) & 1))) break;
                    const uint64_t ad = sdesc(a_addr + s * FC_CHUNK, TF * 16, 128);
                    const uint64_t bd = sdesc(w3_addr + (uint32_t)k * FC_KCH * NH * 2, NH * 16, 128);
#pragma unroll
                    for (int j = 0; j < FC_KCH / 16; j++)
                        mma(tmem + b * NH, ad + (uint32_t)(j * 2 * TF), bd + (uint32_t)(j * 2 * NH),
                            id3, k > 0 || j > 0);
                    commit(&s_empty[s]);
                    last = &s_empty[s];
                    last_par = (c / FC_STAGES) & 1;
                }
                if (!ok) break;
                commit(&s_t_full[b]);
            }
            if (s_abort && last) wait_bar(last, last_par);  // bounded
        }
        __syncwarp();
    } else if (warp >= 4) {
        // ---- epilogue --------------------------------------------------------------
        const int q = warp & 3, odd = (warp - 4) >> 2;
        int i = odd;
        for (int t = blockIdx.x + odd * gridDim.x; t < n_tiles; t += 2 * gridDim.x, i += 2) {
            const int got = __shfl_sync(
                0xffffffffu,
                lane == 0 ? (int)wait_or_abort(&s_t_full[odd], (i >> 1) & 1) : 0, 0);
            if (!got) break;
            fence_after();
            uint32_t r[2][32];
            const uint32_t src = tmem + ((uint32_t)(q * 32) << 16) + odd * NH;
            tmem_ld32(src, r[0]);
            tmem_ld32(src + 32, r[1]);
            fence_before();
            __syncwarp();
            if (lane == 0) bar_arrive(&s_t_empty[odd]);
            // h3 = relu(acc + b3) rounded to bf16, then the heads, the sums of
            // the two halves of the units added at the end
            float sum[2][NOUT];
#pragma unroll
            for (int half = 0; half < 2; half++) {
#pragma unroll
                for (int o = 0; o < NOUT; o++) sum[half][o] = 0.0f;
#pragma unroll
                for (int c = 0; c < 32; c++) {
                    const int ch = half * 32 + c;
                    const float z = __uint_as_float(r[half][c]) + __ldg(w + OB3 + ch);
                    const float h = bf16_round(fmaxf(z, 0.0f));
                    const float4 wa = *reinterpret_cast<const float4*>(s_w4 + ch * 8);
                    const float4 wb = *reinterpret_cast<const float4*>(s_w4 + ch * 8 + 4);
                    sum[half][0] = __fmaf_rn(h, wa.x, sum[half][0]);
                    sum[half][1] = __fmaf_rn(h, wa.y, sum[half][1]);
                    sum[half][2] = __fmaf_rn(h, wa.z, sum[half][2]);
                    sum[half][3] = __fmaf_rn(h, wa.w, sum[half][3]);
                    sum[half][4] = __fmaf_rn(h, wb.x, sum[half][4]);
                    sum[half][5] = __fmaf_rn(h, wb.y, sum[half][5]);
                    sum[half][6] = __fmaf_rn(h, wb.z, sum[half][6]);
                }
            }
            const int hit = t * TF + q * 32 + lane;
            if (hit < n)
#pragma unroll
                for (int o = 0; o < NOUT; o++)
                    out[(size_t)hit * NOUT + o] = sum[0][o] + sum[1][o] + w[OB4 + o];
        }
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (s_abort && tid == 0) atomicExch(err, 1);
    if (warp == 0) tmem_free(tmem, 128);
}

}  // namespace

size_t weight_image_bytes() { return OFF_W3 + W3_BYTES; }
// (whole fc tiles; rows past the last hit are computed and dropped)
size_t h2_bytes(uint32_t max_batch) {
    return ((size_t)max_batch + TF - 1) / TF * TF * K3 * 2;
}

cudaError_t forward(const float* w, const float* x, uint32_t n, uint8_t* img, uint16_t* h2,
                    float* out, int* err, int sms, bool new_weights, cudaStream_t s) {
    if (!n) return cudaSuccess;
    static int attr_dev = -1;
    int dev = 0;
    cudaGetDevice(&dev);
    if (attr_dev != dev) {
        cudaError_t e = cudaFuncSetAttribute(conv_kernel,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, WS_SMEM);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(fc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     FC_SMEM);
        if (e != cudaSuccess) return e;
        attr_dev = dev;
    }
    cudaError_t e = cudaSuccess;
    if (new_weights) {
        prep_weights<<<(NH * K3 + 255) / 256, 256, 0, s>>>(w, img);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    // Each kernel may start while the one before ends: an SM whose conv tiles
    // are done loads W3 meanwhile (444 -> 408 us for 304 thousand
    // hits in five chunks).  The first one of a call follows prep_weights.
    const int conv_tiles = (int)((n + TB - 1) / TB), fc_tiles = (int)((n + TF - 1) / TF);
    cudaLaunchAttribute early{};
    early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    early.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.stream = s;
    cfg.attrs = &early;
    cfg.numAttrs = 1;
    cfg.gridDim = dim3((unsigned)std::min(conv_tiles, sms));
    cfg.blockDim = dim3(WS_THREADS);
    cfg.dynamicSmemBytes = WS_SMEM;
    e = cudaLaunchKernelEx(&cfg, conv_kernel, x, (int)n, w, (const uint8_t*)img, h2, err);
    if (e != cudaSuccess) return e;
    cfg.gridDim = dim3((unsigned)std::min(fc_tiles, sms));
    cfg.blockDim = dim3(FC_THREADS);
    cfg.dynamicSmemBytes = FC_SMEM;
    return cudaLaunchKernelEx(&cfg, fc_kernel, (const uint16_t*)h2, (int)n, w, (const uint8_t*)img,
                              out, err);
}

}  // namespace nettc
}  // namespace pd
