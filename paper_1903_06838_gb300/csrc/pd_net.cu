// pd_net.cu — the learned photon count / subpixel network: its state and
// entry points, patch gather, batch gather, Adam and refinement.
//
// The paper found off-the-shelf deep models lost photon information and
// offered its fixed filters as the seed of future learned models (abstract,
// sections "Methods" and "Conclusions").  This network refines the classical
// count and centre of mass of each hit from the 5x5 neighbourhood of its
// seed: conv3x3x32 -> conv3x3x32 -> FC64 -> {5 count logits, (dx, dy)}.
//
// Loss and gradients are in pd_net_train.cu (mma.sync m16n8k16, bfloat16
// operands rounded to nearest even, float32 accumulation); inference
// (pd_net_forward) runs on tcgen05 with TMEM accumulators (pd_net_tc.cu), with
// the same operand rounding.  Biases, ReLU, the loss and the optimiser are
// float32.  Layouts follow the oracle (oracle/net.py): activations
// [hit][position 0..24][channel].
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <random>
#include <string>
#include <vector>

#include "pd.h"
#include "pd_internal.cuh"
#include "pd_net_tc.cuh"
#include "pd_net_train.cuh"

namespace {

constexpr int NPOS = 25, C1 = 32, C2 = 32, NH = 64, NOUT = 7;
constexpr int NW1 = C1 * 9, NB1 = C1, NW2 = C2 * 9 * C1, NB2 = C2, NW3 = NH * NPOS * C2,
              NB3 = NH, NW4 = NOUT * NH, NB4 = NOUT;
constexpr int OW1 = 0, OB1 = OW1 + NW1, OW2 = OB1 + NB1, OB2 = OW2 + NW2, OW3 = OB2 + NB2,
              OB3 = OW3 + NW3, OW4 = OB3 + NB3, OB4 = OW4 + NW4, NPARAM = OB4 + NB4;

// rows idx[i] of a training set into batch row i (one thread per float of a
// patch row, the labels by the row's first thread)
__global__ void take_kernel(const float* __restrict__ patches, const uint8_t* __restrict__ counts,
                            const float* __restrict__ targets, const uint8_t* __restrict__ mask,
                            const uint32_t* __restrict__ idx, uint32_t n,
                            float* __restrict__ p_out, uint8_t* __restrict__ c_out,
                            float* __restrict__ t_out, uint8_t* __restrict__ m_out) {
    const uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (uint64_t)n * NPOS) return;
    const uint32_t i = (uint32_t)(t / NPOS), k = (uint32_t)(t % NPOS);
    const uint32_t j = idx[i];
    p_out[t] = patches[(size_t)j * NPOS + k];
    if (k == 0) {
        c_out[i] = counts[j];
        m_out[i] = mask[j];
        t_out[2 * (size_t)i] = targets[2 * (size_t)j];
        t_out[2 * (size_t)i + 1] = targets[2 * (size_t)j + 1];
    }
}

__global__ void adam_kernel(float* __restrict__ w, const float* __restrict__ gr,
                            float* __restrict__ m, float* __restrict__ v, int n, float lr,
                            float b1, float b2, float c1, float c2, float eps) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gv = gr[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gv;
    const float vi = b2 * v[i] + (1.0f - b2) * gv * gv;
    m[i] = mi;
    v[i] = vi;
    w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// 5x5 patch of e / photon_kev around each hit's seed (zero outside the
// module): e recomputed exactly as the chain does, with the call's common
// mode of frame - frame_base (unit term, and for the stacked mean the module
// row and column terms).
//
// A warp takes kGatherHits hits, a lane per patch pixel.  With one hit a warp
// the five integer divisions of its place were most of the instructions and
// the kernel waited for one hit's loads at a time; now lane j splits hit j's
// pixel and the others read it from there, units are found by multiplication,
// and the loads of four hits are in flight.  300 thousand hits of 704 x 768
// frames: 63 -> 32 us.
constexpr int kGatherHits = 8;

struct GatherDiv {  // ceil(2^32 / d) of the unit sizes, 0 for 1
    uint32_t unit_rows, unit_cols;
};
// v / d for v < 2^16, d <= 2^16: with q = ceil(2^32 / d), v (q d - 2^32) < 2^32
__device__ __forceinline__ uint32_t div16(uint32_t v, uint32_t q) {
    return q ? __umulhi(v, q) : v;
}

template <bool MG>
__global__ void __launch_bounds__(256)
    gather_kernel(pd::ChainParams p, const uint16_t* __restrict__ raw, uint32_t frame_base,
                  const float* __restrict__ cm, const pd_hit* __restrict__ hits, uint32_t n,
                  float* __restrict__ patches, pd::MultiGain mg, GatherDiv dv) {
    const uint32_t h0 = (blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32) * kGatherHits;
    const int lane = threadIdx.x & 31;
    if (h0 >= n) return;
    const pd_hit* own = hits + min(h0 + (uint32_t)lane % kGatherHits, n - 1);
    const uint32_t own_px = own->pixel, own_f = own->frame - frame_base;
    const uint32_t own_m = own_px / p.module_px, within = own_px - own_m * p.module_px;
    const uint32_t own_r = within / p.cols;
    const uint32_t own_rc = own_r << 16 | (within - own_r * p.cols);
    const int dy = lane / 5 - 2, dx = lane % 5 - 2;
    const int delta = dy * (int)p.cols + dx;
    const bool stacked = cm_kind(p) == PD_CM_MEAN_STACKED;
    const uint32_t per_frame = cm_per_frame(p);
#pragma unroll 4
    for (int j = 0; j < kGatherHits; j++) {
        const uint32_t f = __shfl_sync(0xffffffffu, own_f, j);
        const uint32_t px = __shfl_sync(0xffffffffu, own_px, j);
        const uint32_t m = __shfl_sync(0xffffffffu, own_m, j);
        const uint32_t rc = __shfl_sync(0xffffffffu, own_rc, j);
        if (h0 + j >= n || lane >= NPOS) continue;
        const int r = (int)(rc >> 16) + dy, c = (int)(rc & 0xFFFFu) + dx;
        float v = 0.0f;
        if (r >= 0 && r < (int)p.rows && c >= 0 && c < (int)p.cols) {
            const uint32_t g = px + (uint32_t)delta;
            const uint32_t unit = m * p.units_per_module +
                                  div16((uint32_t)r, dv.unit_rows) * p.units_per_row +
                                  div16((uint32_t)c, dv.unit_cols);
            const float* cmf = cm + (size_t)f * per_frame;
            const uint16_t w = __ldg(raw + (size_t)f * p.frame_px + g);
            float e;
            if (MG) {
                e = pd::mg_energy(mg, p.frame_px, w, g, cmf[unit]);
            } else {
                const float d = __fsub_rn(__uint2float_rn(w), __ldg(p.ped + g));
                const float ig = __ldg(p.inv_gain + g);
                if (stacked)
                    e = pd::energy<true>(cm_after_gain(p), d, ig, cmf[unit],
                                         cmf[p.units_per_frame + (size_t)m * p.rows + r],
                                         cmf[p.units_per_frame + (size_t)p.n_modules * p.rows +
                                             (size_t)m * p.cols + c]);
                else
                    e = pd::energy<false>(cm_after_gain(p), d, ig, cmf[unit], 0.0f, 0.0f);
            }
            v = __fdiv_rn(e, p.photon_kev);
        }
        patches[(size_t)(h0 + j) * NPOS + lane] = v;
    }
}

// Replace count and (dx, dy) of hits the network is confident about; keep
// the classical values elsewhere.
__global__ void refine_kernel(const float* __restrict__ out, const pd_hit* __restrict__ in,
                              uint32_t n, float conf, float count_conf,
                              pd_hit* __restrict__ res) {
    const uint32_t b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= n) return;
    pd_hit h = in[b];
    const float* o = out + (size_t)b * NOUT;
    float mx = o[0];
    int arg = 0;
    for (int k = 1; k < 5; k++)
        if (o[k] > mx) {
            mx = o[k];
            arg = k;
        }
    float s = 0.0f;
    for (int k = 0; k < 5; k++) s += expf(o[k] - mx);
    const float pmax = 1.0f / s;
    if (pmax >= conf && arg >= 1) {
        if (pmax >= count_conf) h.count = (uint8_t)arg;
        h.dx = o[5];
        h.dy = o[6];
        h.flags |= PD_HIT_LEARNED;
    }
    res[b] = h;
}

int net_fail(int code, const std::string& why) { return pd::internal_fail(code, why.c_str()); }
int net_cuda(cudaError_t e, const char* what) {
    return net_fail(PD_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

}  // namespace

struct pd_net {
    uint32_t max_batch = 0;
    float *w = nullptr, *gw = nullptr, *m = nullptr, *v = nullptr;
    uint64_t step = 0;
    // tensor-core inference: bf16 weight image, bf16 h2, timeout flag
    uint8_t* tc_img = nullptr;
    uint16_t* tc_h2 = nullptr;
    int* tc_err = nullptr;
    // training: bf16 weight fragments, bf16 h2 and dz3 rows, gradient sums
    uint4* tr_img = nullptr;
    float* tr_slices = nullptr;
    uint16_t *tr_h2 = nullptr, *tr_dz3 = nullptr;
};

namespace {

void free_net(pd_net* n) {
    if (!n) return;
    for (float* p : {n->w, n->gw, n->m, n->v}) cudaFree(p);
    cudaFree(n->tc_img);
    cudaFree(n->tc_h2);
    cudaFree(n->tc_err);
    cudaFree(n->tr_img);
    cudaFree(n->tr_h2);
    cudaFree(n->tr_dz3);
    cudaFree(n->tr_slices);
    delete n;
}

}  // namespace

extern "C" {

uint32_t pd_net_num_params(void) { return NPARAM; }

int pd_net_create(uint32_t max_batch, uint64_t seed, pd_net** out) {
    if (!out || !max_batch) return net_fail(PD_EINVAL, "pd_net_create: need out and max_batch");
    *out = nullptr;
    pd_net* n = new (std::nothrow) pd_net();
    if (!n) return net_fail(PD_ENOMEM, "host allocation failed");
    n->max_batch = max_batch;
    for (float** p : {&n->w, &n->gw, &n->m, &n->v})
        if (cudaMalloc(p, NPARAM * sizeof(float)) != cudaSuccess) {
            free_net(n);
            return net_fail(PD_ENOMEM, "pd_net_create: device allocation failed");
        }
    if (cudaMalloc(&n->tc_img, pd::nettc::weight_image_bytes()) != cudaSuccess ||
        cudaMalloc(&n->tc_h2, pd::nettc::h2_bytes(max_batch)) != cudaSuccess ||
        cudaMalloc(&n->tc_err, sizeof(int)) != cudaSuccess ||
        cudaMalloc(&n->tr_img, pd::nettrain::image_bytes()) != cudaSuccess ||
        cudaMalloc(&n->tr_h2, pd::nettrain::h2_bytes(max_batch)) != cudaSuccess ||
        cudaMalloc(&n->tr_dz3, pd::nettrain::dz3_bytes(max_batch)) != cudaSuccess ||
        cudaMalloc(&n->tr_slices, pd::nettrain::slice_bytes(max_batch, pd::device_sm_count())) !=
            cudaSuccess ||
        cudaMemset(n->tc_err, 0, sizeof(int)) != cudaSuccess) {
        free_net(n);
        return net_fail(PD_ENOMEM, "pd_net_create: device allocation failed");
    }
    // weights and biases uniform in +-1/sqrt(fan_in), from a seeded generator
    std::vector<float> host(NPARAM, 0.0f);
    std::mt19937_64 rng(seed);
    auto fill = [&](int off, int count, int fan_in) {
        const double b = 1.0 / std::sqrt((double)fan_in);
        std::uniform_real_distribution<double> ud(-b, b);
        for (int i = 0; i < count; i++) host[off + i] = (float)ud(rng);
    };
    fill(OW1, NW1, 9);
    fill(OB1, NB1, 9);
    fill(OW2, NW2, 9 * C1);
    fill(OB2, NB2, 9 * C1);
    fill(OW3, NW3, NPOS * C2);
    fill(OB3, NB3, NPOS * C2);
    fill(OW4, NW4, NH);
    fill(OB4, NB4, NH);
    if (cudaMemcpy(n->w, host.data(), NPARAM * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(n->m, 0, NPARAM * 4) != cudaSuccess ||
        cudaMemset(n->v, 0, NPARAM * 4) != cudaSuccess) {
        free_net(n);
        return net_fail(PD_ECUDA, "pd_net_create: upload failed");
    }
    *out = n;
    return PD_OK;
}

int pd_net_set_params(pd_net* n, const float* host, uint32_t count) {
    if (!n || !host || count != NPARAM) return net_fail(PD_EINVAL, "pd_net_set_params: size");
    cudaError_t e = cudaMemcpy(n->w, host, NPARAM * 4, cudaMemcpyHostToDevice);
    return e == cudaSuccess ? PD_OK : net_cuda(e, "pd_net_set_params");
}

int pd_net_get_params(pd_net* n, float* host, uint32_t count) {
    if (!n || !host || count != NPARAM) return net_fail(PD_EINVAL, "pd_net_get_params: size");
    cudaError_t e = cudaMemcpy(host, n->w, NPARAM * 4, cudaMemcpyDeviceToHost);
    return e == cudaSuccess ? PD_OK : net_cuda(e, "pd_net_get_params");
}

int pd_net_forward(pd_net* n, const float* patches, uint32_t count, float* out_dev, void* stream) {
    if (!n || (count && (!patches || !out_dev))) return net_fail(PD_EINVAL, "pd_net_forward: args");
    cudaStream_t s = (cudaStream_t)stream;
    const int sms = pd::device_sm_count();
    for (uint32_t done = 0; done < count;) {
        const uint32_t b = std::min(n->max_batch, count - done);
        cudaError_t e = pd::nettc::forward(n->w, patches + (size_t)done * NPOS, b, n->tc_img,
                                           n->tc_h2, out_dev + (size_t)done * NOUT, n->tc_err,
                                           sms, done == 0, s);
        if (e) return net_cuda(e, "pd_net_forward");
        done += b;
    }
    if (!count) return PD_OK;
    // a timed-out wait inside the kernels is reported here (this synchronises
    // the stream)
    int flag = 0;
    cudaError_t e = cudaMemcpyAsync(&flag, n->tc_err, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (!e) e = cudaStreamSynchronize(s);
    if (e) return net_cuda(e, "pd_net_forward");
    if (flag) {
        cudaMemsetAsync(n->tc_err, 0, sizeof(int), s);
        return net_fail(PD_ETIMEDOUT, "pd_net_forward: tensor-core pipeline wait timed out");
    }
    return PD_OK;
}

int pd_net_gradients(pd_net* n, const float* patches, const uint8_t* counts, const float* targets,
                     const uint8_t* mask, uint32_t count, float n_reg, float lambda,
                     float* grads_dev, float* loss_dev, void* stream) {
    if (!n || !count || count > n->max_batch || !patches || !counts || !targets || !mask)
        return net_fail(PD_EINVAL, "pd_net_gradients: args (count <= max_batch)");
    cudaStream_t s = (cudaStream_t)stream;
    // straight into the caller's array where its alignment takes the kernels'
    // two-float additions
    float* g = grads_dev && (uintptr_t)grads_dev % 8 == 0 ? grads_dev : n->gw;
    cudaError_t e = pd::nettrain::gradients(n->w, patches, counts, targets, mask, count,
                                            std::max(1.0f, n_reg), lambda, n->tr_img, n->tr_h2,
                                            n->tr_dz3, n->tr_slices, g, loss_dev,
                                            pd::device_sm_count(), s);
    if (!e && grads_dev && g != grads_dev)
        e = cudaMemcpyAsync(grads_dev, g, NPARAM * 4, cudaMemcpyDeviceToDevice, s);
    return e == cudaSuccess ? PD_OK : net_cuda(e, "pd_net_gradients");
}

int pd_net_take(const float* patches, const uint8_t* counts, const float* targets,
                const uint8_t* mask, const uint32_t* idx, uint32_t count, float* p_out,
                uint8_t* c_out, float* t_out, uint8_t* m_out, void* stream) {
    if (!count) return PD_OK;
    if (!patches || !counts || !targets || !mask || !idx || !p_out || !c_out || !t_out || !m_out)
        return net_fail(PD_EINVAL, "pd_net_take: NULL argument");
    const uint64_t threads = (uint64_t)count * NPOS;
    take_kernel<<<(unsigned)((threads + 255) / 256), 256, 0, (cudaStream_t)stream>>>(
        patches, counts, targets, mask, idx, count, p_out, c_out, t_out, m_out);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PD_OK : net_cuda(e, "pd_net_take");
}

int pd_net_train_step(pd_net* n, const float* patches, const uint8_t* counts, const float* targets,
                      const uint8_t* mask, uint32_t count, float n_reg, float lambda, float lr,
                      float* loss_dev, void* stream) {
    int rc = pd_net_gradients(n, patches, counts, targets, mask, count, n_reg, lambda, nullptr,
                              loss_dev, stream);
    if (rc) return rc;
    n->step++;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.0f - (float)std::pow(0.9, (double)n->step);
    const float c2 = 1.0f - (float)std::pow(0.999, (double)n->step);
    adam_kernel<<<(NPARAM + 255) / 256, 256, 0, (cudaStream_t)stream>>>(n->w, n->gw, n->m, n->v,
                                                                        NPARAM, lr, b1, b2, c1, c2,
                                                                        1e-8f);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PD_OK : net_cuda(e, "adam");
}

int pd_net_refine(const float* out_dev, const pd_hit* hits_in, uint32_t count, float conf,
                  float count_conf, pd_hit* hits_out, void* stream) {
    if (count && (!out_dev || !hits_in || !hits_out)) return net_fail(PD_EINVAL, "pd_net_refine");
    if (!count) return PD_OK;
    refine_kernel<<<(count + 255) / 256, 256, 0, (cudaStream_t)stream>>>(
        out_dev, hits_in, count, conf, count_conf, hits_out);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PD_OK : net_cuda(e, "refine");
}

void pd_net_destroy(pd_net* n) {
    if (!n) return;
    cudaDeviceSynchronize();
    free_net(n);
}

}  // extern "C"

namespace pd {
cudaError_t launch_gather(const ChainParams& p, const uint16_t* raw, uint32_t frame_base,
                          const float* cm, const pd_hit* hits, uint32_t n, float* patches,
                          cudaStream_t s, const MultiGain* mg) {
    if (!n) return cudaSuccess;
    const uint32_t per = 8 * kGatherHits;  // hits per 256-thread block
    const MultiGain m = mg ? *mg : MultiGain{};
    auto magic = [](uint32_t d) { return d > 1 ? (uint32_t)(((1ull << 32) + d - 1) / d) : 0u; };
    const GatherDiv dv{magic(p.unit_rows), magic(p.unit_cols)};
    const unsigned blocks = n / per + (n % per != 0);
    if (mg)
        gather_kernel<true><<<blocks, 256, 0, s>>>(p, raw, frame_base, cm, hits, n, patches, m, dv);
    else
        gather_kernel<false><<<blocks, 256, 0, s>>>(p, raw, frame_base, cm, hits, n, patches, m, dv);
    return cudaGetLastError();
}
}  // namespace pd
