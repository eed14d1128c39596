// S7: the learned inverse.  A small 1-D convolutional network reads a
// normalised mean-latency trace over the 512 points of the plan and predicts
// (capacity, line size, ways, policy); an exhaustive least-squares matcher over
// the simulator's miss-rate table is its fallback and its judge.
//
// Network (per trace, channel-last activations [L, C]):
//   4 x [conv1d k=5, stride 2, pad 2, 64 channels, GELU]: 512x1 -> 256 -> 128 -> 64 -> 32
//   flatten 32*64 = 2048 -> FC 256 -> GELU -> FC 31 = heads of 17 + 4 + 7 + 3 logits
// Every product takes BF16 operands with FP32 accumulation; master weights,
// Adam moments and gradients stay FP32.  Inference runs on the tcgen05 tensor
// cores (conv_tc.cu): layers 1 and 2 in one kernel (layer 1 computed on chip
// from the FP32 inputs), layers 3 and 4 in one kernel (layer 3 on chip), then
// FC + heads in one kernel.  The training step (train_tc.cu) runs the
// 64-channel convolutions forward (pre-activations kept) and backward, and
// the FC and heads layers as GEMMs, on the tcgen05 tensor cores too; the
// first convolution (one input channel, five taps) runs on CUDA cores both
// ways.
//
// The synthetic traces follow Sec. 4.1's mean-latency model t = t0 + t_m r
// with r the miss rate the simulator reports for each plan point.
#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include <cuda_bf16.h>

#include "conv_tc.cuh"
#include "pchase_internal.cuh"
#include "tc_common.cuh"

namespace pchase {

namespace {



// --------------------------------------------------------- network plumbing
constexpr int kPoints = 512;
constexpr int kCh = 64;
constexpr int kKer = 5;
constexpr int kHidden = 256;
constexpr int kFlat = 32 * kCh;
constexpr int kLogits = 31;
constexpr int kLogitsPad = 32;  // BF16 logit gradients: rows of 64 bytes
__constant__ int c_head_off[5] = {0, 17, 21, 28, 31};

// dz = dy * gelu'(pre) (FP32 in, BF16 out for the next GEMMs)
__global__ void gelu_back_kernel(const float *dy, const float *pre, size_t n, float *dzf,
                                 __nv_bfloat16 *dzb) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x) {
        const float v = dy[i] * gelu_grad_t(pre[i]);
        if (dzf) dzf[i] = v;
        dzb[i] = __float2bfloat16(v);
    }
}

// softmax cross-entropy over the four heads; loss (mean over the batch and
// heads) accumulated into *loss; dlogits = (softmax - onehot) / (4 batch).  A
// thread per trace and head (a thread per trace left 4096 traces to 32 CTAs:
// 16 us).  A term and a warp's sum of 32 are FP32; the warps' sums are added in
// FP64 to *sum, and the last block to arrive adds that to *loss.
constexpr size_t kLossOffset = 16;  // behind the status word
struct LossSum {
    double sum;
    uint32_t blocks;
};
__global__ void xent_kernel(const float *logits, const uint32_t *labels, int nb, float *dlog,
                            __nv_bfloat16 *dlogb, LossSum *sum, float *loss) {
    const int u = blockIdx.x * blockDim.x + threadIdx.x;
    const int b = u >> 2, h = u & 3;
    float l = 0.0f;
    const float inv = 1.0f / (4.0f * nb);
    if (b < nb) {
        const int o0 = c_head_off[h], o1 = c_head_off[h + 1];
        const float *z = logits + (size_t)b * kLogits;
        float mx = -INFINITY;
        for (int i = o0; i < o1; ++i) mx = fmaxf(mx, z[i]);
        float se = 0.0f;
        for (int i = o0; i < o1; ++i) se += expf(z[i] - mx);
        const uint32_t y = labels[(size_t)b * 4 + h];
        l = (logf(se) + mx - z[o0 + y]) * inv;
        for (int i = o0; i < o1; ++i) {
            const float p = expf(z[i] - mx) / se;
            const float d = (p - (i == (int)(o0 + y) ? 1.0f : 0.0f)) * inv;
            dlog[(size_t)b * kLogits + i] = d;
            dlogb[(size_t)b * kLogitsPad + i] = __float2bfloat16(d);
        }
        if (h == 3) dlogb[(size_t)b * kLogitsPad + kLogits] = __float2bfloat16(0.0f);
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) l += __shfl_xor_sync(kFull, l, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(&sum->sum, (double)l);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(&sum->blocks, 1u) + 1u == gridDim.x) {
        __threadfence();
        atomicAdd(loss, (float)atomicAdd(&sum->sum, 0.0));
    }
}

// Adam (Kingma & Ba 2015) on FP32 master weights; refreshes BF16 copies
__global__ void adam_kernel(float *w, const float *gr, float *m, float *v, __nv_bfloat16 *wb,
                            size_t n, float lr, float b1, float b2, float eps, float c1, float c2) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x) {
        const float g = gr[i];
        const float mi = b1 * m[i] + (1.0f - b1) * g;
        const float vi = b2 * v[i] + (1.0f - b2) * g * g;
        m[i] = mi;
        v[i] = vi;
        const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        w[i] = wi;
        wb[i] = __float2bfloat16(wi);
    }
}

__device__ __forceinline__ uint64_t smix(uint64_t x) { return splitmix64(x); }
__device__ __forceinline__ float unit_f(uint64_t h) { return (float)(h >> 40) * (1.0f / 16777216.0f); }

// Uniform init in +-scale per parameter segment, counter-based (SplitMix64
// keyed on seed and index); biases start at 0 (scale 0).
struct InitSegs {
    unsigned long long end[12];
    float scale[12];
    int n;
};

__global__ void init_kernel(float *w, __nv_bfloat16 *wb, size_t n, const InitSegs segs,
                            uint64_t seed) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x) {
        int s = 0;
        while (s < segs.n - 1 && i >= segs.end[s]) ++s;
        const float u = unit_f(smix(seed ^ (i * 0x9E3779B97F4A7C15ull)));
        const float v = (2.0f * u - 1.0f) * segs.scale[s];
        w[i] = v;
        wb[i] = __float2bfloat16(v);
    }
}

// Synthetic traces: sample i picks a geometry, a (t0, t1) pair, per-point
// jitter and spikes, all from SplitMix64 keyed on (seed, i, point), then
// min-max normalises.  Box-Muller turns two uniforms into a Gaussian.
__global__ void synth_kernel(const float *rates, const uint32_t *targets, uint32_t n_geoms,
                             uint64_t seed, uint64_t first, uint32_t n, float t0_lo, float t0_hi,
                             float lr_lo, float lr_hi, float sigma, float spike_p, float sp_lo,
                             float sp_hi, float *xf, __nv_bfloat16 *xb, uint32_t *labels,
                             uint32_t *truth) {
    const uint32_t s = blockIdx.x;
    if (s >= n) return;
    __shared__ float y[kPoints];
    __shared__ float red[2][32];
    const uint64_t id = first + s;
    const uint64_t base = smix(seed ^ (id * 0xD1B54A32D192ED03ull));
    const uint32_t g = (uint32_t)(((smix(base ^ 1) >> 32) * (uint64_t)n_geoms) >> 32);
    const float t0 = t0_lo + (t0_hi - t0_lo) * unit_f(smix(base ^ 2));
    const float rho = expf(lr_lo + (lr_hi - lr_lo) * unit_f(smix(base ^ 3)));
    const float tm = t0 * (rho - 1.0f);
    float mn = INFINITY, mx = -INFINITY;
    for (int p = threadIdx.x; p < kPoints; p += blockDim.x) {
        const uint64_t hp = smix(base ^ (((uint64_t)p + 16) << 20));
        const float u1 = fmaxf(unit_f(smix(hp ^ 1)), 1e-7f), u2 = unit_f(smix(hp ^ 2));
        const float z = sqrtf(-2.0f * logf(u1)) * cospif(2.0f * u2);
        float v = (t0 + tm * rates[(size_t)g * kPoints + p]) * (1.0f + sigma * z);
        if (unit_f(smix(hp ^ 3)) < spike_p) v *= sp_lo + (sp_hi - sp_lo) * unit_f(smix(hp ^ 4));
        y[p] = v;
        mn = fminf(mn, v);
        mx = fmaxf(mx, v);
    }
    for (int o = 16; o; o >>= 1) {
        mn = fminf(mn, __shfl_xor_sync(kFull, mn, o));
        mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, o));
    }
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = mn;
        red[1][threadIdx.x >> 5] = mx;
    }
    __syncthreads();
    mn = red[0][0];
    mx = red[1][0];
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
        mn = fminf(mn, red[0][w]);
        mx = fmaxf(mx, red[1][w]);
    }
    const float sc = mx > mn ? 1.0f / (mx - mn) : 0.0f;
    for (int p = threadIdx.x; p < kPoints; p += blockDim.x) {
        const float v = (y[p] - mn) * sc;
        if (xf) xf[(size_t)s * kPoints + p] = v;
        if (xb) xb[(size_t)s * kPoints + p] = __float2bfloat16(v);
    }
    if (threadIdx.x < 4) labels[(size_t)s * 4 + threadIdx.x] = targets[(size_t)g * 4 + threadIdx.x];
    if (threadIdx.x == 0 && truth) truth[s] = g;
}

// argmax and confidence (product of the heads' top probabilities)
__global__ void predict_kernel(const float *logits, int nb, uint32_t *pred, float *conf) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nb) return;
    float c = 1.0f;
    for (int h = 0; h < 4; ++h) {
        const int o0 = c_head_off[h], o1 = c_head_off[h + 1];
        const float *z = logits + (size_t)b * kLogits;
        int best = o0;
        for (int i = o0 + 1; i < o1; ++i)
            if (z[i] > z[best]) best = i;
        float se = 0.0f;
        for (int i = o0; i < o1; ++i) se += expf(z[i] - z[best]);
        c *= 1.0f / se;
        pred[(size_t)b * 4 + h] = (uint32_t)(best - o0);
    }
    conf[b] = c;
}

// column sums with atomics (out zeroed by the caller); a thread's rows are
// loads one after the other, so few of them to a block (256 rows: 12 us)
__global__ void colsum_atomic_kernel(const float *x, int rows, int cols, int rows_per_block,
                                     float *out) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= cols) return;
    const int r0 = blockIdx.y * rows_per_block;
    const int r1 = min(rows, r0 + rows_per_block);
    float s = 0.0f;
#pragma unroll 8
    for (int r = r0; r < r1; ++r) s += x[(size_t)r * cols + c];
    atomicAdd(out + c, s);
}

// First convolution (1 input channel) of the training forward pass:
// out[b][p][co] = BF16(GELU(bias[co] + sum_k W[co][k] * x[b][2p + k - 2])) (BF16
// operands, the FP32 inputs rounded here, FP32 sums; the backward pass works
// the pre-activations out again).  One block per trace: the 512 inputs are
// staged in shared memory (zero padding around them); thread t computes
// channels 8 (t % 8) .. +7 at positions t / 8 + 32 i, so that a warp stores
// four whole rows.  32 KB written per trace (with the 64 KB of FP32
// pre-activations 4096 traces took 90 us, 47 us without).
__global__ void __launch_bounds__(256) conv1_kernel(const float *__restrict__ x, int nb,
                                                    const __nv_bfloat16 *__restrict__ W,
                                                    const float *__restrict__ bias,
                                                    __nv_bfloat16 *__restrict__ out) {
    constexpr int lout = kPoints / 2;
    __shared__ float xs[kPoints + 8];  // xs[q + 2] = x[q], zeros outside
    const int t = threadIdx.x, g = t & 7, p0 = t >> 3;
    float w[8][kKer], bs[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        bs[c] = bias[g * 8 + c];
#pragma unroll
        for (int k = 0; k < kKer; ++k) w[c][k] = __bfloat162float(W[(g * 8 + c) * kKer + k]);
    }
    for (int b = blockIdx.x; b < nb; b += gridDim.x) {
        __syncthreads();  // the previous trace's reads are done
        for (int q = t; q < kPoints + 8; q += blockDim.x) {
            const int src = q - 2;
            xs[q] = (src >= 0 && src < kPoints)
                        ? __bfloat162float(__float2bfloat16(x[(size_t)b * kPoints + src])) : 0.0f;
        }
        __syncthreads();
#pragma unroll 2
        for (int i = 0; i < 8; ++i) {
            const int p = p0 + 32 * i;
            float xin[kKer];
#pragma unroll
            for (int k = 0; k < kKer; ++k) xin[k] = xs[2 * p + k];  // x[2p + k - 2]
            const size_t row = (size_t)b * lout + p;
            float v[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                float acc = 0.0f;
#pragma unroll
                for (int k = 0; k < kKer; ++k) acc = fmaf(w[c][k], xin[k], acc);
                v[c] = acc + bs[c];
            }
            uint32_t pk[4];
#pragma unroll
            for (int c = 0; c < 8; c += 2) {
                const __nv_bfloat162 hv = __floats2bfloat162_rn(gelu_t(v[c]), gelu_t(v[c + 1]));
                pk[c >> 1] = *reinterpret_cast<const uint32_t *>(&hv);
            }
            *reinterpret_cast<uint4 *>(out + row * kCh + g * 8) =
                make_uint4(pk[0], pk[1], pk[2], pk[3]);
        }
    }
}

__global__ void f2b_kernel(const float *x, size_t n, __nv_bfloat16 *y) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x)
        y[i] = __float2bfloat16(x[i]);
}

// learned predictions -> candidate index through a label table; low
// confidence or an unknown label combination marks the trace for fallback
__global__ void route_kernel(const uint32_t *pred, const float *conf, uint32_t n,
                             const uint32_t *label_to_cand, float thresh, uint32_t *cand_out,
                             uint32_t *fallback_list, uint32_t *n_fallback) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t *p = pred + (size_t)i * 4;
    const uint32_t key = ((p[0] * 4 + p[1]) * 7 + p[2]) * 3 + p[3];
    const uint32_t c = label_to_cand[key];
    if (conf[i] < thresh || c == 0xFFFFFFFFu) {
        const uint32_t k = atomicAdd(n_fallback, 1u);
        fallback_list[k] = i;
        cand_out[i] = 0xFFFFFFFFu;
    } else {
        cand_out[i] = c;
    }
}

__global__ void gather_rows_kernel(const float *x, const uint32_t *rows, const uint32_t *n_rows,
                                   float *out) {
    const uint32_t r = blockIdx.x;
    if (r >= *n_rows) return;
    const float *src = x + (size_t)rows[r] * kPoints;
    for (int p = threadIdx.x; p < kPoints; p += blockDim.x) out[(size_t)r * kPoints + p] = src[p];
}

__global__ void scatter_fallback_kernel(const uint32_t *rows, const uint32_t *n_rows,
                                        const uint32_t *idx, uint32_t *cand_out) {
    const uint32_t r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= *n_rows) return;
    cand_out[rows[r]] = idx[r];
}

}  // namespace

// ------------------------------------------------------------ host side
struct InverseLayout {
    // parameter segments (FP32 master / BF16 copy / grads / Adam moments share offsets)
    size_t w[6], b[6], n_params;
    int cin[4], lin[4];
};

InverseLayout inverse_layout() {
    InverseLayout L{};
    size_t off = 0;
    const int cins[4] = {1, kCh, kCh, kCh};
    const int lins[4] = {kPoints, kPoints / 2, kPoints / 4, kPoints / 8};
    for (int l = 0; l < 4; ++l) {
        L.cin[l] = cins[l];
        L.lin[l] = lins[l];
        L.w[l] = off;
        off += (size_t)kCh * kKer * cins[l];
        L.b[l] = off;
        off += kCh;
    }
    L.w[4] = off;
    off += (size_t)kHidden * kFlat;
    L.b[4] = off;
    off += kHidden;
    L.w[5] = off;
    off += (size_t)kLogits * kHidden;
    L.b[5] = off;
    off += kLogits;
    L.n_params = off;
    return L;
}


namespace {

int grid_for(size_t n, int threads = 256) {
    size_t b = (n + threads - 1) / threads;
    if (b > 8192) b = 8192;
    return (int)(b ? b : 1);
}

size_t a256(size_t x) { return (x + 255) & ~size_t(255); }

}  // namespace

}  // namespace pchase

using namespace pchase;

struct pchase_inverse {
    InverseLayout L;
    uint32_t max_batch;
    size_t p_w, p_wb, p_g, p_m, p_v, p_bytes;
    size_t status, pre[4], act[4], pre4, h4, logits, dlog, dlogb, tA, tB, tD, w4t, w5t, dh, dzf, dzb, dbig,
        dsmall, work_bytes, infer_bytes;
};

namespace {
thread_local std::string g_inv_err;
int inv_fail(int code, const char *m) {
    g_inv_err = m;
    return code;
}
#define INV_CUDA(call)                                       \
    do {                                                     \
        cudaError_t e_ = (call);                             \
        if (e_ != cudaSuccess) return inv_fail(PCHASE_ECUDA, cudaGetErrorString(e_)); \
    } while (0)

template <typename T>
T *at(void *base, size_t off) {
    return reinterpret_cast<T *>(static_cast<uint8_t *>(base) + off);
}
template <typename T>
const T *at(const void *base, size_t off) {
    return reinterpret_cast<const T *>(static_cast<const uint8_t *>(base) + off);
}

int device_sms() {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 1;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 1;
    return n;
}

int forward(const pchase_inverse *h, const void *params, void *work, uint32_t B, cudaStream_t st,
            bool train, const float *xf) {
    const InverseLayout &L = h->L;
    const __nv_bfloat16 *wb = at<__nv_bfloat16>(params, h->p_wb);
    const float *wf = at<float>(params, h->p_w);
    const __nv_bfloat16 *in = nullptr;
    int l0 = 0;
    if (!train) {
        // inference: layers 1 and 2 in one tcgen05 kernel from the FP32 inputs
        // (layer 1's activations stay on chip)
        __nv_bfloat16 *o = at<__nv_bfloat16>(work, h->act[1]);
        INV_CUDA(conv12_tc(xf, (int)B, wb + L.w[0], wf + L.b[0], wb + L.w[1], wf + L.b[1], o,
                           at<uint32_t>(work, h->status), device_sms(), st));
        // layers 3 and 4 in one tcgen05 kernel (layer 3's activations stay on chip)
        __nv_bfloat16 *o4 = at<__nv_bfloat16>(work, h->act[3]);
        INV_CUDA(conv34_tc(o, (int)B, wb + L.w[2], wf + L.b[2], wb + L.w[3], wf + L.b[3], o4,
                           at<uint32_t>(work, h->status), device_sms(), st));
        in = o4;
        l0 = 4;
    }
    for (int l = l0; l < 4; ++l) {
        const int lin = L.lin[l], cin = L.cin[l], lout = lin / 2;
        if (cin == kCh) {
            // tcgen05 tensor cores, pre-activations kept
            __nv_bfloat16 *o = at<__nv_bfloat16>(work, h->act[l]);
            INV_CUDA(conv_fwd_tc(in, (int)B, lout, wb + L.w[l], wf + L.b[l],
                                 at<float>(work, h->pre[l]), o, at<uint32_t>(work, h->status),
                                 device_sms(), st));
            in = o;
            continue;
        }
        // first layer (one input channel): direct
        __nv_bfloat16 *o = at<__nv_bfloat16>(work, h->act[l]);
        conv1_kernel<<<std::min<uint32_t>(B, 152u * 8u), 256, 0, st>>>(
            xf, (int)B, wb + L.w[l], wf + L.b[l], o);
        INV_CUDA(cudaGetLastError());
        in = o;
    }
    if (!train) {
        // inference: FC on the tcgen05 tensor cores, heads in its epilogue
        INV_CUDA(fc_heads_tc(in, (int)B, wb + L.w[4], wf + L.b[4], wb + L.w[5], wf + L.b[5],
                             at<float>(work, h->logits), at<uint32_t>(work, h->status), st));
        return PCHASE_OK;
    }
    // FC 2048 -> 256 with bias and GELU (pre-activations kept), then the
    // heads, on the tcgen05 tensor cores
    uint32_t *status = at<uint32_t>(work, h->status);
    __nv_bfloat16 *h4 = at<__nv_bfloat16>(work, h->h4);
    INV_CUDA(tc_gemm(in, kFlat, wb + L.w[4], kFlat, (int)B, kHidden, kFlat, 64, 1, wf + L.b[4],
                     nullptr, kHidden, false, false, at<float>(work, h->pre4), h4, status, st));
    INV_CUDA(tc_gemm(h4, kHidden, wb + L.w[5], kHidden, (int)B, kLogits, kHidden, 32, 1,
                     wf + L.b[5], at<float>(work, h->logits), kLogits, false, false, nullptr,
                     nullptr, status, st));
    return PCHASE_OK;
}

}  // namespace

extern "C" {

const char *pchase_inverse_last_error(void) { return g_inv_err.c_str(); }

int pchase_inverse_create(uint32_t max_batch, pchase_inverse **out) {
    if (!out || max_batch == 0 || max_batch > (1u << 16))
        return inv_fail(PCHASE_EINVAL, "max_batch must be in [1, 65536]");
    auto *h = new (std::nothrow) pchase_inverse();
    if (!h) return inv_fail(PCHASE_ENOMEM, "allocation");
    h->L = inverse_layout();
    h->max_batch = max_batch;
    const size_t n = h->L.n_params;
    size_t o = 0;
    h->p_w = o; o = a256(o + 4 * n);
    h->p_wb = o; o = a256(o + 2 * n);
    h->p_g = o; o = a256(o + 4 * n);
    h->p_m = o; o = a256(o + 4 * n);
    h->p_v = o; o = a256(o + 4 * n);
    h->p_bytes = o;
    const size_t B = max_batch;
    // inference's buffers first (a caller that only infers allocates that
    // prefix, pchase_inverse_infer_work_bytes), then the training step's
    o = 0;
    h->status = o; o = a256(o + kLossOffset + sizeof(LossSum));
    for (int l = 0; l < 4; ++l) {
        const size_t lout = h->L.lin[l] / 2;
        h->act[l] = o; o = a256(o + 2 * B * lout * kCh);
    }
    h->logits = o; o = a256(o + 4 * B * kLogits);
    h->infer_bytes = o;
    size_t big = B * kFlat;  // largest per-layer FP32 activation gradient
    for (int l = 0; l < 4; ++l) {
        const size_t lout = h->L.lin[l] / 2;
        if (l > 0) {  // (the first layer's are worked out again)
            h->pre[l] = o;
            o = a256(o + 4 * B * lout * kCh);
        }
        big = std::max(big, B * lout * kCh);
    }
    h->pre4 = o; o = a256(o + 4 * B * kHidden);
    h->h4 = o; o = a256(o + 2 * B * kHidden);
    h->dlog = o; o = a256(o + 4 * B * kLogits);
    h->dlogb = o; o = a256(o + 2 * B * kLogitsPad);
    {
        // transposed operands of the weight gradients (rows of the batch
        // padded to a multiple of 8) and of the input gradients
        const size_t ldk = (B + 7) / 8 * 8;
        h->tA = o; o = a256(o + 2 * kHidden * ldk);
        h->tB = o; o = a256(o + 2 * kFlat * ldk);
        h->tD = o; o = a256(o + 2 * kLogitsPad * ldk);
        h->w4t = o; o = a256(o + 2 * (size_t)kFlat * kHidden);
        h->w5t = o; o = a256(o + 2 * (size_t)kHidden * kLogitsPad);
    }
    h->dh = o; o = a256(o + 4 * B * kHidden);
    h->dzf = o; o = a256(o + 4 * B * kHidden);
    h->dzb = o; o = a256(o + 2 * B * kHidden);
    h->dbig = o; o = a256(o + 4 * big);
    h->dsmall = o; o = a256(o + 4 * big);
    h->work_bytes = o;
    *out = h;
    return PCHASE_OK;
}

void pchase_inverse_destroy(pchase_inverse *h) { delete h; }
uint64_t pchase_inverse_param_count(const pchase_inverse *h) { return h ? h->L.n_params : 0; }
size_t pchase_inverse_param_bytes(const pchase_inverse *h) { return h ? h->p_bytes : 0; }
size_t pchase_inverse_work_bytes(const pchase_inverse *h) { return h ? h->work_bytes : 0; }
size_t pchase_inverse_infer_work_bytes(const pchase_inverse *h) { return h ? h->infer_bytes : 0; }
size_t pchase_inverse_status_offset(const pchase_inverse *h) { return h ? h->status : 0; }
size_t pchase_inverse_activation_offset(const pchase_inverse *h, uint32_t layer) {
    return h && layer < 4 ? h->act[layer] : 0;
}
size_t pchase_inverse_param_offset(const pchase_inverse *h, uint32_t which) {
    if (!h) return (size_t)-1;
    switch (which) {
        case 0: return h->p_w;
        case 1: return h->p_wb;
        case 2: return h->p_g;
        case 3: return h->p_m;
        case 4: return h->p_v;
        default: return (size_t)-1;
    }
}

int pchase_inverse_init(const pchase_inverse *h, void *params, uint64_t seed,
                        pchase_stream_t stream) {
    if (!h || !params) return inv_fail(PCHASE_EINVAL, "NULL argument");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const InverseLayout &L = h->L;
    InitSegs s{};
    int k = 0;
    for (int l = 0; l < 6; ++l) {
        const size_t fan_in = l < 4 ? (size_t)kKer * L.cin[l] : (l == 4 ? kFlat : kHidden);
        s.end[k] = L.b[l];
        s.scale[k++] = sqrtf(6.0f / (float)fan_in) * (l == 5 ? 0.5f : 1.0f);
        s.end[k] = l < 5 ? L.w[l + 1] : L.n_params;
        s.scale[k++] = 0.0f;
    }
    s.n = k;
    const size_t n = L.n_params;
    init_kernel<<<grid_for(n), 256, 0, st>>>(at<float>(params, h->p_w),
                                               at<__nv_bfloat16>(params, h->p_wb), n, s, seed);
    INV_CUDA(cudaMemsetAsync(at<float>(params, h->p_m), 0, 4 * n, st));
    INV_CUDA(cudaMemsetAsync(at<float>(params, h->p_v), 0, 4 * n, st));
    INV_CUDA(cudaGetLastError());
    return PCHASE_OK;
}

int pchase_inverse_synth(const float *rates, const uint32_t *targets, uint32_t n_geoms,
                         uint64_t seed, uint64_t first, uint32_t n, const float *noise,
                         float *x_out, uint32_t *labels_out, uint32_t *truth_out,
                         pchase_stream_t stream) {
    if (!rates || !targets || !x_out || !labels_out || !noise || n_geoms == 0)
        return inv_fail(PCHASE_EINVAL, "NULL argument or no geometries");
    if (n == 0) return PCHASE_OK;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    synth_kernel<<<n, 128, 0, st>>>(rates, targets, n_geoms, seed, first, n, noise[0], noise[1],
                                    logf(noise[2]), logf(noise[3]), noise[4], noise[5], noise[6],
                                    noise[7], x_out, nullptr, labels_out, truth_out);
    INV_CUDA(cudaGetLastError());
    return PCHASE_OK;
}

int pchase_inverse_train_step(const pchase_inverse *h, void *params, void *work, const float *x,
                              const uint32_t *labels, uint32_t B, float lr, uint32_t step,
                              float *loss_accum, pchase_stream_t stream) {
    if (!h || !params || !work || !x || !labels || !loss_accum)
        return inv_fail(PCHASE_EINVAL, "NULL argument");
    if (B == 0 || B > h->max_batch) return inv_fail(PCHASE_ERANGE, "batch above max_batch");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const InverseLayout &L = h->L;
    INV_CUDA(cudaMemsetAsync(at<uint32_t>(work, h->status), 0, kLossOffset + sizeof(LossSum), st));
    int rc = forward(h, params, work, B, st, true, x);
    if (rc) return rc;
    const size_t n = L.n_params;
    float *grad = at<float>(params, h->p_g);
    const __nv_bfloat16 *wb = at<__nv_bfloat16>(params, h->p_wb);
    INV_CUDA(cudaMemsetAsync(grad, 0, 4 * n, st));
    float *dlog = at<float>(work, h->dlog);
    __nv_bfloat16 *dlogb = at<__nv_bfloat16>(work, h->dlogb);
    xent_kernel<<<(B + 31) / 32, 128, 0, st>>>(at<float>(work, h->logits), labels, (int)B, dlog,
                                                 dlogb, at<LossSum>(work, h->status + kLossOffset), loss_accum);
    // heads and FC on the tcgen05 tensor cores.  Products over the batch
    // (weight gradients) take both operands batch-contiguous: transposed
    // copies, rows padded with zeros to a multiple of 8 traces, K split over
    // CTAs with FP32 atomics into the zeroed gradient.
    uint32_t *status = at<uint32_t>(work, h->status);
    const int ldk = (int)((B + 7) / 8 * 8);
    __nv_bfloat16 *h4 = at<__nv_bfloat16>(work, h->h4);
    __nv_bfloat16 *tA = at<__nv_bfloat16>(work, h->tA), *tB = at<__nv_bfloat16>(work, h->tB);
    __nv_bfloat16 *w4t = at<__nv_bfloat16>(work, h->w4t), *w5t = at<__nv_bfloat16>(work, h->w5t);
    __nv_bfloat16 *tD = at<__nv_bfloat16>(work, h->tD);
    {
        // what can be transposed by now, in one launch (five of them: 40 us of
        // a step of 4096 traces)
        const TransposeJob jobs[kTransposeJobs] = {
            transpose_job(at<__nv_bfloat16>(work, h->act[3]), (int)B, kFlat, kFlat, tB, ldk, kFlat),
            transpose_job(wb + L.w[4], kHidden, kFlat, kFlat, w4t, kHidden, kFlat),
            transpose_job(wb + L.w[5], kLogits, kHidden, kHidden, w5t, kLogitsPad, kHidden),
            transpose_job(h4, (int)B, kHidden, kHidden, tA, ldk, kHidden),
            transpose_job(dlogb, (int)B, kLogitsPad, kLogitsPad, tD, ldk, kLogitsPad)};
        INV_CUDA(transpose_bf16(jobs, kTransposeJobs, st));
    }
    {
        // grad W5 [31][256] = dlogb^T h4, as (h4^T) (dlogb^T)^T stored transposed
        INV_CUDA(tc_gemm(tA, ldk, tD, ldk, kHidden, kLogits, ldk, 32, 32, nullptr, grad + L.w[5],
                         kHidden, true, true, nullptr, nullptr, status, st));
        colsum_atomic_kernel<<<dim3(1, (B + 31) / 32), 32, 0, st>>>(dlog, (int)B, kLogits, 32,
                                                                     grad + L.b[5]);
        // dh [B][256] = dlogb W5
        INV_CUDA(tc_gemm(dlogb, kLogitsPad, w5t, kLogitsPad, (int)B, kHidden, kLogitsPad, 128, 1,
                         nullptr, at<float>(work, h->dh), kHidden, false, false, nullptr, nullptr,
                         status, st));
    }
    float *dzf = at<float>(work, h->dzf);
    __nv_bfloat16 *dzb = at<__nv_bfloat16>(work, h->dzb);
    float *dbig = at<float>(work, h->dbig);
    float *dsmall = at<float>(work, h->dsmall);
    {
        const size_t m = (size_t)B * kHidden;
        gelu_back_kernel<<<grid_for(m), 256, 0, st>>>(at<float>(work, h->dh),
                                                      at<float>(work, h->pre4), m, dzf, dzb);
        // grad W4 [256][2048] = dzb^T act3
        const TransposeJob job = transpose_job(dzb, (int)B, kHidden, kHidden, tA, ldk, kHidden);
        INV_CUDA(transpose_bf16(&job, 1, st));
        INV_CUDA(tc_gemm(tA, ldk, tB, ldk, kHidden, kFlat, ldk, 128, 4, nullptr, grad + L.w[4],
                         kFlat, true, false, nullptr, nullptr, status, st));
        colsum_atomic_kernel<<<dim3((kHidden + 127) / 128, (B + 31) / 32), 128, 0, st>>>(
            dzf, (int)B, kHidden, 32, grad + L.b[4]);
        // d(act3) [B][32 x 64] = dzb W4
        INV_CUDA(tc_gemm(dzb, kHidden, w4t, kHidden, (int)B, kFlat, kHidden, 128, 1, nullptr, dbig,
                         kFlat, false, false, nullptr, nullptr, status, st));
    }
    // convolutions, last to first: the three 64-channel layers on the tensor
    // cores (gelu backward, weight and bias gradients, input gradient into
    // the other FP32 buffer), the first layer on CUDA cores
    {
        float *dcur = dbig, *dnext = dsmall;
        const int sms = device_sms();
        for (int l = 3; l >= 1; --l) {
            INV_CUDA(conv_back_tc(dcur, at<float>(work, h->pre[l]),
                                  at<__nv_bfloat16>(work, h->act[l - 1]), (int)B, L.lin[l] / 2,
                                  wb + L.w[l], grad + L.w[l], grad + L.b[l], dnext,
                                  at<uint32_t>(work, h->status), sms, st));
            std::swap(dcur, dnext);
        }
        INV_CUDA(conv0_back(dcur, x, wb + L.w[0], at<float>(params, h->p_w) + L.b[0], (int)B,
                            grad + L.w[0], grad + L.b[0], sms, st));
    }
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.0f - powf(b1, (float)step + 1.0f), c2 = 1.0f - powf(b2, (float)step + 1.0f);
    adam_kernel<<<grid_for(n), 256, 0, st>>>(at<float>(params, h->p_w), grad,
                                              at<float>(params, h->p_m), at<float>(params, h->p_v),
                                              at<__nv_bfloat16>(params, h->p_wb), n, lr, b1, b2,
                                              1e-8f, c1, c2);
    INV_CUDA(cudaGetLastError());
    return PCHASE_OK;
}

int pchase_inverse_infer(const pchase_inverse *h, const void *params, void *work, const float *x,
                         uint32_t n, uint32_t *pred_out, float *conf_out, float *logits_out,
                         pchase_stream_t stream) {
    if (!h || !params || !work || !x || !pred_out || !conf_out)
        return inv_fail(PCHASE_EINVAL, "NULL argument");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    INV_CUDA(cudaMemsetAsync(at<uint32_t>(work, h->status), 0, 4, st));
    for (uint32_t b0 = 0; b0 < n; b0 += h->max_batch) {
        const uint32_t B = std::min(h->max_batch, n - b0);
        int rc = forward(h, params, work, B, st, false, x + (size_t)b0 * kPoints);
        if (rc) return rc;
        const float *lg = at<float>(work, h->logits);
        predict_kernel<<<(B + 127) / 128, 128, 0, st>>>(lg, (int)B, pred_out + (size_t)b0 * 4,
                                                        conf_out + b0);
        if (logits_out)
            INV_CUDA(cudaMemcpyAsync(logits_out + (size_t)b0 * kLogits, lg,
                                     (size_t)B * kLogits * 4, cudaMemcpyDeviceToDevice, st));
    }
    INV_CUDA(cudaGetLastError());
    return PCHASE_OK;
}

size_t pchase_lsq_work_bytes(uint32_t n) { return lsq_work_bytes(n); }

int pchase_lsq_match(const float *rates, uint32_t n_geoms, const float *y, uint32_t n,
                     uint32_t *best_out, float *resid_out, void *work, pchase_stream_t stream) {
    if (!rates || !y || !best_out || !work || n_geoms == 0)
        return inv_fail(PCHASE_EINVAL, "NULL argument or no geometries");
    if (n == 0) return PCHASE_OK;
    INV_CUDA(lsq_run(rates, n_geoms, y, n, nullptr, best_out, resid_out, work, device_sms(),
                     reinterpret_cast<cudaStream_t>(stream)));
    return PCHASE_OK;
}

int pchase_inverse_classify(const pchase_inverse *h, const void *params, void *work,
                            const float *x, uint32_t n, const uint32_t *label_to_cand,
                            const float *rates, uint32_t n_geoms, float conf_thresh,
                            uint32_t *pred_scratch, float *conf_out, uint32_t *cand_out,
                            uint32_t *fallback_list, uint32_t *n_fallback, float *fb_rows,
                            uint32_t *fb_idx, void *lsq_work, pchase_stream_t stream) {
    if (!h || !params || !work || !x || !label_to_cand || !rates || !pred_scratch || !conf_out ||
        !cand_out || !fallback_list || !n_fallback || !fb_rows || !fb_idx || !lsq_work)
        return inv_fail(PCHASE_EINVAL, "NULL argument");
    if (n == 0) return PCHASE_OK;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    int rc = pchase_inverse_infer(h, params, work, x, n, pred_scratch, conf_out, nullptr, stream);
    if (rc) return rc;
    INV_CUDA(cudaMemsetAsync(n_fallback, 0, 4, st));
    route_kernel<<<(n + 255) / 256, 256, 0, st>>>(pred_scratch, conf_out, n, label_to_cand,
                                                  conf_thresh, cand_out, fallback_list, n_fallback);
    // the fallback runs over a compacted copy whose size is known only on the
    // device: the matcher's grids cover n rows and its blocks stop at the count
    gather_rows_kernel<<<n, 128, 0, st>>>(x, fallback_list, n_fallback, fb_rows);
    INV_CUDA(lsq_run(rates, n_geoms, fb_rows, n, n_fallback, fb_idx, nullptr, lsq_work, device_sms(),
                     st));
    scatter_fallback_kernel<<<(n + 255) / 256, 256, 0, st>>>(fallback_list, n_fallback, fb_idx,
                                                             cand_out);
    INV_CUDA(cudaGetLastError());
    return PCHASE_OK;
}

}  // extern "C"

// ------------------------------------------------------- a library-owned model
// inverse_load / inverse_free / inverse_classify: the learned inverse with its
// parameters, work area and fallback scratch in device memory the library
// allocates at load, for callers that hold only a weights blob.  Traces are
// classified in chunks of kModelChunk.
namespace pchase {
namespace {
constexpr uint32_t kModelChunk = 4096;

__global__ void add_count_kernel(uint32_t *total, const uint32_t *part) { *total += *part; }
}  // namespace
}  // namespace pchase

struct pchase_inverse_model {
    pchase_inverse *h = nullptr;
    void *params = nullptr, *work = nullptr, *scratch = nullptr;
    size_t off_pred = 0, off_fl = 0, off_nf = 0, off_rows = 0, off_idx = 0, off_lsq = 0;
};

extern "C" {

void inverse_free(pchase_inverse_model *m) {
    if (!m) return;
    cudaFree(m->params);
    cudaFree(m->work);
    cudaFree(m->scratch);
    pchase_inverse_destroy(m->h);
    delete m;
}

int inverse_load(const void *weights, size_t bytes, pchase_inverse_model **handle) {
    if (!weights || !handle) return inv_fail(PCHASE_EINVAL, "inverse_load: NULL argument");
    *handle = nullptr;
    auto *m = new (std::nothrow) pchase_inverse_model();
    if (!m) return inv_fail(PCHASE_ENOMEM, "inverse_load: allocation");
    int rc = pchase_inverse_create(kModelChunk, &m->h);
    if (rc) {
        delete m;
        return rc;
    }
    const size_t n = m->h->L.n_params;
    if (bytes != 4 * n) {
        inverse_free(m);
        return inv_fail(PCHASE_EINVAL, "inverse_load: bytes must be 4 x pchase_inverse_param_count");
    }
    const size_t B = kModelChunk;
    size_t o = 0;
    m->off_pred = o; o = a256(o + 16 * B);
    m->off_fl = o; o = a256(o + 4 * B);
    m->off_nf = o; o = a256(o + 4);
    m->off_rows = o; o = a256(o + 4 * B * kPoints);
    m->off_idx = o; o = a256(o + 4 * B);
    m->off_lsq = o; o = a256(o + pchase_lsq_work_bytes((uint32_t)B));
    cudaError_t e = cudaMalloc(&m->params, m->h->p_bytes);
    if (e == cudaSuccess) e = cudaMalloc(&m->work, m->h->work_bytes);
    if (e == cudaSuccess) e = cudaMalloc(&m->scratch, o);
    if (e != cudaSuccess) {
        inverse_free(m);
        return inv_fail(PCHASE_ENOMEM, "inverse_load: cudaMalloc failed");
    }
    // FP32 masters from the blob, their BF16 copies by the library's own
    // conversion kernel, zero moments; synchronous (the blob is host memory)
    float *w = at<float>(m->params, m->h->p_w);
    e = cudaMemcpy(w, weights, bytes, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        f2b_kernel<<<grid_for(n), 256>>>(w, n, at<__nv_bfloat16>(m->params, m->h->p_wb));
        e = cudaMemset(at<float>(m->params, m->h->p_m), 0, 4 * n);
    }
    if (e == cudaSuccess) e = cudaMemset(at<float>(m->params, m->h->p_v), 0, 4 * n);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        inverse_free(m);
        return inv_fail(PCHASE_ECUDA, cudaGetErrorString(e));
    }
    *handle = m;
    return PCHASE_OK;
}

int inverse_classify(const pchase_inverse_model *m, const float *x, uint32_t n,
                     const uint32_t *label_to_cand, const float *rates, uint32_t n_geoms,
                     float conf_thresh, uint32_t *cand_out, float *conf_out, uint32_t *n_fallback,
                     pchase_stream_t stream) {
    if (!m || !x || !label_to_cand || !rates || !cand_out || !conf_out || !n_fallback)
        return inv_fail(PCHASE_EINVAL, "inverse_classify: NULL argument");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    INV_CUDA(cudaMemsetAsync(n_fallback, 0, 4, st));
    uint8_t *s = static_cast<uint8_t *>(m->scratch);
    uint32_t *part = reinterpret_cast<uint32_t *>(s + m->off_nf);
    for (uint32_t b0 = 0; b0 < n; b0 += kModelChunk) {
        const uint32_t c = std::min(kModelChunk, n - b0);
        int rc = pchase_inverse_classify(
            m->h, m->params, m->work, x + (size_t)b0 * kPoints, c, label_to_cand, rates, n_geoms,
            conf_thresh, reinterpret_cast<uint32_t *>(s + m->off_pred), conf_out + b0,
            cand_out + b0, reinterpret_cast<uint32_t *>(s + m->off_fl), part,
            reinterpret_cast<float *>(s + m->off_rows), reinterpret_cast<uint32_t *>(s + m->off_idx),
            s + m->off_lsq, stream);
        if (rc) return rc;
        add_count_kernel<<<1, 1, 0, st>>>(n_fallback, part);
    }
    INV_CUDA(cudaGetLastError());
    return PCHASE_OK;
}

}  // extern "C"

