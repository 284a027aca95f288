// mlp.cu -- the learned proposal of the filter polygon: features of a point
// set and a small MLP that picks the direction count K in {8, 16, 32, 64}
// and the angular offsets of the K-direction polygon (kfilter.cu).  The
// paper filters with the fixed octagon; this is the extension its related
// work points to (more directions).  Whatever the MLP outputs, the polygon's
// vertices are extreme input points, so the filter stays exact.
//
// Features: a 32 x 32 occupancy grid of a 4096-point sample (evenly spaced
// indices) over the sample's bounding box, as fractions of the sample.
// MLP: 1024 -> 64 -> 64 -> 68 (4 K-logits, 64 offsets), ReLU between,
// BF16 weights, FP32 accumulation; one parameter array, row-major:
//   W1[64][1024] b1[64] W2[64][64] b2[64] W3[68][64] b3[68].
// Training: one kernel per sample (forward, the loss -- softmax
// cross-entropy on the K-logits, squared error on the offsets of samples
// that carry an offset label -- and the backward pass through the
// activations), and one per parameter (its gradient summed over the batch
// and the Adam step on FP32 master weights, which also writes their BF16
// copy).
#include <cuda_bf16.h>

#include <algorithm>

#include "common.cuh"
#include "launch.h"
#include "mlp.cuh"

namespace ch {
namespace {

using namespace mlp;

// One block of 1024 threads per point set.
__global__ void __launch_bounds__(1024) features_kernel(const float *__restrict__ pts, int64_t n, float *__restrict__ feat)
{
    __shared__ float s_red[4][32];
    __shared__ uint32_t s_cnt[kIn];
    __shared__ float s_box[4];
    const int t = (int)threadIdx.x, lane = t & 31, warp = t >> 5;
    const int m = n < kSample ? (int)n : kSample;
    for (int c = t; c < kIn; c += 1024) s_cnt[c] = 0u;
    // the sample: points floor(j n / m), j < m
    float px[kSample / 1024], py[kSample / 1024];
    float x0 = __int_as_float(0x7f800000), x1 = -x0, y0 = x0, y1 = -x0;
#pragma unroll
    for (int r = 0; r < kSample / 1024; ++r) {
        const int j = r * 1024 + t;
        px[r] = py[r] = 0.0f;
        if (j < m) {
            const int64_t i = (int64_t)j * n / m;
            const float2 v = reinterpret_cast<const float2 *>(pts)[i];
            px[r] = v.x;
            py[r] = v.y;
            x0 = fminf(x0, v.x);
            x1 = fmaxf(x1, v.x);
            y0 = fminf(y0, v.y);
            y1 = fmaxf(y1, v.y);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        x0 = fminf(x0, __shfl_xor_sync(0xffffffffu, x0, o));
        x1 = fmaxf(x1, __shfl_xor_sync(0xffffffffu, x1, o));
        y0 = fminf(y0, __shfl_xor_sync(0xffffffffu, y0, o));
        y1 = fmaxf(y1, __shfl_xor_sync(0xffffffffu, y1, o));
    }
    if (lane == 0) {
        s_red[0][warp] = x0;
        s_red[1][warp] = x1;
        s_red[2][warp] = y0;
        s_red[3][warp] = y1;
    }
    __syncthreads();
    if (t == 0) {
        float a = s_red[0][0], b = s_red[1][0], c = s_red[2][0], d = s_red[3][0];
        for (int w = 1; w < 32; ++w) {
            a = fminf(a, s_red[0][w]);
            b = fmaxf(b, s_red[1][w]);
            c = fminf(c, s_red[2][w]);
            d = fmaxf(d, s_red[3][w]);
        }
        s_box[0] = a;
        s_box[1] = b;
        s_box[2] = c;
        s_box[3] = d;
    }
    __syncthreads();
    const float w = __fsub_rn(s_box[1], s_box[0]), h = __fsub_rn(s_box[3], s_box[2]);
    const float sx = w > 0.0f ? 32.0f / w : 0.0f, sy = h > 0.0f ? 32.0f / h : 0.0f;
#pragma unroll
    for (int r = 0; r < kSample / 1024; ++r) {
        const int j = r * 1024 + t;
        if (j < m) {
            const int cx = min(kGrid - 1, (int)floorf(__fmul_rn(__fsub_rn(px[r], s_box[0]), sx)));
            const int cy = min(kGrid - 1, (int)floorf(__fmul_rn(__fsub_rn(py[r], s_box[2]), sy)));
            atomicAdd(&s_cnt[cy * kGrid + cx], 1u);
        }
    }
    __syncthreads();
    const float inv = 1.0f / (float)m;
    for (int c = t; c < kIn; c += 1024) feat[c] = (float)s_cnt[c] * inv;
}

// Eight consecutive weights (VEC: the parameters are 16-byte aligned, one
// load; else one by one).
template <bool VEC>
__device__ __forceinline__ void weights8(const __nv_bfloat16 *__restrict__ P, int i, float (&w)[8])
{
    if constexpr (VEC) {
        const uint4 v = __ldg(reinterpret_cast<const uint4 *>(P + i));
        const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            w[2 * q] = __uint_as_float(u[q] << 16);
            w[2 * q + 1] = __uint_as_float(u[q] & 0xffff0000u);
        }
    } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) w[q] = wf(P, i + q);
    }
}

template <int W>   // sum over groups of W lanes, in every lane
__device__ __forceinline__ float lanes_sum(float v)
{
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

struct LossArgs {
    const int32_t *label;
    const float *off, *mask;
    float lam;
    float *dOUT, *dH1, *dH2, *loss;
};

// One block of 512 threads per sample: X[b] -> H1[b], H2[b], and OUT[b]
// (forward) or, TRAIN, the sample's loss
//   CE(softmax(OUT[0:4]), label) + lam * mask * mean_j (OUT[4+j] - off[j])^2
// and the gradients of the batch mean with respect to OUT, H2 and H1
// (dH2 = (W3^T dOUT) * [H2 > 0], dH1 = (W2^T dH2) * [H1 > 0]), all of a
// sample's chain in one launch.
// Bound by latency: the weights (144 KB) come from L2 once per sample.
// Layer 1 gives a warp four outputs, each lane 32 inputs of the sample in
// registers and 16-byte weight loads, all in flight together; the later
// layers give an output eight lanes, and their weights are asked for before
// layer 1 is summed.  One thread per output read W1 with a stride of 2 KB
// and summed 1024 terms in a chain: 54 us for 64 samples, and 18 us more
// in two kernels for the loss and the backward pass; a whole training step
// of 64 samples went from 79 to 18 us.
constexpr int MT = 512;

template <bool VEC, bool TRAIN>
__global__ void __launch_bounds__(MT) sample_kernel(const float *__restrict__ X, int B, const __nv_bfloat16 *__restrict__ P,
                                                    float *__restrict__ H1, float *__restrict__ H2,
                                                    float *__restrict__ OUT, LossArgs A)
{
    kernel_entry();
    __shared__ float s_h1[kHid], s_h2[kHid], s_o[kOut], s_d[kOut], s_dh2[kHid], s_part[MT / kHid][kHid];
    const int b = blockIdx.x, t = (int)threadIdx.x, lane = t & 31, warp = t >> 5;
    const float *x = X + row(b, kIn);
    constexpr int PW = kHid / (MT / 32);   // layer-1 outputs per warp
    constexpr int C = kIn / 256;           // 8 inputs per lane and chunk of 256
    float xv[C][8];
#pragma unroll
    for (int c = 0; c < C; ++c) {
        const int i = c * 256 + lane * 8;
        if constexpr (VEC) {
            const float4 u = __ldg(reinterpret_cast<const float4 *>(x + i)), v = __ldg(reinterpret_cast<const float4 *>(x + i) + 1);
            xv[c][0] = u.x, xv[c][1] = u.y, xv[c][2] = u.z, xv[c][3] = u.w;
            xv[c][4] = v.x, xv[c][5] = v.y, xv[c][6] = v.z, xv[c][7] = v.w;
        } else {
#pragma unroll
            for (int q = 0; q < 8; ++q) xv[c][q] = __ldg(x + i + q);
        }
    }
    const int o8 = t >> 3, l8 = t & 7;     // layers 2 and 3: output and its lane
    float w2[8], w3[8];
    weights8<VEC>(P, oW2 + o8 * kHid + l8 * 8, w2);
    weights8<VEC>(P, oW3 + o8 * kHid + l8 * 8, w3);
    float acc[PW];
#pragma unroll
    for (int u = 0; u < PW; ++u) {
        acc[u] = 0.0f;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            float w[8];
            weights8<VEC>(P, oW1 + (warp * PW + u) * kIn + c * 256 + lane * 8, w);
#pragma unroll
            for (int q = 0; q < 8; ++q) acc[u] = __fmaf_rn(w[q], xv[c][q], acc[u]);
        }
    }
#pragma unroll
    for (int u = 0; u < PW; ++u) {
        const float h = fmaxf(lanes_sum<32>(acc[u]) + wf(P, oB1 + warp * PW + u), 0.0f);
        if (lane == u) {
            s_h1[warp * PW + u] = h;
            H1[row(b, kHid) + warp * PW + u] = h;
        }
    }
    __syncthreads();
    {
        float a = 0.0f;
#pragma unroll
        for (int q = 0; q < 8; ++q) a = __fmaf_rn(w2[q], s_h1[l8 * 8 + q], a);
        const float h = fmaxf(lanes_sum<8>(a) + wf(P, oB2 + o8), 0.0f);
        if (l8 == 0) {
            s_h2[o8] = h;
            H2[row(b, kHid) + o8] = h;
        }
    }
    __syncthreads();
    {
        float a = 0.0f;
#pragma unroll
        for (int q = 0; q < 8; ++q) a = __fmaf_rn(w3[q], s_h2[l8 * 8 + q], a);
        a = lanes_sum<8>(a) + wf(P, oB3 + o8);
        if (l8 == 0) s_o[o8] = a;
        if (warp == 0) {   // the last kOut - 64 outputs: eight lanes each again
            const int o = kHid + (lane >> 3);
            weights8<VEC>(P, oW3 + o * kHid + l8 * 8, w3);
            a = 0.0f;
#pragma unroll
            for (int q = 0; q < 8; ++q) a = __fmaf_rn(w3[q], s_h2[l8 * 8 + q], a);
            a = lanes_sum<8>(a) + wf(P, oB3 + o);
            if (l8 == 0) s_o[o] = a;
        }
    }
    __syncthreads();
    if constexpr (!TRAIN) {
        if (t < kOut) OUT[row(b, kOut) + t] = s_o[t];
    } else {
        const float invB = 1.0f / (float)B, w = A.lam * A.mask[b];
        if (warp == 0) {   // loss, and the gradient of the logits
            const float mx = fmaxf(fmaxf(s_o[0], s_o[1]), fmaxf(s_o[2], s_o[3]));
            float e[4], z = 0.0f;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                e[k] = expf(s_o[k] - mx);
                z += e[k];
            }
            const int y = min(max(A.label[b], 0), 3);   // labels are 0..3; the clamp keeps a bad one in bounds
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (lane == k) {
                    s_d[k] = (e[k] / z - (k == y ? 1.0f : 0.0f)) * invB;
                    A.dOUT[row(b, kOut) + k] = s_d[k];
                }
            }
            const float d0 = s_o[4 + lane] - A.off[row(b, 64) + lane], d1 = s_o[36 + lane] - A.off[row(b, 64) + 32 + lane];
            const float l = lanes_sum<32>(w * d0 * d0 / 64.0f + w * d1 * d1 / 64.0f);
            if (lane == 0) A.loss[b] = logf(z) + mx - s_o[y] + l;
        } else if (warp < 3) {   // the gradient of the offsets
            const int j = t - 32;
            const float d = w * 2.0f * (s_o[4 + j] - A.off[row(b, 64) + j]) / 64.0f * invB;
            s_d[4 + j] = d;
            A.dOUT[row(b, kOut) + 4 + j] = d;
        }
        __syncthreads();
        constexpr int NP = MT / kHid;        // rows of a column's sum per thread: every NP-th
        const int col = t % kHid, part = t / kHid;
        float a = 0.0f;
#pragma unroll
        for (int j = part; j < kOut; j += NP) a = __fmaf_rn(wf(P, oW3 + j * kHid + col), s_d[j], a);
        s_part[part][col] = a;
        __syncthreads();
        if (t < kHid) {
            a = 0.0f;
#pragma unroll
            for (int q = 0; q < NP; ++q) a += s_part[q][t];
            const float g = s_h2[t] > 0.0f ? a : 0.0f;
            s_dh2[t] = g;
            A.dH2[row(b, kHid) + t] = g;
        }
        __syncthreads();
        a = 0.0f;
#pragma unroll
        for (int j = part; j < kHid; j += NP) a = __fmaf_rn(wf(P, oW2 + j * kHid + col), s_dh2[j], a);
        s_part[part][col] = a;
        __syncthreads();
        if (t < kHid) {
            a = 0.0f;
#pragma unroll
            for (int q = 0; q < NP; ++q) a += s_part[q][t];
            A.dH1[row(b, kHid) + t] = s_h1[t] > 0.0f ? a : 0.0f;
        }
    }
}

// One thread per parameter: its gradient summed over the batch, then the
// Adam step on the FP32 master weights and their BF16 copy, which is what
// the other kernels read.  Bound by latency (each thread's loads over the
// batch go out 16 at a time); the gradient stays in a register.
struct AdamArgs {
    float *Wm, *M, *V;
    __nv_bfloat16 *P;
    float lr, b1, b2, eps, c1, c2;
};

__global__ void __launch_bounds__(256) wgrad_adam_kernel(const float *__restrict__ X, int B, const float *__restrict__ H1,
                                                         const float *__restrict__ H2, const float *__restrict__ dH1,
                                                         const float *__restrict__ dH2, const float *__restrict__ dOUT,
                                                         AdamArgs A)
{
    kernel_entry();
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= kParams) return;
    // the parameter's factors: column d of the layer's output gradient, and
    // (weights) column x of its input
    const float *d, *x = nullptr;
    int ds, xs = 0;
    if (p < oW2) {
        d = dH1 + (p < oB1 ? p / kIn : p - oB1);
        ds = kHid;
        if (p < oB1) {
            x = X + p % kIn;
            xs = kIn;
        }
    } else if (p < oW3) {
        d = dH2 + (p < oB2 ? (p - oW2) / kHid : p - oB2);
        ds = kHid;
        if (p < oB2) {
            x = H1 + (p - oW2) % kHid;
            xs = kHid;
        }
    } else {
        d = dOUT + (p < oB3 ? (p - oW3) / kHid : p - oB3);
        ds = kOut;
        if (p < oB3) {
            x = H2 + (p - oW3) % kHid;
            xs = kHid;
        }
    }
    const float m0 = A.M[p], v0 = A.V[p], w0 = A.Wm[p];
    float g = 0.0f;
    if (x) {
#pragma unroll 16
        for (int b = 0; b < B; ++b) g = __fmaf_rn(__ldg(d + (int64_t)b * ds), __ldg(x + (int64_t)b * xs), g);
    } else {
#pragma unroll 16
        for (int b = 0; b < B; ++b) g += __ldg(d + (int64_t)b * ds);
    }
    const float m = A.b1 * m0 + (1.0f - A.b1) * g;
    const float v = A.b2 * v0 + (1.0f - A.b2) * g * g;
    A.M[p] = m;
    A.V[p] = v;
    const float w = w0 - A.lr * (m / A.c1) / (sqrtf(v / A.c2) + A.eps);
    A.Wm[p] = w;
    A.P[p] = __float2bfloat16_rn(w);
}

// 16-byte loads of the inputs and weights where both allow them.
inline bool vec16(const float *X, const void *P)
{
    return ((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(P)) & 15u) == 0;
}

}  // namespace

}  // namespace ch

using namespace ch;

extern "C" int32_t ch_mlp_param_count(void) { return mlp::kParams; }

extern "C" ch_status ch_kgon_features(const float *pts, int64_t n, float *feat, void *stream)
{
    if (!pts || !feat || n < 1 || (reinterpret_cast<uintptr_t>(pts) & 7u) || (reinterpret_cast<uintptr_t>(feat) & 3u))
        return CH_ERR_ARG;
    features_kernel<<<1, 1024, 0, reinterpret_cast<cudaStream_t>(stream)>>>(pts, n, feat);
    return cudaGetLastError() == cudaSuccess ? CH_OK : CH_ERR_CUDA;
}

extern "C" ch_status ch_mlp_forward(const float *X, int32_t B, const void *params, float *H1, float *H2, float *OUT,
                                    void *stream)
{
    if (!X || !params || !H1 || !H2 || !OUT || B < 1) return CH_ERR_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const __nv_bfloat16 *P = static_cast<const __nv_bfloat16 *>(params);
    if (vec16(X, params)) sample_kernel<true, false><<<B, MT, 0, st>>>(X, B, P, H1, H2, OUT, LossArgs{});
    else sample_kernel<false, false><<<B, MT, 0, st>>>(X, B, P, H1, H2, OUT, LossArgs{});
    return cudaGetLastError() == cudaSuccess ? CH_OK : CH_ERR_CUDA;
}

extern "C" ch_status ch_mlp_train_step(const float *X, int32_t B, const int32_t *label, const float *off,
                                       const float *mask, float lam, void *params, float *master, float *adam_m,
                                       float *adam_v, int32_t step, float lr, float *scratch, float *loss, void *stream)
{
    if (!X || !label || !off || !mask || !params || !master || !adam_m || !adam_v || !scratch || !loss || B < 1 ||
        step < 1)
        return CH_ERR_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    __nv_bfloat16 *P = static_cast<__nv_bfloat16 *>(params);
    // scratch: H1, H2 (B x 64 each), dOUT (B x 68), dH1, dH2 (B x 64 each)
    float *H1 = scratch, *H2 = H1 + row(B, kHid), *dOUT = H2 + row(B, kHid);
    float *dH1 = dOUT + row(B, kOut), *dH2 = dH1 + row(B, kHid);
    const LossArgs A{label, off, mask, lam, dOUT, dH1, dH2, loss};
    if (vec16(X, params)) sample_kernel<true, true><<<B, MT, 0, st>>>(X, B, P, H1, H2, nullptr, A);
    else sample_kernel<false, true><<<B, MT, 0, st>>>(X, B, P, H1, H2, nullptr, A);
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.0f - powf(b1, (float)step), c2 = 1.0f - powf(b2, (float)step);
    launch_next(wgrad_adam_kernel, (kParams + 255) / 256, 256, 0, st, X, B, H1, H2, dH1, dH2, dOUT,
                                                            AdamArgs{master, adam_m, adam_v, P, lr, b1, b2, 1e-8f, c1, c2});
    return cudaGetLastError() == cudaSuccess ? CH_OK : CH_ERR_CUDA;
}

// Floats of scratch for ch_mlp_train_step with a batch of B.  (It uses B (4
// kHid + kOut) of them; the number is the one that callers have always been
// given, with room for the outputs and the gradients.)
extern "C" int64_t ch_mlp_scratch_floats(int32_t B)
{
    return (int64_t)B * (4 * kHid + 2 * kOut) + kParams;
}
