// Hit-ranking MLP (12 -> 64 ReLU -> 1): bfloat16 conversion, forward, gradient
// of the mean binary cross-entropy, Adam.  FP32 arithmetic with bfloat16-rounded
// weights.  The batch reduction of the gradient is done in a fixed order
// (per-chunk compensated sums, then the chunk partials in order), so results do
// not depend on how blocks are scheduled.
#include <cuda_runtime.h>

#include <algorithm>

#include "mkf_internal.h"

namespace {

constexpr int kIn = MKF_MLP_IN;
constexpr int kHid = MKF_MLP_HIDDEN;
constexpr int kP = MKF_MLP_PARAMS;
constexpr int kOffB1 = kIn * kHid;
constexpr int kOffW2 = kOffB1 + kHid;
constexpr int kOffB2 = kOffW2 + kHid;
constexpr int kChunk = 256;  // samples per reduction chunk

// float -> bfloat16 bits, round to nearest, ties to even (NaN kept quiet)
__device__ __forceinline__ uint16_t to_bf16(float f) {
    const uint32_t u = __float_as_uint(f);
    if ((u & 0x7fffffffu) > 0x7f800000u) return static_cast<uint16_t>((u >> 16) | 0x40u);
    const uint32_t r = u + 0x7fffu + ((u >> 16) & 1u);
    return static_cast<uint16_t>(r >> 16);
}

__device__ __forceinline__ float from_bf16(uint16_t b) { return __uint_as_float(static_cast<uint32_t>(b) << 16); }

__global__ void to_bf16_kernel(const float *w, uint16_t *o, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) o[i] = to_bf16(w[i]);
}

__device__ __forceinline__ void load_weights(const uint16_t *wb, float *ws) {
    for (int i = threadIdx.x; i < kP; i += blockDim.x) ws[i] = from_bf16(wb[i]);
    __syncthreads();
}

__global__ void __launch_bounds__(128) forward_kernel(const uint16_t *wb, const float *feat, int n, float *logit) {
    __shared__ float ws[kP];
    load_weights(wb, ws);
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    float x[kIn];
#pragma unroll
    for (int k = 0; k < kIn; ++k) x[k] = feat[(int64_t)s * kIn + k];
    float z = ws[kOffB2];
    for (int j = 0; j < kHid; ++j) {
        float a = ws[kOffB1 + j];
#pragma unroll
        for (int k = 0; k < kIn; ++k) a = fmaf(ws[j * kIn + k], x[k], a);
        z = fmaf(ws[kOffW2 + j], fmaxf(a, 0.f), z);
    }
    logit[s] = z;
}

// Gradient of one chunk of samples, reduced over the chunk: block (x, y) takes
// chunk y and the kSlice hidden units of slice x.  First one thread per sample:
// forward, d(loss)/d(logit) = (sigmoid(z) - y) / n, the sample's loss and, for
// the slice's units, the activations and the pre-activation gradients, all kept
// in shared memory; then one thread per parameter of the slice sums its samples
// in order (compensated).  wf: FP32 weights, rounded here as to_bf16 does, or
// nullptr to take wb.
// Bound: latency (4096 samples are 16 chunks: too few blocks to fill the chip,
// and a chunk's compensated sum is 256 dependent steps of four additions, 2 us).
// Every slice therefore repeats the chunk's forward pass (1 us) so that 8 blocks
// work on a chunk, and nothing per sample goes through global memory: the
// activations and gradients written there by one kernel and read back by the
// next, one load per addition, made a training step of 4096 samples take 108 us
// (four kernels; 16.3 us with this one and finish_kernel, 12.1 us when both are
// launched while the kernel before them runs; bit for bit the same).
constexpr int kSlice = 8;
constexpr int kSlices = kHid / kSlice;
constexpr int kRow = kChunk + 4;  // a row of the transposed tiles: 16-byte aligned, rows 4 banks apart
constexpr int kSliceParams = kSlice * (kIn + 2);
static_assert(kHid % kSlice == 0 && kSliceParams + 2 <= kChunk && kChunk % 4 == 0, "one thread per parameter");

// Compensated (Kahan) sum in the order of the calls.
struct KahanSum {
    float sum = 0.f, comp = 0.f;
    __device__ __forceinline__ void add(float t) {
        const float yv = t - comp;
        const float tt = sum + yv;
        comp = (tt - sum) - yv;
        sum = tt;
    }
};

__global__ void __launch_bounds__(kChunk) chunk_grad_kernel(const uint16_t *wb, const float *wf, const float *feat,
                                                            const float *label, int n, float *part) {
    __shared__ __align__(16) float xs[kIn * kRow];     // features, [k][sample]
    __shared__ __align__(16) float hs[kSlice * kRow];  // the slice's activations, [unit][sample]
    __shared__ __align__(16) float ds[kSlice * kRow];  // the slice's pre-activation gradients
    __shared__ __align__(16) float gs[kChunk];
    __shared__ __align__(16) float ls[kChunk];
    __shared__ __align__(16) float ws[kP + 3];
    after_previous();
    const int tid = threadIdx.x;
    const int j0 = blockIdx.x * kSlice;
    const int s0 = blockIdx.y * kChunk, ns = min(kChunk, n - s0);
    for (int i = tid; i < kP; i += kChunk) ws[i] = from_bf16(wf ? to_bf16(wf[i]) : wb[i]);
    for (int i = tid; i < ns * kIn; i += kChunk) {
        const int s = i / kIn, k = i - s * kIn;
        xs[k * kRow + s] = feat[(int64_t)s0 * kIn + i];
    }
    __syncthreads();
    if (tid < ns) {
        float x[kIn];
#pragma unroll
        for (int k = 0; k < kIn; ++k) x[k] = xs[k * kRow + tid];
        float z = ws[kOffB2];
#pragma unroll 4
        for (int j = 0; j < kHid; ++j) {
            const float4 *row = reinterpret_cast<const float4 *>(ws + j * kIn);
            const float4 r0 = row[0], r1 = row[1], r2 = row[2];
            const float wr[kIn] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w, r2.x, r2.y, r2.z, r2.w};
            float a = ws[kOffB1 + j];
#pragma unroll
            for (int k = 0; k < kIn; ++k) a = fmaf(wr[k], x[k], a);
            const float h = fmaxf(a, 0.f);
            const int jj = j - j0;
            if (jj >= 0 && jj < kSlice) {
                hs[jj * kRow + tid] = h;
                ds[jj * kRow + tid] = a > 0.f ? 1.f : 0.f;  // ReLU mask, scaled below
            }
            z = fmaf(ws[kOffW2 + j], h, z);
        }
        const float y = label[s0 + tid];
        const float e = expf(-fabsf(z));
        const float sig = z >= 0.f ? 1.f / (1.f + e) : e / (1.f + e);
        const float g = (sig - y) / static_cast<float>(n);
        gs[tid] = g;
        ls[tid] = fmaxf(z, 0.f) - z * y + log1pf(e);
#pragma unroll
        for (int jj = 0; jj < kSlice; ++jj) ds[jj * kRow + tid] *= g * ws[kOffW2 + j0 + jj];
    }
    __syncthreads();
    // the slice's parameters: W1 rows, b1, w2; slice 0 also takes b2 and the loss
    if (tid >= kSliceParams + (blockIdx.x == 0 ? 2 : 0)) return;
    const float *a, *b = nullptr;  // the sum of a[s] b[s], or of a[s]
    int p;
    if (tid < kSlice * kIn) {
        const int jj = tid / kIn, k = tid - jj * kIn;
        a = ds + jj * kRow;
        b = xs + k * kRow;
        p = (j0 + jj) * kIn + k;
    } else if (tid < kSlice * (kIn + 1)) {
        const int jj = tid - kSlice * kIn;
        a = ds + jj * kRow;
        p = kOffB1 + j0 + jj;
    } else if (tid < kSliceParams) {
        const int jj = tid - kSlice * (kIn + 1);
        a = gs;
        b = hs + jj * kRow;
        p = kOffW2 + j0 + jj;
    } else {
        a = tid == kSliceParams ? gs : ls;
        p = tid == kSliceParams ? kOffB2 : kP;
    }
    KahanSum acc;
    int s = 0;
    for (; s + 4 <= ns; s += 4) {
        const float4 u = *reinterpret_cast<const float4 *>(a + s);
        float4 v = make_float4(1.f, 1.f, 1.f, 1.f);
        if (b) v = *reinterpret_cast<const float4 *>(b + s);
        acc.add(__fmul_rn(u.x, v.x));
        acc.add(__fmul_rn(u.y, v.y));
        acc.add(__fmul_rn(u.z, v.z));
        acc.add(__fmul_rn(u.w, v.w));
    }
    for (; s < ns; ++s) acc.add(__fmul_rn(a[s], b ? b[s] : 1.f));
    part[(int64_t)blockIdx.y * (kP + 1) + p] = acc.sum;
}

// Sum the chunk partials in chunk order; optionally apply Adam.  Bound: latency;
// what needs no partial (the bias corrections' powers) is done before the wait.
__global__ void __launch_bounds__(128) finish_kernel(const float *part, int nchunks, int n, float *grad, float *loss,
                                                     float *w, float *m, float *v, int t, mkf_adam hp, uint16_t *wb) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p > kP) return;
    const float bias1 = 1.f - powf(hp.beta1, static_cast<float>(t));
    const float bias2 = 1.f - powf(hp.beta2, static_cast<float>(t));
    after_previous();
    KahanSum acc;
#pragma unroll 8
    for (int c = 0; c < nchunks; ++c) acc.add(part[(int64_t)c * (kP + 1) + p]);
    const float sum = acc.sum;
    if (p == kP) {
        if (loss) *loss = sum / static_cast<float>(n);
        return;
    }
    if (grad) grad[p] = sum;
    if (w) {
        const float mm = hp.beta1 * m[p] + (1.f - hp.beta1) * sum;
        const float vv = hp.beta2 * v[p] + (1.f - hp.beta2) * sum * sum;
        m[p] = mm;
        v[p] = vv;
        const float mh = mm / bias1;
        const float vh = vv / bias2;
        const float nw = w[p] - hp.lr * mh / (sqrtf(vh) + hp.eps);
        w[p] = nw;
        wb[p] = to_bf16(nw);
    }
}

// wb: bfloat16 weights, or nullptr to round the FP32 weights w (a training step).
mkf_status run_grad(mkf_ctx *ctx, const uint16_t *wb, const float *feat, const float *label, int n, float *grad,
                    float *loss, float *w, float *m, float *v, int t, const mkf_adam *hp, uint16_t *wb_out) {
    const int nchunks = (n + kChunk - 1) / kChunk;
    void *scratch = nullptr;
    mkf_status st = mkf_scratch(ctx, (size_t)nchunks * (kP + 1) * sizeof(float), &scratch);
    if (st != MKF_OK) return st;
    float *part = static_cast<float *>(scratch);
    cudaStream_t s = ctx->stream;
    MKF_CUDA_TRY(mkf_launch(chunk_grad_kernel, dim3(kSlices, nchunks), kChunk, 0, s, wb, wb ? nullptr : w, feat, label,
                            n, part));
    mkf_adam h = hp ? *hp : mkf_adam{0.f, 0.f, 0.f, 0.f};
    MKF_CUDA_TRY(mkf_launch(finish_kernel, (kP + 1 + 127) / 128, 128, 0, s, part, nchunks, n, grad, loss, w, m, v, t, h,
                            wb_out));
    return MKF_OK;
}

}  // namespace

extern "C" mkf_status mkf_mlp_to_bf16(mkf_ctx *ctx, const float *w, uint16_t *w_bf16, int32_t n) {
    if (!ctx || n < 0 || (n > 0 && (!w || !w_bf16))) return MKF_ERR_ARG;
    if (n == 0) return MKF_OK;
    DeviceGuard g(ctx->device);
    if (!g.ok) return MKF_ERR_CUDA;
    to_bf16_kernel<<<(n + 255) / 256, 256, 0, ctx->stream>>>(w, w_bf16, n);
    MKF_CUDA_TRY(cudaGetLastError());
    return MKF_OK;
}

extern "C" mkf_status mkf_mlp_forward(mkf_ctx *ctx, const uint16_t *w_bf16, const float *feat, int32_t n,
                                      float *logit) {
    if (!ctx || !w_bf16 || n < 0 || (n > 0 && (!feat || !logit))) return MKF_ERR_ARG;
    if (n == 0) return MKF_OK;
    DeviceGuard g(ctx->device);
    if (!g.ok) return MKF_ERR_CUDA;
    forward_kernel<<<(n + 127) / 128, 128, 0, ctx->stream>>>(w_bf16, feat, n, logit);
    MKF_CUDA_TRY(cudaGetLastError());
    return MKF_OK;
}

extern "C" mkf_status mkf_mlp_grad(mkf_ctx *ctx, const uint16_t *w_bf16, const float *feat, const float *label,
                                   int32_t n, float *grad, float *loss) {
    if (!ctx || !w_bf16 || !feat || !label || !grad || n < 1) return MKF_ERR_ARG;
    DeviceGuard g(ctx->device);
    if (!g.ok) return MKF_ERR_CUDA;
    return run_grad(ctx, w_bf16, feat, label, n, grad, loss, nullptr, nullptr, nullptr, 0, nullptr, nullptr);
}

extern "C" mkf_status mkf_mlp_train_step(mkf_ctx *ctx, const float *feat, const float *label, int32_t n, float *w,
                                         float *m, float *v, int32_t t, const mkf_adam *hp, uint16_t *w_bf16,
                                         float *loss) {
    if (!ctx || !feat || !label || !w || !m || !v || !hp || !w_bf16 || n < 1 || t < 1) return MKF_ERR_ARG;
    DeviceGuard g(ctx->device);
    if (!g.ok) return MKF_ERR_CUDA;
    return run_grad(ctx, nullptr, feat, label, n, nullptr, loss, w, m, v, t, hp, w_bf16);
}
