// mlp.cu -- the troubled-cell network of the gated form: training kernels
// (loss + gradient, Adam), inference on sample batches, and the generation of
// labelled training samples from a solver state.
//
// Network: 5 -> 32 -> 32 -> 1, ReLU hidden layers, logistic output; input is
// a 5-cell stencil of one sensor field (mixture density or pressure)
// normalised as (v_k - v_i)/max_k |v_k - v_i|; a stencil whose variation is
// at most MFC_GATE_FLOOR |v_i| is flat and never shown to the network.
// Parameters (1281 floats): W1[32][5], b1[32], W2[32][32], b2[32], w3[32],
// b3.  Label of a cell and direction: troubled (1) when, for some primitive
// field whose stencil is not flat, a nonlinear WENO5-JS weight at either
// face departs from its linear weight by more than tau relative; smooth (0)
// otherwise (below the floor the two reconstructions differ by round-off).  Loss: weighted binary
// cross-entropy on the logit (positive-class weight wp).  Training is FP32;
// the samples are formed in FP64 from reference-order primitives (this file is
// built with -fmad=false).
#include <cuda_runtime.h>
#include <math.h>

#include "mfc.h"
#include "mfc_internal.cuh"
#include "sweep.cuh"

namespace mfc5 {

constexpr int kMlpH = 32, kMlpIn = 5;
constexpr int kMlpParams = kMlpH * kMlpIn + kMlpH + kMlpH * kMlpH + kMlpH + kMlpH + 1;
constexpr int OW1 = 0, OB1 = kMlpH * kMlpIn, OW2 = OB1 + kMlpH, OB2 = OW2 + kMlpH * kMlpH, OW3 = OB2 + kMlpH,
              OB3 = OW3 + kMlpH;
static_assert(kMlpParams == 1281, "parameter layout");

__device__ __forceinline__ float softplusf(float t) { return t > 0.f ? t + log1pf(expf(-t)) : log1pf(expf(t)); }

// Loss and gradient over n samples.  Lane l of a warp is neuron l: it holds row
// l of W1 and W2, column l of W2 and the gradient sums of row l of W1, column l
// of W2 and its biases in registers, and a warp takes four samples at a time
// through both passes.  What every lane needs of the others (h1 for the forward
// pass, d2 for the backward one) goes through 512 bytes of the warp's own
// shared memory, read as broadcast 16-byte words: one such load feeds four
// FMAs forward, and eight backward (d1 and dW2).  A block's warps add their sums in
// shared memory, one atomic per parameter and block follows.  One block per
// SM: a batch of 8192 gives a warp four or eight samples, and more blocks would
// only add atomics (64 blocks: 14.5 us a call).  Measured per call with the
// zeroing, batch 8192: 20.5 us with one thread per sample, its activations in
// local memory and 128 samples per block, 10.4 now, of which the launches'
// latencies are about half.
constexpr int kGradWarps = 8, kGradGroup = 4;

__global__ void __launch_bounds__(kGradWarps * 32)
mlp_grad_kernel(const float* __restrict__ X, const float* __restrict__ Y, long long n,
                const float* __restrict__ theta, float wp, float inv_n, float* grad, float* loss) {
    __shared__ float part[kGradWarps][kMlpParams + 1];   // and the loss
    __shared__ float4 act[kGradWarps][kGradGroup][kMlpH / 4];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    // the weights come through shared memory (W2 in rows of 33, so that rows and
    // columns are read without bank conflicts): read from global memory by every
    // lane, the rows alone cost 8192 L1 accesses per block
    float* th = part[0];
    for (int k = threadIdx.x; k < kMlpParams; k += blockDim.x) {
        const int o = k < OW2 || k >= OB2 ? k : OW2 + (k - OW2) / kMlpH * (kMlpH + 1) + (k - OW2) % kMlpH;
        th[o + (k >= OB2 ? kMlpH : 0)] = __ldg(theta + k);
    }
    __syncthreads();
    float w1[kMlpIn], w2r[kMlpH], w2c[kMlpH];
#pragma unroll
    for (int i = 0; i < kMlpIn; ++i) w1[i] = th[OW1 + lane * kMlpIn + i];
#pragma unroll
    for (int i = 0; i < kMlpH; ++i) {
        w2r[i] = th[OW2 + lane * (kMlpH + 1) + i];
        w2c[i] = th[OW2 + i * (kMlpH + 1) + lane];
    }
    const float b1 = th[OB1 + lane], b2 = th[OB2 + kMlpH + lane], w3 = th[OW3 + kMlpH + lane];
    const float b3 = th[OB3 + kMlpH];
    __syncthreads();   // part is written again at the end
    float g1[kMlpIn] = {}, g2[kMlpH] = {}, gb1 = 0.f, gb2 = 0.f, g3 = 0.f, gb3 = 0.f, lsum = 0.f;
    float4(*my)[kMlpH / 4] = act[wib];
    const long long step = (long long)gridDim.x * kGradWarps * kGradGroup;
    for (long long base = ((long long)blockIdx.x * kGradWarps + wib) * kGradGroup; base < n; base += step) {
        float x[kGradGroup][kMlpIn], h1[kGradGroup], h2[kGradGroup], z[kGradGroup], dz[kGradGroup];
#pragma unroll
        for (int s = 0; s < kGradGroup; ++s) {
            const long long k = base + s < n ? base + s : n - 1;   // past the end: weight 0 below
            float a = b1;
#pragma unroll
            for (int i = 0; i < kMlpIn; ++i) {
                x[s][i] = __ldg(X + k * kMlpIn + i);
                a = fmaf(w1[i], x[s][i], a);
            }
            h1[s] = fmaxf(a, 0.f);
            reinterpret_cast<float*>(my[s])[lane] = h1[s];
        }
        __syncwarp();
#pragma unroll
        for (int s = 0; s < kGradGroup; ++s) {
            float a = b2;
#pragma unroll
            for (int q = 0; q < kMlpH / 4; ++q) {
                const float4 v = my[s][q];
                a = fmaf(w2r[4 * q], v.x, a);
                a = fmaf(w2r[4 * q + 1], v.y, a);
                a = fmaf(w2r[4 * q + 2], v.z, a);
                a = fmaf(w2r[4 * q + 3], v.w, a);
            }
            h2[s] = fmaxf(a, 0.f);
            z[s] = w3 * h2[s];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int s = 0; s < kGradGroup; ++s) z[s] += __shfl_xor_sync(0xffffffffu, z[s], o);
        // lane s finishes sample s (every lane holds the sums)
        {
            const int s = lane & (kGradGroup - 1);
            float zs = z[0];
#pragma unroll
            for (int k = 1; k < kGradGroup; ++k) zs = s == k ? z[k] : zs;
            zs += b3;
            const bool in = base + s < n;
            const float y = __ldg(Y + (in ? base + s : n - 1));
            const float sg = 1.f / (1.f + expf(-zs));
            const float d = in ? (wp * y * (sg - 1.f) + (1.f - y) * sg) * inv_n : 0.f;
            if (lane < kGradGroup) {
                gb3 += d;
                if (in) lsum += wp * y * softplusf(-zs) + (1.f - y) * softplusf(zs);
            }
#pragma unroll
            for (int k = 0; k < kGradGroup; ++k) dz[k] = __shfl_sync(0xffffffffu, d, k);
        }
        __syncwarp();   // h1 has been read by every lane
#pragma unroll
        for (int s = 0; s < kGradGroup; ++s) {
            const float d2 = h2[s] > 0.f ? dz[s] * w3 : 0.f;
            reinterpret_cast<float*>(my[s])[lane] = d2;
            gb2 += d2;
            g3 = fmaf(dz[s], h2[s], g3);
        }
        __syncwarp();
#pragma unroll
        for (int s = 0; s < kGradGroup; ++s) {
            float a = 0.f;
#pragma unroll
            for (int q = 0; q < kMlpH / 4; ++q) {
                const float4 v = my[s][q];
                a = fmaf(w2c[4 * q], v.x, a);
                a = fmaf(w2c[4 * q + 1], v.y, a);
                a = fmaf(w2c[4 * q + 2], v.z, a);
                a = fmaf(w2c[4 * q + 3], v.w, a);
                g2[4 * q] = fmaf(v.x, h1[s], g2[4 * q]);
                g2[4 * q + 1] = fmaf(v.y, h1[s], g2[4 * q + 1]);
                g2[4 * q + 2] = fmaf(v.z, h1[s], g2[4 * q + 2]);
                g2[4 * q + 3] = fmaf(v.w, h1[s], g2[4 * q + 3]);
            }
            const float d1 = h1[s] > 0.f ? a : 0.f;
            gb1 += d1;
#pragma unroll
            for (int i = 0; i < kMlpIn; ++i) g1[i] = fmaf(d1, x[s][i], g1[i]);
        }
        __syncwarp();   // d2 has been read before the next samples' h1 is written
    }
    float* mine = part[wib];
#pragma unroll
    for (int i = 0; i < kMlpIn; ++i) mine[OW1 + lane * kMlpIn + i] = g1[i];
#pragma unroll
    for (int j = 0; j < kMlpH; ++j) mine[OW2 + j * kMlpH + lane] = g2[j];
    mine[OB1 + lane] = gb1;
    mine[OB2 + lane] = gb2;
    mine[OW3 + lane] = g3;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        gb3 += __shfl_xor_sync(0xffffffffu, gb3, o);
        lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
    }
    if (lane == 0) {
        mine[OB3] = gb3;
        mine[kMlpParams] = lsum;
    }
    __syncthreads();
    for (int k = threadIdx.x; k <= kMlpParams; k += blockDim.x) {
        float a = part[0][k];
#pragma unroll
        for (int w = 1; w < kGradWarps; ++w) a += part[w][k];
        if (k < kMlpParams) atomicAdd(&grad[k], a);
        else atomicAdd(loss, a * inv_n);
    }
}

// grad and loss start from zero
__global__ void mlp_zero_kernel(float* grad, float* loss) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < kMlpParams) grad[k] = 0.f;
    if (k == kMlpParams) *loss = 0.f;
}

__global__ void mlp_adam_kernel(float* theta, const float* __restrict__ g, float* m, float* v, float lr, float b1,
                                float b2, float eps, float c1, float c2) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= kMlpParams) return;
    float gk = g[k];
    float mk = b1 * m[k] + (1.f - b1) * gk;
    float vk = b2 * v[k] + (1.f - b2) * gk * gk;
    m[k] = mk;
    v[k] = vk;
    theta[k] -= lr * (mk / c1) / (sqrtf(vk / c2) + eps);
}

// Logits: one thread per sample, activations in registers (both layers fully
// unrolled), weight rows read from shared memory as broadcast 16-byte words --
// four FMAs a load, where one-word loads bound the kernel.
__global__ void __launch_bounds__(128) mlp_forward_kernel(const float* __restrict__ X, long long n,
                                                          const float* __restrict__ theta, float* z) {
    __shared__ float4 w2[kMlpH][kMlpH / 4];
    __shared__ float4 w1[kMlpH][2];   // W1[j][0..4], b1[j], b2[j], w3[j]
    for (int k = threadIdx.x; k < kMlpH * kMlpH; k += blockDim.x)
        reinterpret_cast<float*>(w2)[k] = __ldg(theta + OW2 + k);
    for (int k = threadIdx.x; k < kMlpH * 8; k += blockDim.x) {
        const int j = k >> 3, i = k & 7;
        reinterpret_cast<float*>(w1)[k] =
            __ldg(theta + (i < kMlpIn ? OW1 + j * kMlpIn + i : (i == 5 ? OB1 : (i == 6 ? OB2 : OW3)) + j));
    }
    __syncthreads();
    const float b3 = __ldg(theta + OB3);
    for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < n;
         s += (long long)gridDim.x * blockDim.x) {
        float x[kMlpIn], h[kMlpH];
#pragma unroll
        for (int i = 0; i < kMlpIn; ++i) x[i] = __ldg(X + s * kMlpIn + i);
#pragma unroll
        for (int j = 0; j < kMlpH; ++j) {
            const float4 a = w1[j][0], b = w1[j][1];
            float v = fmaf(a.x, x[0], b.y);
            v = fmaf(a.y, x[1], v);
            v = fmaf(a.z, x[2], v);
            v = fmaf(a.w, x[3], v);
            h[j] = fmaxf(fmaf(b.x, x[4], v), 0.f);
        }
        float out = b3;
#pragma unroll 4
        for (int j = 0; j < kMlpH; ++j) {
            const float4 b = w1[j][1];
            float v = b.z;
#pragma unroll
            for (int q = 0; q < kMlpH / 4; ++q) {
                const float4 w = w2[j][q];
                v = fmaf(w.x, h[4 * q], v);
                v = fmaf(w.y, h[4 * q + 1], v);
                v = fmaf(w.z, h[4 * q + 2], v);
                v = fmaf(w.w, h[4 * q + 3], v);
            }
            out = fmaf(b.w, fmaxf(v, 0.f), out);
        }
        z[s] = out;
    }
}

// Training samples from an FP64 state: for every cell c and direction d,
// two samples (density sensor, pressure sensor) sharing the cell's label.
// Layout: sample index ((d * ncell + c) * 2 + sensor).
template <int NDIM>
__global__ void gate_samples_kernel(const double* __restrict__ q, int n0, int n1, int n2, int per0, int per1,
                                    int per2, Eos eos, double eps, float tau, float* X, float* Y) {
    using FL = Fields<NDIM>;
    const long long nc = (long long)n0 * n1 * n2;
    const int n[3] = {n0, n1, n2}, per[3] = {per0, per1, per2};
    const long long stride[3] = {1, n0, (long long)n0 * n1};
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < nc * NDIM;
         t += (long long)gridDim.x * blockDim.x) {
        const int d = (int)(t / nc);
        const long long c = t % nc;
        const int idx = (int)((c / stride[d]) % n[d]);
        const long long base = c - (long long)idx * stride[d];
        double w[5][FL::NEQ];
        for (int k = 0; k < 5; ++k) {
            long long cc = base + (long long)bc_index(idx - 2 + k, n[d], per[d]) * stride[d];
            double v[FL::NEQ];
            for (int f = 0; f < FL::NEQ; ++f) v[f] = q[f * nc + cc];
            exact::cons_to_prim<NDIM>(eos, v, w[k]);   // reference-order primitives
        }
        bool troubled = false;
        const double dm[3] = {0.1, 0.6, 0.3}, dp[3] = {0.3, 0.6, 0.1};
        for (int f = 0; f < FL::NEQ; ++f) {
            const double c13 = 13.0 / 12.0;
            double v0 = w[0][f], v1 = w[1][f], v2 = w[2][f], v3 = w[3][f], v4 = w[4][f];
            double mf = 0.0;
            for (int k = 0; k < 5; ++k) mf = fmax(mf, fabs(w[k][f] - v2));
            if (!(mf > MFC_GATE_FLOOR * fabs(v2))) continue;   // flat: round-off only
            double b[3];
            b[0] = c13 * (v0 - 2.0 * v1 + v2) * (v0 - 2.0 * v1 + v2) + 0.25 * (v0 - 4.0 * v1 + 3.0 * v2) * (v0 - 4.0 * v1 + 3.0 * v2);
            b[1] = c13 * (v1 - 2.0 * v2 + v3) * (v1 - 2.0 * v2 + v3) + 0.25 * (v1 - v3) * (v1 - v3);
            b[2] = c13 * (v2 - 2.0 * v3 + v4) * (v2 - 2.0 * v3 + v4) + 0.25 * (3.0 * v2 - 4.0 * v3 + v4) * (3.0 * v2 - 4.0 * v3 + v4);
            double am[3], ap[3], sm = 0.0, sp = 0.0;
            for (int k = 0; k < 3; ++k) {
                double s2 = (eps + b[k]) * (eps + b[k]);
                am[k] = dm[k] / s2;
                ap[k] = dp[k] / s2;
                sm += am[k];
                sp += ap[k];
            }
            for (int k = 0; k < 3; ++k) {
                troubled |= fabs(am[k] / sm - dm[k]) > tau * dm[k];
                troubled |= fabs(ap[k] / sp - dp[k]) > tau * dp[k];
            }
        }
        for (int sensor = 0; sensor < 2; ++sensor) {
            double v[5], m = 0.0;
            for (int k = 0; k < 5; ++k) v[k] = sensor == 0 ? w[k][0] + w[k][1] : w[k][FL::IE];
            for (int k = 0; k < 5; ++k) m = fmax(m, fabs(v[k] - v[2]));
            long long sidx = t * 2 + sensor;
            const bool live = m > MFC_GATE_FLOOR * fabs(v[2]);
            for (int k = 0; k < 5; ++k) X[sidx * 5 + k] = live ? float((v[k] - v[2]) / m) : 0.f;
            Y[sidx] = !live ? -1.f : (troubled ? 1.f : 0.f);
        }
    }
}

cudaError_t launch_gate_samples(int ndim, const double* q, const int* n, const int* periodic, const Eos& e,
                                double eps, float tau, float* X, float* Y, cudaStream_t s) {
    long long total = (long long)n[0] * n[1] * n[2] * ndim;
    long long blocks = (total + 255) / 256;
    if (blocks > 152LL * 64) blocks = 152LL * 64;
    if (blocks < 1) blocks = 1;
    if (ndim == 1)
        gate_samples_kernel<1><<<(unsigned)blocks, 256, 0, s>>>(q, n[0], n[1], n[2], periodic[0], periodic[1],
                                                                periodic[2], e, eps, tau, X, Y);
    else if (ndim == 2)
        gate_samples_kernel<2><<<(unsigned)blocks, 256, 0, s>>>(q, n[0], n[1], n[2], periodic[0], periodic[1],
                                                                periodic[2], e, eps, tau, X, Y);
    else
        gate_samples_kernel<3><<<(unsigned)blocks, 256, 0, s>>>(q, n[0], n[1], n[2], periodic[0], periodic[1],
                                                                periodic[2], e, eps, tau, X, Y);
    return cudaGetLastError();
}

}  // namespace mfc5

using namespace mfc5;

extern "C" int mfc_mlp_nparams(void) { return kMlpParams; }

extern "C" int mfc_mlp_loss_grad(const float* X, const float* Y, long long n, const float* theta, float pos_weight,
                                 float* grad, float* loss, void* cuda_stream) {
    if (!X || !Y || !theta || !grad || !loss || n <= 0 || !(pos_weight > 0.f)) return MFC_EINVAL;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    mlp_zero_kernel<<<(kMlpParams + 256) / 256, 256, 0, s>>>(grad, loss);
    if (cudaGetLastError() != cudaSuccess) return MFC_ECUDA;
    constexpr int kPerBlock = kGradWarps * kGradGroup;
    long long blocks = (n + kPerBlock - 1) / kPerBlock;
    if (blocks > 152) blocks = 152;
    mlp_grad_kernel<<<(unsigned)blocks, kGradWarps * 32, 0, s>>>(X, Y, n, theta, pos_weight, 1.0f / (float)n, grad,
                                                                 loss);
    return cudaGetLastError() == cudaSuccess ? MFC_OK : MFC_ECUDA;
}

extern "C" int mfc_mlp_adam(float* theta, const float* grad, float* m, float* v, int t, float lr, float beta1,
                            float beta2, float eps, void* cuda_stream) {
    if (!theta || !grad || !m || !v || t < 1) return MFC_EINVAL;
    // bias corrections 1 - beta^t formed in FP64: in FP32, 1 - 0.999^t loses
    // about 1e-5 relative to cancellation
    float c1 = (float)(1.0 - pow((double)beta1, (double)t));
    float c2 = (float)(1.0 - pow((double)beta2, (double)t));
    mlp_adam_kernel<<<(kMlpParams + 255) / 256, 256, 0, (cudaStream_t)cuda_stream>>>(theta, grad, m, v, lr, beta1,
                                                                                      beta2, eps, c1, c2);
    return cudaGetLastError() == cudaSuccess ? MFC_OK : MFC_ECUDA;
}

extern "C" int mfc_mlp_forward(const float* X, long long n, const float* theta, float* z, void* cuda_stream) {
    if (!X || !theta || !z || n <= 0) return MFC_EINVAL;
    long long blocks = (n + 127) / 128;
    if (blocks > 152LL * 16) blocks = 152LL * 16;
    mlp_forward_kernel<<<(unsigned)blocks, 128, 0, (cudaStream_t)cuda_stream>>>(X, n, theta, z);
    return cudaGetLastError() == cudaSuccess ? MFC_OK : MFC_ECUDA;
}
