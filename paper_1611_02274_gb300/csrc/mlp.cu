// mlp.cu -- training and inference kernels of the learned proposal.
//
// The network maps the features of a system's initial state (log |y_k| per
// component and the raw parameter, normalised) to (log h0, log sigma,
// log cost): the first accepted step size and the power-method
// spectral-radius bound the FP64 solver found for it, and the number of
// right-hand-side evaluations the whole integration took (the key that
// orders a batch longest-first).  Weights are kept as FP32 masters and used in
// BF16 (round-to-nearest-even) for every forward pass; all sums are FP32.
//
// Losses: squared error on log h0 and log cost; pinball (quantile tau = 0.9)
// on log sigma, so the network leans to over-estimating sigma -- the stable
// side for RKC.
//
// Kernels:
//   k_mlp_grad    tiles of 32 samples through the network as small FP32
//                 matrix products in shared memory; forward, loss, backward
//                 and the weight-gradient sums in registers, one row of
//                 partial sums per block.
//   k_reduce      the blocks' sums in a fixed order, then bias-corrected
//                 Adam on the FP32 masters and their BF16 copies (training)
//                 or the mean gradient.
//   k_mlp_apply   one thread per sample, weights in shared memory.
//   k_pack        the inference copy the integration kernels evaluate
//                 in-kernel (mlp_warp.cuh): B fragments of mma.m16n8k16 in
//                 fragment-major order, biases, normalisation and the box.
//
// A NaN target is no target (no loss, no gradient, not in the statistics),
// so records with a spectral-radius target only train beside full ones.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstddef>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <random>
#include <string>
#include <vector>

#include "batchode.h"
#include "mlp.cuh"
#include "mlp_warp.cuh"

namespace bode {
int set_last_error(int code, const char* msg);
void clear_last_error();
}  // namespace bode

using namespace bode;

namespace {

constexpr int kH = kMlpHidden;
constexpr float kTau = 0.9f;  // pinball quantile of the log-sigma loss

struct Mlp {
    int n_in = 0;
    int nparams = 0;
    int dev = 0, sms = 0;
    float* master = nullptr;
    __nv_bfloat16* w16 = nullptr;
    float* m = nullptr;
    float* v = nullptr;
    float* part = nullptr;  // per-block gradient sums, grow-only
    size_t part_bytes = 0;
    float* loss = nullptr;  // device scalar
    MlpNorm norm;
    bool has_norm = false;
    int64_t step = 0;
    MlpPacked* packed = nullptr;  // inference copy for the integration kernels
};

constexpr float kBoxMargin = 0.05f;  // in-kernel proposals: the training box widened by 5 % of its width

std::mutex g_mu;
std::map<int32_t, Mlp> g_mlps;
int32_t g_next = 1;

int fail(int code, const char* fmt, ...) __attribute__((format(printf, 2, 3)));
int fail(int code, const char* fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    return set_last_error(code, buf);
}

int cuda_fail(cudaError_t e, const char* what) { return fail(ODE_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e)); }

// ---------------------------------------------------------------- kernels

// Weights (BF16 -> float) into shared memory.
__device__ void load_weights(const __nv_bfloat16* w16, float* sw, int np) {
    for (int k = threadIdx.x; k < np; k += blockDim.x) sw[k] = __bfloat162float(w16[k]);
    __syncthreads();
}

__device__ __forceinline__ float loss_grad(int o, float p, float t, float* loss) {
    if (isnan(t)) return 0.0f;  // no target
    if (o != 1) {  // squared error: log h0, log cost
        const float r = p - t;
        *loss += r * r;
        return 2.0f * r;
    }
    const float r = t - p;  // pinball: tau r for r > 0, (tau - 1) r otherwise
    *loss += r > 0.0f ? kTau * r : (kTau - 1.0f) * r;
    return r > 0.0f ? -kTau : (1.0f - kTau);
}

// Training step, first kernel: per-block sums of the gradient of the summed
// loss over samples [0, n) (rows of X / Y, optionally through a permutation)
// and of the loss, to part[block][mlp_nparams + 1].
//
// A block takes tiles of kTile samples through the network at once, as small
// FP32 matrix products out of shared memory: a layer's outputs in 4 neurons
// x 2 samples per thread, the 64 x 64 weight gradient in 4 x 4 elements per
// thread held in registers over all of a block's tiles.  A batch of 4096
// rows is 128 blocks, one per SM.  The products are 31 kFLOP a row, 2 us of
// the FP32 pipe per batch; the kernel before it walked its samples one after
// another with one thread per neuron and six barriers a sample, 32 samples
// deep, and added 5,300 terms per block with atomics.  Rows of the tiles are
// kRow floats long, so that the rows a warp reads at once start in different
// banks.  The whole call on
// 262,144 rows, 2 epochs of 64 batches: 22.0 -> 3.96 ms, of which the host's
// two shuffles take about 1.5.
constexpr int kTile = 32;
constexpr int kTrainThreads = 256;
constexpr int kRow = kH + 4;
constexpr int kXRow = 52;  // inputs padded to 16, 32 or 48 columns
// floats of a block's row of sums: the parameters, the loss, whole 16-byte words
__host__ __device__ constexpr int part_stride(int n_in) { return (mlp_nparams(n_in) + 1 + 3) / 4 * 4; }
struct TrainSmem {
    float w1t[(kMlpMaxIn + 3) / 4 * 4 * kRow];  // W1 by input, zero rows up to a multiple of 4
    float w2[kH * kRow];          // W2 by output neuron
    float w2t[kH * kRow];         // W2 by input neuron
    float w3[kMlpOut * kH];
    float b1[kH], b2[kH], b3[4];
    float x[kTile * kXRow];
    float a1[kTile * kRow], a2[kTile * kRow], d1[kTile * kRow], d2[kTile * kRow];
    float g3[kTile * 4];
    float red[kTrainThreads / 32];
};

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void st4(float* p, const float* v) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
// acc[r][c] += w[c] * v over a run of K inputs (K a multiple of 4): w rows are
// kRow long and hold four outputs, the two samples' inputs are rows v0 and v1
__device__ __forceinline__ void mac_inputs(const float* w, const float* v0, const float* v1, int K, float (&acc)[2][4]) {
#pragma unroll 4
    for (int k = 0; k < K; k += 4) {
        const float4 a4 = ld4(v0 + k), b4 = ld4(v1 + k);
        const float av[4] = {a4.x, a4.y, a4.z, a4.w}, bv[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 q = ld4(w + (k + i) * kRow);
            const float a = av[i], b = bv[i];
            acc[0][0] = fmaf(q.x, a, acc[0][0]);
            acc[0][1] = fmaf(q.y, a, acc[0][1]);
            acc[0][2] = fmaf(q.z, a, acc[0][2]);
            acc[0][3] = fmaf(q.w, a, acc[0][3]);
            acc[1][0] = fmaf(q.x, b, acc[1][0]);
            acc[1][1] = fmaf(q.y, b, acc[1][1]);
            acc[1][2] = fmaf(q.z, b, acc[1][2]);
            acc[1][3] = fmaf(q.w, b, acc[1][3]);
        }
    }
}

__global__ void __launch_bounds__(kTrainThreads) k_mlp_grad(const __nv_bfloat16* __restrict__ w16, const MlpNorm norm,
                                                             int n_in, const float* __restrict__ X,
                                                             const float* __restrict__ Y,
                                                             const int32_t* __restrict__ perm, int64_t n,
                                                             float* __restrict__ part) {
    extern __shared__ __align__(16) unsigned char raw[];
    TrainSmem& sm = *reinterpret_cast<TrainSmem*>(raw);
    const int tid = threadIdx.x;
    // Everything a block reads is asked for before anything is waited for:
    // the chain row index -> inputs is the only one that is two reads long.
    // Eight threads a row: the row's inputs, and its targets on three of them.
    const int rs = tid >> 3, rl = tid & 7;
    auto row_of = [&](int64_t t) -> int64_t {
        const int64_t q = t * kTile + rs;
        return q < n ? (perm ? (int64_t)perm[q] : q) : -1;
    };
    const int64_t row0 = row_of(blockIdx.x);
    // weights (BF16 -> FP32)
    constexpr int kW1 = (kH * kMlpMaxIn + kTrainThreads - 1) / kTrainThreads, kW2 = kH * kH / 8 / kTrainThreads;
    __nv_bfloat16 v1[kW1], v3[2], vb[2];
    uint4 v2[kW2];
#pragma unroll
    for (int i = 0; i < kW2; ++i) {  // lanes take consecutive rows (128 bytes): no bank conflicts in shared memory
        const int q = tid + i * kTrainThreads, j = q & (kH - 1), k = (q / kH) * 8;
        v2[i] = *reinterpret_cast<const uint4*>(w16 + mlp_w2(n_in) + j * kH + k);
    }
#pragma unroll
    for (int i = 0; i < kW1; ++i)
        if (tid + i * kTrainThreads < kH * n_in) v1[i] = w16[mlp_w1(n_in) + tid + i * kTrainThreads];
    if (tid < kMlpOut * kH) v3[0] = w16[mlp_w3(n_in) + tid];
    if (tid < kMlpOut) v3[1] = w16[mlp_b3(n_in) + tid];
    if (tid < kH) {
        vb[0] = w16[mlp_b1(n_in) + tid];
        vb[1] = w16[mlp_b2(n_in) + tid];
    }
#pragma unroll
    for (int i = 0; i < kW1; ++i) {
        const int e = tid + i * kTrainThreads;
        if (e < kH * n_in) sm.w1t[(e % n_in) * kRow + e / n_in] = __bfloat162float(v1[i]);
    }
    for (int e = n_in * kRow + tid; e < (n_in + 3) / 4 * 4 * kRow; e += kTrainThreads) sm.w1t[e] = 0.0f;
#pragma unroll
    for (int q = 0; q < kW2; ++q) {
        const int j = (tid + q * kTrainThreads) & (kH - 1), k = ((tid + q * kTrainThreads) / kH) * 8;
        const uint32_t word[4] = {v2[q].x, v2[q].y, v2[q].z, v2[q].w};
        float v[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            v[2 * i] = __uint_as_float(word[i] << 16);
            v[2 * i + 1] = __uint_as_float(word[i] & 0xffff0000u);
        }
        st4(sm.w2 + j * kRow + k, v);
        st4(sm.w2 + j * kRow + k + 4, v + 4);
#pragma unroll
        for (int i = 0; i < 8; ++i) sm.w2t[(k + i) * kRow + j] = v[i];
    }
    if (tid < kMlpOut * kH) sm.w3[tid] = __bfloat162float(v3[0]);
    if (tid < kMlpOut) sm.b3[tid] = __bfloat162float(v3[1]);
    if (tid < kH) {
        sm.b1[tid] = __bfloat162float(vb[0]);
        sm.b2[tid] = __bfloat162float(vb[1]);
    }

    const int jg = 4 * (tid & 15), s0 = 2 * (tid >> 4);     // layer products: 4 neurons x 2 samples
    const int jt = 4 * (tid >> 4), kt = 4 * (tid & 15);     // W2 gradient: 4 x 4 elements, rows along the lanes
    const int jr = tid & 63, role = tid >> 6;               // W1 gradient: a neuron, a quarter of the inputs
    const int kper = 4 * ((n_in + 15) / 16);                // inputs per quarter: 4, 8 or 12
    float gW2[4][4] = {}, gW1[12] = {}, gB = 0.0f, gW3[kMlpOut] = {}, lsum = 0.0f;
    const int64_t tiles = (n + kTile - 1) / kTile;
    for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        // normalised inputs, zero past n_in and past the last row
        const int64_t r = t == blockIdx.x ? row0 : row_of(t);
        float xin[6], target = 0.0f;
#pragma unroll
        for (int i = 0; i < 6; ++i) xin[i] = r >= 0 && rl + 8 * i < n_in ? X[r * n_in + rl + 8 * i] : 0.0f;
        if (r >= 0 && rl < kMlpOut) target = Y[r * kMlpOut + rl];
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            const int k = rl + 8 * i;
            if (k < 4 * kper)
                sm.x[rs * kXRow + k] = r >= 0 && k < n_in ? (xin[i] - norm.x_mean[k < kMlpMaxIn ? k : 0]) /
                                                                norm.x_scale[k < kMlpMaxIn ? k : 0]
                                                          : 0.0f;
        }
        __syncthreads();
        float z1[2][4], z2[2][4], out[4];
        {
            const float4 b = ld4(sm.b1 + jg);
            for (int r = 0; r < 2; ++r) z1[r][0] = b.x, z1[r][1] = b.y, z1[r][2] = b.z, z1[r][3] = b.w;
            mac_inputs(sm.w1t + jg, sm.x + s0 * kXRow, sm.x + (s0 + 1) * kXRow, (n_in + 3) / 4 * 4, z1);
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
#pragma unroll
            for (int c = 0; c < 4; ++c) out[c] = silu(z1[r][c]);
            st4(sm.a1 + (s0 + r) * kRow + jg, out);
        }
        __syncthreads();
        {
            const float4 b = ld4(sm.b2 + jg);
            for (int r = 0; r < 2; ++r) z2[r][0] = b.x, z2[r][1] = b.y, z2[r][2] = b.z, z2[r][3] = b.w;
            mac_inputs(sm.w2t + jg, sm.a1 + s0 * kRow, sm.a1 + (s0 + 1) * kRow, kH, z2);
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
#pragma unroll
            for (int c = 0; c < 4; ++c) out[c] = silu(z2[r][c]);
            st4(sm.a2 + (s0 + r) * kRow + jg, out);
        }
        __syncthreads();
        {  // outputs: eight lanes a sample, then the loss and its gradient
            const int s = rs, l = rl;
            float z3[kMlpOut] = {};
#pragma unroll
            for (int i = 0; i < kH / 8; ++i) {
                const float a = sm.a2[s * kRow + l + 8 * i];
#pragma unroll
                for (int o = 0; o < kMlpOut; ++o) z3[o] = fmaf(sm.w3[o * kH + l + 8 * i], a, z3[o]);
            }
#pragma unroll
            for (int o = 0; o < kMlpOut; ++o) {
                for (int d = 4; d > 0; d >>= 1) z3[o] += __shfl_xor_sync(0xffffffffu, z3[o], d);
                if (l == o) {
                    float g = 0.0f;
                    if (r >= 0) g = loss_grad(o, z3[o] + sm.b3[o], (target - norm.y_mean[o]) / norm.y_scale[o], &lsum);
                    sm.g3[s * 4 + o] = g;
                }
            }
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const float g0 = sm.g3[(s0 + r) * 4], g1 = sm.g3[(s0 + r) * 4 + 1], g2 = sm.g3[(s0 + r) * 4 + 2];
#pragma unroll
            for (int c = 0; c < 4; ++c)
                out[c] = (sm.w3[jg + c] * g0 + sm.w3[kH + jg + c] * g1 + sm.w3[2 * kH + jg + c] * g2) * silu_grad(z2[r][c]);
            st4(sm.d2 + (s0 + r) * kRow + jg, out);
        }
        __syncthreads();
        {
            float back[2][4] = {};
            mac_inputs(sm.w2 + jg, sm.d2 + s0 * kRow, sm.d2 + (s0 + 1) * kRow, kH, back);
#pragma unroll
            for (int r = 0; r < 2; ++r) {
#pragma unroll
                for (int c = 0; c < 4; ++c) out[c] = back[r][c] * silu_grad(z1[r][c]);
                st4(sm.d1 + (s0 + r) * kRow + jg, out);
            }
        }
#pragma unroll 4
        for (int s = 0; s < kTile; ++s) {
            const float4 d = ld4(sm.d2 + s * kRow + jt), a = ld4(sm.a1 + s * kRow + kt);
            const float dv[4] = {d.x, d.y, d.z, d.w}, av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) gW2[r][c] = fmaf(dv[r], av[c], gW2[r][c]);
        }
        __syncthreads();
#pragma unroll 2
        for (int s = 0; s < kTile; ++s) {  // a warp has one role
            const float d = sm.d1[s * kRow + jr];
            const float* xr = sm.x + s * kXRow + role * kper;
#pragma unroll
            for (int q = 0; q < 3; ++q)
                if (4 * q < kper) {
                    const float4 v = ld4(xr + 4 * q);
                    gW1[4 * q] = fmaf(d, v.x, gW1[4 * q]);
                    gW1[4 * q + 1] = fmaf(d, v.y, gW1[4 * q + 1]);
                    gW1[4 * q + 2] = fmaf(d, v.z, gW1[4 * q + 2]);
                    gW1[4 * q + 3] = fmaf(d, v.w, gW1[4 * q + 3]);
                }
            if (role == 0) gB += d;
            if (role == 1) gB += sm.d2[s * kRow + jr];
            if (role == 2) {
                const float a = sm.a2[s * kRow + jr];
#pragma unroll
                for (int o = 0; o < kMlpOut; ++o) gW3[o] = fmaf(sm.g3[s * 4 + o], a, gW3[o]);
            }
            if (role == 3 && jr < kMlpOut) gB += sm.g3[s * 4 + jr];
        }
        __syncthreads();  // the tile is read before the next one is written
    }
    // the block's row of sums, written in whole sectors: W2 as 16-byte words
    // of consecutive lanes, W1 by way of shared memory (scattered 4-byte
    // stores cost the kernel more than its products did)
    float* p = part + (int64_t)blockIdx.x * part_stride(n_in);
#pragma unroll
    for (int i = 0; i < 12; ++i)
        if (i < kper && role * kper + i < n_in) sm.w1t[(role * kper + i) * kRow + jr] = gW1[i];
#pragma unroll
    for (int r = 0; r < 4; ++r) st4(p + mlp_w2(n_in) + (jt + r) * kH + kt, gW2[r]);
    __syncthreads();
    for (int e = tid; e < kH * n_in; e += kTrainThreads) p[mlp_w1(n_in) + e] = sm.w1t[(e % n_in) * kRow + e / n_in];
    if (role == 0) p[mlp_b1(n_in) + jr] = gB;
    if (role == 1) p[mlp_b2(n_in) + jr] = gB;
    if (role == 2)
#pragma unroll
        for (int o = 0; o < kMlpOut; ++o) p[mlp_w3(n_in) + o * kH + jr] = gW3[o];
    if (role == 3 && jr < kMlpOut) p[mlp_b3(n_in) + jr] = gB;
    for (int d = 16; d > 0; d >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, d);
    if ((tid & 31) == 0) sm.red[tid >> 5] = lsum;
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < kTrainThreads / 32; ++w) lsum += sm.red[w];
        p[mlp_nparams(n_in)] = lsum;
    }
}

// Second kernel: the blocks' sums in a fixed order (eight lanes of blocks a
// parameter), 32 parameters per block; the word past the parameters is the
// loss.  ADAM: bias-corrected Adam on the mean gradient, writes the FP32
// master and its BF16 copy and adds to *loss; otherwise the mean gradient to
// out and the summed loss to *loss.
template <bool ADAM>
__global__ void __launch_bounds__(256) k_reduce(const float* __restrict__ part, int blocks, int stride, int np, float n_rows,
                                                float* __restrict__ out, float* master, __nv_bfloat16* w16, float* m,
                                                float* v, float lr, float b1, float b2, float eps, float c1, float c2,
                                                float* loss) {
    __shared__ float sums[8][32];
    const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5, k = blockIdx.x * 32 + lane;
    float s = 0.0f, m0 = 0.0f, v0 = 0.0f, w0 = 0.0f;
    if (ADAM && slice == 0 && k < np) {  // asked for before the sums are waited for
        m0 = m[k];
        v0 = v[k];
        w0 = master[k];
    }
    if (k <= np)
#pragma unroll 16
        for (int b = slice; b < blocks; b += 8) s += part[(int64_t)b * stride + k];
    sums[slice][lane] = s;
    __syncthreads();
    if (slice || k > np) return;
    for (int q = 1; q < 8; ++q) s += sums[q][lane];
    if (k == np) {
        *loss = ADAM ? *loss + s : s;
        return;
    }
    if constexpr (!ADAM) {
        out[k] = s / n_rows;
        return;
    }
    const float g = s * (1.0f / n_rows);
    const float mk = b1 * m0 + (1.0f - b1) * g;
    const float vk = b2 * v0 + (1.0f - b2) * g * g;
    m[k] = mk;
    v[k] = vk;
    const float w = w0 - lr * (mk / c1) / (sqrtf(vk / c2) + eps);
    master[k] = w;
    w16[k] = __float2bfloat16_rn(w);
}

__global__ void k_to_bf16(const float* master, __nv_bfloat16* w16, int np) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < np) w16[k] = __float2bfloat16_rn(master[k]);
}

// Forward pass of one normalised input row; returns the de-normalised
// outputs (log h0, log sigma, log cost).
__device__ void mlp_forward(const float* sw, int n_in, const float* x, const MlpNorm& norm, float* out) {
    const float* W1 = sw + mlp_w1(n_in);
    const float* B1 = sw + mlp_b1(n_in);
    const float* W2 = sw + mlp_w2(n_in);
    const float* B2 = sw + mlp_b2(n_in);
    const float* W3 = sw + mlp_w3(n_in);
    const float* B3 = sw + mlp_b3(n_in);
    float a1[kH];
#pragma unroll
    for (int jj = 0; jj < kH; ++jj) {
        float z = B1[jj];
        for (int k = 0; k < n_in; ++k) z += W1[jj * n_in + k] * x[k];
        a1[jj] = silu(z);
    }
    float o[kMlpOut];
#pragma unroll
    for (int q = 0; q < kMlpOut; ++q) o[q] = B3[q];
    for (int jj = 0; jj < kH; ++jj) {
        float z = B2[jj];
#pragma unroll
        for (int k = 0; k < kH; ++k) z += W2[jj * kH + k] * a1[k];
        const float a2 = silu(z);
#pragma unroll
        for (int q = 0; q < kMlpOut; ++q) o[q] += W3[q * kH + jj] * a2;
    }
#pragma unroll
    for (int q = 0; q < kMlpOut; ++q) out[q] = o[q] * norm.y_scale[q] + norm.y_mean[q];
}

// Outputs for feature rows X [n][n_in] (raw features, normalised here).
__global__ void k_mlp_apply(const __nv_bfloat16* w16, const MlpNorm norm, int n_in, const float* X, int64_t n,
                            float* out) {
    extern __shared__ float sw[];
    load_weights(w16, sw, mlp_nparams(n_in));
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    float x[kMlpMaxIn];
    for (int k = 0; k < n_in; ++k) x[k] = (X[r * n_in + k] - norm.x_mean[k]) / norm.x_scale[k];
    mlp_forward(sw, n_in, x, norm, out + r * kMlpOut);
}

// Proposals for an SoA batch: features log max(|y_k|, 1e-30) and the raw
// parameter; NaN outputs (no proposal) outside the training input box
// (widened by `margin` of its width) or when not finite.  The predicted
// cost (optional) is written wherever it is finite.
__global__ void k_mlp_propose(const __nv_bfloat16* w16, const MlpNorm norm, int n_in, int64_t nsys, int neq,
                              const double* y0, const double* params, float margin, float* h0, float* sigma0,
                              float* cost) {
    extern __shared__ float sw[];
    load_weights(w16, sw, mlp_nparams(n_in));
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nsys) return;
    float x[kMlpMaxIn];
    bool inside = true;
    for (int k = 0; k < n_in; ++k) {
        const double raw = k < neq ? log(fmax(fabs(y0[i + nsys * (int64_t)k]), 1e-30)) : params[i];
        const float xr = (float)raw;
        const float w = norm.x_max[k] - norm.x_min[k];
        if (!(xr >= norm.x_min[k] - margin * w && xr <= norm.x_max[k] + margin * w)) inside = false;
        x[k] = (xr - norm.x_mean[k]) / norm.x_scale[k];
    }
    float out[kMlpOut];
    mlp_forward(sw, n_in, x, norm, out);
    const float h = expf(out[0]), s = expf(out[1]);
    const bool ok = inside && isfinite(h) && isfinite(s) && h > 0.f && s > 0.f;
    h0[i] = ok ? h : __int_as_float(0x7fffffff);
    sigma0[i] = ok ? s : __int_as_float(0x7fffffff);
    if (cost) {
        const float c = expf(out[2]);
        cost[i] = isfinite(c) ? c : __int_as_float(0x7fffffff);
    }
}

// Per-block partial sums / extrema / counts of the finite values of the
// feature and target columns.
__global__ void k_stats(const float* X, const float* Y, int64_t n, int n_in, double* part) {
    const int F = n_in + kMlpOut;
    const int f = threadIdx.x;  // one column per thread
    if (f >= F) return;
    double s = 0.0, ss = 0.0, cnt = 0.0;
    float lo = 3.0e38f, hi = -3.0e38f;
    for (int64_t r = blockIdx.x; r < n; r += gridDim.x) {
        const float x = f < n_in ? X[r * n_in + f] : Y[r * kMlpOut + (f - n_in)];
        if (!isfinite(x)) continue;
        s += x;
        ss += (double)x * x;
        cnt += 1.0;
        lo = fminf(lo, x);
        hi = fmaxf(hi, x);
    }
    double* p = part + ((int64_t)blockIdx.x * F + f) * 5;
    p[0] = s;
    p[1] = ss;
    p[2] = lo;
    p[3] = hi;
    p[4] = cnt;
}

// The inference copy: B fragments (lane l of n-tile nt, k-step ks holds
// W[8 nt + l / 4][16 ks + 2 (l % 4) + {0, 1, 8, 9}], BF16 pairs, the lower
// column in the low half), zero outside the layer; biases as the BF16
// values the other kernels use, widened to FP32.
__global__ void k_pack(const __nv_bfloat16* __restrict__ w16, int n_in, MlpPacked* out) {
    const uint16_t* w = reinterpret_cast<const uint16_t*>(w16);
    auto el = [&](int off, int rows, int cols, int r, int c) -> uint32_t {
        return (r < rows && c < cols) ? (uint32_t)w[off + r * cols + c] : 0u;
    };
    auto frag = [&](int off, int rows, int cols, int KS, int idx) {
        const int nt = idx / (KS * 32), ks = (idx / 32) % KS, l = idx % 32;
        const int r = 8 * nt + (l >> 2), c = 16 * ks + 2 * (l & 3);
        return make_uint2(el(off, rows, cols, r, c) | (el(off, rows, cols, r, c + 1) << 16),
                          el(off, rows, cols, r, c + 8) | (el(off, rows, cols, r, c + 9) << 16));
    };
    for (int k = threadIdx.x; k < 8 * kMlpWarpKs1 * 32; k += blockDim.x)
        out->w1[k] = frag(mlp_w1(n_in), kH, n_in, kMlpWarpKs1, k);
    for (int k = threadIdx.x; k < 8 * 4 * 32; k += blockDim.x) out->w2[k] = frag(mlp_w2(n_in), kH, kH, 4, k);
    for (int k = threadIdx.x; k < 4 * 32; k += blockDim.x) out->w3[k] = frag(mlp_w3(n_in), kMlpOut, kH, 4, k);
    for (int k = threadIdx.x; k < kH; k += blockDim.x) {
        out->b1[k] = __bfloat162float(w16[mlp_b1(n_in) + k]);
        out->b2[k] = __bfloat162float(w16[mlp_b2(n_in) + k]);
    }
    if (threadIdx.x < 8) out->b3[threadIdx.x] = threadIdx.x < kMlpOut ? __bfloat162float(w16[mlp_b3(n_in) + threadIdx.x]) : 0.0f;
}

// Outputs 0 and 1 of raw feature rows through the in-kernel evaluation:
// one warp per 32 rows (KS k-steps of 16 inputs), the BF16 features staged
// in a shared-memory row per thread as the integration kernels stage them.
template <int KS>
__global__ void __launch_bounds__(128) k_mlp_apply_warp(const MlpPacked* __restrict__ net, const float* __restrict__ X,
                                                         int64_t n, float* __restrict__ out) {
    constexpr int kStride = 8 * KS + 1;  // words per row (odd: fewer bank conflicts)
    __shared__ uint32_t rows[128 * kStride];
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool have = r < n;
    const unsigned take = __ballot_sync(0xffffffffu, have);
    const int n_in = net->n_in;
    uint32_t* mine = rows + threadIdx.x * kStride;
    uint16_t* fr = reinterpret_cast<uint16_t*>(mine);
    for (int k = 0; k < 16 * KS; ++k)
        fr[k] = to_bf16((have && k < n_in) ? (X[r * n_in + k] - net->x_mean[k]) * net->x_iscale[k] : 0.0f);
    __syncwarp();
    float o0 = 0.0f, o1 = 0.0f;
    mlp_warp_eval<KS>(net, take, mine, kStride, o0, o1);
    if (!have) return;
    out[2 * r] = o0 * net->y_scale[0] + net->y_mean[0];
    out[2 * r + 1] = o1 * net->y_scale[1] + net->y_mean[1];
}

size_t apply_smem(int n_in) { return sizeof(float) * mlp_nparams(n_in); }

int get(int32_t h, Mlp** out) {
    auto it = g_mlps.find(h);
    if (it == g_mlps.end()) return fail(ODE_ERR_HANDLE, "unknown mlp handle %d", h);
    *out = &it->second;
    return ODE_OK;
}

// Rebuilds the inference copy from the BF16 weights and the normalisation
// (after every change of either); synchronous on s.
int refresh_packed(Mlp& net, cudaStream_t s) {
    if (!net.packed) return ODE_OK;
    k_pack<<<1, 256, 0, s>>>(net.w16, net.n_in, net.packed);
    MlpPacked h;  // the host-built part: normalisation and the widened box
    std::memset(&h, 0, sizeof(h));
    for (int k = 0; k < kMlpMaxIn; ++k) {
        h.x_mean[k] = net.norm.x_mean[k];
        h.x_iscale[k] = 1.0f / net.norm.x_scale[k];
        const float w = net.norm.x_max[k] - net.norm.x_min[k];
        h.x_lo[k] = net.norm.x_min[k] - kBoxMargin * w;
        h.x_hi[k] = net.norm.x_max[k] + kBoxMargin * w;
    }
    for (int k = 0; k < kMlpOut; ++k) {
        h.y_mean[k] = net.norm.y_mean[k];
        h.y_scale[k] = net.norm.y_scale[k];
    }
    h.n_in = net.n_in;
    const size_t off = offsetof(MlpPacked, x_mean);
    cudaError_t e = cudaMemcpyAsync(reinterpret_cast<char*>(net.packed) + off, reinterpret_cast<const char*>(&h) + off,
                                    sizeof(MlpPacked) - off, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e == cudaSuccess) e = cudaGetLastError();
    return e == cudaSuccess ? ODE_OK : cuda_fail(e, "network inference copy");
}

// blocks a gradient over n rows takes: a tile each, at most two per SM
int grad_blocks(const Mlp& net, int64_t n) {
    return (int)std::min<int64_t>((n + kTile - 1) / kTile, 2 * (int64_t)net.sms);
}

// room for the block sums of gradients over up to n rows
int reserve_part(Mlp& net, int64_t n) {
    const size_t need = sizeof(float) * (size_t)grad_blocks(net, n) * part_stride(net.n_in);
    if (net.part_bytes >= need) return ODE_OK;
    cudaFree(net.part);
    net.part = nullptr;
    net.part_bytes = 0;
    if (cudaMalloc(&net.part, need) != cudaSuccess) return fail(ODE_ERR_NOMEM, "gradient buffer of %zu bytes", need);
    net.part_bytes = need;
    return ODE_OK;
}

// block sums of the gradient of the summed loss over n rows (device X, Y)
cudaError_t run_grad(Mlp& net, const float* X, const float* Y, const int32_t* perm, int64_t n, cudaStream_t s) {
    k_mlp_grad<<<grad_blocks(net, n), kTrainThreads, sizeof(TrainSmem), s>>>(net.w16, net.norm, net.n_in, X, Y, perm, n,
                                                                              net.part);
    return cudaGetLastError();
}

}  // namespace

namespace bode {
// The inference copy of network `handle` for an integration whose systems
// have n_in - 1 components (ODE_ERR_HANDLE / ODE_ERR_ARG otherwise).
int mlp_packed_for(int32_t handle, int n_in, const MlpPacked** out) {
    std::lock_guard<std::mutex> lk(g_mu);
    Mlp* net;
    int rc = get(handle, &net);
    if (rc) return rc;
    if (net->n_in != n_in) return fail(ODE_ERR_ARG, "network takes %d inputs, the systems have %d + 1", net->n_in, n_in - 1);
    *out = net->packed;
    return ODE_OK;
}
}  // namespace bode

extern "C" {

int ode_mlp_create(int32_t n_in, uint64_t seed, int32_t* handle) {
    clear_last_error();
    if (!handle) return fail(ODE_ERR_ARG, "handle is NULL");
    if (n_in < 1 || n_in > kMlpMaxIn) return fail(ODE_ERR_ARG, "n_in must be in [1, %d]", kMlpMaxIn);
    Mlp net;
    net.n_in = n_in;
    net.nparams = mlp_nparams(n_in);
    cudaError_t e = cudaGetDevice(&net.dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&net.sms, cudaDevAttrMultiProcessorCount, net.dev);
    if (e == cudaSuccess)  // above the default dynamic shared-memory limit: opt in
        e = cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TrainSmem));
    if (e != cudaSuccess) return cuda_fail(e, "device set-up");
    // Glorot-uniform weights, zero biases
    std::vector<float> w(net.nparams, 0.0f);
    std::mt19937_64 rng(seed);
    auto fill = [&](int off, int rows, int cols) {
        const float a = std::sqrt(6.0f / (float)(rows + cols));
        std::uniform_real_distribution<float> u(-a, a);
        for (int k = 0; k < rows * cols; ++k) w[off + k] = u(rng);
    };
    fill(mlp_w1(n_in), kH, n_in);
    fill(mlp_w2(n_in), kH, kH);
    fill(mlp_w3(n_in), kMlpOut, kH);
    const size_t nb = sizeof(float) * net.nparams;
    e = cudaMalloc(&net.master, nb);
    if (e == cudaSuccess) e = cudaMalloc(&net.w16, sizeof(__nv_bfloat16) * net.nparams);
    if (e == cudaSuccess) e = cudaMalloc(&net.m, nb);
    if (e == cudaSuccess) e = cudaMalloc(&net.v, nb);
    if (e == cudaSuccess) e = cudaMalloc(&net.loss, sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc(&net.packed, sizeof(MlpPacked));
    if (e != cudaSuccess) return fail(ODE_ERR_NOMEM, "mlp allocation failed");
    cudaMemcpy(net.master, w.data(), nb, cudaMemcpyHostToDevice);
    cudaMemset(net.m, 0, nb);
    cudaMemset(net.v, 0, nb);
    k_to_bf16<<<(net.nparams + 255) / 256, 256>>>(net.master, net.w16, net.nparams);
    for (int k = 0; k < kMlpMaxIn; ++k) {
        net.norm.x_mean[k] = 0.f;
        net.norm.x_scale[k] = 1.f;
        net.norm.x_min[k] = -3.0e38f;
        net.norm.x_max[k] = 3.0e38f;
    }
    for (int k = 0; k < kMlpOut; ++k) {
        net.norm.y_mean[k] = 0.f;
        net.norm.y_scale[k] = 1.f;
    }
    e = cudaDeviceSynchronize();
    if (e != cudaSuccess) return cuda_fail(e, "mlp initialisation");
    if (int rc = refresh_packed(net, nullptr)) return rc;
    std::lock_guard<std::mutex> lk(g_mu);
    *handle = g_next++;
    g_mlps[*handle] = net;
    return ODE_OK;
}

int ode_mlp_release(int32_t handle) {
    clear_last_error();
    std::lock_guard<std::mutex> lk(g_mu);
    Mlp* net;
    int rc = get(handle, &net);
    if (rc) return rc;
    cudaFree(net->master);
    cudaFree(net->w16);
    cudaFree(net->m);
    cudaFree(net->v);
    cudaFree(net->part);
    cudaFree(net->loss);
    cudaFree(net->packed);
    g_mlps.erase(handle);
    return ODE_OK;
}

int ode_mlp_fit_normalization(int32_t handle, const float* X, const float* Y, int64_t n, void* stream) {
    clear_last_error();
    std::lock_guard<std::mutex> lk(g_mu);
    Mlp* net;
    int rc = get(handle, &net);
    if (rc) return rc;
    if (!X || !Y || n < 2) return fail(ODE_ERR_ARG, "need device X, Y and n >= 2");
    const int F = net->n_in + kMlpOut;
    const int blocks = 1024;
    double* part = nullptr;
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = cudaMalloc(&part, sizeof(double) * blocks * F * 5);
    if (e != cudaSuccess) return fail(ODE_ERR_NOMEM, "statistics buffer");
    k_stats<<<blocks, 64, 0, s>>>(X, Y, n, net->n_in, part);
    std::vector<double> h((size_t)blocks * F * 5);
    e = cudaMemcpyAsync(h.data(), part, sizeof(double) * h.size(), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(part);
    if (e != cudaSuccess) return cuda_fail(e, "statistics");
    for (int f = 0; f < F; ++f) {
        double sum = 0, sq = 0, lo = 3e38, hi = -3e38, cnt = 0;
        for (int b = 0; b < blocks; ++b) {
            const double* p = &h[((size_t)b * F + f) * 5];
            sum += p[0];
            sq += p[1];
            lo = std::min(lo, p[2]);
            hi = std::max(hi, p[3]);
            cnt += p[4];
        }
        if (cnt < 2) {  // no statistics: identity normalisation, unbounded box
            sum = sq = 0;
            cnt = 1;
            lo = -3e38;
            hi = 3e38;
        }
        const double mean = sum / cnt;
        const double sd = std::sqrt(std::max(sq / cnt - mean * mean, 0.0));
        const float scale = (float)(sd > 1e-12 ? sd : 1.0);
        if (f < net->n_in) {
            net->norm.x_mean[f] = (float)mean;
            net->norm.x_scale[f] = scale;
            net->norm.x_min[f] = (float)lo;
            net->norm.x_max[f] = (float)hi;
        } else {
            net->norm.y_mean[f - net->n_in] = (float)mean;
            net->norm.y_scale[f - net->n_in] = scale;
        }
    }
    net->has_norm = true;
    return refresh_packed(*net, s);
}

int ode_mlp_gradient(int32_t handle, const float* X, const float* Y, int64_t n, float* grad_out, float* loss_out,
                     void* stream) {
    clear_last_error();
    std::lock_guard<std::mutex> lk(g_mu);
    Mlp* net;
    int rc = get(handle, &net);
    if (rc) return rc;
    if (!X || !Y || !grad_out || n < 1) return fail(ODE_ERR_ARG, "need device X, Y, grad_out and n >= 1");
    cudaStream_t s = (cudaStream_t)stream;
    if ((rc = reserve_part(*net, n))) return rc;
    cudaError_t e = run_grad(*net, X, Y, nullptr, n, s);
    if (e != cudaSuccess) return cuda_fail(e, "gradient kernel");
    // mean over the rows
    k_reduce<false><<<net->nparams / 32 + 1, 256, 0, s>>>(net->part, grad_blocks(*net, n), part_stride(net->n_in), net->nparams, (float)n, grad_out,
                                                          nullptr, nullptr, nullptr, nullptr, 0, 0, 0, 0, 1, 1, net->loss);
    float l = 0;
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(&l, net->loss, sizeof(float), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(e, "gradient reduction");
    if (loss_out) *loss_out = l / (float)n;
    return ODE_OK;
}

int ode_mlp_train(int32_t handle, const float* X, const float* Y, int64_t n, const ode_train_opts* o,
                  float* loss_history, void* stream) {
    clear_last_error();
    std::lock_guard<std::mutex> lk(g_mu);
    Mlp* net;
    int rc = get(handle, &net);
    if (rc) return rc;
    if (!X || !Y || !o || n < 1) return fail(ODE_ERR_ARG, "need device X, Y, options and n >= 1");
    if (o->epochs < 1 || o->batch < 1 || !(o->lr > 0)) return fail(ODE_ERR_ARG, "need epochs >= 1, batch >= 1, lr > 0");
    if (!net->has_norm) return fail(ODE_ERR_ARG, "call ode_mlp_fit_normalization first");
    cudaStream_t s = (cudaStream_t)stream;
    if ((rc = reserve_part(*net, std::min<int64_t>(n, o->batch)))) return rc;
    int32_t* perm = nullptr;  // the epoch's permutation, then the epochs' losses
    cudaError_t e = cudaMalloc(&perm, sizeof(int32_t) * (size_t)(n + o->epochs));
    if (e != cudaSuccess) return fail(ODE_ERR_NOMEM, "permutation buffer");
    float* losses = reinterpret_cast<float*>(perm + n);
    std::vector<int32_t> hp(n);
    std::mt19937_64 rng(o->seed);
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    e = cudaMemsetAsync(losses, 0, sizeof(float) * o->epochs, s);
    for (int ep = 0; ep < o->epochs && e == cudaSuccess; ++ep) {
        // shuffled while the previous epoch's batches run
        for (int64_t k = 0; k < n; ++k) hp[k] = (int32_t)k;
        std::shuffle(hp.begin(), hp.end(), rng);
        e = cudaMemcpyAsync(perm, hp.data(), sizeof(int32_t) * n, cudaMemcpyHostToDevice, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);  // the copy has read hp
        for (int64_t b0 = 0; b0 < n && e == cudaSuccess; b0 += o->batch) {
            const int64_t bn = std::min<int64_t>(o->batch, n - b0);
            e = run_grad(*net, X, Y, perm + b0, bn, s);
            net->step += 1;
            const float c1 = 1.0f - std::pow(b1, (float)net->step), c2 = 1.0f - std::pow(b2, (float)net->step);
            if (e != cudaSuccess) break;
            k_reduce<true><<<net->nparams / 32 + 1, 256, 0, s>>>(net->part, grad_blocks(*net, bn), part_stride(net->n_in), net->nparams, (float)bn,
                                                                 nullptr, net->master, net->w16, net->m, net->v, o->lr, b1,
                                                                 b2, eps, c1, c2, losses + ep);
            e = cudaGetLastError();
        }
    }
    std::vector<float> l(o->epochs);
    if (e == cudaSuccess) e = cudaMemcpyAsync(l.data(), losses, sizeof(float) * o->epochs, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
        cudaFree(perm);
        return cuda_fail(e, "training");
    }
    for (int ep = 0; loss_history && ep < o->epochs; ++ep) loss_history[ep] = l[ep] / (float)n;
    cudaFree(perm);
    return refresh_packed(*net, s);
}

int ode_mlp_apply(int32_t handle, const float* X, int64_t n, float* out, void* stream) {
    clear_last_error();
    std::lock_guard<std::mutex> lk(g_mu);
    Mlp* net;
    int rc = get(handle, &net);
    if (rc) return rc;
    if (!X || !out || n < 0) return fail(ODE_ERR_ARG, "need device X and out");
    if (n == 0) return ODE_OK;
    k_mlp_apply<<<(unsigned)((n + 127) / 128), 128, apply_smem(net->n_in), (cudaStream_t)stream>>>(
        net->w16, net->norm, net->n_in, X, n, out);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? ODE_OK : cuda_fail(e, "mlp apply");
}

int ode_mlp_propose(int32_t handle, int64_t nsys, int32_t neq, const double* y0, const double* params, float margin,
                    float* h0, float* sigma0, float* cost, void* stream) {
    clear_last_error();
    std::lock_guard<std::mutex> lk(g_mu);
    Mlp* net;
    int rc = get(handle, &net);
    if (rc) return rc;
    if (neq + 1 != net->n_in) return fail(ODE_ERR_ARG, "network takes %d inputs, state has %d + 1", net->n_in, neq);
    if (!y0 || !params || !h0 || !sigma0 || nsys < 0) return fail(ODE_ERR_ARG, "need device y0, params, h0, sigma0");
    if (nsys == 0) return ODE_OK;
    k_mlp_propose<<<(unsigned)((nsys + 127) / 128), 128, apply_smem(net->n_in), (cudaStream_t)stream>>>(
        net->w16, net->norm, net->n_in, nsys, neq, y0, params, margin, h0, sigma0, cost);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? ODE_OK : cuda_fail(e, "mlp proposal");
}

int ode_mlp_get_params(int32_t handle, float* params, float* norm) {
    clear_last_error();
    std::lock_guard<std::mutex> lk(g_mu);
    Mlp* net;
    int rc = get(handle, &net);
    if (rc) return rc;
    if (params) {
        cudaError_t e = cudaMemcpy(params, net->master, sizeof(float) * net->nparams, cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) return cuda_fail(e, "parameter copy");
    }
    if (norm) std::memcpy(norm, &net->norm, sizeof(MlpNorm));
    return ODE_OK;
}

int ode_mlp_set_params(int32_t handle, const float* params, const float* norm) {
    clear_last_error();
    std::lock_guard<std::mutex> lk(g_mu);
    Mlp* net;
    int rc = get(handle, &net);
    if (rc) return rc;
    if (params) {
        cudaError_t e = cudaMemcpy(net->master, params, sizeof(float) * net->nparams, cudaMemcpyHostToDevice);
        if (e != cudaSuccess) return cuda_fail(e, "parameter copy");
        k_to_bf16<<<(net->nparams + 255) / 256, 256>>>(net->master, net->w16, net->nparams);
        e = cudaDeviceSynchronize();
        if (e != cudaSuccess) return cuda_fail(e, "parameter copy");
    }
    if (norm) {
        std::memcpy(&net->norm, norm, sizeof(MlpNorm));
        net->has_norm = true;
    }
    return refresh_packed(*net, nullptr);
}

int ode_mlp_apply_warp(int32_t handle, const float* X, int64_t n, float* out, void* stream) {
    clear_last_error();
    std::lock_guard<std::mutex> lk(g_mu);
    Mlp* net;
    int rc = get(handle, &net);
    if (rc) return rc;
    if (!X || !out || n < 0) return fail(ODE_ERR_ARG, "need device X and out");
    if (n == 0) return ODE_OK;
    const unsigned blocks = (unsigned)((n + 127) / 128);
    cudaStream_t s = (cudaStream_t)stream;
    const int ks = (net->n_in + 15) / 16;
    if (ks == 1)
        k_mlp_apply_warp<1><<<blocks, 128, 0, s>>>(net->packed, X, n, out);
    else if (ks == 2)
        k_mlp_apply_warp<2><<<blocks, 128, 0, s>>>(net->packed, X, n, out);
    else
        k_mlp_apply_warp<3><<<blocks, 128, 0, s>>>(net->packed, X, n, out);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? ODE_OK : cuda_fail(e, "mlp warp apply");
}

int ode_mlp_num_params(int32_t n_in) { return n_in >= 1 && n_in <= kMlpMaxIn ? mlp_nparams(n_in) : -1; }

}  // extern "C"
