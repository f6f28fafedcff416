// Training and batched inference of the restart-schedule network (eik_mlp.cuh).
//
// One thread per sample, the weights in shared memory, the activations in
// registers.  The gradient kernel keeps its samples' activations and deltas in
// shared memory and adds up their outer products there, one partial sum per
// parameter and block of kChunk samples; a second kernel adds the blocks' sums.
// Both sum in a fixed order (no atomics), so repeated training runs give the same
// weights bit for bit.
//
// What bounds them: instruction issue (about 2400 fused multiply-adds and 64 tanh
// per sample, 1800 more for the outer products).  32768 samples, forward and
// gradient: 255 us with one thread per parameter walking over the samples and the
// activations in local and global memory, 53 us with this layout (three launches).
#include "eik.h"
#include "eik_mlp.cuh"

#include <cstdint>
#include <string>

namespace {

using namespace eikg;

thread_local std::string g_mlp_err;

eik_status mlp_fail(eik_status s, const std::string& m) {
    g_mlp_err = m;
    return s;
}

constexpr int kChunk = 128;            // samples per block of the gradient kernel
constexpr int kPitch = kChunk + 4;     // row pitch of the sample arrays (float4 rows on different banks)

inline int64_t grad_blocks(int32_t B) { return B > 0 ? (static_cast<int64_t>(B) + kChunk - 1) / kChunk : 0; }

// The weights as the threads read them (the same address in every lane, four at a time).
struct __align__(16) NetSmem {
    float w1t[kIn][kHid];              // W1 transposed
    float w2t[kHid][kHid];             // W2 transposed
    float w2[kHid][kHid];
    float b1[kHid], b2[kHid];
    float w3[kAct][kHid + 1];          // (rows taken by action: a padded pitch)
    float b3[kAct];
};

__device__ __forceinline__ void load_net(NetSmem& N, const float* __restrict__ w) {
    for (int t = threadIdx.x; t < kHid * kIn; t += blockDim.x) N.w1t[t % kIn][t / kIn] = w[kOffW1 + t];
    for (int t = threadIdx.x; t < kHid * kHid; t += blockDim.x) {
        const float v = w[kOffW2 + t];
        N.w2[t / kHid][t % kHid] = v;
        N.w2t[t % kHid][t / kHid] = v;
    }
    for (int t = threadIdx.x; t < kAct * kHid; t += blockDim.x) N.w3[t / kHid][t % kHid] = w[kOffW3 + t];
    for (int t = threadIdx.x; t < kHid; t += blockDim.x) N.b1[t] = w[kOffB1 + t], N.b2[t] = w[kOffB2 + t];
    for (int t = threadIdx.x; t < kAct; t += blockDim.x) N.b3[t] = w[kOffB3 + t];
    __syncthreads();
}

// o[i] = c[i] + sum_j m[j][i] v[j], j ascending
template <int J>
__device__ __forceinline__ void layer(const float (*m)[kHid], const float* v, float* o) {
#pragma unroll
    for (int j = 0; j < J; ++j)
#pragma unroll
        for (int i = 0; i < kHid; i += 4) {
            const float4 q = *reinterpret_cast<const float4*>(&m[j][i]);
            o[i] = __fmaf_rn(q.x, v[j], o[i]);
            o[i + 1] = __fmaf_rn(q.y, v[j], o[i + 1]);
            o[i + 2] = __fmaf_rn(q.z, v[j], o[i + 2]);
            o[i + 3] = __fmaf_rn(q.w, v[j], o[i + 3]);
        }
}

__device__ __forceinline__ void hidden(const NetSmem& N, const float* x, float* h1, float* h2) {
#pragma unroll
    for (int i = 0; i < kHid; ++i) h1[i] = N.b1[i];
    layer<kIn>(N.w1t, x, h1);
#pragma unroll
    for (int i = 0; i < kHid; ++i) h1[i] = tanhf(h1[i]);
#pragma unroll
    for (int i = 0; i < kHid; ++i) h2[i] = N.b2[i];
    layer<kHid>(N.w2t, h1, h2);
#pragma unroll
    for (int i = 0; i < kHid; ++i) h2[i] = tanhf(h2[i]);
}

__global__ void __launch_bounds__(64) k_mlp_forward(const float* __restrict__ w, const float* __restrict__ X, int B,
                                                    float* __restrict__ Y) {
    __shared__ NetSmem N;
    load_net(N, w);
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= B) return;
    float x[kIn], h1[kHid], h2[kHid];
#pragma unroll
    for (int j = 0; j < kIn; ++j) x[j] = X[static_cast<size_t>(s) * kIn + j];
    hidden(N, x, h1, h2);
#pragma unroll
    for (int a = 0; a < kAct; ++a) {
        float y = N.b3[a];
#pragma unroll
        for (int j = 0; j < kHid; ++j) y = __fmaf_rn(N.w3[a][j], h2[j], y);
        Y[static_cast<size_t>(s) * kAct + a] = y;
    }
}

// A block's samples, one column each.
struct __align__(16) GradSmem {
    NetSmem net;
    float x[kIn][kPitch], h1[kHid][kPitch], h2[kHid][kPitch], d1[kHid][kPitch], d2[kHid][kPitch];
    float dy[kAct][kPitch];            // d loss / d y: the taken action's, else 0
    float e2[kPitch];                  // squared errors
};

// sum over the block's samples of p[s] q[s], four interleaved partial sums
__device__ __forceinline__ float dot(const float* p, const float* q) {
    float a0 = 0.0f, a1 = 0.0f, a2 = 0.0f, a3 = 0.0f;
#pragma unroll 8
    for (int s = 0; s < kChunk; s += 4) {
        const float4 u = *reinterpret_cast<const float4*>(p + s), v = *reinterpret_cast<const float4*>(q + s);
        a0 = __fmaf_rn(u.x, v.x, a0);
        a1 = __fmaf_rn(u.y, v.y, a1);
        a2 = __fmaf_rn(u.z, v.z, a2);
        a3 = __fmaf_rn(u.w, v.w, a3);
    }
    return (a0 + a1) + (a2 + a3);
}
__device__ __forceinline__ float total(const float* p) {
    float a0 = 0.0f, a1 = 0.0f, a2 = 0.0f, a3 = 0.0f;
#pragma unroll 8
    for (int s = 0; s < kChunk; s += 4) {
        const float4 u = *reinterpret_cast<const float4*>(p + s);
        a0 += u.x;
        a1 += u.y;
        a2 += u.z;
        a3 += u.w;
    }
    return (a0 + a1) + (a2 + a3);
}

// Block c: forward, error of the taken action and backpropagated deltas of its
// samples, then partial[c][p] = their sum for every parameter p (and, for p ==
// kParams, of the squared errors).  Places without a sample hold zeros, and a sample
// counts only for its action: neither spreads a value that is not finite.
__global__ void __launch_bounds__(kChunk) k_mlp_partial(const float* __restrict__ w, const float* __restrict__ X,
                                                        const int* __restrict__ act, const float* __restrict__ tgt, int B,
                                                        float* __restrict__ partial) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    GradSmem& S = *reinterpret_cast<GradSmem*>(smem_raw);
    load_net(S.net, w);
    const int t = threadIdx.x, s = blockIdx.x * kChunk + t;
    {
        float x[kIn], u[kHid], v[kHid];
        const bool in = s < B;
#pragma unroll
        for (int j = 0; j < kIn; ++j) {
            x[j] = in ? X[static_cast<size_t>(s) * kIn + j] : 0.0f;
            S.x[j][t] = x[j];
        }
        hidden(S.net, x, u, v);                                  // u = h1, v = h2
#pragma unroll
        for (int j = 0; j < kHid; ++j) S.h1[j][t] = u[j], S.h2[j][t] = v[j];
        const int a = in ? act[s] : 0;
        float y = S.net.b3[a];
#pragma unroll
        for (int j = 0; j < kHid; ++j) y = __fmaf_rn(S.net.w3[a][j], v[j], y);
        const float e = in ? y - tgt[s] : 0.0f;
        const float dy = 2.0f * e / static_cast<float>(B);       // d loss / d y_a, loss = mean e^2
        S.e2[t] = e * e;
#pragma unroll
        for (int q = 0; q < kAct; ++q) S.dy[q][t] = q == a ? dy : 0.0f;
#pragma unroll
        for (int j = 0; j < kHid; ++j) {
            v[j] = dy * S.net.w3[a][j] * (1.0f - v[j] * v[j]);   // d2
            S.d2[j][t] = v[j];
        }
#pragma unroll
        for (int j = 0; j < kHid; ++j) u[j] = 0.0f;
        layer<kHid>(S.net.w2, v, u);                             // sum_i d2_i W2[i][j]
#pragma unroll
        for (int j = 0; j < kHid; ++j) {
            const float h = S.h1[j][t];
            S.d1[j][t] = u[j] * (1.0f - h * h);
        }
        // A hidden value that is not a number makes y and with it dy none either, so W3's
        // row of the action taken is lost; the other rows multiply it by 0.  (Guarded
        // where they are stored, the values of all samples took 0.2 us of 53.)
        if (!in || !(dy == dy)) {
            for (int j = 0; j < kHid; ++j) {
                S.h2[j][t] = 0.0f;
                if (!in) S.h1[j][t] = S.d1[j][t] = S.d2[j][t] = 0.0f;
            }
        }
    }
    __syncthreads();
    float* out = partial + static_cast<size_t>(blockIdx.x) * (kParams + 1);
    {   // W2[i][j]: d2_i h1_j, eight j a thread
        const int i = t >> 2, j0 = (t & 3) * 8;
        float acc[8][2] = {};
#pragma unroll 2
        for (int q = 0; q < kChunk; q += 4) {
            const float4 d = *reinterpret_cast<const float4*>(&S.d2[i][q]);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float4 h = *reinterpret_cast<const float4*>(&S.h1[j0 + j][q]);
                acc[j][0] = __fmaf_rn(d.y, h.y, __fmaf_rn(d.x, h.x, acc[j][0]));
                acc[j][1] = __fmaf_rn(d.w, h.w, __fmaf_rn(d.z, h.z, acc[j][1]));
            }
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) out[kOffW2 + i * kHid + j0 + j] = acc[j][0] + acc[j][1];
    }
    for (int p = t; p < kHid * kIn; p += kChunk) out[kOffW1 + p] = dot(S.d1[p / kIn], S.x[p % kIn]);       // d1_i x_j
    for (int p = t; p < kAct * kHid; p += kChunk) out[kOffW3 + p] = dot(S.dy[p / kHid], S.h2[p % kHid]);   // dy_a h2_j
    if (t < kHid) out[kOffB1 + t] = total(S.d1[t]);
    else if (t < 2 * kHid) out[kOffB2 + t - kHid] = total(S.d2[t - kHid]);
    else if (t < 2 * kHid + kAct) out[kOffB3 + t - 2 * kHid] = total(S.dy[t - 2 * kHid]);
    else if (t == 2 * kHid + kAct) out[kParams] = total(S.e2);
}

// The blocks' partial sums: 32 parameters a CTA, warp r adding the blocks r, r + 8,
// ..., then the eight sums in order.
constexpr int kSumWarps = 8;
__global__ void k_mlp_total(int nchunks, const float* __restrict__ partial, int B, float* __restrict__ grad,
                            float* __restrict__ loss) {
    __shared__ float sum[kSumWarps][33];
    const int lane = threadIdx.x & 31, r = threadIdx.x >> 5, p = blockIdx.x * 32 + lane;
    float acc = 0.0f;
    if (p <= kParams) {
#pragma unroll 8
        for (int c = r; c < nchunks; c += kSumWarps) acc += partial[static_cast<size_t>(c) * (kParams + 1) + p];
    }
    sum[r][lane] = acc;
    __syncthreads();
    if (r != 0 || p > kParams) return;
#pragma unroll
    for (int q = 1; q < kSumWarps; ++q) acc += sum[q][lane];
    if (p == kParams) {
        if (loss) *loss = acc / static_cast<float>(B);
    } else {
        grad[p] = acc;
    }
}

// Adam (Kingma and Ba, 2015), element-wise
__global__ void k_mlp_adam(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m,
                           float* __restrict__ v, int n, float lr, float b1, float b2, float eps, float c1, float c2) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const float gp = g[p];
    const float mp = b1 * m[p] + (1.0f - b1) * gp;
    const float vp = b2 * v[p] + (1.0f - b2) * gp * gp;
    m[p] = mp;
    v[p] = vp;
    w[p] -= lr * (mp / c1) / (sqrtf(vp / c2) + eps);
}

}  // namespace

extern "C" {

const char* eik_mlp_last_error(void) { return g_mlp_err.c_str(); }

int32_t eik_mlp_work_floats(int32_t B) {
    const int64_t n = grad_blocks(B) * (kParams + 1);
    return n <= INT32_MAX ? static_cast<int32_t>(n) : 0;
}

eik_status eik_mlp_forward(const float* w, const float* X, int32_t B, float* Y, void* stream) {
    if (!w || !X || !Y || B < 1) return mlp_fail(EIK_EINVAL, "eik_mlp_forward: bad argument");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    k_mlp_forward<<<(B + 63) / 64, 64, 0, s>>>(w, X, B, Y);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return mlp_fail(EIK_ECUDA, cudaGetErrorString(e));
    return EIK_OK;
}

eik_status eik_mlp_grad(const float* w, const float* X, const int32_t* act, const float* tgt, int32_t B, float* grad,
                        float* loss, float* work, void* stream) {
    if (!w || !X || !act || !tgt || !grad || !work || B < 1) return mlp_fail(EIK_EINVAL, "eik_mlp_grad: bad argument");
    if (eik_mlp_work_floats(B) == 0)
        return mlp_fail(EIK_EINVAL, "eik_mlp_grad: more samples than a work space of 2^31 - 1 floats serves");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int nchunks = static_cast<int>(grad_blocks(B));
    const cudaError_t attr = cudaFuncSetAttribute(k_mlp_partial, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                  static_cast<int>(sizeof(GradSmem)));
    if (attr != cudaSuccess) return mlp_fail(EIK_ECUDA, cudaGetErrorString(attr));
    k_mlp_partial<<<nchunks, kChunk, sizeof(GradSmem), s>>>(w, X, act, tgt, B, work);
    k_mlp_total<<<(kParams + 1 + 31) / 32, 32 * kSumWarps, 0, s>>>(nchunks, work, B, grad, loss);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return mlp_fail(EIK_ECUDA, cudaGetErrorString(e));
    return EIK_OK;
}

eik_status eik_mlp_adam(float* w, const float* grad, float* m, float* v, int32_t n, float lr, float b1, float b2,
                        float eps, int32_t t, void* stream) {
    if (!w || !grad || !m || !v || n < 1 || t < 1) return mlp_fail(EIK_EINVAL, "eik_mlp_adam: bad argument");
    const float c1 = 1.0f - powf(b1, static_cast<float>(t));
    const float c2 = 1.0f - powf(b2, static_cast<float>(t));
    k_mlp_adam<<<(n + 255) / 256, 256, 0, static_cast<cudaStream_t>(stream)>>>(w, grad, m, v, n, lr, b1, b2, eps, c1,
                                                                                c2);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return mlp_fail(EIK_ECUDA, cudaGetErrorString(e));
    return EIK_OK;
}

eik_status eik_sched_actions(double* stride_h, int32_t* block_dim, int32_t cap, int32_t* n) {
    if (!n) return mlp_fail(EIK_EINVAL, "eik_sched_actions: n is NULL");
    *n = kAct;
    for (int a = 0; a < kAct && a < cap; ++a) {
        if (stride_h) stride_h[a] = action_stride_h(a);
        if (block_dim) block_dim[a] = action_block(a);
    }
    return EIK_OK;
}

}  // extern "C"
