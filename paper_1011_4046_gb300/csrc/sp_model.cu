// sp_model.cu -- the region cost model: a 16-64-64-1 ReLU network trained on
// measured region times, and the bucketing of a launch's regions by its
// predictions (the learned ordering of the device queue).
//
// The paper's manager issues regions so that expensive ones do not finish
// last (Sec. 4; uneven region costs, Sec. 6).  Here the network predicts the
// log of a region's time from 16 features (feature_kernel in sp_kernels.cu);
// regions go into one of four priority buckets and the persistent kernel pops
// the highest non-empty bucket first.  Only the schedule changes, never the
// arithmetic of a region, so results stay bit-identical.
//
// Kernels (FP32, hand-written):
//   mlp_infer_kernel    forward of one or two samples per thread, to outputs
//                       or (with the thresholds) priority buckets;
//   train_kernel        an epoch of minibatch Adam steps on one cluster;
//   mlp_grad_kernel     per block of <= 128 samples: forward, reverse pass and
//                       the block's sum of parameter gradients of the mean
//                       squared error, in a fixed order (deterministic);
//   grad_reduce_kernel  sums the blocks' partial gradients in block order;
//   adam_kernel         one Adam step per parameter (Kingma & Ba 2015).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "sp.h"
#include "sp_device.cuh"

namespace {

constexpr int kIn = 16, kHid = 64;
constexpr int kW1 = 0, kB1 = kW1 + kHid * kIn, kW2 = kB1 + kHid, kB2 = kW2 + kHid * kHid, kW3 = kB2 + kHid,
              kB3 = kW3 + kHid, kParams = kB3 + 1;
static_assert(kParams == SP_MODEL_PARAMS, "parameter count");
constexpr int kGradBlock = 128;   // samples per gradient block
constexpr int kPitch = kGradBlock + 1;  // sample-minor rows, padded against bank conflicts

__device__ __forceinline__ void load_params(float *s, const float *theta)
{
    for (int i = threadIdx.x; i < kParams; i += blockDim.x) s[i] = theta[i];
}

// Network outputs, or (PRIO) priority buckets: 0 for a prediction >= thr[0]
// (most expensive), 1 for >= thr[1], 2 for >= thr[2], else 3.
//
// Bound by the FP32 pipe (5184 fused multiply-adds a sample).  A thread holds
// S samples with all 64 sums of a layer in registers and steps through the
// layer's inputs: a weight row (transposed in shared memory) is read by 16-byte
// broadcasts, each feeding four multiply-adds per sample as two packed ones,
// where one 4-byte broadcast per multiply-add bound it before.  Each sum takes
// its terms in the order of the inputs, as one chain of fused multiply-adds.
// Blocks stay and loop over the samples, so the weights are laid out once a
// block.  2^20 samples, call and synchronisation: 557 us before, 238 now (141
// at the FP32 rate); one sample a thread 335 us (its broadcasts bound it
// again), three 245 us.  Two pay from the size at which one already fills
// every SM with two blocks.
constexpr int kInferThreads = 128;
constexpr int kInferPerSm = 2;

struct InferWeights {
    float w1[kIn][kHid], w2[kHid][kHid];  // by input, then output
    float b1[kHid], b2[kHid], w3[kHid], b3, pad[3];
};

template <int S, int N_IN, class In>
__device__ __forceinline__ void layer(float2 (&acc)[S][kHid / 2], const float (*w)[kHid], const float *b, In in)
{
#pragma unroll
    for (int j = 0; j < kHid / 2; ++j) {
        const float2 v = *reinterpret_cast<const float2 *>(b + 2 * j);
#pragma unroll
        for (int s = 0; s < S; ++s) acc[s][j] = v;
    }
#pragma unroll 4
    for (int i = 0; i < N_IN; ++i) {
        float2 x[S];
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const float v = in(s, i);
            x[s] = make_float2(v, v);
        }
#pragma unroll
        for (int j = 0; j < kHid / 4; ++j) {
            const float4 r = *reinterpret_cast<const float4 *>(w[i] + 4 * j);
#pragma unroll
            for (int s = 0; s < S; ++s) {
                acc[s][2 * j] = __ffma2_rn(make_float2(r.x, r.y), x[s], acc[s][2 * j]);
                acc[s][2 * j + 1] = __ffma2_rn(make_float2(r.z, r.w), x[s], acc[s][2 * j + 1]);
            }
        }
    }
}

template <int S, bool PRIO>
__global__ void __launch_bounds__(kInferThreads, kInferPerSm)
    mlp_infer_kernel(const float *__restrict__ theta, const float *__restrict__ thr, const float *__restrict__ X, long long n,
                     float *__restrict__ out, unsigned char *__restrict__ prio)
{
    extern __shared__ __align__(16) unsigned char smem[];
    InferWeights &W = *reinterpret_cast<InferWeights *>(smem);
    float *const h = reinterpret_cast<float *>(smem + sizeof(InferWeights)) + threadIdx.x;  // [input][sample][thread]
    for (int p = threadIdx.x; p < kIn * kHid; p += kInferThreads) W.w1[p / kHid][p % kHid] = theta[kW1 + (p % kHid) * kIn + p / kHid];
    for (int p = threadIdx.x; p < kHid * kHid; p += kInferThreads) W.w2[p / kHid][p % kHid] = theta[kW2 + (p % kHid) * kHid + p / kHid];
    for (int p = threadIdx.x; p < kHid; p += kInferThreads) {
        W.b1[p] = theta[kB1 + p];
        W.b2[p] = theta[kB2 + p];
        W.w3[p] = theta[kW3 + p];
    }
    if (threadIdx.x == 0) W.b3 = theta[kB3];
    const bool vec = ((uintptr_t)X & 15) == 0;
    __syncthreads();
    for (long long base = (long long)blockIdx.x * (S * kInferThreads); base < n;
         base += (long long)gridDim.x * (S * kInferThreads)) {
        float2 acc[S][kHid / 2];
#pragma unroll
        for (int s = 0; s < S; ++s) {  // inputs, through the thread's own column of shared memory
            const long long k = base + s * kInferThreads + threadIdx.x;
            const float *x = X + kIn * (k < n ? k : n - 1);
            float4 v[kIn / 4];
#pragma unroll
            for (int i = 0; i < kIn / 4; ++i)
                v[i] = vec ? __ldg(reinterpret_cast<const float4 *>(x) + i)
                           : make_float4(x[4 * i], x[4 * i + 1], x[4 * i + 2], x[4 * i + 3]);
#pragma unroll
            for (int i = 0; i < kIn / 4; ++i) {
                h[((4 * i + 0) * S + s) * kInferThreads] = v[i].x;
                h[((4 * i + 1) * S + s) * kInferThreads] = v[i].y;
                h[((4 * i + 2) * S + s) * kInferThreads] = v[i].z;
                h[((4 * i + 3) * S + s) * kInferThreads] = v[i].w;
            }
        }
        auto in = [&](int s, int i) { return h[(i * S + s) * kInferThreads]; };
        layer<S, kIn>(acc, W.w1, W.b1, in);
#pragma unroll
        for (int j = 0; j < kHid / 2; ++j)
#pragma unroll
            for (int s = 0; s < S; ++s) {
                h[(2 * j * S + s) * kInferThreads] = fmaxf(acc[s][j].x, 0.0f);
                h[((2 * j + 1) * S + s) * kInferThreads] = fmaxf(acc[s][j].y, 0.0f);
            }
        layer<S, kHid>(acc, W.w2, W.b2, in);
#pragma unroll
        for (int s = 0; s < S; ++s) {
            float y = W.b3;
#pragma unroll
            for (int j = 0; j < kHid / 2; ++j) {
                y = fmaf(W.w3[2 * j], fmaxf(acc[s][j].x, 0.0f), y);
                y = fmaf(W.w3[2 * j + 1], fmaxf(acc[s][j].y, 0.0f), y);
            }
            const long long k = base + s * kInferThreads + threadIdx.x;
            if (k >= n) continue;
            if (PRIO)
                prio[k] = (unsigned char)(y >= thr[0] ? 0 : (y >= thr[1] ? 1 : (y >= thr[2] ? 2 : 3)));
            else
                out[k] = y;
        }
    }
}

template <int S, bool PRIO>
cudaError_t infer_t(const float *theta, const float *thr, const float *X, long long n, float *out, unsigned char *prio,
                    int sms, cudaStream_t st)
{
    const size_t smem = sizeof(InferWeights) + sizeof(float) * kHid * S * kInferThreads;
    cudaError_t e =
        cudaFuncSetAttribute(mlp_infer_kernel<S, PRIO>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const long long tiles = (n + S * kInferThreads - 1) / (S * kInferThreads);
    const unsigned grid = (unsigned)std::min<long long>(tiles, (long long)kInferPerSm * sms);
    mlp_infer_kernel<S, PRIO><<<grid, kInferThreads, smem, st>>>(theta, thr, X, n, out, prio);
    return cudaGetLastError();
}

template <bool PRIO>
cudaError_t infer(const float *theta, const float *thr, const float *X, long long n, float *out, unsigned char *prio, int sms,
                  cudaStream_t st)
{
    if (n <= (long long)kInferPerSm * sms * kInferThreads) return infer_t<1, PRIO>(theta, thr, X, n, out, prio, sms, st);
    return infer_t<2, PRIO>(theta, thr, X, n, out, prio, sms, st);
}

// Gradient of L = (1/n) sum (yhat - y)^2 over the samples idx[0..count) (or
// 0..count when idx is null), block b taking samples [128 b, 128 b + 128).
// partial[b][p] = block b's share of dL/dtheta_p; partial[b][kParams] = its
// share of L.  Shared memory: the parameters, then sample-minor arrays
// x[16], h1[64], h2[64], dL/dz1[64], dL/dz2[64], dL/dyhat, r^2/n.
__global__ void __launch_bounds__(kGradBlock) mlp_grad_kernel(const float *__restrict__ theta,
                                                              const float *__restrict__ X, const float *__restrict__ Y,
                                                              const int *__restrict__ idx, int count, float inv_n,
                                                              float *__restrict__ partial)
{
    extern __shared__ float sm[];
    float *P = sm;
    float *xs = P + kParams;
    float *h1s = xs + kIn * kPitch;
    float *h2s = h1s + kHid * kPitch;
    float *g1s = h2s + kHid * kPitch;
    float *g2s = g1s + kHid * kPitch;
    float *gos = g2s + kHid * kPitch;
    float *ls = gos + kPitch;
    load_params(P, theta);
    __syncthreads();
    const int t = threadIdx.x;
    const int k = blockIdx.x * kGradBlock + t;
    if (k < count) {
        const long long s = idx ? idx[k] : k;
        const float *x = X + kIn * s;
        float in[kIn];
#pragma unroll
        for (int i = 0; i < kIn; ++i) {
            in[i] = x[i];
            xs[i * kPitch + t] = in[i];
        }
        unsigned long long m1 = 0ull, m2 = 0ull;  // ReLU masks
        for (int j = 0; j < kHid; ++j) {
            float z = P[kB1 + j];
#pragma unroll
            for (int i = 0; i < kIn; ++i) z = fmaf(P[kW1 + j * kIn + i], in[i], z);
            if (z > 0.0f) m1 |= 1ull << j;
            h1s[j * kPitch + t] = fmaxf(z, 0.0f);
        }
        float yhat = P[kB3];
        for (int j = 0; j < kHid; ++j) {
            float z = P[kB2 + j];
            for (int i = 0; i < kHid; ++i) z = fmaf(P[kW2 + j * kHid + i], h1s[i * kPitch + t], z);
            if (z > 0.0f) m2 |= 1ull << j;
            const float h = fmaxf(z, 0.0f);
            h2s[j * kPitch + t] = h;
            yhat = fmaf(P[kW3 + j], h, yhat);
        }
        const float r = yhat - Y[s];
        const float go = 2.0f * r * inv_n;
        gos[t] = go;
        ls[t] = r * r * inv_n;
        for (int j = 0; j < kHid; ++j) g2s[j * kPitch + t] = ((m2 >> j) & 1ull) ? go * P[kW3 + j] : 0.0f;
        for (int i = 0; i < kHid; ++i) {
            float gh = 0.0f;
            for (int j = 0; j < kHid; ++j) gh = fmaf(P[kW2 + j * kHid + i], g2s[j * kPitch + t], gh);
            g1s[i * kPitch + t] = ((m1 >> i) & 1ull) ? gh : 0.0f;
        }
    } else {
        for (int i = 0; i < kIn; ++i) xs[i * kPitch + t] = 0.0f;
        for (int j = 0; j < kHid; ++j) {
            h1s[j * kPitch + t] = 0.0f;
            h2s[j * kPitch + t] = 0.0f;
            g1s[j * kPitch + t] = 0.0f;
            g2s[j * kPitch + t] = 0.0f;
        }
        gos[t] = 0.0f;
        ls[t] = 0.0f;
    }
    __syncthreads();
    float *out = partial + (size_t)blockIdx.x * (kParams + 1);
    for (int p = t; p <= kParams; p += kGradBlock) {
        const float *a, *b = nullptr;  // sum over samples of a[s] * b[s] (b null: of a[s])
        if (p < kB1) {
            a = g1s + (p / kIn) * kPitch;
            b = xs + (p % kIn) * kPitch;
        } else if (p < kW2) {
            a = g1s + (p - kB1) * kPitch;
        } else if (p < kB2) {
            a = g2s + ((p - kW2) / kHid) * kPitch;
            b = h1s + ((p - kW2) % kHid) * kPitch;
        } else if (p < kW3) {
            a = g2s + (p - kB2) * kPitch;
        } else if (p < kB3) {
            a = gos;
            b = h2s + (p - kW3) * kPitch;
        } else if (p == kB3) {
            a = gos;
        } else {
            a = ls;
        }
        float acc = 0.0f;
        if (b)
            for (int s = 0; s < kGradBlock; ++s) acc = fmaf(a[s], b[s], acc);
        else
            for (int s = 0; s < kGradBlock; ++s) acc += a[s];
        out[p] = acc;
    }
}

__global__ void grad_reduce_kernel(const float *__restrict__ partial, int blocks, float *__restrict__ grad,
                                   float *__restrict__ loss_out)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p > kParams) return;
    float acc = 0.0f;
    for (int b = 0; b < blocks; ++b) acc += partial[(size_t)b * (kParams + 1) + p];
    if (p < kParams)
        grad[p] = acc;
    else if (loss_out)
        *loss_out = acc;
}

__global__ void adam_kernel(float *__restrict__ theta, float *__restrict__ m, float *__restrict__ v,
                            const float *__restrict__ grad, float lr, float beta1, float beta2, float eps, float c1,
                            float c2)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= kParams) return;
    const float g = grad[p];
    const float mp = beta1 * m[p] + (1.0f - beta1) * g;
    const float vp = beta2 * v[p] + (1.0f - beta2) * g * g;
    m[p] = mp;
    v[p] = vp;
    theta[p] -= lr * (mp * c1) / (sqrtf(vp * c2) + eps);
}

// A whole epoch of minibatch Adam steps in one launch of one thread-block
// cluster.  A step's work is small (256 samples: 4e6 multiply-adds) and each
// step depends on the last, so its latency counts: as three launches (a
// gradient kernel on batch / 128 blocks, a sum over blocks, Adam) a step of 256
// samples took 90 us, 79 of them two blocks' gradient; here 7.0 us (3.4 of them
// the barriers and the stores between CTAs).  Each
// CTA of the cluster takes its share of the minibatch, 16 samples at a time,
// with the parameters in its shared memory, and sends its part of the gradient
// into the shared memory of the CTA that owns that slice of the parameters
// (stores: a remote read would wait for its round trip).  The owner sums the
// parts in rank order (deterministic), updates its slice, whose Adam moments
// its threads keep in registers, and stores it into every CTA's shared memory.
// Two hardware cluster barriers a step order this.
//
// A warp's pass over the 16 samples: eight outputs times four groups of four
// samples, so that a 16-byte read of weights (pitches odd in 16-byte units)
// and one of activations are each one wavefront; the gradient of W2 as 4 x 4
// tiles over the samples.
constexpr int kTrainThreads = 256;
constexpr int kTrainChunk = 16;  // samples of a pass
#ifndef SP_TRAIN_CTAS  // a test builds the kernel of 8
#define SP_TRAIN_CTAS 16
#endif
constexpr int kTrainCtas = SP_TRAIN_CTAS;  // most CTAs of the cluster (8 where 16 do not fit)
// Largest minibatch of this path (4096 samples: 59 us a step, 76 as launches
// over many SMs, which take 8192 in 83)
constexpr int kTrainMaxBatch = 4096;
constexpr int kActPitch = kHid + 4;

// Parameters of a CTA's slice: a multiple of four, so that four consecutive
// parameters from a multiple of four on have one owner.
__host__ __device__ constexpr int train_slice(int ctas) { return ((kParams + 1 + ctas - 1) / ctas + 3) & ~3; }

struct alignas(16) TrainSmem {
    float w1[kHid][kIn + 4], w2[kHid][kHid + 4];  // [output][input]
    float b1[kHid], b2[kHid], w3[kHid], b3[4];
    float x[kTrainChunk][kIn + 4];
    float h1[kTrainChunk][kActPitch], h2[kTrainChunk][kActPitch], g1[kTrainChunk][kActPitch], g2[kTrainChunk][kActPitch];
    float parts[kTrainCtas * train_slice(kTrainCtas) + 8 * 4];  // [CTA][slice] of the gradient (last: the loss)
    float out[kTrainThreads / 32][kTrainChunk], go[kTrainChunk], sq[kTrainChunk], y[kTrainChunk];
};
static_assert(8 * train_slice(8) <= kTrainCtas * train_slice(kTrainCtas) + 8 * 4, "room for the parts of either cluster");

struct TrainArgs {
    float *theta, *m, *v;
    const float *X, *Y;
    const int *order;      // sample indices of the epoch
    const float2 *corr;    // bias corrections of each step
    float *losses;
    int n, batch, steps;
    float lr, beta1, beta2, eps;
};

// Where parameter p sits; four consecutive ones from a multiple of four on are
// contiguous (those after the last are padding).
__device__ __forceinline__ float *train_param(TrainSmem &S, int p)
{
    if (p < kB1) return &S.w1[p / kIn][p % kIn];
    if (p < kW2) return &S.b1[p - kB1];
    if (p < kB2) return &S.w2[(p - kW2) / kHid][(p - kW2) % kHid];
    if (p < kW3) return &S.b2[p - kB2];
    if (p < kB3) return &S.w3[p - kW3];
    return &S.b3[p - kB3];
}

__device__ __forceinline__ void st_cluster(unsigned addr, float v)
{
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}

__device__ __forceinline__ void st_cluster4(unsigned addr, float4 v)
{
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
}

__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }

__device__ __forceinline__ float dot4(float4 a, float4 b, float acc)
{
    return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, acc))));
}

template <int R>
__global__ void __launch_bounds__(kTrainThreads, 1) train_kernel(const TrainArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    TrainSmem &S = *reinterpret_cast<TrainSmem *>(smem);
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int rank = (int)sp::cluster_ctarank();
    constexpr int kSlice = train_slice(R);
    static_assert(kSlice / 4 <= kTrainThreads, "a thread updates four parameters");
    for (int p = t; p < kParams; p += kTrainThreads) *train_param(S, p) = a.theta[p];
    // the four parameters this thread updates, and their moments
    const int own = rank * kSlice + 4 * t;
    const bool owner = 4 * t < kSlice && own <= kParams;
    float am[4], av[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        am[q] = owner && own + q < kParams ? a.m[own + q] : 0.0f;
        av[q] = owner && own + q < kParams ? a.v[own + q] : 0.0f;
    }
    const int j = warp * 8 + (lane & 7), s0 = (lane >> 3) * 4;  // layers: output j of samples s0 .. s0 + 3
    const int xs = t >> 4, xi = t & (kIn - 1);         // inputs: value xi of sample xs
    const int tj = (t >> 4) * 4, ti = (t & 15) * 4;    // gradient of W2: rows tj .., columns ti ..
    const int wj = t >> 2, wi = (t & 3) * 4;           // gradient of W1: row wj, columns wi ..
    const int bj = t & (kHid - 1), bk = t >> 6;        // gradients of b1, b2, W3 (bk 0, 1, 2), b3 and loss
    const float *const Xi = a.X + xi;
    // a part of the gradient to its owner
    auto part_of = [&](int p) {
        const int to = p / kSlice;
        return sp::map_shared(&S.parts[rank * kSlice + (p - to * kSlice)], to);
    };
    const unsigned to_w1 = part_of(kW1 + wj * kIn + wi);
    unsigned to_w2[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) to_w2[q] = part_of(kW2 + (tj + q) * kHid + ti);
    const unsigned to_b = part_of(bk == 0 ? kB1 + bj : bk == 1 ? kB2 + bj : bk == 2 ? kW3 + bj : kB3 + (bj & 1));
    // This CTA's samples of a step: [k0, k1) of the epoch's order, taken in
    // passes of 16.  A pass's values are requested a pass ahead, and their
    // places in the order (which the requests wait for) two ahead.
    struct Pass {
        int step, k, k1, count;
    };
    auto enter = [&](Pass &p, int step) {
        const int first = step * a.batch;
        p.step = step;
        p.count = min(a.batch, a.n - first);
        const int per = (p.count + R - 1) / R;
        p.k = first + min(p.count, rank * per);
        p.k1 = first + min(p.count, rank * per + per);
    };
    auto advance = [&](Pass &p) {
        if (p.step >= a.steps) return;
        if (p.k + kTrainChunk < p.k1)
            p.k += kTrainChunk;
        else if (p.step + 1 < a.steps)
            enter(p, p.step + 1);
        else
            p.step = a.steps;
    };
    auto place = [&](const Pass &p) { return p.step < a.steps && p.k + xs < p.k1 ? a.order[p.k + xs] : -1; };
    auto fetch = [&](int s, float &x, float &y) {
        x = s >= 0 ? Xi[kIn * (long long)s] : 0.0f;
        y = s >= 0 && xi == 0 ? a.Y[s] : 0.0f;
    };
    Pass cur, ahead;
    enter(cur, 0);
    float xv, yv;
    fetch(place(cur), xv, yv);
    ahead = cur;
    advance(ahead);
    int next_place = place(ahead);
    sp::cluster_barrier();
    for (int step = 0; step < a.steps; ++step) {
        const float inv_n = 1.0f / (float)cur.count;
        const float2 corr = a.corr[step];
        float gw2[4][4] = {}, gw1[4] = {}, gb = 0.0f;
        for (bool last = false; !last; advance(cur)) {
            S.x[xs][xi] = xv;
            if (xi == 0) S.y[xs] = yv;
            const int live = min(kTrainChunk, cur.k1 - cur.k);  // samples of this pass (at most 0: none)
            last = cur.k + kTrainChunk >= cur.k1;
            __syncthreads();
            fetch(next_place, xv, yv);
            advance(ahead);
            next_place = place(ahead);
            if (live > 0) {
                {  // layer 1
                    float4 w[kIn / 4];
#pragma unroll
                    for (int i = 0; i < kIn / 4; ++i) w[i] = ld4(&S.w1[j][4 * i]);
                    const float b = S.b1[j];
#pragma unroll
                    for (int s = 0; s < 4; ++s) {
                        float z = b;
#pragma unroll
                        for (int i = 0; i < kIn / 4; ++i) z = dot4(w[i], ld4(&S.x[s0 + s][4 * i]), z);
                        S.h1[s0 + s][j] = fmaxf(z, 0.0f);
                    }
                }
                __syncthreads();
                const float w3 = S.w3[j];
                float h2[4];
                {  // layer 2 and the output
                    float z[4];
#pragma unroll
                    for (int s = 0; s < 4; ++s) z[s] = S.b2[j];
#pragma unroll
                    for (int i = 0; i < kHid; i += 4) {
                        const float4 w = ld4(&S.w2[j][i]);
#pragma unroll
                        for (int s = 0; s < 4; ++s) z[s] = dot4(w, ld4(&S.h1[s0 + s][i]), z[s]);
                    }
#pragma unroll
                    for (int s = 0; s < 4; ++s) {
                        h2[s] = fmaxf(z[s], 0.0f);
                        S.h2[s0 + s][j] = h2[s];
                        float y = w3 * h2[s];
#pragma unroll
                        for (int o = 4; o > 0; o >>= 1) y += __shfl_xor_sync(~0u, y, o);
                        if ((lane & 7) == 0) S.out[warp][s0 + s] = y;
                    }
                }
                __syncthreads();
#pragma unroll
                for (int s = 0; s < 4; ++s) {  // dL/dyhat, dL/dz2
                    float y = S.b3[0];
#pragma unroll
                    for (int w = 0; w < kTrainThreads / 32; ++w) y += S.out[w][s0 + s];
                    const float r = y - S.y[s0 + s];
                    const float go = s0 + s < live ? 2.0f * r * inv_n : 0.0f;
                    S.g2[s0 + s][j] = h2[s] > 0.0f ? go * w3 : 0.0f;
                    if (j == 0) {
                        S.go[s0 + s] = go;
                        S.sq[s0 + s] = s0 + s < live ? r * r * inv_n : 0.0f;
                    }
                }
                __syncthreads();
                {  // dL/dz1: j is the hidden unit of layer 1
                    float g[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
                    for (int i = 0; i < kHid; i += 4) {
                        const float4 w = make_float4(S.w2[i][j], S.w2[i + 1][j], S.w2[i + 2][j], S.w2[i + 3][j]);
#pragma unroll
                        for (int s = 0; s < 4; ++s) g[s] = dot4(w, ld4(&S.g2[s0 + s][i]), g[s]);
                    }
#pragma unroll
                    for (int s = 0; s < 4; ++s) S.g1[s0 + s][j] = S.h1[s0 + s][j] > 0.0f ? g[s] : 0.0f;
                }
                __syncthreads();
                // sums over the samples, in order (those past the last have zero derivatives)
#pragma unroll
                for (int s = 0; s < kTrainChunk; ++s) {
                    const float4 u = ld4(&S.g2[s][tj]), h = ld4(&S.h1[s][ti]), x = ld4(&S.x[s][wi]);
                    const float uu[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        gw2[q][0] = fmaf(uu[q], h.x, gw2[q][0]);
                        gw2[q][1] = fmaf(uu[q], h.y, gw2[q][1]);
                        gw2[q][2] = fmaf(uu[q], h.z, gw2[q][2]);
                        gw2[q][3] = fmaf(uu[q], h.w, gw2[q][3]);
                    }
                    const float g = S.g1[s][wj];
                    gw1[0] = fmaf(g, x.x, gw1[0]);
                    gw1[1] = fmaf(g, x.y, gw1[1]);
                    gw1[2] = fmaf(g, x.z, gw1[2]);
                    gw1[3] = fmaf(g, x.w, gw1[3]);
                }
                if (bk == 2) {
#pragma unroll
                    for (int s = 0; s < kTrainChunk; ++s) gb = fmaf(S.go[s], S.h2[s][bj], gb);
                } else {
                    const float *const v = bk == 0 ? &S.g1[0][bj] : bk == 1 ? &S.g2[0][bj] : (bj & 1) ? S.sq : S.go;
                    const int pitch = bk < 2 ? kActPitch : 1;
#pragma unroll
                    for (int s = 0; s < kTrainChunk; ++s) gb += v[s * pitch];
                }
                __syncthreads();  // the next pass overwrites the samples' values
            }
        }
        st_cluster4(to_w1, make_float4(gw1[0], gw1[1], gw1[2], gw1[3]));
#pragma unroll
        for (int q = 0; q < 4; ++q) st_cluster4(to_w2[q], make_float4(gw2[q][0], gw2[q][1], gw2[q][2], gw2[q][3]));
        if (bk < 3 || bj < 2) st_cluster(to_b, gb);
        __syncwarp();
        sp::cluster_barrier();  // every part has arrived
        if (owner) {
            float g[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float4 v = ld4(&S.parts[r * kSlice + 4 * t]);
                g[0] += v.x;
                g[1] += v.y;
                g[2] += v.z;
                g[3] += v.w;
            }
            float *const w = train_param(S, own);
            float next[4] = {w[0], w[1], w[2], w[3]};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (own + q == kParams) a.losses[step] = g[q];
                if (own + q >= kParams) continue;
                am[q] = a.beta1 * am[q] + (1.0f - a.beta1) * g[q];
                av[q] = a.beta2 * av[q] + (1.0f - a.beta2) * g[q] * g[q];
                next[q] -= a.lr * (am[q] * corr.x) / (sqrtf(av[q] * corr.y) + a.eps);
            }
#pragma unroll
            for (int r = 0; r < R; ++r)
                st_cluster4(sp::map_shared(w, r), make_float4(next[0], next[1], next[2], next[3]));
        }
        __syncwarp();
        sp::cluster_barrier();  // the parts have been read, the new parameters are everywhere
    }
    if (owner) {
        const float *const w = train_param(S, own);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (own + q >= kParams) continue;
            a.theta[own + q] = w[q];
            a.m[own + q] = am[q];
            a.v[own + q] = av[q];
        }
    }
}

template <int R>
cudaError_t train_launch_t(const TrainArgs &a, cudaStream_t st, bool probe)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = R;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(R);
    cfg.blockDim = dim3(kTrainThreads);
    cfg.dynamicSmemBytes = sizeof(TrainSmem);
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaFuncSetAttribute(train_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TrainSmem));
    if (e == cudaSuccess && R > 8) e = cudaFuncSetAttribute(train_kernel<R>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    if (!probe) return cudaLaunchKernelEx(&cfg, train_kernel<R>, a);
    int clusters = 0;
    e = cudaOccupancyMaxActiveClusters(&clusters, train_kernel<R>, &cfg);
    return e != cudaSuccess ? e : clusters > 0 ? cudaSuccess : cudaErrorInvalidConfiguration;
}

// CTAs of the training cluster on the current device, 0: none fits.  A size that
// does not fit is an answer, not an error of the call: it is cleared.
int train_ctas()
{
    const TrainArgs none = {};
    if (train_launch_t<kTrainCtas>(none, nullptr, true) == cudaSuccess) return kTrainCtas;
    cudaGetLastError();
    if (train_launch_t<8>(none, nullptr, true) == cudaSuccess) return 8;
    cudaGetLastError();
    return 0;
}

cudaError_t train_launch(int ctas, const TrainArgs &a, cudaStream_t st)
{
    return ctas == kTrainCtas ? train_launch_t<kTrainCtas>(a, st, false) : train_launch_t<8>(a, st, false);
}

size_t grad_smem_bytes() { return sizeof(float) * (kParams + (kIn + 4 * kHid) * kPitch + 2 * kPitch); }

// SplitMix64 (Steele, Lea and Flood, OOPSLA 2014) as a counter-based stream:
// output i of the stream at `seed` is mix(seed + (i + 1) * golden).
uint64_t splitmix64(uint64_t seed, uint64_t i)
{
    uint64_t z = seed + (i + 1) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Order of epoch ep: the stable argsort of the uniforms 2^42 + ep 2^32 + i of
// the stream.  The 53-bit outputs sort as the uniforms do and are spread
// evenly, so one counting pass by their leading bits leaves about one sample a
// bucket, and sorting within buckets is next to nothing (16384 samples:
// comparison sort 0.85 ms, this 0.03 ms).
void epoch_order(uint64_t seed, int ep, int64_t n, std::vector<int> *order)
{
    int bits = 1;
    while (((int64_t)1 << bits) < n) ++bits;
    std::vector<uint64_t> key((size_t)n), sorted((size_t)n);
    std::vector<int> first(((size_t)1 << bits) + 1, 0);
    for (int64_t i = 0; i < n; ++i) {
        key[(size_t)i] = splitmix64(seed, (1ull << 42) + ((uint64_t)ep << 32) + (uint64_t)i) >> 11;
        ++first[(size_t)(key[(size_t)i] >> (53 - bits)) + 1];
    }
    for (size_t b = 1; b < first.size(); ++b) first[b] += first[b - 1];
    order->resize((size_t)n);
    for (int64_t i = 0; i < n; ++i) {
        // the next place of the bucket, moved up past larger keys (equal ones keep their order)
        const uint64_t k = key[(size_t)i];
        int at = first[(size_t)(k >> (53 - bits))]++;
        while (at > 0 && sorted[(size_t)at - 1] > k && (sorted[(size_t)at - 1] >> (53 - bits)) == (k >> (53 - bits))) {
            sorted[(size_t)at] = sorted[(size_t)at - 1];
            (*order)[(size_t)at] = (*order)[(size_t)at - 1];
            --at;
        }
        sorted[(size_t)at] = k;
        (*order)[(size_t)at] = (int)i;
    }
}

// Waits for a stream on the way out of a call, so that host values its queued
// copies still read outlive them whichever way the call ends (declared after
// those values).
struct Drain {
    cudaStream_t stream;
    ~Drain() { cudaStreamSynchronize(stream); }
};

double uniform01(uint64_t seed, uint64_t i) { return (double)(splitmix64(seed, i) >> 11) * 0x1.0p-53; }

}  // namespace

struct sp_model {
    cudaStream_t stream = nullptr;
    int sms = 0;  // SMs of its device
    float *theta = nullptr, *m = nullptr, *v = nullptr, *grad = nullptr, *thr = nullptr;
    float *partial = nullptr;
    size_t cap_partial = 0;
    float *losses = nullptr;
    size_t cap_losses = 0;
    int *order = nullptr;
    size_t cap_order = 0;
    float2 *corr = nullptr;  // bias corrections of every step of a training call
    size_t cap_corr = 0;
    float *pred = nullptr;   // predictions on the training set
    size_t cap_pred = 0;
    int train_ctas = -1;     // of the training cluster; 0: none fits, -1: not asked yet
    int64_t adam_t = 0;
    float thr_host[3] = {0.0f, 0.0f, 0.0f};
};

namespace {

template <class T>
cudaError_t grow_buf(T **p, size_t *cap, size_t need)
{
    if (*cap >= need && *p) return cudaSuccess;
    if (*p) cudaFree(*p);
    *p = nullptr;
    *cap = 0;
    cudaError_t e = cudaMalloc((void **)p, std::max<size_t>(need, 1) * sizeof(T));
    if (e == cudaSuccess) *cap = std::max<size_t>(need, 1);
    return e;
}

int upload_params(sp_model *m, const float *host)
{
    cudaError_t e = cudaMemcpyAsync(m->theta, host, kParams * sizeof(float), cudaMemcpyHostToDevice, m->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->m, 0, kParams * sizeof(float), m->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->v, 0, kParams * sizeof(float), m->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(m->thr, m->thr_host, 3 * sizeof(float), cudaMemcpyHostToDevice, m->stream);
    m->adam_t = 0;
    return e == cudaSuccess ? SP_OK : SP_ECUDA;
}

// Gradient of the mean squared error over `count` samples into m->grad and
// the loss into *loss_dev (device, may be null).
int enqueue_grad(sp_model *m, const float *X, const float *Y, const int *idx, int count, float *loss_dev)
{
    const int blocks = (count + kGradBlock - 1) / kGradBlock;
    if (grow_buf(&m->partial, &m->cap_partial, (size_t)blocks * (kParams + 1)) != cudaSuccess) return SP_ENOMEM;
    const size_t smem = grad_smem_bytes();
    cudaError_t e = cudaFuncSetAttribute(mlp_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return SP_ECUDA;
    mlp_grad_kernel<<<blocks, kGradBlock, smem, m->stream>>>(m->theta, X, Y, idx, count, 1.0f / (float)count,
                                                              m->partial);
    grad_reduce_kernel<<<(kParams + 1 + 255) / 256, 256, 0, m->stream>>>(m->partial, blocks, m->grad, loss_dev);
    return cudaGetLastError() == cudaSuccess ? SP_OK : SP_ECUDA;
}

}  // namespace

extern "C" {

int sp_model_create(uint64_t seed, void *cuda_stream, sp_model **out)
{
    if (!out) return SP_EINVAL;
    *out = nullptr;
    sp_model *m = new (std::nothrow) sp_model();
    if (!m) return SP_ENOMEM;
    m->stream = (cudaStream_t)cuda_stream;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&m->sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaMalloc((void **)&m->theta, kParams * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc((void **)&m->m, kParams * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc((void **)&m->v, kParams * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc((void **)&m->grad, kParams * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc((void **)&m->thr, 3 * sizeof(float));
    if (e != cudaSuccess) {
        sp_model_destroy(m);
        return SP_ENOMEM;
    }
    // He-uniform weights: parameter k draws uniform k of the stream; a weight
    // of a layer with fan-in f is (2u - 1) sqrt(6 / f) in FP64, rounded once.
    std::vector<float> init(kParams, 0.0f);
    const int layer_off[3] = {kW1, kW2, kW3}, fan_in[3] = {kIn, kHid, kHid}, count[3] = {kHid * kIn, kHid * kHid, kHid};
    for (int l = 0; l < 3; ++l)
        for (int i = 0; i < count[l]; ++i) {
            const int k = layer_off[l] + i;
            init[k] = (float)((2.0 * uniform01(seed, (uint64_t)k) - 1.0) * std::sqrt(6.0 / fan_in[l]));
        }
    const int rc = upload_params(m, init.data());
    if (rc != SP_OK) {
        sp_model_destroy(m);
        return rc;
    }
    if (cudaStreamSynchronize(m->stream) != cudaSuccess) {
        sp_model_destroy(m);
        return SP_ECUDA;
    }
    *out = m;
    return SP_OK;
}

int sp_model_destroy(sp_model *m)
{
    if (!m) return SP_EINVAL;
    cudaFree(m->theta);
    cudaFree(m->m);
    cudaFree(m->v);
    cudaFree(m->grad);
    cudaFree(m->thr);
    cudaFree(m->partial);
    cudaFree(m->losses);
    cudaFree(m->order);
    cudaFree(m->corr);
    cudaFree(m->pred);
    delete m;
    return SP_OK;
}

int sp_model_get_params(sp_model *m, float *params_host, float *thresholds_host)
{
    if (!m || !params_host) return SP_EINVAL;
    cudaError_t e = cudaMemcpyAsync(params_host, m->theta, kParams * sizeof(float), cudaMemcpyDeviceToHost, m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    if (e != cudaSuccess) return SP_ECUDA;
    if (thresholds_host) std::memcpy(thresholds_host, m->thr_host, sizeof m->thr_host);
    return SP_OK;
}

int sp_model_set_params(sp_model *m, const float *params_host, const float *thresholds_host)
{
    if (!m || !params_host) return SP_EINVAL;
    if (thresholds_host) {
        if (!(thresholds_host[0] >= thresholds_host[1] && thresholds_host[1] >= thresholds_host[2])) return SP_EINVAL;
        std::memcpy(m->thr_host, thresholds_host, sizeof m->thr_host);
    }
    const int rc = upload_params(m, params_host);
    if (rc != SP_OK) return rc;
    return cudaStreamSynchronize(m->stream) == cudaSuccess ? SP_OK : SP_ECUDA;
}

int sp_model_predict(sp_model *m, const float *x_dev, int64_t n, float *y_dev)
{
    if (!m || n < 0 || (n > 0 && (!x_dev || !y_dev))) return SP_EINVAL;
    if (n == 0) return SP_OK;
    if (infer<false>(m->theta, nullptr, x_dev, n, y_dev, nullptr, m->sms, m->stream) != cudaSuccess) return SP_ECUDA;
    return cudaStreamSynchronize(m->stream) == cudaSuccess ? SP_OK : SP_ECUDA;
}

int sp_model_grad(sp_model *m, const float *x_dev, const float *y_dev, int64_t n, float *grad_host, double *loss)
{
    if (!m || n < 1 || n > (1 << 24) || !x_dev || !y_dev || !grad_host) return SP_EINVAL;
    if (grow_buf(&m->losses, &m->cap_losses, 1) != cudaSuccess) return SP_ENOMEM;
    int rc = enqueue_grad(m, x_dev, y_dev, nullptr, (int)n, m->losses);
    if (rc != SP_OK) return rc;
    float l = 0.0f;
    cudaError_t e = cudaMemcpyAsync(grad_host, m->grad, kParams * sizeof(float), cudaMemcpyDeviceToHost, m->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&l, m->losses, sizeof l, cudaMemcpyDeviceToHost, m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    if (e != cudaSuccess) return SP_ECUDA;
    if (loss) *loss = l;
    return SP_OK;
}

int sp_model_adam_step(sp_model *m, const float *grad_host, float lr, float beta1, float beta2, float eps)
{
    if (!m || !grad_host || !(lr > 0) || !(beta1 >= 0 && beta1 < 1) || !(beta2 >= 0 && beta2 < 1) || !(eps > 0))
        return SP_EINVAL;
    cudaError_t e = cudaMemcpyAsync(m->grad, grad_host, kParams * sizeof(float), cudaMemcpyHostToDevice, m->stream);
    if (e != cudaSuccess) return SP_ECUDA;
    ++m->adam_t;
    const float c1 = (float)(1.0 / (1.0 - std::pow((double)beta1, (double)m->adam_t)));
    const float c2 = (float)(1.0 / (1.0 - std::pow((double)beta2, (double)m->adam_t)));
    adam_kernel<<<(kParams + 255) / 256, 256, 0, m->stream>>>(m->theta, m->m, m->v, m->grad, lr, beta1, beta2, eps,
                                                              c1, c2);
    if (cudaGetLastError() != cudaSuccess) return SP_ECUDA;
    return cudaStreamSynchronize(m->stream) == cudaSuccess ? SP_OK : SP_ECUDA;
}

int sp_model_train(sp_model *m, const float *x_dev, const float *y_dev, int64_t n, int32_t epochs, int32_t batch,
                   float lr, uint64_t order_seed, const int32_t *order_host, float *losses_host)
{
    if (!m || !x_dev || !y_dev || n < 1 || n > (1 << 24) || epochs < 1 || batch < 1 || batch > (1 << 20) || !(lr > 0))
        return SP_EINVAL;
    const size_t total = (size_t)n * (size_t)epochs;
    const int64_t per_epoch = (n + batch - 1) / batch;
    const size_t steps = (size_t)per_epoch * epochs;
    if (order_host)
        for (size_t i = 0; i < total; ++i)
            if (order_host[i] < 0 || order_host[i] >= n) return SP_EINVAL;
    if (grow_buf(&m->order, &m->cap_order, total) != cudaSuccess) return SP_ENOMEM;
    if (grow_buf(&m->losses, &m->cap_losses, steps) != cudaSuccess) return SP_ENOMEM;
    const float beta1 = 0.9f, beta2 = 0.999f, eps = 1e-8f;
    // What the call's copies read or write on the host.  An asynchronous copy from
    // pageable memory may read it as late as its turn on the stream, behind the
    // training before it, so every epoch's order stands by itself.
    std::vector<float2> corr(steps);
    std::vector<std::vector<int>> orders(order_host ? 0 : (size_t)epochs);
    std::vector<float> pred((size_t)n);
    const Drain drain{m->stream};
    for (size_t k = 0; k < steps; ++k) {
        const double t = (double)(m->adam_t + (int64_t)k + 1);
        corr[k] = make_float2((float)(1.0 / (1.0 - std::pow((double)beta1, t))), (float)(1.0 / (1.0 - std::pow((double)beta2, t))));
    }
    if (m->train_ctas < 0) m->train_ctas = train_ctas();
    const int ctas = std::min<int64_t>(batch, n) <= kTrainMaxBatch ? m->train_ctas : 0;
    cudaError_t e = cudaSuccess;
    if (ctas) {
        if (grow_buf(&m->corr, &m->cap_corr, steps) != cudaSuccess) return SP_ENOMEM;
        e = cudaMemcpyAsync(m->corr, corr.data(), steps * sizeof(float2), cudaMemcpyHostToDevice, m->stream);
        if (e != cudaSuccess) return SP_ECUDA;
    }
    // epoch by epoch: while the GPU trains one, the host makes the next one's order
    size_t step = 0;
    for (int ep = 0; ep < epochs; ++ep) {
        const int *src = order_host ? order_host + (size_t)ep * n : nullptr;
        if (!src) {
            epoch_order(order_seed, ep, n, &orders[(size_t)ep]);
            src = orders[(size_t)ep].data();
        }
        int *const d_order = m->order + (size_t)ep * n;
        e = cudaMemcpyAsync(d_order, src, (size_t)n * sizeof(int), cudaMemcpyHostToDevice, m->stream);
        if (e != cudaSuccess) return SP_ECUDA;
        if (ctas) {
            TrainArgs a = {};
            a.theta = m->theta, a.m = m->m, a.v = m->v;
            a.X = x_dev, a.Y = y_dev, a.order = d_order;
            a.corr = m->corr + step, a.losses = m->losses + step;
            a.n = (int)n, a.batch = batch, a.steps = (int)per_epoch;
            a.lr = lr, a.beta1 = beta1, a.beta2 = beta2, a.eps = eps;
            if (train_launch(ctas, a, m->stream) != cudaSuccess) return SP_ECUDA;
            step += (size_t)per_epoch;
            m->adam_t += per_epoch;
            continue;
        }
        for (int64_t s0 = 0; s0 < n; s0 += batch, ++step) {
            const int count = (int)std::min<int64_t>(batch, n - s0);
            int rc = enqueue_grad(m, x_dev, y_dev, d_order + s0, count, m->losses + step);
            if (rc != SP_OK) return rc;
            ++m->adam_t;
            adam_kernel<<<(kParams + 255) / 256, 256, 0, m->stream>>>(m->theta, m->m, m->v, m->grad, lr, beta1, beta2, eps,
                                                                      corr[step].x, corr[step].y);
        }
    }
    if (cudaGetLastError() != cudaSuccess) return SP_ECUDA;
    if (losses_host) {
        e = cudaMemcpyAsync(losses_host, m->losses, steps * sizeof(float), cudaMemcpyDeviceToHost, m->stream);
        if (e != cudaSuccess) return SP_ECUDA;
    }
    // bucket thresholds: quartiles of the trained network's predictions on the
    // training set (order statistics, largest first)
    if (grow_buf(&m->pred, &m->cap_pred, (size_t)n) != cudaSuccess) return SP_ENOMEM;
    e = infer<false>(m->theta, nullptr, x_dev, n, m->pred, nullptr, m->sms, m->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(pred.data(), m->pred, (size_t)n * sizeof(float), cudaMemcpyDeviceToHost, m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    if (e != cudaSuccess) return SP_ECUDA;
    auto end = pred.end();
    for (int q = 0; q < 3; ++q) {
        const auto at = pred.begin() + (n - 1) * (3 - q) / 4;
        if (at < end) std::nth_element(pred.begin(), at, end);
        m->thr_host[q] = *at;
        end = at;
    }
    e = cudaMemcpyAsync(m->thr, m->thr_host, 3 * sizeof(float), cudaMemcpyHostToDevice, m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    return e == cudaSuccess ? SP_OK : SP_ECUDA;
}

// File: "SPMLP001", int32 parameter count, float params[count], float thresholds[3].
int sp_model_save(sp_model *m, const char *path)
{
    if (!m || !path) return SP_EINVAL;
    std::vector<float> p(kParams);
    int rc = sp_model_get_params(m, p.data(), nullptr);
    if (rc != SP_OK) return rc;
    FILE *f = std::fopen(path, "wb");
    if (!f) return SP_EINVAL;
    const int32_t cnt = kParams;
    bool ok = std::fwrite("SPMLP001", 1, 8, f) == 8 && std::fwrite(&cnt, sizeof cnt, 1, f) == 1 &&
              std::fwrite(p.data(), sizeof(float), kParams, f) == (size_t)kParams &&
              std::fwrite(m->thr_host, sizeof(float), 3, f) == 3;
    ok = (std::fclose(f) == 0) && ok;
    return ok ? SP_OK : SP_EINVAL;
}

int sp_model_load(const char *path, void *cuda_stream, sp_model **out)
{
    if (!path || !out) return SP_EINVAL;
    *out = nullptr;
    FILE *f = std::fopen(path, "rb");
    if (!f) return SP_EINVAL;
    char magic[8];
    int32_t cnt = 0;
    std::vector<float> p(kParams);
    float thr[3];
    bool ok = std::fread(magic, 1, 8, f) == 8 && std::memcmp(magic, "SPMLP001", 8) == 0 &&
              std::fread(&cnt, sizeof cnt, 1, f) == 1 && cnt == kParams &&
              std::fread(p.data(), sizeof(float), kParams, f) == (size_t)kParams &&
              std::fread(thr, sizeof(float), 3, f) == 3;
    std::fclose(f);
    if (!ok) return SP_EINVAL;
    sp_model *m = nullptr;
    int rc = sp_model_create(0, cuda_stream, &m);
    if (rc != SP_OK) return rc;
    rc = sp_model_set_params(m, p.data(), thr);
    if (rc != SP_OK) {
        sp_model_destroy(m);
        return rc;
    }
    *out = m;
    return SP_OK;
}

}  // extern "C"

namespace sp {

// Priority bucket of every region of a launch from its features (used by
// sp_evolve with the learned ordering).
cudaError_t model_buckets(const sp_model *m, const float *X, long long n, unsigned char *prio, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    return infer<true>(m->theta, m->thr, X, n, nullptr, prio, m->sms, st);
}

}  // namespace sp
