// k_mlp.cu -- the learned k-ladder predictor: a 64 -> 128 -> 128 -> 33 ReLU MLP
// trained on the GPU (FP32 master weights, Adam) and run for inference in
// BF16 (a component of this library, not of the paper).
//
// Loss of a batch: mean over its samples of the cross-entropy between
// softmax(y[0:32]) and the target fractions t[0:32], plus (y[32] - t[32])^2.
//
// Training is one cooperative launch per call of qsg_mlp_train (up to 256
// steps): per step, the blocks compute the gradients of the batch's tiles of 16
// samples (forward, loss, backward) into a partial-gradient buffer, meet at a
// grid barrier, sum the tiles' partial gradients in tile order and apply Adam
// (one thread per parameter), and meet again.  Every sum runs in a fixed
// order, so training is deterministic.  A step is a few MFLOP on 29k
// parameters, so what counts is latency: the weights are staged in shared
// memory once per tile with 16-byte loads, in rows padded so that both the
// forward products (16-byte reads along a row, one row per lane) and the
// backward ones (4-byte reads along a column index, one column per lane) are
// free of bank conflicts, and 512 threads share a tile.  With one thread per
// hidden unit, weights read from global memory for every sample and two
// launches per step, a step of 128 samples took 280 us; it takes 28 us now.
#include <cmath>

#include <cuda_bf16.h>

#include "qsg_launch.h"

namespace qsg {

constexpr int kIn = 64, kH = 128, kOut = 33, kTile = 16;
constexpr int oW1 = 0, oB1 = oW1 + kH * kIn, oW2 = oB1 + kH, oB2 = oW2 + kH * kH, oW3 = oB2 + kH,
              oB3 = oW3 + kOut * kH, kParams = oB3 + kOut;
static_assert(kParams == 29089, "parameter layout");

constexpr int kMlpThreads = 512;
// rows padded by 16 bytes: a quarter warp's eight 16-byte reads of eight
// consecutive rows fall into different banks
constexpr int kP1 = kIn + 4, kPH = kH + 4;

// The weights in shared memory.
struct Weights {
    float W1[kH][kP1];
    float W2[kH][kPH];
    float W3[kOut][kPH];
    float b1[kH], b2[kH], b3[kOut + 3];
};

// Activations and gradients of one tile.
struct Tile {
    float x[kTile][kP1];
    float z1[kTile][kPH], z2[kTile][kPH];  // before the ReLU
    float y[kTile][kOut + 3];
    float dyT[kOut + 3][kTile], d2T[kH][kTile], d1T[kH][kTile];  // dL/dy, dL/dz2, dL/dz1 by unit
    float lsum[kTile];
};

int mlp_param_count() { return kParams; }

// Copy the parameters to shared memory, asynchronously (every load in flight
// at once) and past L1 (the previous step of the same launch wrote them). The
// caller's next barrier follows stage_wait.
__device__ __forceinline__ void stage_weights(const float *P, Weights &w) {
    const int tid = threadIdx.x;
    auto rows = [&](const float *src, float *dst, int n, int len, int pitch) {
        const int q = len / 4;
#pragma unroll 8
        for (int e = tid; e < n * q; e += kMlpThreads)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(
                             (unsigned)__cvta_generic_to_shared(dst + (e / q) * pitch + 4 * (e % q))),
                         "l"(src + 4 * e)
                         : "memory");
    };
    rows(P + oW1, &w.W1[0][0], kH, kIn, kP1);
    rows(P + oW2, &w.W2[0][0], kH, kH, kPH);
    rows(P + oW3, &w.W3[0][0], kOut, kH, kPH);
    if (tid < kH) {
        w.b1[tid] = __ldcg(P + oB1 + tid);
        w.b2[tid] = __ldcg(P + oB2 + tid);
        if (tid < kOut) w.b3[tid] = __ldcg(P + oB3 + tid);
    }
}
__device__ __forceinline__ void stage_wait() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// acc[k] += row . a[k] over n (a multiple of 4) terms in increasing order; `in`
// maps an activation before it is used.
template <int S, class In>
__device__ __forceinline__ void dots(const float *row, const float *const (&a)[S], int n, float (&acc)[S], In &&in) {
#pragma unroll 4
    for (int i = 0; i < n; i += 4) {
        const float4 w = *reinterpret_cast<const float4 *>(row + i);
#pragma unroll
        for (int k = 0; k < S; ++k) {
            const float4 v = *reinterpret_cast<const float4 *>(a[k] + i);
            acc[k] = fmaf(w.x, in(v.x), acc[k]);
            acc[k] = fmaf(w.y, in(v.y), acc[k]);
            acc[k] = fmaf(w.z, in(v.z), acc[k]);
            acc[k] = fmaf(w.w, in(v.w), acc[k]);
        }
    }
}

__device__ __forceinline__ float relu(float v) { return fmaxf(v, 0.0f); }

// Forward, loss and backward of samples idx[t0 .. t0 + nt) (nt <= 16); the
// tile's gradient goes to G, its loss to *loss.  Units of the padding samples
// are computed from zeros and never written.
__device__ void tile_gradient(const Weights &w, Tile &t, const float *__restrict__ X, const float *__restrict__ T,
                              const int *__restrict__ idx, int t0, int nt, float inv_b, float *__restrict__ G,
                              float *loss) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int e = tid; e < kTile * (kIn / 4); e += kMlpThreads) {
        const int s = e / (kIn / 4), q = e % (kIn / 4);
        const float4 v = s < nt ? __ldg(reinterpret_cast<const float4 *>(X + (size_t)idx[t0 + s] * kIn) + q)
                                : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        *reinterpret_cast<float4 *>(&t.x[s][4 * q]) = v;
    }
    __syncthreads();
    // layers 1 and 2: thread = (hidden unit, four samples)
    const int j = tid & (kH - 1), s0 = 4 * (tid >> 7);
    {
        float a[4] = {w.b1[j], w.b1[j], w.b1[j], w.b1[j]};
        const float *const in[4] = {t.x[s0], t.x[s0 + 1], t.x[s0 + 2], t.x[s0 + 3]};
        dots<4>(w.W1[j], in, kIn, a, [](float v) { return v; });
#pragma unroll
        for (int k = 0; k < 4; ++k) t.z1[s0 + k][j] = a[k];
    }
    __syncthreads();
    {
        float a[4] = {w.b2[j], w.b2[j], w.b2[j], w.b2[j]};
        const float *const in[4] = {t.z1[s0], t.z1[s0 + 1], t.z1[s0 + 2], t.z1[s0 + 3]};
        dots<4>(w.W2[j], in, kH, a, relu);
#pragma unroll
        for (int k = 0; k < 4; ++k) t.z2[s0 + k][j] = a[k];
    }
    __syncthreads();
    // layer 3: thread = (output, sample); 33 outputs x 16 samples
    for (int e = tid; e < kOut * kTile; e += kMlpThreads) {
        const int s = e / kOut, o = e % kOut;
        float a[1] = {w.b3[o]};
        const float *const in[1] = {t.z2[s]};
        dots<1>(w.W3[o], in, kH, a, relu);
        t.y[s][o] = a[0];
    }
    __syncthreads();
    // loss and dL/dy: warp = sample, lane = output; sums in output order
    {
        const int s = warp;
        if (s < nt) {
            const float *tt = T + (size_t)idx[t0 + s] * kOut;
            const float yo = t.y[s][lane], to = __ldg(tt + lane);
            float mx = yo;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            const float ex = expf(yo - mx);
            float se = 0.0f, tsum = 0.0f;
#pragma unroll
            for (int o = 0; o < 32; ++o) {
                se += __shfl_sync(0xffffffffu, ex, o);
                tsum += __shfl_sync(0xffffffffu, to, o);
            }
            const float lse = logf(se);
            const float logp = yo - mx - lse;
            float ce = 0.0f;
#pragma unroll
            for (int o = 0; o < 32; ++o)
                ce -= __shfl_sync(0xffffffffu, to, o) * __shfl_sync(0xffffffffu, logp, o);
            t.dyT[lane][s] = (expf(logp) * tsum - to) * inv_b;
            if (lane == 0) {
                const float r = t.y[s][32] - __ldg(tt + 32);
                t.dyT[32][s] = 2.0f * r * inv_b;
                t.lsum[s] = ce + r * r;
            }
        } else {
            t.dyT[lane][s] = 0.0f;
            if (lane == 0) t.dyT[32][s] = 0.0f;
        }
    }
    __syncthreads();
    if (tid == 0) {
        float l = 0.0f;
        for (int s = 0; s < nt; ++s) l += t.lsum[s];
        *loss = l * inv_b;
    }
    // dL/dz2: thread = (unit, four samples)
    {
        float a[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 3
        for (int o = 0; o < kOut; ++o) {
            const float4 d = *reinterpret_cast<const float4 *>(&t.dyT[o][s0]);
            const float wv = w.W3[o][j];
            a[0] = fmaf(d.x, wv, a[0]);
            a[1] = fmaf(d.y, wv, a[1]);
            a[2] = fmaf(d.z, wv, a[2]);
            a[3] = fmaf(d.w, wv, a[3]);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) a[k] = t.z2[s0 + k][j] > 0.0f ? a[k] : 0.0f;
        *reinterpret_cast<float4 *>(&t.d2T[j][s0]) = make_float4(a[0], a[1], a[2], a[3]);
    }
    // weight gradient rows [0, n) of a layer: thread = (input i, every step-th
    // row); the inputs of the sixteen samples stay in registers
    auto weight_grad = [&](const float (*dT)[kTile], int n, const float (&v)[kTile], int i, int r0, int step, int len,
                           float *Gw) {
        for (int r = r0; r < n; r += step) {
            float a = 0.0f;
            const float4 *d = reinterpret_cast<const float4 *>(dT[r]);
#pragma unroll
            for (int q = 0; q < kTile / 4; ++q) {
                const float4 dv = d[q];
                if (4 * q + 0 < nt) a = fmaf(dv.x, v[4 * q + 0], a);
                if (4 * q + 1 < nt) a = fmaf(dv.y, v[4 * q + 1], a);
                if (4 * q + 2 < nt) a = fmaf(dv.z, v[4 * q + 2], a);
                if (4 * q + 3 < nt) a = fmaf(dv.w, v[4 * q + 3], a);
            }
            Gw[r * len + i] = a;
        }
    };
    auto bias_grad = [&](const float (*dT)[kTile], int n, float *Gb) {
        if (tid < n) {
            float a = 0.0f;
            for (int s = 0; s < nt; ++s) a += dT[tid][s];
            Gb[tid] = a;
        }
    };
    float v[kTile];
#pragma unroll
    for (int s = 0; s < kTile; ++s) v[s] = relu(t.z2[s][j]);
    weight_grad(t.dyT, kOut, v, j, tid >> 7, kMlpThreads / kH, kH, G + oW3);
    bias_grad(t.dyT, kOut, G + oB3);
    __syncthreads();
    // dL/dz1
    {
        float a[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 4
        for (int k = 0; k < kH; ++k) {
            const float4 d = *reinterpret_cast<const float4 *>(&t.d2T[k][s0]);
            const float wv = w.W2[k][j];
            a[0] = fmaf(d.x, wv, a[0]);
            a[1] = fmaf(d.y, wv, a[1]);
            a[2] = fmaf(d.z, wv, a[2]);
            a[3] = fmaf(d.w, wv, a[3]);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) a[k] = t.z1[s0 + k][j] > 0.0f ? a[k] : 0.0f;
        *reinterpret_cast<float4 *>(&t.d1T[j][s0]) = make_float4(a[0], a[1], a[2], a[3]);
    }
#pragma unroll
    for (int s = 0; s < kTile; ++s) v[s] = relu(t.z1[s][j]);
    weight_grad(t.d2T, kH, v, j, tid >> 7, kMlpThreads / kH, kH, G + oW2);
    bias_grad(t.d2T, kH, G + oB2);
    __syncthreads();
#pragma unroll
    for (int s = 0; s < kTile; ++s) v[s] = t.x[s][tid & (kIn - 1)];
    weight_grad(t.d1T, kH, v, tid & (kIn - 1), tid >> 6, kMlpThreads / kIn, kIn, G + oW1);
    bias_grad(t.d1T, kH, G + oB1);
}

// Barrier over the blocks of a cooperative launch: `count` is the number of
// arrivals so far of the launch (a multiple of the grid before the first).
// False, and *status set, when the wait gives up after `limit` polls.
__device__ __forceinline__ bool grid_barrier(unsigned *count, unsigned goal, int *status, unsigned limit) {
    __shared__ int ok;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        atomicAdd(count, 1u);
        int got = 0;
        for (unsigned it = 0; it < limit && !got; ++it) got = *(volatile unsigned *)count >= goal;
        if (!got) atomicExch(status, (int)DEVERR_TIMEOUT);
        ok = got;
    }
    __syncthreads();
    __threadfence();
    return ok != 0;
}

// `steps` training steps (adam != 0) or one gradient (adam = 0, grad_out).
// idx: [steps][batch] sample indices; corr: [steps][2] Adam's 1 - 0.9^t and
// 1 - 0.999^t (host FP64, rounded once); sync: {barrier count, status}, zero
// at launch.
__global__ void __launch_bounds__(kMlpThreads, 1)
    k_mlp_train(float *P, float *__restrict__ M, float *__restrict__ V, const float *__restrict__ X,
                const float *__restrict__ T, const int *__restrict__ idx, int steps, int batch, float *partial,
                float *loss_partial, float *grad_out, int adam, float lr, const float *__restrict__ corr,
                float *loss_out, unsigned *sync, unsigned wait_limit) {
    extern __shared__ __align__(16) unsigned char mlp_smem[];
    Weights &w = *reinterpret_cast<Weights *>(mlp_smem);
    Tile &t = *reinterpret_cast<Tile *>(mlp_smem + sizeof(Weights));
    const int ntiles = (batch + kTile - 1) / kTile;
    const float inv_b = 1.0f / (float)batch;
    unsigned goal = 0;
    for (int step = 0; step < steps; ++step) {
        const int *ix = idx + (size_t)step * batch;
        if ((int)blockIdx.x < ntiles) {
            stage_weights(P, w);
            stage_wait();  // the barrier after the tile's inputs follows
            for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
                const int t0 = tile * kTile;
                tile_gradient(w, t, X, T, ix, t0, min(kTile, batch - t0), inv_b, partial + (size_t)tile * kParams,
                              loss_partial + tile);
                __syncthreads();  // the tile's buffers are reused
            }
        }
        goal += gridDim.x;
        if (!grid_barrier(sync, goal, reinterpret_cast<int *>(sync + 1), wait_limit)) return;
        const float c1 = corr[2 * step], c2 = corr[2 * step + 1];
        for (int p = blockIdx.x * kMlpThreads + threadIdx.x; p < kParams; p += gridDim.x * kMlpThreads) {
            float g = 0.0f;
#pragma unroll 8
            for (int b = 0; b < ntiles; ++b) g += __ldcg(partial + (size_t)b * kParams + p);
            if (grad_out) grad_out[p] = g;
            if (adam) {
                // Adam (Kingma & Ba 2015)
                const float m = 0.9f * M[p] + 0.1f * g;
                const float v = 0.999f * V[p] + 0.001f * g * g;
                M[p] = m;
                V[p] = v;
                P[p] -= lr * (m / c1) / (sqrtf(v / c2) + 1e-8f);
            }
        }
        if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {
            float l = 0.0f;
            for (int b = 0; b < ntiles; ++b) l += __ldcg(loss_partial + b);
            loss_out[step] = l;
        }
        if (step + 1 == steps) break;
        goal += gridDim.x;
        if (!grid_barrier(sync, goal, reinterpret_cast<int *>(sync + 1), wait_limit)) return;
    }
}

cudaError_t launch_mlp_steps(float *P, float *M, float *V, const float *X, const float *T, const int *idx, int steps,
                             int batch, float *partial, float *loss_partial, float *grad_out, int adam, float lr,
                             const float *corr, float *loss_out, unsigned *sync, cudaStream_t st) {
    constexpr int sm = (int)(sizeof(Weights) + sizeof(Tile));
    static_assert(sm <= 227 * 1024, "one block per SM");
    int dev = 0, nsm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_mlp_train, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
    if (e == cudaSuccess) e = cudaMemsetAsync(sync, 0, 2 * sizeof(unsigned), st);
    if (e != cudaSuccess) return e;
    // a block per tile, and enough for one parameter per thread (57 blocks);
    // one block per SM at most (the blocks wait for one another)
    const int ntiles = (batch + kTile - 1) / kTile, nparam = (kParams + kMlpThreads - 1) / kMlpThreads;
    int blocks = ntiles > nparam ? ntiles : nparam;
    if (blocks > nsm) blocks = nsm;
    unsigned limit = kDefaultWaitLimit;
    void *args[] = {&P, &M, &V, &X, &T, &idx, &steps, &batch, &partial, &loss_partial, &grad_out, &adam, &lr, &corr,
                    &loss_out, &sync, &limit};
    count_launches(1);
    return cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(k_mlp_train), dim3((unsigned)blocks),
                                       dim3(kMlpThreads), args, (size_t)sm, st);
}

// ---------------------------------------------------------------------------
// Inference.  FP32: plain forward.  BF16: weights, inputs and hidden
// activations rounded to bfloat16 (nearest even), products and sums in FP32.
// A block stages the weights once (rounding them on the way) and runs tiles
// of 4 S samples, one hidden unit and S samples per thread; with a block and a
// pass over the weights in global memory per sample, 256 samples took 33 us.
// ---------------------------------------------------------------------------
template <int S>
struct InferTile {
    float x[4 * S][kP1], h1[4 * S][kPH], h2[4 * S][kPH];
};

template <bool BF16, int S>
__global__ void __launch_bounds__(kMlpThreads, 1) k_mlp_infer(const float *P, const float *__restrict__ X,
                                                              float *__restrict__ Y, long long n) {
    extern __shared__ __align__(16) unsigned char mlp_smem[];
    Weights &w = *reinterpret_cast<Weights *>(mlp_smem);
    InferTile<S> &t = *reinterpret_cast<InferTile<S> *>(mlp_smem + sizeof(Weights));
    constexpr int TS = 4 * S;
    const int tid = threadIdx.x;
    auto act = [](float v) { return BF16 ? __bfloat162float(__float2bfloat16_rn(v)) : v; };
    auto same = [](float v) { return v; };
    stage_weights(P, w);
    stage_wait();
    if (BF16) {
        // round in place: every thread its share of all of it
        __syncthreads();
        float *all = reinterpret_cast<float *>(mlp_smem);
        for (int e = tid; e < (int)(sizeof(Weights) / sizeof(float)); e += kMlpThreads) all[e] = act(all[e]);
    }
    const int j = tid & (kH - 1), s0 = S * (tid >> 7);
    for (long long base = (long long)blockIdx.x * TS; base < n; base += (long long)gridDim.x * TS) {
        const int nt = (int)(n - base < TS ? n - base : TS);
        for (int e = tid; e < TS * (kIn / 4); e += kMlpThreads) {
            const int s = e / (kIn / 4), q = e % (kIn / 4);
            float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (s < nt) v = __ldg(reinterpret_cast<const float4 *>(X + (size_t)(base + s) * kIn) + q);
            *reinterpret_cast<float4 *>(&t.x[s][4 * q]) = make_float4(act(v.x), act(v.y), act(v.z), act(v.w));
        }
        __syncthreads();
        {
            float a[S];
            const float *in[S];
#pragma unroll
            for (int k = 0; k < S; ++k) {
                a[k] = w.b1[j];
                in[k] = t.x[s0 + k];
            }
            dots<S>(w.W1[j], in, kIn, a, same);
#pragma unroll
            for (int k = 0; k < S; ++k) t.h1[s0 + k][j] = act(relu(a[k]));
        }
        __syncthreads();
        {
            float a[S];
            const float *in[S];
#pragma unroll
            for (int k = 0; k < S; ++k) {
                a[k] = w.b2[j];
                in[k] = t.h1[s0 + k];
            }
            dots<S>(w.W2[j], in, kH, a, same);
#pragma unroll
            for (int k = 0; k < S; ++k) t.h2[s0 + k][j] = act(relu(a[k]));
        }
        __syncthreads();
        for (int e = tid; e < nt * kOut; e += kMlpThreads) {
            const int s = e / kOut, o = e % kOut;
            float a[1] = {w.b3[o]};
            const float *const in[1] = {t.h2[s]};
            dots<1>(w.W3[o], in, kH, a, same);
            Y[(size_t)base * kOut + e] = a[0];
        }
        __syncthreads();
    }
}

template <bool BF16, int S>
static cudaError_t launch_infer(const float *P, const float *X, float *Y, long long n, int nsm, cudaStream_t st) {
    constexpr int sm = (int)(sizeof(Weights) + sizeof(InferTile<S>));
    const cudaError_t e = cudaFuncSetAttribute(k_mlp_infer<BF16, S>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
    if (e != cudaSuccess) return e;
    const long long tiles = (n + 4 * S - 1) / (4 * S);
    count_launches(1);
    k_mlp_infer<BF16, S><<<(unsigned)(tiles < nsm ? tiles : nsm), kMlpThreads, sm, st>>>(P, X, Y, n);
    return cudaGetLastError();
}

cudaError_t launch_mlp_infer(const float *P, const float *X, float *Y, long long n, int bf16, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    int dev = 0, nsm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    // one sample per thread while every tile of four has an SM of its own,
    // else four (a weight read then serves four products)
    const bool wide = n > 4LL * nsm;
    if (bf16) return wide ? launch_infer<true, 4>(P, X, Y, n, nsm, st) : launch_infer<true, 1>(P, X, Y, n, nsm, st);
    return wide ? launch_infer<false, 4>(P, X, Y, n, nsm, st) : launch_infer<false, 1>(P, X, Y, n, nsm, st);
}

}  // namespace qsg
