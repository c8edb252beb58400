// k_mlp.cu -- the learned k-ladder predictor: a 64 -> 128 -> 128 -> 33 ReLU MLP
// trained on the GPU (FP32 master weights, Adam) and run for inference in
// BF16 (a component of this library, not of the paper).
//
// Loss of a batch: mean over its samples of the cross-entropy between
// softmax(y[0:32]) and the target fractions t[0:32], plus (y[32] - t[32])^2.
//
// Training is one cooperative launch per call of qsg_mlp_train (up to 256
// steps).  A step has two halves with a grid barrier after each.  In the first
// a block runs four samples through the network and back (forward, loss, dL/dz
// of every layer) and writes their activations and dL/dz; in the second every
// parameter's gradient is summed over the batch and Adam applied at once: four
// warps share two rows and 32 columns of a weight matrix (an activation then serves
// both rows), each taking every fourth tile of 16 samples.  Every sum runs in a
// fixed order (samples within tiles, tiles in order), so training is deterministic.
//
// A step is a few MFLOP on 29k parameters, so what counts is latency.  The
// weights are staged in shared memory with 16-byte loads, layer by layer behind
// the products, in rows padded so that both the forward products (16-byte reads
// along a row, one row per lane) and the backward ones (4-byte reads along a
// column index, one column per lane) are free of bank conflicts.  Four samples per
// block spread a batch of 128 over 32 SMs and the parameter sums over all of
// them; whole rows per sample go out, because dL/dz written by unit, a few bytes to
// each of 128 rows, cost 2 us at a batch of 128 and 11 at 608.
//
// A step of 128 samples, us: one thread per hidden unit, weights read from global
// memory for every sample and two launches 280; blocks of 16 samples that also sum
// their own weight gradients, added up across tiles by a second pass, 28; this form
// 13.6 (11.7 for 16 samples, 16.4 for 256, 24 for 608; the form before 27, 28, 31.
// Past about a thousand samples that one reads less, 3,000: 88 against 60, but such
// batches are no use to a predictor trained on a few thousand samples).
#include <cmath>

#include <cuda_bf16.h>

#include "coop_launch.h"
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

constexpr int kOutP = kOut + 3;  // a row of dL/dy, padded
constexpr int kUnit = 4;  // samples a block takes through the network at a time

// Activations and gradients of one unit.
struct Unit {
    float x[kUnit][kP1];
    float z1[kUnit][kPH], z2[kUnit][kPH];  // before the ReLU
    float y[kUnit][kOut + 3];
    float dyT[kOut + 3][kUnit], d2T[kH][kUnit];  // dL/dy, dL/dz2 by unit
};

// What the parameter sums read, for n samples (the batch rounded up to whole tiles):
// inputs, ReLU outputs and dL/dz, a row per sample.
struct Acts {
    float *x, *h1, *h2, *d1, *d2, *dy, *loss;
    int n;
    __host__ __device__ Acts(float *base, int batch) {
        n = (batch + kTile - 1) / kTile * kTile;
        x = base;
        h1 = x + (size_t)n * kIn;
        h2 = h1 + (size_t)n * kH;
        d1 = h2 + (size_t)n * kH;
        d2 = d1 + (size_t)n * kH;
        dy = d2 + (size_t)n * kH;
        loss = dy + (size_t)n * kOutP;
    }
};
constexpr int kActWords = kIn + 4 * kH + kOutP + 1;  // per sample

int mlp_param_count() { return kParams; }
size_t mlp_act_words(int batch) { return (size_t)((batch + kTile - 1) / kTile * kTile) * kActWords; }

// Copy the parameters to shared memory, asynchronously (every load in flight
// at once, a group per layer) and past L1 (the previous step of the same launch
// wrote them). A barrier follows the stage_wait of a layer, whose N is the number
// of later layers.
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
    auto commit = [] { asm volatile("cp.async.commit_group;\n" ::: "memory"); };
    rows(P + oW1, &w.W1[0][0], kH, kIn, kP1);
    commit();
    rows(P + oW2, &w.W2[0][0], kH, kH, kPH);
    commit();
    rows(P + oW3, &w.W3[0][0], kOut, kH, kPH);
    commit();
    if (tid < kH) {
        w.b1[tid] = __ldcg(P + oB1 + tid);
        w.b2[tid] = __ldcg(P + oB2 + tid);
        if (tid < kOut) w.b3[tid] = __ldcg(P + oB3 + tid);
    }
}
template <int N>
__device__ __forceinline__ void stage_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

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

// Forward, loss and backward of samples s0 .. s0 + nt of the batch (nt <= 4);
// the padding samples are computed from zeros, and their results never read.
// Called with the weights' copies in flight.
__device__ void unit_pass(const Weights &w, Unit &t, const float *__restrict__ X, const float *__restrict__ T,
                          const int *__restrict__ idx, int s0, int nt, float inv_b, const Acts &A) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int e = tid; e < kUnit * (kIn / 4); e += kMlpThreads) {
        const int s = e / (kIn / 4), q = e % (kIn / 4);
        const float4 v = s < nt ? __ldg(reinterpret_cast<const float4 *>(X + (size_t)idx[s0 + s] * kIn) + q)
                                : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        *reinterpret_cast<float4 *>(&t.x[s][4 * q]) = v;
        *reinterpret_cast<float4 *>(A.x + (size_t)(s0 + s) * kIn + 4 * q) = v;
    }
    stage_wait<2>();
    __syncthreads();
    // hidden layers: thread = (unit, two samples), in half of the warps
    const bool half = tid < 2 * kH;
    const int j = tid & (kH - 1), k0 = 2 * (tid >> 7 & 1);
    if (half) {
        float a[2] = {w.b1[j], w.b1[j]};
        const float *const in[2] = {t.x[k0], t.x[k0 + 1]};
        dots<2>(w.W1[j], in, kIn, a, [](float v) { return v; });
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            t.z1[k0 + k][j] = a[k];
            A.h1[(size_t)(s0 + k0 + k) * kH + j] = relu(a[k]);
        }
    }
    stage_wait<1>();
    __syncthreads();
    if (half) {
        float a[2] = {w.b2[j], w.b2[j]};
        const float *const in[2] = {t.z1[k0], t.z1[k0 + 1]};
        dots<2>(w.W2[j], in, kH, a, relu);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            t.z2[k0 + k][j] = a[k];
            A.h2[(size_t)(s0 + k0 + k) * kH + j] = relu(a[k]);
        }
    }
    stage_wait<0>();
    __syncthreads();
    // layer 3: thread = (output, sample); 33 outputs x 4 samples
    if (tid < kOut * kUnit) {
        const int s = tid / kOut, o = tid % kOut;
        float a[1] = {w.b3[o]};
        const float *const in[1] = {t.z2[s]};
        dots<1>(w.W3[o], in, kH, a, relu);
        t.y[s][o] = a[0];
    }
    __syncthreads();
    // loss and dL/dy: warp = sample, lane = output; sums in output order
    if (warp < kUnit) {
        const int s = warp;
        float d = 0.0f, d32 = 0.0f;
        if (s < nt) {
            const float *tt = T + (size_t)idx[s0 + s] * kOut;
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
            d = (expf(logp) * tsum - to) * inv_b;
            const float r = t.y[s][32] - __ldg(tt + 32);
            d32 = 2.0f * r * inv_b;
            if (lane == 0) A.loss[s0 + s] = ce + r * r;
        }
        t.dyT[lane][s] = d;
        A.dy[(size_t)(s0 + s) * kOutP + lane] = d;
        if (lane == 0) {
            t.dyT[32][s] = d32;
            A.dy[(size_t)(s0 + s) * kOutP + 32] = d32;
        }
    }
    __syncthreads();
    // dL/dz2 and dL/dz1: thread = (unit, two samples)
    if (half) {
        float a[2] = {0.0f, 0.0f};
#pragma unroll 11
        for (int o = 0; o < kOut; ++o) {
            const float2 d = *reinterpret_cast<const float2 *>(&t.dyT[o][k0]);
            const float wv = w.W3[o][j];
            a[0] = fmaf(d.x, wv, a[0]);
            a[1] = fmaf(d.y, wv, a[1]);
        }
        const float2 d = make_float2(t.z2[k0][j] > 0.0f ? a[0] : 0.0f, t.z2[k0 + 1][j] > 0.0f ? a[1] : 0.0f);
        *reinterpret_cast<float2 *>(&t.d2T[j][k0]) = d;
        A.d2[(size_t)(s0 + k0) * kH + j] = d.x;
        A.d2[(size_t)(s0 + k0 + 1) * kH + j] = d.y;
    }
    __syncthreads();
    if (half) {
        float a[2] = {0.0f, 0.0f};
#pragma unroll 16
        for (int k = 0; k < kH; ++k) {
            const float2 d = *reinterpret_cast<const float2 *>(&t.d2T[k][k0]);
            const float wv = w.W2[k][j];
            a[0] = fmaf(d.x, wv, a[0]);
            a[1] = fmaf(d.y, wv, a[1]);
        }
        A.d1[(size_t)(s0 + k0) * kH + j] = t.z1[k0][j] > 0.0f ? a[0] : 0.0f;
        A.d1[(size_t)(s0 + k0 + 1) * kH + j] = t.z1[k0 + 1][j] > 0.0f ? a[1] : 0.0f;
    }
    __syncthreads();
}

// The parameter sums' work items, four warps each: two rows and 32 columns of a
// weight matrix, or 32 biases, or the loss.
constexpr int kItems1 = kH / 2 * (kIn / 32), kItems2 = kH / 2 * (kH / 32), kItems3 = (kOut + 1) / 2 * (kH / 32);
constexpr int kItemsB = (2 * kH + kOut + 31) / 32, kItems = kItems1 + kItems2 + kItems3 + kItemsB + 1;
constexpr int kTeam = 4, kTeams = kMlpThreads / 32 / kTeam;
constexpr int kRound = 32;  // tiles summed between two meetings of a team
struct Sums {
    float of[kTeams][kRound][2][32];
};

// What a team sums: dL/dz of two neighbouring units (rows dstride apart) times
// this lane's input (rows istride apart), or (no input) dL/dz of this lane's unit.
struct Item {
    const float *d, *in;
    int dstride, istride;
};

// The tile of samples t .. t + nt of one item; reads past L1.
__device__ __forceinline__ void tile_sum(const Item &it, int t, int nt, float &a0, float &a1) {
    a0 = a1 = 0.0f;
    if (it.in) {
        float v[kTile];
        float2 e[kTile];
#pragma unroll
        for (int s = 0; s < kTile; ++s) {
            v[s] = __ldcg(it.in + (size_t)(t + s) * it.istride);
            e[s] = __ldcg(reinterpret_cast<const float2 *>(it.d + (size_t)(t + s) * it.dstride));
        }
#pragma unroll
        for (int s = 0; s < kTile; ++s)
            if (s < nt) {
                a0 = fmaf(e[s].x, v[s], a0);
                a1 = fmaf(e[s].y, v[s], a1);
            }
    } else {
#pragma unroll
        for (int s = 0; s < kTile; ++s) {
            const float d = __ldcg(it.d + (size_t)(t + s) * it.dstride);
            if (s < nt) a0 += d;
        }
    }
}

// Sum over the batch, in tile order, by the four warps of a team: each takes every
// fourth tile of a round, then warps 0 and 1 add a row's tiles.  In warps 0 and 1
// the result is the sum of row 0 and 1.
__device__ __forceinline__ float team_sum(const Item &it, int batch, float (&of)[kRound][2][32], int team, int part,
                                          int lane) {
    float g = 0.0f;
    const int tiles = (batch + kTile - 1) / kTile;
    for (int r0 = 0; r0 < tiles; r0 += kRound) {
        const int n = min(kRound, tiles - r0);
        for (int b = part; b < n; b += kTeam) {
            const int t = (r0 + b) * kTile;
            tile_sum(it, t, min(kTile, batch - t), of[b][0][lane], of[b][1][lane]);
        }
        asm volatile("bar.sync %0, %1;\n" ::"r"(1 + team), "n"(32 * kTeam) : "memory");
        if (part < 2)
#pragma unroll 8
            for (int b = 0; b < n; ++b) g += of[b][part][lane];
        asm volatile("bar.sync %0, %1;\n" ::"r"(1 + team), "n"(32 * kTeam) : "memory");
    }
    return g;
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
// idx: [steps][batch] sample indices; act: mlp_act_words(batch) floats; corr:
// [steps][2] Adam's 1 - 0.9^t and 1 - 0.999^t (host FP64, rounded once); sync:
// {barrier count, status}, zero at launch.
__global__ void __launch_bounds__(kMlpThreads, 1)
    k_mlp_train(float *P, float *__restrict__ M, float *__restrict__ V, const float *__restrict__ X,
                const float *__restrict__ T, const int *__restrict__ idx, int steps, int batch, float *act,
                float *grad_out, int adam, float lr, const float *__restrict__ corr, float *loss_out, unsigned *sync,
                unsigned wait_limit) {
    extern __shared__ __align__(16) unsigned char mlp_smem[];
    Weights &w = *reinterpret_cast<Weights *>(mlp_smem);
    Unit &t = *reinterpret_cast<Unit *>(mlp_smem + sizeof(Weights));
    Sums &sums = *reinterpret_cast<Sums *>(mlp_smem + sizeof(Weights) + sizeof(Unit));
    const Acts A(act, batch);
    const int units = (batch + kUnit - 1) / kUnit;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const float inv_b = 1.0f / (float)batch;
    unsigned goal = 0;
    for (int step = 0; step < steps; ++step) {
        const int *ix = idx + (size_t)step * batch;
        if ((int)blockIdx.x < units) {
            stage_weights(P, w);
            for (int u = blockIdx.x; u < units; u += gridDim.x)
                unit_pass(w, t, X, T, ix, u * kUnit, min(kUnit, batch - u * kUnit), inv_b, A);
        }
        goal += gridDim.x;
        if (!grid_barrier(sync, goal, reinterpret_cast<int *>(sync + 1), wait_limit)) return;
        const float c1 = corr[2 * step], c2 = corr[2 * step + 1];
        auto apply = [&](int p, float g) {
            if (grad_out) grad_out[p] = g;
            if (adam) {
                // Adam (Kingma & Ba 2015)
                const float m = 0.9f * M[p] + 0.1f * g;
                const float v = 0.999f * V[p] + 0.001f * g * g;
                M[p] = m;
                V[p] = v;
                P[p] -= lr * (m / c1) / (sqrtf(v / c2) + 1e-8f);
            }
        };
        const int team = warp / kTeam, part = warp % kTeam;
        // two rows (the last of an odd number: one) and 32 columns
        auto weights = [&](int item, const float *d, int dstride, const float *in, int rows, int len, int base) {
            const int r = item / (len / 32) * 2, i = item % (len / 32) * 32 + lane;
            const float g = team_sum(Item{d + r, in + i, dstride, len}, batch, sums.of[team], team, part, lane);
            if (part < 2 && r + part < rows) apply(base + (r + part) * len + i, g);
        };
        for (int item = team * (int)gridDim.x + (int)blockIdx.x; item < kItems; item += (int)gridDim.x * kTeams) {
            int k = item;
            if (k < kItems2) {
                weights(k, A.d2, kH, A.h1, kH, kH, oW2);
            } else if ((k -= kItems2) < kItems3) {
                weights(k, A.dy, kOutP, A.h2, kOut, kH, oW3);
            } else if ((k -= kItems3) < kItems1) {
                weights(k, A.d1, kH, A.x, kH, kIn, oW1);
            } else if ((k -= kItems1) < kItemsB) {
                const int b = min(32 * k + lane, 2 * kH + kOut - 1);
                const Item it{b < kH ? A.d1 + b : (b < 2 * kH ? A.d2 + b - kH : A.dy + b - 2 * kH), nullptr,
                              b < 2 * kH ? kH : kOutP, 0};
                const float g = team_sum(it, batch, sums.of[team], team, part, lane);
                if (part == 0 && b == 32 * k + lane)
                    apply(b < kH ? oB1 + b : (b < 2 * kH ? oB2 + b - kH : oB3 + b - 2 * kH), g);
            } else if (part == 0) {
                // a tile's loss per lane, then the tiles in order
                float l = 0.0f;
                for (int t0 = 0; t0 < batch; t0 += 32 * kTile) {
                    const int t1 = t0 + lane * kTile;
                    float a = 0.0f;
#pragma unroll
                    for (int q = 0; q < kTile; ++q) {
                        const float v = t1 + q < batch ? __ldcg(A.loss + t1 + q) : 0.0f;
                        if (t1 + q < batch) a += v;
                    }
                    a *= inv_b;
                    const int n = min(32, (batch - t0 + kTile - 1) / kTile);
                    for (int b = 0; b < n; ++b) l += __shfl_sync(0xffffffffu, a, b);
                }
                if (lane == 0) loss_out[step] = l;
            }
        }
        if (step + 1 == steps) break;
        goal += gridDim.x;
        if (!grid_barrier(sync, goal, reinterpret_cast<int *>(sync + 1), wait_limit)) return;
    }
}

cudaError_t launch_mlp_steps(float *P, float *M, float *V, const float *X, const float *T, const int *idx, int steps,
                             int batch, float *act, float *grad_out, int adam, float lr, const float *corr,
                             float *loss_out, unsigned *sync, cudaStream_t st) {
    constexpr int sm = (int)(sizeof(Weights) + sizeof(Unit) + sizeof(Sums));
    static_assert(sm <= 227 * 1024, "one block per SM");
    int dev = 0, nsm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_mlp_train, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
    if (e == cudaSuccess) e = cudaMemsetAsync(sync, 0, 2 * sizeof(unsigned), st);
    if (e != cudaSuccess) return e;
    // a block per unit, and one for as many items of the parameter sums as it has
    // teams; one block per SM at most (the blocks wait for one another).  The sums do
    // not depend on the number of blocks.
    const int units = (batch + kUnit - 1) / kUnit, share = (kItems + kTeams - 1) / kTeams;
    int blocks = units > share ? units : share;
    if (blocks > nsm) blocks = nsm;
    unsigned limit = kDefaultWaitLimit;
    void *args[] = {&P, &M, &V, &X, &T, &idx, &steps, &batch, &act, &grad_out, &adam, &lr, &corr, &loss_out, &sync, &limit};
    count_launches(1);
    return launch_resident_grid(blocks, [&](int n) {
        return cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(k_mlp_train), dim3((unsigned)n),
                                           dim3(kMlpThreads), args, (size_t)sm, st);
    });
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
    stage_wait<0>();
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
