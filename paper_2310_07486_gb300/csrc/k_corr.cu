// k_corr.cu -- imaginary-time correlators C(tau), Q2(tau) and the equal-time
// replica overlap (Eqs. (C_A_transfer), (def-C-Q2-tau)), accumulated exactly
// in int64, and their FP64 finish.
//
// The multispin words hold 64 samples per site.  The correlators need, per
// sample, the overlap of two tau slices summed over sites, so the slices are
// first transposed into x-packed words (64 sites per word, one sample per
// row) in a scratch buffer; an overlap is then L^2 - 2 popc(a ^ b).
#include "qsg_launch.h"

namespace qsg {

size_t measure_scratch_words_per_pair(const Group &g) {
    return (size_t)g.R * 64 * g.Ltau * g.nwx;
}

// Bit matrix transpose step of half-size j across lanes l and l ^ j: bits
// whose index has bit j clear (mask m) stay in the lower row; the lower row
// takes the partner's low-half bits shifted up, the upper row the partner's
// high-half bits shifted down.  Five such steps (j = 16 .. 1) and the
// in-register step j = 32 swap the bits of (row, column): (s, b) -> (b, s).
template <int J>
__device__ __forceinline__ uint64_t transpose_step(uint64_t w, bool upper, uint64_t m) {
    const uint64_t p = __shfl_xor_sync(0xffffffffu, w, J);
    return upper ? ((w & ~m) | ((p >> J) & m)) : ((w & m) | ((p << J) & ~m));
}

// scratch layout for a batch of (w, j) pairs: [pair][r][b][tau][nwx].
// One block per (slot of the batch, run of kTrRun tau planes), one warp per
// plane: for every 64-site group the warp's lane l loads the multispin words
// of sites l and l + 32 (bit b = sample b, one coalesced 512-byte read),
// transposes the 64 x 64 bit block in registers and holds the x-packed words
// of samples l and l + 32, which it puts in shared memory.  The block then
// writes each sample's kTrRun x nwx words, contiguous in the scratch, as one
// coalesced run (a sample's words of one plane are nwx words long and the
// next sample's begin L_tau nwx words later, so a warp storing its two words
// straight would write 64 separate 8-byte pieces).
constexpr int kTrRun = 8;  // tau planes per block (warps of 32 threads)

__global__ void __launch_bounds__(32 * kTrRun) k_transpose(Group g, int p0, int npairs, uint64_t *P) {
    extern __shared__ uint64_t trs[];  // [64 samples][kTrRun * nwx + 1 (padding)]
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int nwx = g.nwx, Lt = g.Ltau, L2 = g.L * g.L;
    const int pitch = kTrRun * nwx + 1;
    const int sb = blockIdx.x;  // slot of the batch: (pair, replica)
    const int t0 = blockIdx.y * kTrRun, nt = min(kTrRun, Lt - t0);
    const int pb = sb / g.R, r = sb % g.R;
    const int p = p0 + pb, w = p / g.K, j = p % g.K;
    const size_t s = ((size_t)w * g.R + r) * g.K + j;
    if (sb >= npairs * g.R) return;  // the grid is exact: never taken
    if (wp < nt) {
        const int t = t0 + wp;
        const uint64_t *src = g.S + s * g.N + (size_t)t * L2;
        for (int gx = 0; gx < nwx; ++gx) {
            const int s0 = gx * 64 + lane, s1 = s0 + 32;
            const uint64_t w0 = s0 < L2 ? src[s0] : 0ull;
            const uint64_t w1 = s1 < L2 ? src[s1] : 0ull;
            // j = 32: rows l and l + 32 are both in this lane
            uint64_t a0 = (w0 & 0xFFFFFFFFull) | (w1 << 32);
            uint64_t a1 = (w0 >> 32) | (w1 & 0xFFFFFFFF00000000ull);
            a0 = transpose_step<16>(a0, lane & 16, 0x0000FFFF0000FFFFull);
            a1 = transpose_step<16>(a1, lane & 16, 0x0000FFFF0000FFFFull);
            a0 = transpose_step<8>(a0, lane & 8, 0x00FF00FF00FF00FFull);
            a1 = transpose_step<8>(a1, lane & 8, 0x00FF00FF00FF00FFull);
            a0 = transpose_step<4>(a0, lane & 4, 0x0F0F0F0F0F0F0F0Full);
            a1 = transpose_step<4>(a1, lane & 4, 0x0F0F0F0F0F0F0F0Full);
            a0 = transpose_step<2>(a0, lane & 2, 0x3333333333333333ull);
            a1 = transpose_step<2>(a1, lane & 2, 0x3333333333333333ull);
            a0 = transpose_step<1>(a0, lane & 1, 0x5555555555555555ull);
            a1 = transpose_step<1>(a1, lane & 1, 0x5555555555555555ull);
            trs[(size_t)lane * pitch + wp * nwx + gx] = a0;
            trs[(size_t)(lane + 32) * pitch + wp * nwx + gx] = a1;
        }
    }
    __syncthreads();
    // sample b's words of planes t0 .. t0 + nt - 1 are contiguous in the scratch
    const int n = nt * nwx;
    uint64_t *dst = P + ((size_t)sb * 64 * Lt + t0) * nwx;
    for (int b = wp; b < 64; b += kTrRun)
        for (int o = lane; o < n; o += 32) dst[(size_t)b * Lt * nwx + o] = trs[(size_t)b * pitch + o];
}

// One block per (slot of the batch, sample bit): all lags of one sample.
__global__ void __launch_bounds__(256) k_gram(Group g, int p0, const uint64_t *P, int use_smem) {
    extern __shared__ uint64_t sh[];
    const int sb = blockIdx.x / 64, b = blockIdx.x % 64;
    const int pb = sb / g.R, r = sb % g.R;
    const int p = p0 + pb, w = p / g.K, j = p % g.K;
    const int Lt = g.Ltau, nwx = g.nwx, L2 = g.L * g.L;
    const uint64_t *src = P + ((size_t)sb * 64 + b) * Lt * nwx;
    if (use_smem) {
        for (int i = threadIdx.x; i < Lt * nwx; i += blockDim.x) sh[i] = src[i];
        __syncthreads();
        src = sh;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    for (int lag = warp; lag < g.nlag; lag += nwarp) {
        long long cs = 0, qs = 0;
        for (int t1 = lane; t1 < Lt; t1 += 32) {
            int t2 = t1 + lag;
            int sgn = 1;
            if (t2 >= Lt) {
                t2 -= Lt;
                if (g.boundary == 1) sgn = -1;
            }
            int d = 0;
            for (int x = 0; x < nwx; ++x) d += __popcll(src[t1 * nwx + x] ^ src[t2 * nwx + x]);
            const long long c = (long long)(L2 - 2 * d);
            cs += sgn * c;
            qs += c * c;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            cs += __shfl_down_sync(0xffffffffu, cs, o);
            qs += __shfl_down_sync(0xffffffffu, qs, o);
        }
        if (lane == 0) {
            const size_t idx = ((((size_t)r * g.W * 64) + (size_t)w * 64 + b) * g.K + j) * g.nlag + lag;
            g.Cacc[idx] += cs;
            g.Qacc[idx] += qs;
        }
    }
}

// Short extents of tau: all lags of a few samples per block on the integer pipes.
// A 128 x 128 tensor tile has (L_tau / 128)^2 of its elements in use, and a unit of
// one step leaves its fold to the lag bins unhidden, so small lattices spent 8,000
// cycles per sample where XOR and popcount take a few hundred: L = 8, L_tau = 48,
// 81,920 samples 2,110 us with tensor tiles, 72 us here.
//
// The rows of kShortSamples(..) samples are staged in shared memory, followed by
// the first L_tau / 2 + 1 of them again as t >= L_tau (complemented under APBC: an
// overlap with them then has its sign flipped), so a lag is a plain row offset.  A
// thread owns the lags l, l + ng, l + 2 ng, l + 3 ng of one sample and walks the
// rows: one read of row t1 serves four lags, consecutive lanes read consecutive
// rows (an odd pitch keeps the banks apart).  Words are joined three at a time by a
// full adder (two popcounts for three words), the popcount's rate being a quarter
// of the logic's.  With n differing sites of L^2, c = L^2 - 2 n: the sums of n and
// n^2 give those of c and c^2.
constexpr int kShortThreads = 256;
constexpr int kShortWords = 4;  // 64-site words of a slice at most (L <= 16)

struct ShortShape {
    int ng;       // lag groups (threads) per sample
    int rows;     // rows staged per sample
    int samples;  // samples per block
    size_t bytes;
};
static ShortShape short_shape(const Group &g) {
    ShortShape s;
    s.ng = (g.nlag + 3) / 4;
    s.rows = g.Ltau + g.nlag;
    const int pitch = g.nwx | 1;
    const size_t per = ((size_t)s.rows * pitch | 1) * sizeof(uint64_t);
    s.samples = kShortThreads / s.ng;
    while (s.samples > 1 && s.samples * per > 40 * 1024) --s.samples;
    s.bytes = s.samples * per;
    return s;
}

template <int NX>
__device__ __forceinline__ int differing(const uint64_t (&x)[NX], const uint64_t *y) {
    uint32_t d[2 * NX];
#pragma unroll
    for (int k = 0; k < NX; ++k) {
        const uint64_t v = x[k] ^ y[k];
        d[2 * k] = (uint32_t)v;
        d[2 * k + 1] = (uint32_t)(v >> 32);
    }
    int one = 0, two = 0;
    constexpr int T = 2 * NX / 3;
#pragma unroll
    for (int k = 0; k < T; ++k) {
        one += __popc(d[3 * k] ^ d[3 * k + 1] ^ d[3 * k + 2]);
        two += __popc(maj3(d[3 * k], d[3 * k + 1], d[3 * k + 2]));
    }
#pragma unroll
    for (int k = 3 * T; k < 2 * NX; ++k) one += __popc(d[k]);
    return one + 2 * two;
}

template <int NX>
__global__ void __launch_bounds__(kShortThreads) k_gram_short(Group g, int p0, const uint64_t *__restrict__ P,
                                                              int nsamples, ShortShape sh) {
    extern __shared__ uint64_t rows[];
    constexpr int pitch = NX | 1;
    const int Lt = g.Ltau, L2 = g.L * g.L, nl = g.nlag;
    const int per = sh.rows * pitch | 1;
    const int s0 = blockIdx.x * sh.samples, ns = min(sh.samples, nsamples - s0);
    const uint64_t *src = P + (size_t)s0 * Lt * NX;
    const int n = Lt * NX;
    for (int i = threadIdx.x; i < ns * n; i += kShortThreads) {
        const int s = i / n, rk = i - s * n, t = rk / NX, k = rk - t * NX;
        uint64_t v = src[i];
        uint64_t *d = rows + (size_t)s * per + k;
        d[t * pitch] = v;
        if (t < nl) {
            if (g.boundary == 1) {
                const int left = L2 - 64 * k;  // sites of the lattice in this word
                v ^= left >= 64 ? ~0ull : (1ull << left) - 1;
            }
            d[(t + Lt) * pitch] = v;
        }
    }
    __syncthreads();
    const int sl = threadIdx.x / sh.ng, lg = threadIdx.x - sl * sh.ng;
    if (sl >= ns) return;
    const uint64_t *base = rows + (size_t)sl * per;
    unsigned sn[4] = {0u, 0u, 0u, 0u}, sq[4] = {0u, 0u, 0u, 0u};
    const uint64_t *y[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) y[j] = base + min(lg + j * sh.ng, nl - 1) * pitch;
#pragma unroll 2
    for (int t = 0; t < Lt; ++t) {
        uint64_t x[NX];
#pragma unroll
        for (int k = 0; k < NX; ++k) x[k] = base[t * pitch + k];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const unsigned d = (unsigned)differing<NX>(x, y[j] + t * pitch);
            sn[j] += d;
            sq[j] += d * d;
        }
    }
    const int sample = s0 + sl, sb = sample / 64, b = sample % 64;
    const int pb = sb / g.R, r = sb % g.R;
    const int p = p0 + pb, w = p / g.K, jj = p % g.K;
    const size_t idx = ((((size_t)r * g.W * 64) + (size_t)w * 64 + b) * g.K + jj) * nl;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int lag = lg + j * sh.ng;
        if (lag < nl) {
            const long long all = (long long)Lt * L2;
            g.Cacc[idx + lag] += all - 2 * (long long)sn[j];
            g.Qacc[idx + lag] += all * L2 - 4LL * L2 * sn[j] + 4LL * sq[j];
        }
    }
}

// Where the integer form is the faster one: its time grows as words x L_tau^2, that
// of a short tensor unit hardly at all.  2,048 sample bits, us here / with tensor
// tiles: L = 8, L_tau = 32 11 / 65, 128 20 / 71, 256 42 / 87; L = 10, L_tau = 128 29 / 73,
// 256 79 / 91; L = 12, L_tau = 128 40 / 77, 192 58 / 94, 256 111 / 97; L = 16, L_tau = 128
// 51 / 77, 192 112 / 95.  From two whole row blocks (L_tau = 256) on the tensor units
// have steps to overlap and keep the work.  So they do where the samples are few: the
// rows of one sample are a serial walk here, and a tile takes no longer for 152 samples
// than for one.  The line lies at L_tau (2 + 1.9 words) sample bits, 256 at least: whole
// measurements, us here / with tensor tiles, L = 4, L_tau = 32 22 / 18 for 128 bits; L = 8, L_tau = 64 24 / 19 for 128 bits, 26 / 42 for 1,024; L = 8,
// L_tau = 240 45 / 37 for 512, 46 / 54 for 1,024; L = 16, L_tau = 128 48 / 36 for 512, 62 / 54
// for 1,024, 91 / 104 for 2,048.
static bool use_short(const Group &g, int nsamples) {
    if (g.nwx > kShortWords || g.Ltau >= 2 * 128 || g.nwx * g.Ltau > 576) return false;
    return nsamples >= 256 && 10LL * nsamples >= (long long)g.Ltau * (20 + 19 * g.nwx);
}

static cudaError_t launch_gram_short(const Group &g, int p0, int npairs, const uint64_t *P, cudaStream_t st) {
    const ShortShape sh = short_shape(g);
    const int nsamples = npairs * g.R * 64, blocks = (nsamples + sh.samples - 1) / sh.samples;
    count_launches(1);
    switch (g.nwx) {
        case 1: k_gram_short<1><<<blocks, kShortThreads, sh.bytes, st>>>(g, p0, P, nsamples, sh); break;
        case 2: k_gram_short<2><<<blocks, kShortThreads, sh.bytes, st>>>(g, p0, P, nsamples, sh); break;
        case 3: k_gram_short<3><<<blocks, kShortThreads, sh.bytes, st>>>(g, p0, P, nsamples, sh); break;
        default: k_gram_short<4><<<blocks, kShortThreads, sh.bytes, st>>>(g, p0, P, nsamples, sh); break;
    }
    return cudaGetLastError();
}

constexpr size_t kGramSmem = 200 * 1024;  // rows of a sample that k_gram keeps in shared memory at most

cudaError_t launch_measure(const Group &g, uint64_t *scratch, size_t scratch_words, int tensor, int triples,
                           int *status, unsigned wait_limit, cudaStream_t st) {
    const size_t per_pair = measure_scratch_words_per_pair(g);
    int batch = (int)(scratch_words / per_pair);
    if (batch < 1) return cudaErrorInvalidValue;
    const int npairs_total = g.W * g.K;
    const size_t sh_bytes = (size_t)g.Ltau * g.nwx * sizeof(uint64_t);
    const int use_smem = sh_bytes <= kGramSmem ? 1 : 0;
    if (use_smem && !tensor) {
        cudaError_t e = cudaFuncSetAttribute(k_gram, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGramSmem);
        if (e != cudaSuccess) return e;
    }
    for (int p0 = 0; p0 < npairs_total; p0 += batch) {
        const int np = min(batch, npairs_total - p0);
        const size_t tr_smem = (size_t)64 * (kTrRun * g.nwx + 1) * sizeof(uint64_t);
        if (tr_smem > 48 * 1024) {
            const cudaError_t ea = cudaFuncSetAttribute(k_transpose, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                        64 * (kTrRun * 16 + 1) * (int)sizeof(uint64_t));
            if (ea != cudaSuccess) return ea;
        }
        count_launches(1);
        // slots along x (up to 2^31 - 1), runs of planes along y (L_tau / 8 <= 8192)
        k_transpose<<<dim3((unsigned)(np * g.R), (unsigned)((g.Ltau + kTrRun - 1) / kTrRun)), 32 * kTrRun, tr_smem,
                      st>>>(g, p0, np, scratch);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        if (tensor && use_short(g, np * g.R * 64)) {
            e = launch_gram_short(g, p0, np, scratch, st);
        } else if (tensor) {
            e = launch_gram_tc(g, p0, np, scratch, status, wait_limit, st);
        } else {
            count_launches(1);
            k_gram<<<np * g.R * 64, 256, use_smem ? sh_bytes : 0, st>>>(g, p0, scratch, use_smem);
            e = cudaGetLastError();
        }
        if (e != cudaSuccess) return e;
        // equal-time replica overlaps and the other one-time sums (k_onetime.cu)
        e = launch_onetime(g, p0, np, scratch, triples, st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Division of many numbers by one, correctly rounded (Markstein, Computation of
// elementary functions on the IBM RISC System/6000 processor, IBM J. Res. Dev. 34,
// 1990): with y = 1 / d rounded and q within an ulp of x / d, q + (x - q d) y,
// by fused multiply-adds, is x / d rounded.  q here is x (y + yl) with the
// reciprocal's own error yl, so it is within an ulp.  FP64 arithmetic is what the
// finish consists of (two operations per SM and clock): a quotient costs four
// operations instead of a division's ten or so (6,144 sample bits of 257 lags: 73 ->
// 40 us).
struct Divisor {
    double d, y, yl;
    __device__ __forceinline__ void set(double by) {
        d = by;
        y = __drcp_rn(by);
        yl = __dmul_rn(__fma_rn(-d, y, 1.0), y);
    }
    __device__ __forceinline__ double into(double x) const {
        const double q = __fma_rn(x, y, __dmul_rn(x, yl));
        return __fma_rn(__fma_rn(-q, d, x), y, q);
    }
};

// C = C_acc / (n_meas L^2 L_tau), Q2 = Q_acc / (n_meas L^4 L_tau),
// q2 = P_acc / (n_meas n_pairs L^4 L_tau), each one correctly rounded division by a
// product rounded operation by operation.
__global__ void k_finish(Group g, double nm) {
    const double L2 = (double)(g.L * g.L), Lt = (double)g.Ltau;
    const double pairs = (double)(g.R * (g.R - 1) / 2);
    const size_t nc = (size_t)g.R * g.W * 64 * g.K * g.nlag;
    const size_t np = (size_t)g.W * 64 * g.K;
    __shared__ Divisor by[2];  // set once per block: a reciprocal costs as much as a division
    if (threadIdx.x == 0) {
        by[0].set(__dmul_rn(__dmul_rn(nm, L2), Lt));
        by[1].set(__dmul_rn(__dmul_rn(__dmul_rn(nm, L2), L2), Lt));
    }
    __syncthreads();
    const Divisor c = by[0], q = by[1];
    if (nm == 0.0) {  // a count set to zero: the infinities and NaN of a division
        for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nc; i += (size_t)gridDim.x * blockDim.x) {
            g.outC[i] = __ddiv_rn((double)g.Cacc[i], 0.0);
            g.outQ[i] = __ddiv_rn((double)g.Qacc[i], 0.0);
            if (i < np) g.outP[i] = __ddiv_rn((double)g.Pacc[i], 0.0);
        }
        return;
    }
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nc; i += (size_t)gridDim.x * blockDim.x) {
        g.outC[i] = c.into((double)g.Cacc[i]);
        g.outQ[i] = q.into((double)g.Qacc[i]);
        if (i < np)
            g.outP[i] = __ddiv_rn((double)g.Pacc[i],
                                  __dmul_rn(__dmul_rn(__dmul_rn(__dmul_rn(nm, pairs), L2), L2), Lt));
    }
}

cudaError_t launch_finish(const Group &g, long long n_meas, cudaStream_t st) {
    const size_t nc = (size_t)g.R * g.W * 64 * g.K * g.nlag;
    long long blocks = (long long)((nc + 255) / 256);
    if (blocks > 152 * 8) blocks = 152 * 8;
    count_launches(1);
    k_finish<<<(int)blocks, 256, 0, st>>>(g, (double)n_meas);
    return cudaGetLastError();
}

}  // namespace qsg
