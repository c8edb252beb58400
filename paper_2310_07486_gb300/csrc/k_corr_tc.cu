// k_corr_tc.cu -- imaginary-time correlators on the 5th-generation tensor cores.
//
// For one sample (one bit of one slot) the correlators of Eq. (def-C-Q2-tau)
// are sums along the cyclic diagonals of the Gram matrix of its tau slices,
//     G(t1, t2) = sum_x S_x,t1 S_x,t2,
//     C(d) = sum_t1 s G(t1, t1 + d),   Q(d) = sum_t1 G(t1, t1 + d)^2,
// a dense contraction over the L^2 sites.  The spins are +-1, exact in FP8
// E4M3, and every partial sum is an integer of magnitude <= L^2 < 2^24, so a
// tcgen05.mma (kind::f8f6f4, FP32 accumulation in tensor memory) computes G
// exactly.
//
// Order of the work.  A 128 x 128 tile (i, e) holds the rows t1 = 128 i + m and
// the columns t2 = 128 (i + e) + q (mod L_tau), so its element (m, q) has the
// offset d = 128 e + q - m whatever i is.  A work unit is one sample and one
// column offset e, or two neighbouring ones (e, e + 1), and runs over every row
// block i: the epilogue keeps the sums of G and of G^2 over i in registers, one
// FP32 add and one FP32 multiply-add per element straight on the accumulator
// values (integers below 2^24, exact), and folds them into per-lag bins once
// per unit.  With the tensor-memory loads in the 16 x 256 bit shape a thread's
// elements lie in rows r, r + 8, r + 16, r + 24 and the same columns of every
// octet, so elements of equal offset meet in one thread and 38 sums of each
// kind cover its 128 elements of a tile.  (The form before this one ordered
// the tiles by row block and folded every tile with two shared-memory atomics
// per element: 3.92 ms for 2,048 sample bits at L = 24, L_tau = 2048, where
// this one takes 2.31 ms.)  The wrap past L_tau is taken where the rows
// are loaded: the row of t2 >= L_tau is that of t2 - L_tau, with its sign
// flipped under APBC, so C needs no sign in the epilogue.
//
// One persistent CTA per SM, specialised warps:
//   producers (8 warps, a thread per row of A or of B) load the x-packed bit
//     rows of the transposed scratch one step ahead into registers and expand
//     them to E4M3 in shared memory, +-1 (0 for padding) in A and +-1/2 in B (G
//     is even, so the accumulators hold the integers G / 2 and the running sums
//     of squares stay exact four times as long), K-major with the 128-byte
//     swizzle, sites in a bit-interleaved order shared by A and B;
//   one thread issues the MMAs of a step (one i) in 128-site chunks, two tiles
//     as one N = 256 MMA per 32 sites.  In a unit of two offsets the column
//     block i + e + 1 of one step is the block i + e of the next: it stays in
//     shared memory (slots used in turn), so a step expands two blocks for two
//     tiles;
//   the epilogue (8 warps, two per TMEM lane quadrant, one per tile of the
//     step) reads the accumulators, double-buffered in tensor memory.
// Per step of two tiles at L = 24 the MMAs read 216 KB and the producers write 144
// KB of shared memory (2,880 cycles at 128 B per cycle) beside 2,304 cycles of
// tensor work; measured, a step takes 4,700.  The MMAs alone, without waits, run at
// 2,300 (1.16 ms for the batch above); with the hand-over but neither expansion nor
// reads 2.02 ms, so most of what is left is the hand-over of chunks between the
// roles.  A fourth chunk in flight (both slots' half-empty last chunks in one) did not
// help, nor did one polling lane per warp (6.7 ms).  Lattices of more than five chunks
// (L > 24), whose column blocks do not fit, take every offset as a unit of its own,
// both operands streamed.
#include "qsg_launch.h"

namespace qsg {

namespace {

constexpr int kTile = 128;                   // rows of A (t1) and of B (t2) per tile
constexpr int kChunk = 128;                  // sites (bytes) per K chunk = one swizzled row
constexpr int kChunkBytes = kTile * kChunk;  // 16 KB per operand chunk
constexpr int kPairNc = 5;                   // chunks up to which column blocks stay resident
// Slots of resident column blocks: two, or more for rows of few chunks, whose
// steps are so short that the hand-over of a stage (about 1,500 cycles from the
// wait for it to its release) needs several steps in flight.
__host__ __device__ constexpr int block_slots(int nc) { return nc == 1 ? 6 : (nc == 2 ? 4 : 2); }
constexpr int kMaxStages = 6;                // chunks in flight at most
constexpr int kProducers = 256;              // warps 0-7: threads 0-127 A rows, 128-255 B rows
constexpr int kProducerWarps = kProducers / 32;
constexpr int kEpilogueWarps = 8;
constexpr int kEpilogue = 256;               // warps 8-15: quadrant = warp & 3, tile = (warp >> 2) & 1
constexpr int kMmaWarp = 16;
constexpr int kThreads = 17 * 32;
// registers: 17 warps put five on one scheduler, so the launch gets 96 a
// thread; the epilogue's 76 running sums and 32 loaded values want more, which
// the producers give up (256 x 80 + 256 x 112 + 32 x 96 = 544 x 96)
constexpr int kLaunchRegs = 96, kProducerRegs = 80, kEpilogueRegs = 112;
static_assert(kProducers * kProducerRegs + kEpilogue * kEpilogueRegs + 32 * kLaunchRegs == kThreads * kLaunchRegs,
              "register shares");
constexpr int kBins = 384;                   // lags of a unit: 128 e - 127 .. 128 e + 255
constexpr int kOct = kTile / 8 + 3;          // distinct octet offsets of a thread's elements
constexpr unsigned kSpinLimit = 1u << 22;    // polls of the wait for issued MMAs before TMEM is freed

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups 1024 B
// apart.  Its upper half is constant; the lower half is the address / 16 (below 2^14)
// and a constant, so a step along K or to another chunk is one 32-bit addition.  (With
// 64-bit descriptors built per MMA the issuing thread was late: 2,507 -> 2,313 us at L =
// 24, L_tau = 2048, 665 -> 622 us at L = 20, L_tau = 1024, 576 -> 562 us at L = 16, L_tau =
// 512.)
constexpr uint32_t kDescHigh = (1024u >> 4) | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint32_t desc_low(uint32_t saddr) { return (saddr >> 4) | (1u << 16); }

// Instruction descriptor: D = FP32, A = B = E4M3, both K-major, M = 128, N = n.
__device__ __forceinline__ uint32_t idesc_e4m3(int n) {
    return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kTile >> 4) << 24);
}

struct Ctl {
    uint64_t full[kMaxStages], empty[kMaxStages];  // chunk written / multiplied
    uint64_t accfull[2], accempty[2];              // accumulator computed / read
    uint64_t done;                                 // every MMA of the CTA completed
    uint32_t tmem;
    int abort;  // a wait gave up: every role skips its work and runs out its loops
};

// Wait for the phase of the given parity; false (and the abort flag set) when
// `limit` polls are used up, or when another thread has given up already (the
// flag is read every 64 polls, after the barrier itself).
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, int *abort, unsigned limit) {
    const uint32_t a = smem_u32(bar);
    volatile int *ab = abort;
    for (unsigned it = 0; it < limit; ++it) {
        uint32_t done;
        asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
                     : "=r"(done)
                     : "r"(a), "r"(parity)
                     : "memory");
        if (done) return true;
        if ((it & 63u) == 63u && *ab) return false;
    }
    *ab = 1;
    return false;
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(smem_u32(bar))
                 : "memory");
}

// 32 spin bits -> 32 E4M3 bytes (`one` = four bytes of the magnitude; a set bit
// is spin -1, the sign bit) in the site order of the contraction: byte k of
// output word j is bit 8k + j.  The Gram sums over sites, so any order serves
// that A and B share; this one takes one shift and one mask per output word.
// The shift is a multiplication by unit << (7 - j), unit = 1 unknown to the
// compiler: the multiplier's pipe is idle here and the integer one is not.
__device__ __forceinline__ uint32_t spread_e4m3(uint32_t b, int j, uint32_t one, uint32_t unit) {
    return ((b * (unit << (7 - j))) & 0x80808080u) | one;
}

// Bytes of spread_e4m3's output word j whose bits are set in the site mask vm
// are 0xFF, the others 0.
__device__ __forceinline__ uint32_t spread_mask(uint32_t vm, int j) {
    return (((vm << (7 - j)) & 0x80808080u) >> 7) * 0xFFu;
}

// The 64 sites of word wv into granules 4 hh .. 4 hh + 3 of the swizzled
// 128-byte row `row` at rowp; sites >= valid (outside the lattice, or every
// site of a row past L_tau) become 0.  Output words 8 e + j (e = half of the
// word) fill granules 4 hh + 2 e + (j >> 2).
__device__ __forceinline__ void expand_full(uint8_t *rowp, uint64_t wv, int hh, int row, uint32_t one, uint32_t unit) {
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const uint32_t b = (uint32_t)(wv >> (32 * e));
#pragma unroll
        for (int hq = 0; hq < 2; ++hq) {
            const int gr = 4 * hh + 2 * e + hq;
            *reinterpret_cast<uint4 *>(rowp + ((gr ^ (row & 7)) << 4)) =
                make_uint4(spread_e4m3(b, 4 * hq, one, unit), spread_e4m3(b, 4 * hq + 1, one, unit),
                           spread_e4m3(b, 4 * hq + 2, one, unit), spread_e4m3(b, 4 * hq + 3, one, unit));
        }
    }
}

__device__ __noinline__ void expand_part(uint8_t *rowp, uint64_t wv, int valid, int hh, int row, uint32_t one) {
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const uint32_t b = (uint32_t)(wv >> (32 * e));
        const int v32 = valid - 32 * e;
        const uint32_t vm = v32 >= 32 ? 0xFFFFFFFFu : (v32 <= 0 ? 0u : (1u << v32) - 1u);
#pragma unroll
        for (int hq = 0; hq < 2; ++hq) {
            const int gr = 4 * hh + 2 * e + hq;
            uint32_t o[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) o[k] = spread_e4m3(b, 4 * hq + k, one, 1u) & spread_mask(vm, 4 * hq + k);
            *reinterpret_cast<uint4 *>(rowp + ((gr ^ (row & 7)) << 4)) = make_uint4(o[0], o[1], o[2], o[3]);
        }
    }
}

__device__ __forceinline__ void expand_word(uint8_t *rowp, uint64_t wv, int valid, int hh, int row, uint32_t one,
                                            uint32_t unit) {
    if (valid >= 64)
        expand_full(rowp, wv, hh, row, one, unit);
    else
        expand_part(rowp, wv, valid, hh, row, one);
}

__device__ __forceinline__ void mma_f8(uint32_t d, uint32_t da, uint32_t db, uint32_t idesc, uint32_t acc) {
    asm volatile("{\n.reg .pred p;\n.reg .b64 a, b;\nmov.b64 a, {%1, %5};\nmov.b64 b, {%2, %5};\nsetp.ne.u32 p, %4, 0;\n"
                 "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], a, b, %3, p;\n}\n" ::"r"(d),
                 "r"(da), "r"(db), "r"(idesc), "r"(acc), "r"(kDescHigh));
}

// How the offsets of one sample are cut into units and steps.
struct GramPlan {
    int nsamples;
    int nb;       // row blocks
    int npair;    // units of two offsets per sample: e = 0, 2, ..
    int nsingle;  // units of one offset per sample, the first of them e = e_single
    int e_single;
    int e_mirror;  // offset whose steps stop at nb / 2 (each tile is the transpose of another), or -1
    int triangle;  // one row block: only the tile of t2 >= t1, without the wrap past L_tau
    int nstages;
    int flush;     // steps after which the FP32 sums must be folded
    uint32_t unit;  // 1 (see spread_e4m3)
};

struct Unit {
    int sample, e, steps;
    bool pair, mirror;
};

// Units of two offsets of every sample first (a sample's units on neighbouring
// SMs at the same time, so that they share its rows in L2), then the others;
// a static round robin over each kind keeps the SMs balanced.
__device__ __forceinline__ Unit unit_of(const GramPlan &pl, int u) {
    Unit r;
    const int np = pl.nsamples * pl.npair;
    r.pair = u < np;
    if (r.pair) {
        r.sample = u / pl.npair;
        r.e = 2 * (u - r.sample * pl.npair);
        r.mirror = false;
    } else {
        r.sample = (u - np) / pl.nsingle;
        r.e = pl.e_single + (u - np) - r.sample * pl.nsingle;
        r.mirror = pl.triangle || r.e == pl.e_mirror;
    }
    r.steps = r.mirror && !pl.triangle ? pl.nb / 2 : pl.nb;
    return r;
}
__device__ __forceinline__ int unit_count(const GramPlan &pl) { return pl.nsamples * (pl.npair + pl.nsingle); }

// The steps a CTA runs, in order: of every unit the steps 0 .. steps - 1, before
// them (i = -1) the load of the first column block in a unit of two offsets.
struct Cursor {
    int u, i;
    bool valid;
    Unit un;
};
__device__ __forceinline__ void cursor_unit(const GramPlan &pl, Cursor &c) {
    c.valid = c.u < unit_count(pl);
    if (!c.valid) return;
    c.un = unit_of(pl, c.u);
    c.i = c.un.pair ? -1 : 0;
}
__device__ __forceinline__ void cursor_next(const GramPlan &pl, Cursor &c) {
    if (!c.valid || ++c.i < c.un.steps) return;
    c.u += gridDim.x;
    cursor_unit(pl, c);
}

// Source row of a producer thread at a step: row `row` of the A block
// (t1 = 128 i + row) or of the column block the step brings in (t2 =
// 128 (i + e [+ 1]) + row, wrapped).
struct Row {
    const uint64_t *src;
    uint64_t flip;  // all ones where B's row wraps under APBC
    bool live;      // B, or an A row that exists (t1 < L_tau)
};
__device__ __forceinline__ Row row_of(const Cursor &c, const uint64_t *__restrict__ P, int Lt, int nwx, int apbc,
                                      bool isB, int row) {
    Row r;
    int t = c.valid ? kTile * (c.i + (isB ? c.un.e + (c.un.pair ? 1 : 0) : 0)) + row : 0;
    r.flip = 0ull;
    r.live = true;
    if (isB) {
        if (t >= Lt) {
            t = t < 2 * Lt ? t - Lt : t % Lt;  // beyond 2 L_tau: no lag of this row is used
            if (apbc) r.flip = ~0ull;
        }
    } else if (c.i < 0 || t >= Lt) {
        r.live = false;
        t = 0;
    }
    r.src = P + ((size_t)(c.valid ? c.un.sample : 0) * Lt + t) * nwx;
    return r;
}
// 64 accumulator columns of 16 TMEM lanes: octet o of the columns is v[4 o ..
// 4 o + 3] = (row r, columns 2 c, 2 c + 1), (row r + 8, the same), with r =
// lane / 4 and c = lane % 4
__device__ __forceinline__ void tmem_ld_oct8(uint32_t taddr, uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x8.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
          "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
          "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr)
        : "memory");
}

// Shift a warp's sums of both kinds, c[0 .. N) and q[0 .. N), one level down a tree
// over its lanes: add to every lane the sums (fc, fq) of lane `src`, whose elements
// lie at offsets 8 higher where that lane's row wrapped (then its sum k belongs to k +
// 1).  c[N], q[N] are new.  Two sums of each kind at a time: four shuffles in flight
// (one at a time, the fold took 11,000 cycles a unit, most of them their latency).
template <int N>
__device__ __forceinline__ void fold_level(float (&c)[22], int (&q)[22], const float (&fc)[22], const int (&fq)[22],
                                           bool wraps, int src) {
    auto sc = [&](int k) { return wraps ? (k > 0 ? fc[k > 0 ? k - 1 : 0] : 0.0f) : (k < N ? fc[k] : 0.0f); };
    auto sq = [&](int k) { return wraps ? (k > 0 ? fq[k > 0 ? k - 1 : 0] : 0) : (k < N ? fq[k] : 0); };
#pragma unroll
    for (int k = N; k >= 0; k -= 2) {
        const float c0 = __shfl_sync(0xffffffffu, sc(k), src);
        const int q0 = __shfl_sync(0xffffffffu, sq(k), src);
        float c1 = 0.0f;
        int q1 = 0;
        if (k > 0) {
            c1 = __shfl_sync(0xffffffffu, sc(k - 1), src);
            q1 = __shfl_sync(0xffffffffu, sq(k - 1), src);
        }
        c[k] = (k < N ? c[k] : 0.0f) + c0;
        q[k] = (k < N ? q[k] : 0) + q0;
        if (k > 0) {
            c[k - 1] += c1;
            q[k - 1] += q1;
        }
    }
}

// The warp's sums, index kappa of column 2 c (c, q) and of column 2 c + 1 (c1, q1) of
// every lane (row r = lane / 4, c = lane % 4), element offset 8 kappa + 2 c + q - r,
// summed over lanes of equal offset: lane 4 r then holds in c[k], q[k] the sums of
// offset 8 k - r.
__device__ __forceinline__ void fold_lanes(float (&c)[22], int (&q)[22], const float (&c1)[22], const int (&q1)[22],
                                           int lane) {
    static_assert(kOct == 19, "levels of 19, 20 and 21 sums");
    const int r = lane >> 2, l = lane & 3;
    fold_level<19>(c, q, c1, q1, r < 1, (((r + 1) & 7) << 2) | l);              // second column into first
    fold_level<20>(c, q, c, q, r < 2, (((r + 2) & 7) << 2) | ((l + 1) & 3));  // odd lanes into even ones
    fold_level<21>(c, q, c, q, r < 4, (((r + 4) & 7) << 2) | ((l + 2) & 3));
}

}  // namespace

// P: [sample][Ltau][nwx] transposed bits of the batch (sample = (pair, r, bit)).
// NC = 128-site chunks of a row (L^2 / 128 rounded up).
template <int NC>
__global__ void __launch_bounds__(kThreads, 1)
    k_gram_tc(Group g, int p0, const uint64_t *__restrict__ P, const GramPlan pl, int *status, unsigned wait_limit) {
    constexpr bool RESIDENT = NC <= kPairNc;  // column blocks in resident slots, else streamed with A
    constexpr int NS = block_slots(NC);
    extern __shared__ __align__(16) uint8_t dyn_raw[];
    uint8_t *dyn = dyn_raw + ((1024u - (smem_u32(dyn_raw) & 1023u)) & 1023u);
    __shared__ Ctl ctl;
    __shared__ int binC[kBins];
    __shared__ unsigned binQ[kBins];
    const int Lt = g.Ltau, L2 = g.L * g.L, half = Lt / 2, nl = g.nlag, nwx = g.nwx;
    const int nunits = unit_count(pl), nst = pl.nstages;
    uint8_t *sA = dyn;                               // nst chunks of 128 rows x 128 sites
    uint8_t *sB = sA + (size_t)nst * kChunkBytes;  // RESIDENT: [chunk][slot], else nst chunks

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int s = 0; s < kMaxStages; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(&ctl.full[s])), "r"(kProducerWarps));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&ctl.empty[s])));
        }
        for (int a = 0; a < 2; ++a) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&ctl.accfull[a])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(&ctl.accempty[a])), "r"(kEpilogueWarps));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&ctl.done)));
        asm volatile("fence.mbarrier_init.release.cluster;\n");
        ctl.abort = 0;
    }
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;\n" ::"r"(smem_u32(&ctl.tmem)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    for (int l = tid; l < kBins; l += kThreads) {
        binC[l] = 0;
        binQ[l] = 0u;
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n");
    const uint32_t tmem = ctl.tmem;

    if (warp < kProducerWarps) {
        // ------------------------------------------------------------ producers
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(kProducerRegs));
        const bool isB = tid >= kTile;
        const int row = tid & (kTile - 1);
        Cursor cur, ahead;
        cur.u = blockIdx.x;
        cursor_unit(pl, cur);
        ahead = cur;
        Row now = row_of(cur, P, Lt, nwx, g.boundary, isB, row);
        uint64_t w[2 * NC];
#pragma unroll
        for (int k = 0; k < 2 * NC; ++k) w[k] = k < nwx ? __ldg(now.src + k) : 0ull;
        // (a triangle leaves out the rows that wrap: +-0)
        const uint32_t one = isB ? (pl.triangle && row >= Lt ? 0u : 0x30303030u) : 0x38383838u, unit = pl.unit;
        // the first use of a stage waits for the phase before the first
        // (complete at initialisation)
        uint32_t par = 1u;
        int st = 0, slot = 0;  // slot: of the column block a step brings in, in turn over all steps
        while (cur.valid) {
            cursor_next(pl, ahead);
            const Row next = row_of(ahead, P, Lt, nwx, g.boundary, isB, row);
            const bool write = isB || cur.i >= 0;  // no A block before the first step
            const uint64_t flip = now.flip;
            // unrolled, so that a chunk's words are replaced by those of the
            // next step as soon as they are used: the loads have a whole step
            // to land and need no registers of their own (in a rolled loop
            // they were waited for before its first pass, 1,900 cycles a step)
#pragma unroll
            for (int kc = 0; kc < NC; ++kc) {
                const bool ok = mbar_wait(&ctl.empty[st], par, &ctl.abort, wait_limit);
                uint8_t *rowp = (!isB ? sA + (size_t)st * kChunkBytes
                                      : (RESIDENT ? sB + (size_t)(NS * kc + slot) * kChunkBytes
                                                  : sB + (size_t)st * kChunkBytes)) +
                                row * kChunk;
                if (ok && write) {
                    // a word past the lattice's last site is never read (the
                    // MMAs of the last chunk stop at its last word with a
                    // site); zeros in A alone blank the sites past L^2 and
                    // the rows past L_tau
                    const int left = L2 - kc * kChunk;
                    const int valid = isB ? kChunk : (now.live ? left : 0);
                    expand_word(rowp, w[2 * kc] ^ flip, valid, 0, row, one, unit);
                    if (left > 64) expand_word(rowp, w[2 * kc + 1] ^ flip, valid - 64, 1, row, one, unit);
                }
                asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                __syncwarp();  // the warp's rows are written: one arrival per warp
                if (lane == 0) mbar_arrive(&ctl.full[st]);
                if (++st == nst) {
                    st = 0;
                    par ^= 1u;
                }
                w[2 * kc] = __ldg(next.src + 2 * kc);
                if (2 * kc + 1 < nwx) w[2 * kc + 1] = __ldg(next.src + 2 * kc + 1);
            }
            now = next;
            cur = ahead;
            if (++slot == NS) slot = 0;
        }
    } else if (warp < kMmaWarp) {
        // ------------------------------------------------------------- epilogue
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(kEpilogueRegs));
        const int etid = tid - kProducers;
        const int quad = warp & 3;                       // TMEM lanes 32 quad .. 32 quad + 31
        const int half_w = (warp >> 2) & 1;              // of two tiles of a step, or of two steps
        const int r = lane >> 2;                         // the thread's row of an octet pair
        uint32_t n_t = 0;
        int parity = 0;  // of the step, the loads of a unit's first column block counted
        for (int u = blockIdx.x; u < nunits; u += gridDim.x) {
            const Unit un = unit_of(pl, u);
            if (un.pair) parity ^= 1;
            const int e = un.pair ? un.e + half_w : un.e;
            const int lag0 = max(0, kTile * un.e - (kTile - 1));  // lag of bin 0
            const int sb = un.sample / 64, bit = un.sample % 64;
            const int pb = sb / g.R, rr = sb % g.R;
            const int pidx = p0 + pb, w = pidx / g.K, j = pidx % g.K;
            const size_t gbase = ((((size_t)rr * g.W * 64) + (size_t)w * 64 + bit) * g.K + j) * nl;
            float accC[kOct][2], accQ[kOct][2];
#pragma unroll
            for (int k = 0; k < kOct; ++k) accC[k][0] = accC[k][1] = accQ[k][0] = accQ[k][1] = 0.0f;
            int in_flush = 0, in_push = 0;
            for (int i = 0; i < un.steps; ++i, ++n_t, parity ^= 1) {
                const int a = (int)(n_t & 1u);
                // warp-uniform: the tensor-memory loads below are .sync.aligned
                const bool ok =
                    __all_sync(0xFFFFFFFFu, mbar_wait(&ctl.accfull[a], (n_t >> 1) & 1u, &ctl.abort, wait_limit));
                asm volatile("tcgen05.fence::after_thread_sync;\n");
                // the tile of this warp: the columns of the slot that holds its
                // offset (two offsets), or every second step (one offset)
                const bool mine = un.pair || (i & 1) == half_w;
                // (of two slots, the step's new block, offset e + 1, is in slot `parity`)
                const int slot = !un.pair ? 0 : (NS == 2 ? (half_w ? parity : parity ^ 1) : half_w);
                if (ok && mine) {
                    const uint32_t ta = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(a * 256 + slot * kTile);
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int kg = 0; kg < 2; ++kg) {
                            uint32_t v[32];
                            tmem_ld_oct8(ta + ((uint32_t)(h * 16) << 16) + (uint32_t)(kg * 64), v);
#pragma unroll
                            for (int o = 0; o < 8; ++o)
#pragma unroll
                                for (int q = 0; q < 4; ++q) {
                                    const int k = kg * 8 + o - (2 * h + (q >> 1)) + 3;
                                    const float x = __uint_as_float(v[4 * o + q]);
                                    accC[k][q & 1] += x;
                                    accQ[k][q & 1] = fmaf(x, x, accQ[k][q & 1]);
                                }
                        }
                }
                asm volatile("tcgen05.fence::before_thread_sync;\n");
                __syncwarp();
                if (lane == 0) mbar_arrive(&ctl.accempty[a]);
                // fold the sums before they could leave FP32's exact integers,
                // and add the 32-bit bins to the int64 sums before they wrap
                const bool last = i + 1 == un.steps;
                if (++in_flush == pl.flush || last) {
                    in_flush = 0;
                    // sums of G over lanes stay exact in FP32 (magnitudes
                    // below 2^24), those of squares need integers
                    const int dbase = kTile * e - 32 * quad - 24 - r;
                    const bool owner = (lane & 3) == 0;
                    // every offset of the tile is a lag: no tests per element
                    const bool inside = !un.mirror && kTile * e >= kTile && kTile * e + kTile - 1 <= half;
                    float vc[22], wc[22];
                    int vq[22], wq[22];
#pragma unroll
                    for (int k = 0; k < 22; ++k) {
                        vc[k] = k < kOct ? accC[k < kOct ? k : 0][0] : 0.0f;
                        wc[k] = k < kOct ? accC[k < kOct ? k : 0][1] : 0.0f;
                        vq[k] = k < kOct ? __float2int_rn(accQ[k < kOct ? k : 0][0]) : 0;
                        wq[k] = k < kOct ? __float2int_rn(accQ[k < kOct ? k : 0][1]) : 0;
                    }
                    fold_lanes(vc, vq, wc, wq, lane);
                    if (inside) {
                        // (sums past the tile's last offset, k > 18, are of nothing)
#pragma unroll
                        for (int k = 0; k < 22; ++k)
                            if (owner && (k <= 18 || dbase + 8 * k <= kTile * e + kTile - 1)) {
                                atomicAdd(binC + (dbase - lag0) + 8 * k, __float2int_rn(vc[k]));
                                atomicAdd(binQ + (dbase - lag0) + 8 * k, (unsigned)vq[k]);
                            }
                    } else if (owner) {
#pragma unroll
                        for (int k = 0; k < 22; ++k) {
                            const int d = dbase + 8 * k;
                            int cv = __float2int_rn(vc[k]), lag = d;
                            unsigned qv = (unsigned)vq[k];
                            if (un.mirror && d >= half) {
                                // half the row blocks, or the tile of t2 >= t1: an
                                // element past L_tau / 2 is the wrapped pair of lag
                                // L_tau - d, and one at L_tau / 2 stands for both
                                // directions
                                lag = Lt - d;
                                if (d == half) qv *= 2u;
                                cv = d == half ? (g.boundary == 1 ? 0 : 2 * cv) : (g.boundary == 1 ? -cv : cv);
                            }
                            if (d >= 0 && lag >= lag0 && lag <= half) {
                                atomicAdd(&binC[lag - lag0], cv);
                                atomicAdd(&binQ[lag - lag0], qv);
                            }
                        }
                    }
#pragma unroll
                    for (int k = 0; k < kOct; ++k) accC[k][0] = accC[k][1] = accQ[k][0] = accQ[k][1] = 0.0f;
                    if (++in_push == 2 || last) {
                        in_push = 0;
                        asm volatile("bar.sync 1, %0;\n" ::"n"(kEpilogue) : "memory");
                        const bool write = !*(volatile int *)&ctl.abort;
                        for (int l = etid; l < kBins; l += kEpilogue) {
                            // sums of G / 2 and of its square
                            const long long cs = 2LL * binC[l];
                            const unsigned long long qs = 4ull * binQ[l];
                            if (write && cs)
                                atomicAdd(reinterpret_cast<unsigned long long *>(&g.Cacc[gbase + lag0 + l]),
                                          (unsigned long long)cs);
                            if (write && qs)
                                atomicAdd(reinterpret_cast<unsigned long long *>(&g.Qacc[gbase + lag0 + l]), qs);
                            binC[l] = 0;
                            binQ[l] = 0u;
                        }
                        asm volatile("bar.sync 1, %0;\n" ::"n"(kEpilogue) : "memory");
                    }
                }
            }
        }
    } else {
        // ------------------------------------------------------------------ MMA
        // one thread issues every MMA; a commit after a chunk's MMAs frees its
        // stage (and the older column block's slot of that chunk)
        if (lane == 0) {
            const uint32_t id128 = idesc_e4m3(128), id256 = idesc_e4m3(256);
            // 32-site steps of the last chunk: those of its 64-site words that
            // hold a lattice site (the bit-interleaved order spreads a word's
            // sites over its whole 64-byte span)
            const int nk_last = min(kChunk / 32, 2 * ((L2 - (NC - 1) * kChunk + 63) / 64));
            constexpr uint32_t kC = kChunkBytes / 16;  // a chunk in descriptor units
            const uint32_t sA0 = desc_low(smem_u32(sA)), sB0 = desc_low(smem_u32(sB));
            uint32_t par = 0u, n_t = 0;
            int st = 0, slot = 0, older = NS - 1;  // slots of the step's new column block and of the one before
            bool issued = false;
            for (int u = blockIdx.x; u < nunits; u += gridDim.x) {
                const Unit un = unit_of(pl, u);
                for (int i = un.pair ? -1 : 0; i < un.steps; ++i) {
                    const int a = (int)(n_t & 1u);
                    bool ok = true;
                    if (i >= 0) {
                        ok = mbar_wait(&ctl.accempty[a], ((n_t >> 1) & 1u) ^ 1u, &ctl.abort, wait_limit);
                        asm volatile("tcgen05.fence::after_thread_sync;\n");
                    }
                    const uint32_t d = tmem + (uint32_t)(a * 256);
                    // two slots: both column blocks as one N = 256 MMA; more: one
                    // N = 128 MMA per column block, the older block's first
                    const uint32_t idesc = un.pair && NS == 2 ? id256 : id128;
                    const uint32_t b0 =
                        un.pair ? (NS == 2 ? 0u : (uint32_t)older * kC) : (uint32_t)slot * kC;
                    const uint32_t b1 = (uint32_t)slot * kC;
                    const bool second = un.pair && NS > 2;
#pragma unroll 1  // rolled: the three roles' code shares the instruction cache
                    for (int kc = 0; kc < NC; ++kc) {
                        ok = mbar_wait(&ctl.full[st], par, &ctl.abort, wait_limit) && ok;
                        asm volatile("tcgen05.fence::after_thread_sync;\n");
                        if (ok && i >= 0) {
                            const uint32_t ab = sA0 + (uint32_t)st * kC;
                            const uint32_t bb = RESIDENT ? sB0 + (uint32_t)(NS * kc) * kC : sB0 + (uint32_t)st * kC;
                            const uint32_t bb0 = RESIDENT ? bb + b0 : bb;
                            const int nk = kc == NC - 1 ? nk_last : kChunk / 32;
                            const uint32_t acc0 = kc > 0 ? 1u : 0u;
                            mma_f8(d, ab, bb0, idesc, acc0);
                            mma_f8(d, ab + 2u, bb0 + 2u, idesc, 1u);
                            if (nk > 2) {
                                mma_f8(d, ab + 4u, bb0 + 4u, idesc, 1u);
                                mma_f8(d, ab + 6u, bb0 + 6u, idesc, 1u);
                            }
                            if (NS > 2 && second) {
                                mma_f8(d + kTile, ab, bb + b1, id128, acc0);
                                mma_f8(d + kTile, ab + 2u, bb + b1 + 2u, id128, 1u);
                                if (nk > 2) {
                                    mma_f8(d + kTile, ab + 4u, bb + b1 + 4u, id128, 1u);
                                    mma_f8(d + kTile, ab + 6u, bb + b1 + 6u, id128, 1u);
                                }
                            }
                            issued = true;
                        }
                        mma_commit(&ctl.empty[st]);
                        if (++st == nst) {
                            st = 0;
                            par ^= 1u;
                        }
                    }
                    if (i >= 0) {
                        mma_commit(&ctl.accfull[a]);
                        ++n_t;
                    }
                    older = slot;
                    if (++slot == NS) slot = 0;
                }
            }
            // every MMA issued has completed before the tensor memory is released
            // (a commit tracks all earlier MMAs of the issuing thread)
            mma_commit(&ctl.done);
            if (issued) {
                uint32_t done = 0;
                for (unsigned it = 0; it < kSpinLimit && !done; ++it)
                    asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\nselp.u32 %0, 1, 0, p;\n}\n"
                                 : "=r"(done)
                                 : "r"(smem_u32(&ctl.done))
                                 : "memory");
                if (!done) ctl.abort = 1;
            }
        }
        __syncwarp();
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n");
    if (warp == kMmaWarp) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\n" ::"r"(tmem));
    if (tid == 0 && ctl.abort) atomicExch(status, DEVERR_TIMEOUT);
}

namespace {

constexpr size_t kSmemLimit = 227 * 1024 - 4096;  // dynamic, beside the static control block and bins

GramPlan gram_plan(const Group &g, int nsamples) {
    GramPlan pl;
    const int nc = (g.L * g.L + kChunk - 1) / kChunk, half = g.Ltau / 2;
    const int mmax = g.Ltau < kTile ? g.Ltau - 1 : kTile - 1;
    const int ne = (mmax + half + kTile) / kTile;  // column offsets that hold a lag <= L_tau / 2
    pl.nsamples = nsamples;
    pl.nb = (g.Ltau + kTile - 1) / kTile;
    pl.npair = nc <= kPairNc ? ne / 2 : 0;
    pl.nsingle = ne - 2 * pl.npair;
    pl.e_single = 2 * pl.npair;
    // where L_tau / 2 is a whole number of blocks, the tiles (i, e) and
    // (i + nb / 2, e) of the last offset are each other's transpose
    pl.e_mirror = half % kTile == 0 && pl.nb > 1 ? half / kTile : -1;
    // One row block of a lattice whose units have one offset and stream both operands (L >
    // 24): the triangle of t2 >= t1 holds every pair of rows once, the offsets past L_tau
    // / 2 standing for the wrapped ones, in one tile where the offsets up to L_tau / 2 take
    // two (L_tau = 86 .. 128).  2,048 sample bits, us of a measurement with the offsets / the
    // triangle: L = 26, L_tau = 112 214 / 159, L = 32, L_tau = 112 312 / 234.  With two row
    // blocks (three tiles for four) the shorter units cost more than the tile saves (L = 26,
    // L_tau = 160 302 / 371), and so they do with resident column blocks (L = 24, L_tau = 86
    // 129 / 144).
    pl.triangle = pl.nb == 1 && ne == 2 && nc > kPairNc;
    if (pl.triangle) {
        pl.e_single = 0;
        pl.nsingle = 1;
    }
    // resident: the slots' chunks, and no more stages than a stage's release
    // can stand for (it must imply that of the slot to be overwritten, block_slots
    // - 1 steps back); streamed: A and B chunks
    const int ns = block_slots(nc);
    const size_t fixed = 1024 + (nc <= kPairNc ? (size_t)ns * nc * kChunkBytes : 0);
    const size_t per = (nc <= kPairNc ? 1 : 2) * (size_t)kChunkBytes;
    int s = kMaxStages;
    if (nc <= kPairNc && s > (ns - 1) * nc) s = (ns - 1) * nc;
    while (s > 1 && fixed + s * per > kSmemLimit) --s;
    pl.nstages = s;
    // a thread's sum takes up to four squares (G / 2)^2 <= L^4 / 4 per step
    // (exact in FP32 up to 2^24); two flushes of 256 squares per step stay
    // below 2^31
    const long long l4 = (long long)g.L * g.L * g.L * g.L;
    const long long f = (1LL << 24) / l4;
    pl.flush = (int)(f < 1 ? 1 : (f > 1024 ? 1024 : f));
    pl.unit = 1u;
    return pl;
}

template <int NC>
cudaError_t launch_nc(const Group &g, int p0, const GramPlan &pl, const uint64_t *P, int *status, unsigned wait_limit,
                      int nsm, cudaStream_t st) {
    const size_t sm =
        1024 + (NC <= kPairNc ? (size_t)(block_slots(NC) * NC + pl.nstages) : (size_t)(2 * pl.nstages)) * kChunkBytes;
    cudaError_t e = cudaFuncSetAttribute(k_gram_tc<NC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    const long long nunits = (long long)pl.nsamples * (pl.npair + pl.nsingle);
    const int grid = (int)(nunits < nsm ? nunits : nsm);
    count_launches(1);
    k_gram_tc<NC><<<grid, kThreads, sm, st>>>(g, p0, P, pl, status, wait_limit);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_gram_tc(const Group &g, int p0, int npairs, const uint64_t *P, int *status, unsigned wait_limit,
                           cudaStream_t st) {
    int dev = 0, nsm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const GramPlan pl = gram_plan(g, npairs * g.R * 64);
    switch ((g.L * g.L + kChunk - 1) / kChunk) {
        case 1: return launch_nc<1>(g, p0, pl, P, status, wait_limit, nsm, st);
        case 2: return launch_nc<2>(g, p0, pl, P, status, wait_limit, nsm, st);
        case 3: return launch_nc<3>(g, p0, pl, P, status, wait_limit, nsm, st);
        case 4: return launch_nc<4>(g, p0, pl, P, status, wait_limit, nsm, st);
        case 5: return launch_nc<5>(g, p0, pl, P, status, wait_limit, nsm, st);
        case 6: return launch_nc<6>(g, p0, pl, P, status, wait_limit, nsm, st);
        case 7: return launch_nc<7>(g, p0, pl, P, status, wait_limit, nsm, st);
        default: return launch_nc<8>(g, p0, pl, P, status, wait_limit, nsm, st);
    }
}

}  // namespace qsg
