// k_sweep_unit.cuh -- the fused one-pass checkerboard sweep, lattice size known
// at compile time (instantiated per algorithm in k_sweep_unit_*.cu).
//
// A unit is one slot and a chunk [a, b) of its tau planes (even a, b), streamed
// through a ring of 16 shared-memory planes, so every word crosses HBM once each
// way.  A thread owns the column pair (x0, x0 + 1) of a row y, x0 = 2 xh + (y &
// 1), so that on every plane one column is colour 0 and the other colour 1, and
// one Philox call feeds the thread's 2 x 2 (x, tau) block of four sites.  A step
// updates colour 0 of planes q .. q + 3, then (after one block barrier) colour 1
// of planes q - 1 .. q + 2: the order of a colour-0 half sweep followed by a
// colour-1 half sweep.  The colour-1 sites of a chunk's first plane and of the
// plane before it wait for both chunks: whichever of the two units finishes
// second updates them (an arrival counter, no waiting).
//
// Data path.  Planes lie in shared memory as they do in HBM, and bulk copies
// move them, four planes at a time in each direction, issued by one thread per
// unit: group i (planes a - 1 + 4 i .. a + 2 + 4 i) is final after step i, stored
// at step i + 1 and its ring slots refilled with group i + 4, which step i + 3
// needs: a whole step of lead.  The threads spend no instruction on moving
// data.  (Per-thread 8-byte cp.async into planes split by colour class and
// stores read back from shared memory made the data path alone take 0.94 ms of
// the 1.11 ms of an L = 24, L_tau = 2048, 256-slot sweep; this one alone takes
// 0.73 ms, the HBM copy time.)  So that natural-order planes are read without the
// two-way bank conflicts of columns two words apart, neighbouring lanes take
// neighbouring rows: even rows use even words (x0 even), odd rows odd words, and
// sixteen lanes touch sixteen banks (but for wraps).
//
// What bounds it now: the integer pipes.  About 43 of its 66 instructions per
// site word run there, 66 % of the pipe's rate, the block barrier being the
// largest stall; see qsg_sweep.cuh for the update itself.
//
// A block serves chunks of one slot, so everything that depends on the slot is
// uniform (the thresholds stay in uniform registers) and 72 registers suffice,
// three blocks of 288 threads per SM at L = 24 (the ring of 74 KB allows three too).
// Where 80 registers cost no resident block they are given, see unit_regs.
// L = 6 has 18 threads per chunk and runs 14 neighbouring chunks per block, in
// lockstep, so that its eight warps are full (92 slots of L_tau = 1024, us per sweep:
// a chunk per block 50, 16 chunks in nine warps of 72 registers, which spill more, 34.0
// Metropolis and 30.1 heat bath, 14 in eight warps of 80 27.1 and 25.5).  From
// L = 10 on that is no gain: five chunks per block at L = 10 (L_tau = 736, 348 slots)
// 100 against 96 us, four at L = 12 (L_tau = 256, 192 slots) 46 / 44, two at L = 14
// (L_tau = 400, 64 slots) 37 / 31: what the idle lanes cost is less than the coarser
// cut and the spills of per-chunk registers.
#pragma once
#include <type_traits>

#include "qsg_launch.h"
#include "qsg_sweep.cuh"

namespace qsg {
namespace unit {

using namespace sweep;

constexpr int kRing = 16;                  // planes in the ring
constexpr unsigned kDrainPolls = 1u << 24; // polls of the wait for copies in flight after a wait gave up

// Chunks per block.
__host__ __device__ constexpr int units_per_block(int L) {
    return L <= 6 ? 14 : 1;
}
// Registers of a thread: 80, which nearly every size needs to be free of spills, where
// as many blocks fit an SM as with 72 (by registers, 24 against 28 warps, or by the
// ring), else 72.  72 / 80, us per sweep: L = 18, L_tau = 2048, 92 slots 239 / 235; L = 16,
// L_tau = 512, 96 slots 51.3 / 49.8 (heat bath), L_tau = 2048, 128 slots 205.6 / 202.3.
__host__ __device__ constexpr int unit_regs(int L) {
    const int warps = (units_per_block(L) * L * L / 2 + 31) / 32;
    const int ring = 227 * 1024 / (units_per_block(L) * kRing * L * L * 8 + 1280);
    const int at72 = 28 / warps < ring ? 28 / warps : ring, at80 = 24 / warps < ring ? 24 / warps : ring;
    return at80 >= at72 ? 80 : 72;
}

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bar_init(uint64_t *b) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_addr(b)) : "memory");
}
__device__ __forceinline__ void bar_expect(uint64_t *b, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_addr(b)), "r"(bytes) : "memory");
}
// Wait for the phase of the given parity; false after `limit` polls.
__device__ __forceinline__ bool bar_wait(uint64_t *b, uint32_t parity, unsigned limit) {
    const uint32_t a = smem_addr(b);
    for (; limit != 0; --limit) {
        uint32_t done;
        asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
                     : "=r"(done)
                     : "r"(a), "r"(parity)
                     : "memory");
        if (done) return true;
    }
    return false;
}
// Block barrier with the conjunction of v.  Not the .aligned form of
// __syncthreads_and: threads of one warp wait for different units' copies and may
// arrive apart (that form let L = 6 blocks through early).
__device__ __forceinline__ bool block_and(bool v) {
    uint32_t r;
    asm volatile("{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbarrier.cta.red.and.pred q, 0, p;\nselp.u32 %0, 1, 0, q;\n}\n"
                 : "=r"(r)
                 : "r"((uint32_t)v)
                 : "memory");
    return r != 0;
}
// Bulk copies: 16-byte aligned on both sides, sizes multiples of 16 (a plane is
// 8 L^2 bytes, L even).
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                     smem_addr(dst)),
                 "l"(src), "r"(bytes), "r"(smem_addr(bar))
                 : "memory");
}
__device__ __forceinline__ void bulk_store(void *dst, const void *src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n" ::"l"(dst), "r"(smem_addr(src)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory"); }
__device__ __forceinline__ void fence_async() { asm volatile("fence.proxy.async;\n" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

// A thread's two columns and their neighbours as words of a plane; threads of
// even and odd position take the even and odd row of a row pair.
struct Cols {
    int o0, o1, l0, u0, d0, r1, u1, d1;
    int qrow;  // Philox block index within a tau pair
    __device__ __forceinline__ Cols(int L, int c) {
        const int rp = c / L, e = c - rp * L;
        const int y = 2 * rp + (e & 1), xh = e >> 1;
        const int x0 = 2 * xh + (y & 1);
        const int x1 = x0 + 1 == L ? 0 : x0 + 1;
        const int x0m = x0 == 0 ? L - 1 : x0 - 1, x1p = x1 + 1 == L ? 0 : x1 + 1;
        const int yp = y + 1 == L ? 0 : y + 1, ym = y == 0 ? L - 1 : y - 1;
        o0 = y * L + x0;
        o1 = y * L + x1;
        l0 = y * L + x0m;
        u0 = yp * L + x0;
        d0 = ym * L + x0;
        r1 = y * L + x1p;
        u1 = yp * L + x1;
        d1 = ym * L + x1;
        qrow = y * (L / 2) + xh;
    }
};
// The seven couplings of the two sites (r0 is also the left one of column x1).
struct Couplings {
    uint64_t r0, l0, u0, d0, r1, u1, d1;
    __device__ __forceinline__ Couplings(const Group &g, int w, const Cols &k) {
        const uint64_t *Jx = g.Jx + (size_t)w * g.L * g.L, *Jy = g.Jy + (size_t)w * g.L * g.L;
        r0 = __ldg(Jx + k.o0);
        l0 = __ldg(Jx + k.l0);
        u0 = __ldg(Jy + k.o0);
        d0 = __ldg(Jy + k.d0);
        r1 = __ldg(Jx + k.o1);
        u1 = __ldg(Jy + k.o1);
        d1 = __ldg(Jy + k.d1);
    }
};

// Colour-1 sites (x0, pb - 1) and (x0 + 1, pb) around chunk boundary pb; spins
// are read from global memory past L1 (the neighbouring unit wrote them).
template <int ALGO, int L>
__device__ __forceinline__ void boundary_sites(const Group &g, const Cols &k, const Couplings &J, uint64_t *Sg, int pb,
                                               const Thresh &T, uint32_t sweep, uint32_t slot, uint32_t k0,
                                               uint32_t k1) {
    constexpr int L2 = L * L;
    const int Lt = g.Ltau;
    const uint32_t tag = (STREAM_SWEEP << 24) | ((uint32_t)g.gid << 8);
    const uint64_t apbc = g.boundary == 1 ? ~0ull : 0ull;
    {
        const int p = pb == 0 ? Lt - 1 : pb - 1;  // odd plane: x0 is colour 1
        const uint64_t *P = Sg + (size_t)p * L2;
        const uint64_t *Pp = Sg + (size_t)(p + 1 == Lt ? 0 : p + 1) * L2;
        const uint64_t *Pm = Sg + (size_t)(p - 1) * L2;
        const uint64_t fp = p == Lt - 1 ? apbc : 0ull;
        const uint4 r = philox4x32_10(make_uint4((uint32_t)(p >> 1) * (uint32_t)(L2 / 2) + (uint32_t)k.qrow, sweep, slot,
                                                 tag), k0, k1);
        Sg[(size_t)p * L2 + k.o0] =
            update_site<ALGO>(__ldcg(P + k.o0), __ldcg(P + k.o1), __ldcg(P + k.l0), __ldcg(P + k.u0), __ldcg(P + k.d0),
                              __ldcg(Pp + k.o0) ^ fp, __ldcg(Pm + k.o0), J.r0, J.l0, J.u0, J.d0, r.z, T);
    }
    {
        const int p = pb;  // even plane: x0 + 1 is colour 1
        const uint64_t *P = Sg + (size_t)p * L2;
        const uint64_t *Pp = Sg + (size_t)(p + 1) * L2;
        const uint64_t *Pm = Sg + (size_t)(p == 0 ? Lt - 1 : p - 1) * L2;
        const uint64_t fm = p == 0 ? apbc : 0ull;
        const uint4 r = philox4x32_10(make_uint4((uint32_t)(p >> 1) * (uint32_t)(L2 / 2) + (uint32_t)k.qrow, sweep, slot,
                                                 tag), k0, k1);
        Sg[(size_t)p * L2 + k.o1] =
            update_site<ALGO>(__ldcg(P + k.o1), __ldcg(P + k.r1), __ldcg(P + k.o0), __ldcg(P + k.u1), __ldcg(P + k.d1),
                              __ldcg(Pp + k.o1), __ldcg(Pm + k.o1) ^ fm, J.r1, J.r0, J.u1, J.d1, r.y, T);
    }
}

// Slots [0, S1) run nch chunks, slots [S1, nslots) nch2, every slot's chunks of
// nearly equal length, P consecutive ones per block; the boundary counter at the start of chunk ch of slot s is
// arrivals[s * astride + ch].  When a wait for a copy gives up, the block starts no
// further copy, neither way, and updates no boundary site; it runs out its loop on
// what the ring holds, waits for the copies in flight, leaves the counters as a
// finished block would and sets *err (may be null) to DEVERR_TIMEOUT.
template <int ALGO, int L, int P, int NREG>
__global__ void __launch_bounds__(P *L *L / 2) __maxnreg__(NREG)
    k_sweep_unit(const Group g, const int nch, const int S1, const int nch2, const uint32_t *sweep_base,
                 const uint32_t sweep_off, const uint32_t k0, const uint32_t k1, unsigned *__restrict__ arrivals,
                 const int astride, int *err) {
    constexpr int L2 = L * L, NT = L2 / 2, SLOT = L2;
    constexpr uint32_t kPlaneBytes = 8u * L2;
    extern __shared__ __align__(128) uint64_t smem[];
    __shared__ uint64_t full_all[P][4];
    __shared__ int do_boundary[P], loaded[P];  // loaded: groups of planes, of each unit
    const uint32_t sweep = (sweep_base ? *sweep_base : 0u) + sweep_off;
    const int un = P == 1 ? 0 : (int)threadIdx.x / NT, c = (int)threadIdx.x - un * NT;
    const int bps1 = (nch + P - 1) / P, bps2 = (nch2 + P - 1) / P;  // blocks per slot
    const int n1 = S1 * bps1;
    const bool first = (int)blockIdx.x < n1;
    const int nu = first ? nch : nch2, bps = first ? bps1 : bps2;
    const int v = (int)blockIdx.x - (first ? 0 : n1);
    const int s = (first ? 0 : S1) + v / bps;
    const int ch = (v % bps) * P + un;
    const bool active = P == 1 || ch < nu;  // the last block of a slot may lack chunks
    const int Lt = g.Ltau, hp = Lt / 2;
    const int a = active ? 2 * (int)((long long)ch * hp / nu) : 0;
    const int b = active ? 2 * (int)((long long)(ch + 1) * hp / nu) : 0;
    const int Cmin = P == 1 ? b - a : 2 * (hp / nu), Cmax = P == 1 ? b - a : 2 * ((hp + nu - 1) / nu);
    const int M = (Cmax + 3) / 4;
    const int w = s / (g.R * g.K), j = s % g.K;
    uint64_t *Sg = g.S + (size_t)s * g.N;
    uint64_t *ring = smem + (size_t)un * kRing * SLOT;
    uint64_t *full = full_all[un];
    const bool leader = c == 0 && active;

    // group gi: planes a - 1 + 4 gi .. a + 2 + 4 gi (those up to b) into ring slots 4 (gi & 3) ..
    auto load_group = [&](int gi) {
        const int p0 = a - 1 + 4 * gi;
        const int n = min(4, b + 1 - p0);
        if (n <= 0) return;
        uint64_t *dst = ring + (gi & 3) * 4 * SLOT;
        bar_expect(&full[gi & 3], (uint32_t)n * kPlaneBytes);
        if (p0 >= 0 && p0 + n <= Lt) {
            bulk_load(dst, Sg + (size_t)p0 * L2, (uint32_t)n * kPlaneBytes, &full[gi & 3]);
        } else {
            for (int i = 0; i < n; ++i) {
                const int p = p0 + i;
                bulk_load(dst + i * SLOT, Sg + (size_t)(p < 0 ? p + Lt : (p >= Lt ? p - Lt : p)) * L2, kPlaneBytes,
                          &full[gi & 3]);
            }
        }
    };
    // group gi back to global memory: its planes in [a, b)
    auto store_group = [&](int gi) {
        const int p0 = a - 1 + 4 * gi;
        const int lo = max(p0, a), hi = min(p0 + 4, b);
        if (lo < hi)
            bulk_store(Sg + (size_t)lo * L2, ring + ((gi & 3) * 4 + lo - p0) * SLOT, (uint32_t)(hi - lo) * kPlaneBytes);
    };

    if (leader) {
#pragma unroll
        for (int i = 0; i < 4; ++i) bar_init(&full[i]);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        fence_async_smem();
        load_group(0);
        load_group(1);
        load_group(2);
        load_group(3);
    }
    if (leader) loaded[un] = (b - a + 1) / 4 + 1;
    const Cols k(L, c);
    const Couplings J(g, w, k);
    Thresh T;
#pragma unroll
    for (int n = 0; n < 7; ++n) T.t[n] = g.thr[j * 16 + (ALGO == 0 ? n % 3 : 8 + n)];
    const uint32_t tag = (STREAM_SWEEP << 24) | ((uint32_t)g.gid << 8);
    const uint64_t apbc = g.boundary == 1 ? ~0ull : 0ull;
    auto draw = [&](int q) {
        return philox4x32_10(make_uint4((uint32_t)(q >> 1) * (uint32_t)NT + (uint32_t)k.qrow, sweep, (uint32_t)s, tag),
                             k0, k1);
    };
    uint4 ra = draw(a), rb = draw(a + 2);
    uint32_t carry = 0;
    __syncthreads();  // the barriers are initialised
    // no wait of this thread gave up; from the first step's barrier on, of the block.
    // (Leaving the loop, or looking at a flag in shared memory while waiting, made the
    // compiler spill, and a frame in local memory alone costs a launch of few slots 2 us:
    // the host bounds the polls of all steps together instead, see step_polls.)
    bool ok = !active || bar_wait(&full[0], 0u, g.wait_limit);
    uint64_t W0[8], W1[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) W0[i] = W1[i] = 0;
    W0[7] = ring[k.o0];
    W1[7] = ring[k.o1];
    W0[0] = ring[SLOT + k.o0];
    W1[0] = ring[SLOT + k.o1];

    // one step: planes q .. q + 3, q = a + 4 m; slot of plane a + i is (i + 1) & 15
    auto step = [&](int m, auto mm, auto edge) {
        constexpr bool EDGE = decltype(edge)::value;
        constexpr int Q = 4 * decltype(mm)::value;
        const int q = a + 4 * m;
        auto slot = [&](auto ic) -> uint64_t * { return ring + ((decltype(ic)::value + 1) & 15) * SLOT; };
#define IC(N) std::integral_constant<int, Q + (N)>{}
        if (active && (!EDGE || q + 3 <= b))
            ok = bar_wait(&full[(m + 1) & 3], (uint32_t)((m + 1) >> 2) & 1u, g.wait_limit) && ok;
        auto own = [&](auto ic) {
            W0[decltype(ic)::value & 7] = slot(ic)[k.o0];
            W1[decltype(ic)::value & 7] = slot(ic)[k.o1];
        };
        own(IC(1));
        own(IC(2));
        own(IC(3));
        own(IC(4));
        const uint4 r0 = ra, r1 = rb;
        // column x0 of plane a + i (colour 0 on even planes, 1 on odd ones)
        auto col0 = [&](auto ic, uint32_t u, uint64_t fm) {
            constexpr int I = decltype(ic)::value, R = I & 7, RP = (I + 1) & 7, RM = (I + 7) & 7;
            uint64_t *pp = slot(ic);
            W0[R] = update_site<ALGO>(W0[R], W1[R], pp[k.l0], pp[k.u0], pp[k.d0], W0[RP], W0[RM] ^ fm, J.r0, J.l0, J.u0, J.d0,
                                      u, T);
            pp[k.o0] = W0[R];
        };
        auto col1 = [&](auto ic, uint32_t u, uint64_t fp) {
            constexpr int I = decltype(ic)::value, R = I & 7, RP = (I + 1) & 7, RM = (I + 7) & 7;
            uint64_t *pp = slot(ic);
            W1[R] = update_site<ALGO>(W1[R], pp[k.r1], W0[R], pp[k.u1], pp[k.d1], W1[RP] ^ fp, W1[RM], J.r1, J.r0, J.u1, J.d1,
                                      u, T);
            pp[k.o1] = W1[R];
        };
        {
            if (!EDGE || q < b) col0(IC(0), r0.x, EDGE && q == 0 ? apbc : 0ull);
            if (!EDGE || q + 1 < b) col1(IC(1), r0.w, EDGE && q + 2 == Lt ? apbc : 0ull);
            if (!EDGE || q + 2 < b) col0(IC(2), r1.x, 0ull);
            if (!EDGE || q + 3 < b) col1(IC(3), r1.w, EDGE && q + 4 == Lt ? apbc : 0ull);
        }
        fence_async_smem();
        ok = block_and(ok);
        if (leader && ok && (!EDGE || m > 0)) {
            store_group(m - 1);
            bulk_commit();
        }
        {
            if (!EDGE || (q - 1 > a && q - 1 < b - 1)) col0(IC(-1 + 16), carry, 0ull);
            if (!EDGE || (q > a && q < b - 1)) col1(IC(0), r0.y, 0ull);
            if (!EDGE || (q + 1 < b - 1)) col0(IC(1), r0.z, 0ull);
            if (!EDGE || (q + 2 < b - 1)) col1(IC(2), r1.y, 0ull);
        }
        ra = draw(q + 4);
        rb = draw(q + 6);
        carry = r1.z;
        if (leader && (!EDGE || m > 0)) {
            if (ok) {
                bulk_wait_read();
                load_group(m + 3);
            } else {
                loaded[un] = min(loaded[un], m + 3);
            }
        }
#undef IC
    };
    // steps whose planes q - 1 .. q + 4 are all inside the chunk run without the
    // edge checks
    for (int m0 = 0; m0 < M; m0 += 4) {
        if (m0 == 0 || 4 * (m0 + 3) + 5 > Cmin) {
            step(m0, std::integral_constant<int, 0>{}, std::true_type{});
            if (P > 1 || m0 + 1 < M) step(m0 + 1, std::integral_constant<int, 1>{}, std::true_type{});
            if (P > 1 || m0 + 2 < M) step(m0 + 2, std::integral_constant<int, 2>{}, std::true_type{});
            if (P > 1 || m0 + 3 < M) step(m0 + 3, std::integral_constant<int, 3>{}, std::true_type{});
        } else {
            step(m0, std::integral_constant<int, 0>{}, std::false_type{});
            step(m0 + 1, std::integral_constant<int, 1>{}, std::false_type{});
            step(m0 + 2, std::integral_constant<int, 2>{}, std::false_type{});
            step(m0 + 3, std::integral_constant<int, 3>{}, std::false_type{});
        }
    }
    // steps run: no more than the planes need (up to three idle ones cost 3 % at L = 24,
    // L_tau = 2048, 1,005 -> 970 us, 10 % at L = 16, L_tau = 512, 96 slots, 55 -> 50 us; with
    // several chunks per block the checks cost more than they save)
    const int Mr = P > 1 ? (M + 3) / 4 * 4 : M;
    fence_async_smem();
    __syncthreads();
    const int chn = ch + 1 == nu ? 0 : ch + 1;  // the chunk after the last is the first
    if (c == 0) {
        int flags = 0;
        if (active) {
            if (ok) {
                store_group(Mr - 1);
                store_group(Mr);
                bulk_commit();
            } else {
                const int n = loaded[un];
                for (int gi = max(n - 4, 0); gi < n; ++gi) bar_wait(&full[gi & 3], (uint32_t)(gi >> 2) & 1u, kDrainPolls);
                if (err) atomicExch(err, (int)DEVERR_TIMEOUT);
            }
            bulk_wait_all();
            fence_async();
            __threadfence();
            if (atomicAdd(&arrivals[s * astride + ch], 1u) == 1u) flags |= 1;
            if (atomicAdd(&arrivals[s * astride + chn], 1u) == 1u) flags |= 2;
            __threadfence();
        }
        do_boundary[un] = ok ? flags : flags | 4;
    }
    __syncthreads();
    const int flags = do_boundary[un];
    if (flags) {
        if ((flags & 5) == 1)
            boundary_sites<ALGO, L>(g, k, J, Sg, a, T, sweep, (uint32_t)s, k0, k1);
        if ((flags & 6) == 2)
            boundary_sites<ALGO, L>(g, k, J, Sg, b == Lt ? 0 : b, T, sweep, (uint32_t)s, k0, k1);
        if (c == 0) {
            if (flags & 1) arrivals[s * astride + ch] = 0u;
            if (flags & 2) arrivals[s * astride + chn] = 0u;
        }
    }
}

// Polls of a step's wait: a block whose wait gave up runs out its steps, each of which
// may wait in vain, so that they share eight limits; but no less than 1,024 polls a wait
// (a poll suspends the thread for a while), unless the limit itself is smaller.
inline unsigned step_polls(unsigned limit, int steps) {
    const unsigned long long share = 8ull * limit / (unsigned)(steps < 8 ? 8 : steps);
    const unsigned long long least = limit < 1024u ? limit : 1024u;
    return (unsigned)(share > least ? share : least);
}

// The launch of one sweep: nch chunks per slot for the first S1 slots, nch2 for
// the others; with arrivals == nullptr only *resident is set, to (SMs x 64 + the
// blocks of this instance an SM holds) x 64 + the chunks of a block.
template <int ALGO, int L>
cudaError_t launch_unit(const Group &g, int nch, int nch2, int S1, const uint32_t *sweep_base, uint32_t sweep,
                        uint64_t seed, unsigned *arrivals, int *err, int *resident, cudaStream_t st) {
    constexpr int P = units_per_block(L);
    constexpr int threads = P * L * L / 2;
    constexpr size_t sm = (size_t)P * kRing * L * L * sizeof(uint64_t);
    auto kern = k_sweep_unit<ALGO, L, P, unit_regs(L)>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
    if (!arrivals) {
        int dev = 0, nsm = 0, per = 0;
        e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, threads, sm);
        *resident = (nsm * 64 + per) * 64 + P;
        return e;
    }
    Group gw = g;
    const int shortest = nch < nch2 ? nch : nch2;  // chunks of a slot
    gw.wait_limit = step_polls(g.wait_limit, (g.Ltau / 2 + shortest - 1) / shortest / 2 + 2);
    const int blocks = S1 * ((nch + P - 1) / P) + (g.nslots - S1) * ((nch2 + P - 1) / P);
    count_launches(1);
    kern<<<blocks, threads, sm, st>>>(gw, nch, S1, nch2, sweep_base, sweep, (uint32_t)seed, (uint32_t)(seed >> 32),
                                      arrivals, nch > nch2 ? nch : nch2, err);
    return cudaGetLastError();
}

template <int ALGO>
cudaError_t launch_unit_L(const Group &g, int nch, int nch2, int S1, const uint32_t *sb, uint32_t sweep, uint64_t seed,
                          unsigned *arrivals, int *err, int *resident, cudaStream_t st) {
#define QSG_UNIT(N) \
    case N: return launch_unit<ALGO, N>(g, nch, nch2, S1, sb, sweep, seed, arrivals, err, resident, st);
    switch (g.L) {
        QSG_UNIT(6)
        QSG_UNIT(8)
        QSG_UNIT(10)
        QSG_UNIT(12)
        QSG_UNIT(14)
        QSG_UNIT(16)
        QSG_UNIT(18)
        QSG_UNIT(20)
        QSG_UNIT(22)
        QSG_UNIT(24)
        QSG_UNIT(26)
        QSG_UNIT(28)
        QSG_UNIT(30)
        QSG_UNIT(32)
    }
#undef QSG_UNIT
    return cudaErrorInvalidValue;
}

}  // namespace unit
}  // namespace qsg
