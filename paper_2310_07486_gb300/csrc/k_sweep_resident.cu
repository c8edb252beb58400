// k_sweep_resident.cu -- several checkerboard sweeps of small lattices in one
// launch: a block holds one slot in shared memory from the first sweep to the
// last, so a call of n sweeps reads and writes HBM once and launches once.
//
// The small lattices of the k-ladder study and of short test runs were bound by
// launches, by filling and draining the plane ring and by the deferred chunk
// boundaries, not by their updates.  A sweep, in calls of 30, before and here: L = 8,
// L_tau = 48, 1,280 slots 25 / 16 us; L = 12, L_tau = 64, 128 slots 27 / 5.3 us; L = 10,
// L_tau = 200, 128 slots (no multiple of 16: two one-site-per-thread launches) 44 /
// 11.5 us.
//
// A thread owns the column pair (x0, x0 + 1) of a row (the geometry of
// k_sweep_unit.cuh: bank-conflict-free natural-order planes) on up to IP pairs of
// tau planes, so one Philox call feeds its 2 x 2 (x, tau) block: two colour-0
// updates, a block barrier, two colour-1 updates, a block barrier.  Blocks are
// sized so that an SM's resident blocks have about 1,024 threads together: with
// several slots per SM the barriers of one are hidden behind the others.
#include "k_sweep_unit.cuh"

namespace qsg {

namespace {

using namespace sweep;
using namespace unit;

constexpr size_t kSlotLimit = 226 * 1024;  // bytes of a slot that fit beside the static barrier
// Time of a launch at most, us, and that of a sweep of a slot of N words alone on an
// SM (measured: 0.64 for N = 576, 1.4 for 2,304, 3.5 for 6,400; slots that share an SM
// take less than the sum of theirs).
constexpr double kLaunchTime = 250e3;
constexpr double sweep_time(int N) { return 0.3 + 0.55e-3 * N; }

// A value the compiler knows nothing about: keeps it from carrying the addresses
// of every plane pair from one half sweep to the next in registers (they spilled).
__device__ __forceinline__ int opaque(int v) {
    asm volatile("" : "+r"(v));
    return v;
}

template <int ALGO, int IP>
__global__ void __launch_bounds__(1024, 1) k_sweep_resident(const Group g, const int count, const uint32_t *sweep_base,
                                                            const uint32_t sweep_off, const uint32_t k0,
                                                            const uint32_t k1) {
    extern __shared__ __align__(128) uint64_t smem[];
    __shared__ uint64_t full;
    const int L = g.L, L2 = L * L, ncol = L2 / 2, Lt = g.Ltau, M = Lt / 2;
    const int s = blockIdx.x;
    const int c = (int)threadIdx.x % ncol, m0 = (int)threadIdx.x / ncol, mt = (int)blockDim.x / ncol;
    const int w = s / (g.R * g.K), j = s % g.K;
    uint64_t *Sg = g.S + (size_t)s * g.N;
    const uint32_t bytes = 8u * (uint32_t)g.N;
    const uint32_t sweep0 = (sweep_base ? *sweep_base : 0u) + sweep_off;
    if (threadIdx.x == 0) {
        bar_init(&full);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        fence_async_smem();
        bar_expect(&full, bytes);
        bulk_load(smem, Sg, bytes, &full);
    }
    const Cols k(L, c);
    const Couplings J(g, w, k);
    Thresh T;
#pragma unroll
    for (int n = 0; n < 7; ++n) T.t[n] = g.thr[j * 16 + (ALGO == 0 ? n % 3 : 8 + n)];
    const uint32_t tag = (STREAM_SWEEP << 24) | ((uint32_t)g.gid << 8);
    const uint64_t apbc = g.boundary == 1 ? ~0ull : 0ull;
    __syncthreads();
    // a wait that gives up leaves the slot as it is, once the copy is no longer in flight
    if (!block_and(bar_wait(&full, 0u, g.wait_limit))) {
        if (threadIdx.x == 0) {
            bar_wait(&full, 0u, kDrainPolls);
            if (g.err) atomicExch(g.err, (int)DEVERR_TIMEOUT);
        }
        return;
    }
    for (int it = 0; it < count; ++it) {
        uint32_t ry[IP], rz[IP];
#pragma unroll
        for (int i = 0; i < IP; ++i) {
            const int m = opaque(m0 + mt * i);
            if (m < M) {
                const uint4 r = philox4x32_10(make_uint4((uint32_t)(m * ncol + k.qrow), sweep0 + (uint32_t)it, (uint32_t)s,
                                                         tag), k0, k1);
                ry[i] = r.y;
                rz[i] = r.z;
                uint64_t *p0 = smem + 2 * m * L2, *p1 = p0 + L2;
                const uint64_t *pm = m == 0 ? smem + (Lt - 1) * L2 : p0 - L2, *pn = m == M - 1 ? smem : p1 + L2;
                const uint64_t B0 = p0[k.o1], A1 = p1[k.o0];
                p0[k.o0] = update_site<ALGO>(p0[k.o0], B0, p0[k.l0], p0[k.u0], p0[k.d0], A1,
                                             pm[k.o0] ^ (m == 0 ? apbc : 0ull), J.r0, J.l0, J.u0, J.d0, r.x, T);
                p1[k.o1] = update_site<ALGO>(p1[k.o1], p1[k.r1], A1, p1[k.u1], p1[k.d1],
                                             pn[k.o1] ^ (m == M - 1 ? apbc : 0ull), B0, J.r1, J.r0, J.u1, J.d1, r.w, T);
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < IP; ++i) {
            const int m = opaque(m0 + mt * i);
            if (m < M) {
                uint64_t *p0 = smem + 2 * m * L2, *p1 = p0 + L2;
                const uint64_t *pm = m == 0 ? smem + (Lt - 1) * L2 : p0 - L2, *pn = m == M - 1 ? smem : p1 + L2;
                const uint64_t A0 = p0[k.o0], B1 = p1[k.o1];
                p0[k.o1] = update_site<ALGO>(p0[k.o1], p0[k.r1], A0, p0[k.u1], p0[k.d1], B1,
                                             pm[k.o1] ^ (m == 0 ? apbc : 0ull), J.r1, J.r0, J.u1, J.d1, ry[i], T);
                p1[k.o0] = update_site<ALGO>(p1[k.o0], B1, p1[k.l0], p1[k.u0], p1[k.d0],
                                             pn[k.o0] ^ (m == M - 1 ? apbc : 0ull), A0, J.r0, J.l0, J.u0, J.d0, rz[i], T);
            }
        }
        if (it + 1 == count) fence_async_smem();
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        bulk_store(Sg, smem, bytes);
        bulk_commit();
        bulk_wait_all();
    }
}

template <int ALGO, int IP>
cudaError_t launch(const Group &g, int threads, size_t sm, int count, const uint32_t *sb, uint32_t sweep, uint64_t seed,
                   cudaStream_t st) {
    auto kern = k_sweep_resident<ALGO, IP>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSlotLimit);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
    count_launches(1);
    kern<<<g.nslots, threads, sm, st>>>(g, count, sb, sweep, (uint32_t)seed, (uint32_t)(seed >> 32));
    return cudaGetLastError();
}

template <int ALGO>
cudaError_t launch_ip(int ip, const Group &g, int threads, size_t sm, int count, const uint32_t *sb, uint32_t sweep,
                      uint64_t seed, cudaStream_t st) {
    switch (ip) {
        case 1: return launch<ALGO, 1>(g, threads, sm, count, sb, sweep, seed, st);
        case 2: return launch<ALGO, 2>(g, threads, sm, count, sb, sweep, seed, st);
        case 3: return launch<ALGO, 3>(g, threads, sm, count, sb, sweep, seed, st);
        case 4: return launch<ALGO, 4>(g, threads, sm, count, sb, sweep, seed, st);
        case 6: return launch<ALGO, 6>(g, threads, sm, count, sb, sweep, seed, st);
        default: return launch<ALGO, 8>(g, threads, sm, count, sb, sweep, seed, st);
    }
}

}  // namespace

// Block shape: rows of threads (one per column pair) and plane pairs per thread.
struct ResidentShape {
    int rows, ip;
};
static ResidentShape resident_shape(const Group &g, int nsm) {
    const size_t sm = (size_t)g.N * sizeof(uint64_t);
    const int ncol = g.L * g.L / 2, M = g.Ltau / 2;
    // blocks an SM holds, by shared memory and by the slots there are
    int per = (int)(227 * 1024 / (sm + 1024 + 64));
    const int need = (g.nslots + nsm - 1) / nsm;
    if (per > need) per = need;
    if (per > 16) per = 16;
    if (per < 1) per = 1;
    // 1,024 threads per SM shared out, then the fewest rows that need the same
    // number of plane pairs per thread
    int rows = 1024 / per / ncol;
    if (rows < 1) rows = 1;
    if (rows > M) rows = M;
    int ip = (M + rows - 1) / rows;
    if (ip > 8) ip = 8;
    if (ip == 5) ip = 6;
    if (ip == 7) ip = 8;
    rows = (M + ip - 1) / ip;
    return ResidentShape{rows, ip};
}

// A slot fits one SM's shared memory, and 1,024 threads of eight plane pairs each
// cover it.
bool sweep_resident_fits(const Group &g) {
    if ((size_t)g.N * sizeof(uint64_t) > kSlotLimit || ((uintptr_t)g.S & 15u) != 0) return false;
    return resident_shape(g, 1).rows * (g.L * g.L / 2) <= 1024;
}

cudaError_t launch_sweep_resident(const Group &g, int count, const uint32_t *sweep_base, uint32_t sweep, uint64_t seed,
                                  cudaStream_t st) {
    if (!sweep_resident_fits(g)) return cudaErrorInvalidValue;
    if (count <= 0) return cudaSuccess;
    const size_t sm = (size_t)g.N * sizeof(uint64_t);
    int dev = 0, nsm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const ResidentShape r = resident_shape(g, nsm);
    const int threads = r.rows * (g.L * g.L / 2);
    if (threads > 1024) return cudaErrorInvalidValue;
    // launches of a bounded length, however many sweeps are asked for: an SM serves its
    // share of the slots, so few slots take as long as one per SM
    const long long most = (long long)(kLaunchTime / ((g.nslots + nsm - 1) / nsm * sweep_time(g.N)));
    for (int done = 0; done < count && e == cudaSuccess;) {
        const int n = most < 1 ? 1 : (int)(most < count - done ? most : count - done);
        const uint32_t first = sweep + (uint32_t)done;
        e = g.algo == 0 ? launch_ip<0>(r.ip, g, threads, sm, n, sweep_base, first, seed, st)
                        : launch_ip<1>(r.ip, g, threads, sm, n, sweep_base, first, seed, st);
        done += n;
    }
    return e;
}

}  // namespace qsg
