// k_sweep_unit.cu -- host side of the fused sweep (k_sweep_unit.cuh): which groups
// it serves and how their slots are cut into chunks of tau planes.
#include <atomic>
#include <cmath>

#include "qsg_launch.h"

namespace qsg {

cudaError_t launch_sweep_unit_hb(const Group &g, int nch, int nch2, int S1, const uint32_t *sweep_base, uint32_t sweep,
                                 uint64_t seed, unsigned *arrivals, int *err, int *resident, cudaStream_t st);
cudaError_t launch_sweep_unit_met(const Group &g, int nch, int nch2, int S1, const uint32_t *sweep_base, uint32_t sweep,
                                  uint64_t seed, unsigned *arrivals, int *err, int *resident, cudaStream_t st);

// L = 6 .. 32, any even L_tau; the bulk copies need 16-byte aligned planes.
bool sweep_unit_supported(const Group &g) { return g.L >= 6 && ((uintptr_t)g.S & 15u) == 0; }

static cudaError_t launch(const Group &g, int nch, int nch2, int S1, const uint32_t *sweep_base, uint32_t sweep,
                          uint64_t seed, unsigned *arrivals, int *resident, cudaStream_t st) {
    return g.algo == 0 ? launch_sweep_unit_met(g, nch, nch2, S1, sweep_base, sweep, seed, arrivals, g.err, resident, st)
                       : launch_sweep_unit_hb(g, nch, nch2, S1, sweep_base, sweep, seed, arrivals, g.err, resident, st);
}

// SMs, blocks an SM holds for the group's instance (0 if unknown) and chunks per
// block.
static void residency(const Group &g, int *nsm, int *per, int *chunks) {
    static std::atomic<int> known[2][33];
    int r = known[g.algo][g.L].load(std::memory_order_relaxed);
    if (r == 0) {
        if (launch(g, 1, 1, 0, nullptr, 0, 0, nullptr, &r, nullptr) != cudaSuccess) r = 0;
        known[g.algo][g.L].store(r, std::memory_order_relaxed);
    }
    *nsm = r / 4096;
    *per = r / 64 % 64;
    *chunks = r % 64;
}

// Chunks per slot, chosen so that the blocks fill whole waves of resident ones
// while chunks stay long: a chunk costs its planes plus about kOverhead planes
// (filling the ring, the deferred boundary sites); a last wave that puts x of an
// SM's `per` blocks on the fullest SM takes x / per of a full one, but not below
// kThin (one block alone does not fill an SM).  Against measured times (L = 24,
// L_tau = 2048, 256 slots; 3, 4, 5, 7, 12, 16 chunks) the ratios agree within 4 %, for a
// single chunk within 8 %; seven chunks are the best of them, and the choice.  Chunks
// need not divide L_tau: they differ by two planes at most.
// Blocks of one warp (L = 8) are the load of one of an SM's four schedulers, so they are
// counted per scheduler, and x of the `per` blocks there take (x / per)^0.9 of a full
// wave.  Counted per SM, the choice for L_tau = 1024, 92 slots was 18 chunks in 31.4 us
// per sweep, where 26 take 29.2 and the best count, 33, 28.7.
int sweep_unit_chunks(const Group &g) {
    constexpr double kOverhead = 8.0, kThin = 0.45;
    int nsm = 0, per = 0, P = 1;
    residency(g, &nsm, &per, &P);
    if (nsm <= 0 || per <= 0) return 1;
    const bool one_warp = P == 1 && g.L * g.L / 2 <= 32 && per >= 4;
    if (one_warp) {
        nsm *= 4;
        per /= 4;
    }
    const long long R = (long long)nsm * per;
    int best = 1;
    double best_cost = 1e300;
    const int most = g.Ltau / 16 < 1 ? 1 : g.Ltau / 16;
    // whole blocks of chunks, and the most chunks there can be
    for (int n = most < P ? most : P; n <= most; n = n < most && n + P > most ? most : n + P) {
        const long long blocks = (long long)g.nslots * ((n + P - 1) / P), rest = blocks % R;
        double waves = (double)(blocks / R);
        if (rest > 0) {
            double part = (double)((rest + nsm - 1) / nsm) / per;
            if (one_warp) part = std::pow(part, 0.9);
            waves += part > kThin ? part : kThin;
        }
        const double cost = waves * ((double)g.Ltau / n + kOverhead);
        if (cost < best_cost * 0.999) {
            best_cost = cost;
            best = n;
        }
        if (blocks > 24 * R) break;
    }
    return best;
}

cudaError_t launch_sweep_unit(const Group &g, int nch, int nch2, int S1, const uint32_t *sweep_base, uint32_t sweep,
                              uint64_t seed, unsigned *arrivals, cudaStream_t st) {
    // the boundary counters: L_tau / 4 per slot (one for L_tau = 2)
    const int most = g.Ltau >= 4 ? g.Ltau / 4 : 1;
    if (!sweep_unit_supported(g) || nch < 1 || nch2 < 1 || nch > most || nch2 > most) return cudaErrorInvalidValue;
    return launch(g, nch, nch2, S1, sweep_base, sweep, seed, arrivals, nullptr, st);
}

}  // namespace qsg
