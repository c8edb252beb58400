// k_sweep_unit_hb.cu -- heat bath instances of the fused sweep (k_sweep_unit.cuh).
#include "k_sweep_unit.cuh"

namespace qsg {

cudaError_t launch_sweep_unit_hb(const Group &g, int nch, int nch2, int S1, const uint32_t *sweep_base, uint32_t sweep,
                                uint64_t seed, unsigned *arrivals, int *err, int *resident, cudaStream_t st) {
    return unit::launch_unit_L<1>(g, nch, nch2, S1, sweep_base, sweep, seed, arrivals, err, resident, st);
}

}  // namespace qsg
