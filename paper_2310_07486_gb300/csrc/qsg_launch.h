// qsg_launch.h -- host-side launchers of the sm_103a kernels (internal).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "qsg_device.cuh"

namespace qsg {

// Process-wide count of kernel launches (qsg_kernel_launches()).
void count_launches(int n);

// Shared-memory limits of kernels (cudaFuncAttributeMaxDynamicSharedMemorySize) are set
// to the largest size that any launch of the kernel takes, never to that of one
// launch: contexts of other shapes on other host threads, or later nodes of the same
// graph, would otherwise lower the limit before the launch that needs it.

// Acceptance tables of a ladder k[0..K) (host FP64, integer results), 16 words
// per ladder position: [0..2] Metropolis thresholds for S h = 2, 4, 6, [8..14]
// heat-bath thresholds for h = 6 - 2 n, the rest zero.  False if the ladder is
// not 0 < k_0 < ... < k_{K-1} < 3 or a table is not monotone (the bitsliced
// comparison of the sweep kernels relies on monotone tables).
bool build_accept_tables(const double *k, int K, uint32_t *table);

// Device-side status word: non-zero after a bounded wait gave up.
enum : int { DEVERR_NONE = 0, DEVERR_TIMEOUT = 1 };
// Polls of each bounded device wait (QSG_OPT_WAIT_LIMIT replaces it).
constexpr unsigned kDefaultWaitLimit = 1u << 22;

cudaError_t launch_init_couplings(const Group &g, uint64_t seed, cudaStream_t st);
cudaError_t launch_init_spins(const Group &g, uint64_t seed, cudaStream_t st);

// One full sweep (colour 0 then colour 1) of every slot of the group.
// The "reference" variant runs one launch per colour with one thread per site.
cudaError_t launch_sweep_reference(const Group &g, uint32_t sweep, uint64_t seed, cudaStream_t st);

// Planes per work unit of the generic wavefront kernel (0 if the group cannot use
// it: L_tau no multiple of 16, or `requested` > 0 no multiple of 16 dividing it).
int wavefront_chunk(const Group &g, int requested);
// 0, 1, 3: the fused kernel with the lattice size compiled in (k_sweep_unit.cuh)
// where it exists; 2: the generic wavefront kernel
extern int g_wavefront_variant;
// One fused sweep, arrivals = nslots * (L_tau / 4) zeroed counters.  The sweep
// index is *sweep_base + sweep (sweep_base may be null), so that a captured CUDA
// graph of several sweeps can be replayed later.  requested: planes per work unit
// (0 = automatic); the last `tail` slots (0 = none) run chunks of a quarter of
// that after every other unit.
bool sweep_fused_supported(const Group &g, int requested);
cudaError_t launch_sweep_wavefront(const Group &g, const uint32_t *sweep_base, uint32_t sweep, uint64_t seed,
                                   unsigned *arrivals, int requested, int tail, cudaStream_t st);
// The form with the lattice size compiled in (L >= 6, any L_tau): slots [0, S1)
// in nch chunks, the others in nch2.
bool sweep_unit_supported(const Group &g);
int sweep_unit_chunks(const Group &g);  // the automatic choice of nch
cudaError_t launch_sweep_unit(const Group &g, int nch, int nch2, int S1, const uint32_t *sweep_base, uint32_t sweep,
                              uint64_t seed, unsigned *arrivals, cudaStream_t st);
// `count` sweeps in one launch, each slot in one block's shared memory.
bool sweep_resident_fits(const Group &g);
cudaError_t launch_sweep_resident(const Group &g, int count, const uint32_t *sweep_base, uint32_t sweep, uint64_t seed,
                                  cudaStream_t st);
cudaError_t launch_set_word(uint32_t *p, uint32_t value, cudaStream_t st);
// dst[0..words) = src[0..words), device to device, by a kernel when both are
// 16-byte aligned and words is even (else by cudaMemcpyAsync).
cudaError_t launch_copy_words(uint64_t *dst, const uint64_t *src, size_t words, cudaStream_t st);
cudaError_t launch_add_word(uint32_t *p, uint32_t value, cudaStream_t st);

// All groups of a context in one persistent launch per sweep (same algorithm,
// L <= 24, L_tau % 16 == 0).  Device arrays: the Group structs, the group
// order (largest first), the prefix sums of work units in that order, the
// chunk length of every group, and two queue counters (zero between launches).
struct PersistentPlan {
    const Group *groups;
    const int *order, *prefix, *chunk;
    unsigned *queue;
    int ngroups, total_units, algo;
};
cudaError_t launch_sweep_persistent(const PersistentPlan &plan, const uint32_t *sweep_base, uint32_t sweep,
                                    uint64_t seed, cudaStream_t st);

// Unsatisfied-bond counts U[slot][bit] of the current configurations.
cudaError_t launch_energy(const Group &g, cudaStream_t st);

// Tempering step `m`: decisions (and U bookkeeping), then the spin-bit moves.
cudaError_t launch_tempering(const Group &g, uint32_t m, uint64_t seed, cudaStream_t st);

// Correlator accumulation through the x-packed transposed scratch buffer;
// tensor = 1 computes the Gram tiles with tcgen05 (k_corr_tc.cu), 0 with
// XOR/popcount on the integer pipes.  status receives DEVERR_TIMEOUT if a
// bounded wait of the tensor path gave up (after wait_limit polls).
// triples = 1 also accumulates the three-replica one-time sums (3 <= R <= 8).
cudaError_t launch_measure(const Group &g, uint64_t *scratch, size_t scratch_words, int tensor, int triples,
                           int *status, unsigned wait_limit, cudaStream_t st);
// One-time observable sums of a batch of (w, j) pairs from the transposed scratch.
cudaError_t launch_onetime(const Group &g, int p0, int np, const uint64_t *P, int triples, cudaStream_t st);
// FP64 finish of the one-time observables into g.outO and g.outK.
cudaError_t launch_onetime_finish(const Group &g, long long n_meas, int triples, cudaStream_t st);
// Tensor-core Gram path over the transposed bits P of a batch: folds every
// 128 x 128 tile of the Gram matrices into the lag sums.
cudaError_t launch_gram_tc(const Group &g, int p0, int npairs, const uint64_t *P, int *status, unsigned wait_limit,
                           cudaStream_t st);

// FP64 finish into g.outC / g.outQ / g.outP.
cudaError_t launch_finish(const Group &g, long long n_meas, cudaStream_t st);

// Scratch words the correlator path needs for one (w, j) pair of the group.
size_t measure_scratch_words_per_pair(const Group &g);

// The 64 coupling features of every sample bit of the group, out [W*64][64].
cudaError_t launch_features(const Group &g, float *out, cudaStream_t st);

// Learned-ladder MLP (k_mlp.cu).  P: FP32 parameters, M, V: Adam moments;
// `steps` steps over the batches idx[steps][batch] (activations and dL/dz in act,
// mlp_act_words(batch) floats), Adam's bias corrections in corr[steps][2]; adam = 0 only writes
// the gradient to grad_out (device, may be null).  loss_out: [steps] (device);
// sync: two device words, the second a status (DEVERR_TIMEOUT after a bounded
// grid wait gave up).  X, T, P and act are 16-byte aligned.
int mlp_param_count();
size_t mlp_act_words(int batch);
cudaError_t launch_mlp_steps(float *P, float *M, float *V, const float *X, const float *T, const int *idx, int steps,
                             int batch, float *act, float *grad_out, int adam, float lr, const float *corr,
                             float *loss_out, unsigned *sync, cudaStream_t st);
cudaError_t launch_mlp_infer(const float *P, const float *X, float *Y, long long n, int bf16, cudaStream_t st);

}  // namespace qsg
