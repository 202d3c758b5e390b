// kernels.h -- host-side launchers of the SLPIC kernels (kernels.cu).
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "slpic_internal.cuh"

namespace slpic {

constexpr int kParticleThreads = 256;
constexpr int kFieldThreads = 1024;        // k_potential (one CTA)
constexpr int kFieldClusterCtas = 8;       // k_field: one cluster of 8 CTAs
constexpr int kFieldClusterCtasWide = 16;  // k_field_wide: 16 (non-portable cluster size)
constexpr int kFieldClusterThreads = 256;

size_t particle_smem_bytes(int nn);         // E + one int64 per node (allocation-free kernel)
size_t particle_kernel_smem_bytes(int nn);  // k_particles_compact: E + split deposit
size_t particle_inplace_smem_bytes(int nn); // k_particles: E + split deposit
constexpr int kCompactEvery = 16;           // one compacting particle step per this many
size_t field_smem_bytes(int nn);
size_t field_cluster_smem_bytes(int nn, int ns, int ctas);
int field_max_nodes();
cudaError_t configure_kernels(int nn);
cudaError_t particle_ctas_per_sm(int nn, int *inplace, int *compacting);

void launch_particles(const StepParams &p, int ctas_per_species, bool compact, cudaStream_t st);
// k_particles_tma: the in-place step with the particle stream staged by TMA bulk
// copies, one CTA of kTmaThreads per SM (kTmaConsumers consumer threads, one
// producer warp), tiles of kTmaTile particles in a ring of `stages` stages.
constexpr int kTmaThreads = 1024;
constexpr int kTmaConsumers = 992;
constexpr int kTmaPer = 2;                         // particles per consumer thread per tile
constexpr int kTmaTile = kTmaConsumers * kTmaPer;  // 1,984 particles: 7,936 B of cells
size_t particle_tma_smem_bytes(int nn, int stages);
// ring stages that fit beside an nn-node grid (at most 4); 0 if fewer than 2 fit
cudaError_t configure_particles_tma(int nn, int *stages);
void launch_particles_tma(const StepParams &p, int ctas, int stages, cudaStream_t st);
// k_steps (steps.cu): many steps in one cooperative launch of `ctas` CTAs; scratch of
// steps_scratch_bytes on the device; max_smem: dynamic shared memory it may take
constexpr int kStepsThreads = 1024;
// Where the line lies (us a step, three kernels against k_steps): 2,560 particles 27 / 9,
// 51,200 30 / 12, 5.2e5 42 / 25, 2.0e6 62 / 47, 4.9e6 83 / 75, 8.1e6 104 / 107.5.  The host
// knows the slots, of which a third to all are in use: at 7e6 it is no slower for any count.
// (A species' sums also have to fit 64 bits: fewer than 2^24 particles.)
constexpr long long kStepsMaxSlots = 7000000;  // most slots, all species
static_assert(kStepsMaxSlots < (1LL << 24), "steps_field");
// Every CTA does the whole field, which the cheaper steps of a periodic grid (no walls, no
// source, every slot in use) do not hide on many nodes (beta = 1: 3,000 nodes 6.9e6 81 / 83;
// 4,000 5.0e6 72 / 69, 6.9e6 84 / 85; 6,000 3.5e6 62 / 61, 5.0e6 72 / 75; 8,400 1.0e6 46 / 46,
// 2.0e6 53 / 56; between plates it holds at 8,400 and 6.9e6), so there the line comes down.
constexpr long long steps_max_slots(int nn, bool periodic)
{
    const long long line = 1150LL * (9000 - nn);
    return periodic && line < kStepsMaxSlots ? line : kStepsMaxSlots;
}
constexpr int kStepsFewest = 4, kStepsMost = 4096;  // steps of a launch
size_t steps_scratch_bytes(int nn, int ns);
size_t steps_smem_bytes(int nn, int ns, bool profile);
cudaError_t configure_steps(int *max_smem);
cudaError_t launch_steps(const StepParams &p, int nsteps, int every, int ctas, void *scratch, cudaStream_t st);
void launch_hard(const StepParams &p, int ctas, bool compact, cudaStream_t st);
void launch_field(const StepParams &p, int mode, cudaStream_t st);
// copy of a deposit ([species][nn], ndep words) and of E, for an overlapped read-back
void launch_snapshot(const unsigned long long *dep, unsigned long long *dep_out, size_t ndep,
                     const float *E, float *E_out, int nn, cudaStream_t st);
// rho and phi (p.rho, p.phi) from the deposit dep ([species][nn]) of time level step
void launch_potential(const StepParams &p, const unsigned long long *dep, long long step,
                      cudaStream_t st);
// batched forms over many instances: d_params[m] on the device.  A CTA b of a particle
// kernel takes the work items first[b] .. first[b+1]-1, {instance, species, f0, f1} each: the
// instance's tiles of that species from f0 to f1 of kBatchParts.
constexpr int kBatchParts = 1 << 24;
struct BatchWork {
    int4 *items = nullptr;
    int *first = nullptr;
    int ctas = 0;
};
// CTAs per SM of the batched particle kernels; stages: of the TMA-staged in-place one (0: the
// per-warp one)
cudaError_t configure_batch_kernels(int max_nn, int *inplace_per_sm, int *compact_per_sm, int *stages);
void launch_particles_batch(const StepParams *d_params, const BatchWork &w, int max_nn, bool compact,
                            int stages, cudaStream_t st);
void launch_hard_batch(const StepParams *d_params, int m, int ctas, bool compact, cudaStream_t st);
void launch_field_batch(const StepParams *d_params, int m, int max_nn, int max_ns, int mode,
                        cudaStream_t st);
void launch_deposit(const StepParams &p, int ctas_per_species, cudaStream_t st);
void launch_diag(const StepParams &p, double *out, int ctas_per_species, cudaStream_t st);
void launch_validate(const int32_t *cell, const float *off, const float *v, long long n,
                     int n_cells, int *bad, cudaStream_t st);
void launch_pack(const int32_t *cell, const float *off, const float *v, long long n,
                 int32_t *cdst, float4 *pdst, cudaStream_t st);
void launch_unpack(const int32_t *csrc, const float4 *psrc, long long n, int32_t *cell,
                   float *off, float *v, cudaStream_t st);

}  // namespace slpic
