// mixed.h -- the MIXED32 particle half (int cell + FP32 offset, FP32 gather/push/deposit,
// tile-binned particles with shared-memory field and current windows), for one or many
// simulations sharing each launch.
#pragma once

#include <cuda_runtime.h>

#include <string>

#include "pic.h"
#include "pic_internal.cuh"

namespace pic {

struct MixedState;

// Temporaries of the library's stream-ordered pool (mixed.cu), which keeps what it was given for
// the next load or re-sort. Those of read-backs and diagnostics (scratch_alloc) are in it up
// to kScratchKept bytes each; larger ones come from the device's default pool and go back to the
// device. temp_free releases either.
constexpr size_t kScratchKept = 64u << 20;
cudaError_t temp_alloc(void** p, size_t bytes, cudaStream_t st);
cudaError_t scratch_alloc(void** p, size_t bytes, cudaStream_t st);
void temp_free(void* p, cudaStream_t st);

// Choose tiles and allocate bins for ngrids simulations (fills the tile fields of the
// host descriptors G[0..ngrids), which the caller then copies to dgrids).
int mixed_create(MixedState** out, const pic_params* p, int ngrids, GridDev* G,
                 const GridDev* dgrids, long long ntot, float* F32, long long* Jfix, CgState* cg,
                 DevStatus* st, std::string& err);
void mixed_destroy(MixedState* m);
// Replace one species' particles of simulation g (FP64 physical positions and momenta,
// host or device).
int mixed_load(MixedState* m, int g, int sp, const double* x, const double* y, const double* ux,
               const double* uy, const double* uz, long long n, cudaStream_t s, std::string& err);
// Enqueue one part of a step: part 0 = its start (stop flag, counters, J = 0) and the
// overflow-list push, 1 = tile kernels, 2 = the injector's pairs, 3 = its end (buffer
// swap, PCG statistics).
void mixed_enqueue(MixedState* m, cudaStream_t s, int part);
// Host bookkeeping around a pic_step call: lost bins are refused before it, overflowed ones
// sorted anew after it.
int mixed_before_steps(MixedState* m, cudaStream_t s, std::string& err);
// hs: the device status as it is after the steps
int mixed_after_steps(MixedState* m, const DevStatus& hs, cudaStream_t s, std::string& err);

// Kernels mixed_enqueue launches per step (all parts together).
int mixed_step_kernels(const MixedState* m);
long long mixed_count(MixedState* m, int g, int sp);
// Add simulation g's node density into rho (device, ncell values; may be null), each
// particle of species s contributing q[s] (0: the species is left out), and w * its
// total momentum into mom (device, 3 values; may be null).
int mixed_rho_momentum(MixedState* m, int g, const double q[2], double* rho, double* mom, cudaStream_t s,
                       std::string& err);
long long mixed_rebins(MixedState* m);
// Bumped whenever device buffers are reallocated: step graphs captured before hold stale
// pointers and must be rebuilt.
long long mixed_generation(MixedState* m);
// Copy out one species of simulation g as FP64 [x, y, ux, uy, uz] (physical units).
int mixed_particles(MixedState* m, int g, int sp, double* out5xn, long long n, cudaStream_t s,
                    std::string& err);

}  // namespace pic
