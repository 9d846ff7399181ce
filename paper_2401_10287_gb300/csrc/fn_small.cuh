// Single-kernel value pass and Metropolis chain of small FP64 networks (fn_small.cu).
#pragma once
#include "fn_internal.cuh"

namespace fn {

// FP64 mode, at most 8 electrons, 64 columns and 16 determinants, activations within 96 KB (one CTA
// holds whole walkers), and no more walkers than it is the faster path for.
bool small_covers(const fn_system* s, int B);
void launch_small_log_psi(const fn_system* s, const void* walkers, int B, double* log_psi, int8_t* sign, cudaStream_t st);
void launch_small_mcmc(const fn_system* s, void* walkers, double* log_psi, int B, int n_steps, double step_size,
                       uint64_t seed, uint64_t step_offset, int64_t* accept, cudaStream_t st);

}  // namespace fn
