// Coarse end of the V-cycle in one launch (all levels from the first that fits).
#pragma once

#include "mx_internal.cuh"

#define COARSE_MAX_LEVELS 8
#define COARSE_MAX_CELLS 4096  // largest bottom level
#define COARSE_MAX_SMEM (160 * 1024)

// true if levels [0, nl) of `levs` (the last one the bottom) fit the kernel: on
// one CTA, or spread over a cluster
template <typename T>
bool coarse_fits(const Level<T> *levs, int nl, int clustered);

// V-cycle on levs[0..nl): reads levs[0].f, writes levs[0].e (global memory)
template <typename T>
void k_coarse_vcycle(cudaStream_t s, const Level<T> *levs, int nl, int nu1, int nu2, int bot_iters, int singular);

cudaError_t coarse_init();

// batched coarse ends, one CTA per box: argument blocks for one box each (host
// fills and returns the shared memory it needs, device reads)
size_t coarse_args_bytes();
size_t coarse_fill_args(void *dst, const Level<float> *levs, int nl, int nu1, int nu2, int bot_iters, int singular);
void k_coarse_vcycle_batch(cudaStream_t s, const void *dev_args, const SolveState *st, int nbox, size_t smem);
