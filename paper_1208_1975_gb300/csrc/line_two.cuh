// FP32 x-line Jacobi, two sweeps per pass (line_two.cu).
#pragma once
#include "brs_internal.cuh"

// Sets c->two_stages (0: the context does not take the form).
int line_two_setup(brs_ctx* c);
// Pairs of sweeps that a call of nsweeps runs as one pass each.
int line_two_pairs(const brs_ctx* c, int nsweeps);
// Two sweeps from uin into uout (different arrays).
int line_two_launch(brs_ctx* c, const void* uin, void* uout, const void* b, cudaStream_t s);
