// FP64 x-line sweeps on the caller's layout (line_tile.cu).
#pragma once
#include <vector>

#include "brs_internal.cuh"

int line_tile_setup(brs_ctx* c);
void line_tile_teardown(brs_ctx* c);
int line_tile_sweep(brs_ctx* c, void* u, const void* b, int nsweeps, cudaStream_t s);
// On a Jacobi context with omega = 1: out = M^{-1}(b + N u), and out = M^{-1} r.
int line_tile_undamped(brs_ctx* c, const double* u, double* out, const double* b, cudaStream_t s);
int line_tile_solve(brs_ctx* c, const double* r, double* out, cudaStream_t s);
// The buffer for scaled b belongs to the line-major form, where the context has it.
void line_tile_borrow(brs_ctx* c, double* bs);
// Release what only calls of several sweeps use.
void line_tile_trim(brs_ctx* c);

// Pivots of the elimination from both ends (line_seq.cu).
std::vector<double> seq_line_pivots(int n, double ax, double ay, double az);
