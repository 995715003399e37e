// FP64 x-line sweeps on the caller's layout (line_tile.cu).
#pragma once
#include <vector>

#include "brs_internal.cuh"

int line_tile_setup(brs_ctx* c);
void line_tile_teardown(brs_ctx* c);
int line_tile_sweep(brs_ctx* c, void* u, const void* b, int nsweeps, cudaStream_t s);

// Pivots of the elimination from both ends (line_seq.cu).
std::vector<double> seq_line_pivots(int n, double ax, double ay, double az);
