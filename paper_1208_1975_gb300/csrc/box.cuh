// Box-block path (box.cu): setup, teardown and one sweep launch.
#pragma once
#include "brs_internal.cuh"

int box_setup(brs_ctx* c);
void box_teardown(brs_ctx* c);
int box_sweep_launch(brs_ctx* c, const void* uin, void* uout, const void* b, cudaStream_t s);

// One-pass form of box sweeps in the box's sine basis (box_sine.cu), for boxes with sides of at
// most 16.  The pass updates the M boxes of `rows` (packed box coordinates) from u into uout.
bool box_sine_takes(const brs_params& p);
int box_sine_setup(const brs_params& p, double omega, void** out);
void box_sine_teardown(void* state);
int box_sine_pass(const void* state, int dtype, const void* u, void* uout, const void* b,
                  const long long* rows, long long M, cudaStream_t s);
