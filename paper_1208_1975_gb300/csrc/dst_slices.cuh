// FP64 sine transforms on the tensor cores (dst_slices.cu).
#pragma once
#include "brs_internal.cuh"

struct DstSlices;

// The orthonormal DST-I S of rows of n doubles, in calls of about `rows` rows (more run in
// blocks).  *out stays null where the form does not apply (short rows, or digit sums that could
// leave the exact range of the accumulators).
int dst_slices_create(int n, long long rows, int device, int* status, DstSlices** out);
void dst_slices_destroy(DstSlices* d);

// dst[row][p] = sum_x S[p][x] src[row][x], times scale[(row % period) * n + p] if scale is set.
// src and dst: [rows][n], not overlapping.
int dst_slices_run(const DstSlices* d, const double* src, double* dst, const double* scale,
                   int period, long long rows, cudaStream_t s);

// The same transform of the plane right-hand sides R_k = b_k + az (u_{k-1} + u_{k+1}) (zero outside
// the grid) of planes k0, k0 + kstep, ... of [nz][ny][n] grids: dst[plane][y][p], planes packed,
// times scale[y * n + p].
int dst_slices_rhs(const DstSlices* d, const double* u, const double* b, double az, double* dst,
                   const double* scale, int ny, int nz, int k0, int kstep, int planes,
                   cudaStream_t s);

// uout_k = om1 u_k + S src for planes k0, k0 + kstep, ...; src [plane][y][p] packed, u and uout
// grids (may be the same).
int dst_slices_update(const DstSlices* d, const double* src, const double* u, double om1,
                      double* uout, int ny, int k0, int kstep, int planes, cudaStream_t s);
