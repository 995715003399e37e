// Sine transforms along x by digits on the tensor cores (dst_slices.cu).
#pragma once
#include "brs_internal.cuh"

// Shortest rows taken: below, the digits' passes cost more than the products they replace (FP32,
// one sweep per call: 64x61x50 36 us against 32 for two sweeps of FP32 products, 100x90x80 51
// against 71; from 96 on FP32 contexts choose by their grid, digits_rule in plane.cu).  Longest: 511,
// without 503 (the digits' sums, dst_slices.cu).
constexpr int dst_slices_min(int element_size) { return element_size == 8 ? 48 : 96; }

template <typename T>
struct DstSlices;

// The orthonormal DST-I S of rows of n values (double or float), in calls of about `rows` rows
// (more run in blocks).  *out stays null where the form does not apply (short rows, or digit sums
// that could leave the exact range of the accumulators).
template <typename T>
int dst_slices_create(int n, long long rows, int device, int* status, DstSlices<T>** out);
template <typename T>
void dst_slices_destroy(DstSlices<T>* d);

// FP64: dst[row][p] = sum_x S[p][x] src[row][x], times scale[(row % period) * n + p] if scale is set.
// src and dst: [rows][n], not overlapping.
int dst_slices_run(const DstSlices<double>* d, const double* src, double* dst, const double* scale,
                   int period, long long rows, cudaStream_t s);

// The same transform of the plane right-hand sides R_k = b_k + az (u_{k-1} + u_{k+1}) (zero outside
// the grid) of planes k0, k0 + kstep, ... of [nz][ny][n] grids: dst[plane][y][p], planes packed,
// times scale[y * n + p] if set; modes: dst[plane][p][y].
template <typename T>
int dst_slices_rhs(const DstSlices<T>* d, const T* u, const T* b, double az, T* dst, const T* scale,
                   int ny, int nz, int k0, int kstep, int planes, bool modes, cudaStream_t s);

// uout_k = om1 u_k + om S src for planes k0, k0 + kstep, ...; src [plane][y][p] packed, u and uout
// grids (may be the same).
template <typename T>
int dst_slices_update(const DstSlices<T>* d, const T* src, const T* u, double om1, double om,
                      T* uout, int ny, int k0, int kstep, int planes, cudaStream_t s);

// Between rows src[plane][y][x] and modes dst[plane][p][y], and back.
int dst_slices_to_modes(const DstSlices<float>* d, const float* src, float* dst, int ny, int planes,
                        cudaStream_t s);
int dst_slices_from_modes(const DstSlices<float>* d, const float* src, float* dst, int ny,
                          int planes, cudaStream_t s);
