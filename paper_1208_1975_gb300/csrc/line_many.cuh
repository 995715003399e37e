// Several line solves side by side in one line group.
#pragma once
#include "line_impl.cuh"

namespace brs {

// line_solve (line_impl.cuh) of M lines at once, step by step side by side: one line's chain of
// multiply-adds and shuffles leaves most issue slots of its warp empty.
template <int E, int G, int M>
__device__ __forceinline__ void line_solve_many(float (&r)[M][E], const LineTables<float, E, G>& tb,
                                                int lane)
{
    constexpr int LG = Log2<G>::value;
    float z[M], B[M];
#pragma unroll
    for (int m = 0; m < M; ++m)
        z[m] = 0.0f;
#pragma unroll
    for (int q = 0; q < E; ++q)
#pragma unroll
        for (int m = 0; m < M; ++m)
            z[m] = fma(tb.c[q], z[m], r[m][q]);
#pragma unroll
    for (int m = 0; m < M; ++m)
        B[m] = z[m];
#pragma unroll
    for (int t = 0; t < LG; ++t) {
        const int d = 1 << t;
        float Bp[M];
#pragma unroll
        for (int m = 0; m < M; ++m)
            Bp[m] = __shfl_up_sync(0xffffffffu, B[m], d, G);
#pragma unroll
        for (int m = 0; m < M; ++m)
            if (lane >= d)
                B[m] = fma(tb.af[t], Bp[m], B[m]);
    }
#pragma unroll
    for (int m = 0; m < M; ++m) {
        z[m] = __shfl_up_sync(0xffffffffu, B[m], 1, G);
        if (lane == 0)
            z[m] = 0.0f;
    }
#pragma unroll
    for (int q = 0; q < E; ++q)
#pragma unroll
        for (int m = 0; m < M; ++m) {
            z[m] = fma(tb.c[q], z[m], r[m][q]);
            r[m][q] = z[m];
        }
#pragma unroll
    for (int m = 0; m < M; ++m)
        z[m] = 0.0f;
#pragma unroll
    for (int q = E - 1; q >= 0; --q)
#pragma unroll
        for (int m = 0; m < M; ++m)
            z[m] = fma(tb.e[q], z[m], r[m][q]);
#pragma unroll
    for (int m = 0; m < M; ++m)
        B[m] = z[m];
#pragma unroll
    for (int t = 0; t < LG; ++t) {
        const int d = 1 << t;
        float Bn[M];
#pragma unroll
        for (int m = 0; m < M; ++m)
            Bn[m] = __shfl_down_sync(0xffffffffu, B[m], d, G);
#pragma unroll
        for (int m = 0; m < M; ++m)
            if (lane + d < G)
                B[m] = fma(tb.ab[t], Bn[m], B[m]);
    }
#pragma unroll
    for (int m = 0; m < M; ++m) {
        z[m] = __shfl_down_sync(0xffffffffu, B[m], 1, G);
        if (lane == G - 1)
            z[m] = 0.0f;
    }
#pragma unroll
    for (int q = E - 1; q >= 0; --q)
#pragma unroll
        for (int m = 0; m < M; ++m) {
            z[m] = fma(tb.e[q], z[m], r[m][q]);
            r[m][q] = z[m];
        }
}

}  // namespace brs
