// Rows of line cells in shared memory, a lane's E consecutive cells at lane * E, for E = 8 with the
// lane's two 16-byte halves trading places when lane / 4 is odd: the 8 lanes of a 16-byte access
// phase then cover all banks, without the register selects that reading halves in either order
// would need.
#pragma once
#include "brs_internal.cuh"

namespace brs {

template <int E>
__device__ __forceinline__ int row_pos(int y)  // place of cell y in its row
{
    return E == 8 ? y ^ ((y >> 3) & 4) : y;
}

template <int E>
__device__ __forceinline__ void row_ld(float (&v)[E], const float* row, int lane)
{
    const float4* p = reinterpret_cast<const float4*>(row + lane * E);
    const int h = E == 8 ? (lane >> 2) & 1 : 0;
#pragma unroll
    for (int m = 0; m < E / 4; ++m) {
        const float4 t = p[m ^ h];
        v[4 * m] = t.x, v[4 * m + 1] = t.y, v[4 * m + 2] = t.z, v[4 * m + 3] = t.w;
    }
}

template <int E>
__device__ __forceinline__ void row_st(float* row, const float (&v)[E], int lane)
{
    float4* p = reinterpret_cast<float4*>(row + lane * E);
    const int h = E == 8 ? (lane >> 2) & 1 : 0;
#pragma unroll
    for (int m = 0; m < E / 4; ++m)
        p[m ^ h] = make_float4(v[4 * m], v[4 * m + 1], v[4 * m + 2], v[4 * m + 3]);
}

}  // namespace brs
