// Sine transforms along x on the tensor cores, exact to the element type's rounding: dst = src S
// for rows of n doubles or floats and the symmetric DST-I matrix S.
//
// GB300 retires 2 FP64 FMAs per clock per SM, 626 G/s, so the n/2 FMAs per cell of the folded
// product (plane_modes_f64.cu) take 3.6 ms per transform at 256^3, 55 % of a 50-sweep FP64 plane
// call.  Here every factor is split into 7 signed digits of 8 bits (the Ozaki scheme: K. Ozaki,
// T. Ogita, S. Oishi, S. M. Rump, "Error-free transformations of matrix multiplication by using
// fast routines of matrix multiplication and its applications", Numer. Algorithms 59, 2012):
//   x = 2^e sum_s d_s 2^(-8 s),  |d_s| <= 128,  s = 1..7   (56 bits; e from the row's largest)
// and the digit products are summed on the tensor cores in bf16 with FP32 accumulators, which hold
// integers below 2^24 exactly.  Products of equal weight, s + t = const, share an accumulator; the
// 28 pairs with s + t <= 8 are summed.  A pair left out is at most 2^-58 of 2^(e + eb), the scale of
// the row's digits and S's, which is 4 to 16 times the row's largest product: the six of weight 9 come
// to at most 6 n 2^-58 of it, and as digits fall to about (6 n)^(1/2) 2^-60 (2^-55 at n = 256), where a
// product on the FP64 pipe rounds n/2 partial sums by up to 2^-53 each.  One output is 7 exact
// integers, joined in 64-bit integer arithmetic and rounded: no FP64 instruction at all per output.
// Rows of wide range keep the 2-norm error of the others (one spike, decaying cells, random exponents
// over 3 to 30 decades, n = 130: FP64 1.7 .. 2.9e-16 against 5.1 .. 7.1e-16 by products, FP32 6 .. 8e-8
// against 2.4 .. 3.9e-7).
//
// Rows of n = 48 (FP32 96) to 511 values, 503 excepted.  From 512 on S's largest value falls below the
// next power of two, eb drops with it, and the sums of the first four weights could pass 2^24 (1.18
// times at 512); those of 503 could by its digits (1.07 times).
//
// Measured at 256^3, same box: 0.41 ms per transform (0.07 slicing, 0.34 products, whose digit
// tiles, 84 KB per 56 instructions, come from L2 at about 7 TB/s) against 3.6; calls of 50 FP64
// plane sweeps 20.1 -> 9.2 ms, of one 14.2 -> 1.09.  Errors against extended precision, u uniform,
// n = 48 .. 480, products on the FP64 pipe -> here: one sweep 7e-17 -> 5e-17 of the 2-norm, two
// 4.7 .. 8.4e-16 -> 1.2 .. 2.1e-16.
//
// FP32 (contexts on CUDA cores: sides that are not whole 32-cell blocks) takes 4 digits, 10 pairs
// with s + t <= 5, every accumulator exact: 200x190x180 one sweep per call 354 -> 230 us, and half the error
// (2-norm against FP64, u uniform, n = 100 .. 480: one sweep 5 .. 6e-8 -> 3e-8).
//
// Two kernels per block of rows, sized so that the digits stay in L2:
//  * slice_rows: a warp per row finds the row's largest exponent and writes the 7 digit planes
//    [s][row][Kp] as bf16 (integer arithmetic only).
//  * slices_gemm: persistent, one CTA per SM.  128 rows x 64 columns per tile, K in steps of 32
//    (64-byte swizzled rows) through a two-stage TMA ring that holds all 14 digit tiles of a step
//    (84 KB), 56 tcgen05.mma per step into 7 accumulators (448 TMEM columns), then the epilogue:
//    lane = row, eight columns at a time by two warps per lane quarter.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <new>
#include <type_traits>
#include <vector>

#include "dst_slices.cuh"
#include "plane_tc.cuh"

namespace {

constexpr int kTileM = 128, kTileN = 64, kStepK = 32;
constexpr int kGemmThreads = 320;  // producer warp, MMA warp, 8 epilogue warps
constexpr int kABytes = kTileM * kStepK * 2, kBBytes = kTileN * kStepK * 2;

// Digits per factor (8 bits each), the ring and the accumulator sets by element type.
template <typename T>
struct Dig;
template <>
struct Dig<double> {
    static constexpr int N = 7, MANT = 52, EXPS = 0x7ff, BIAS = 1023;
    using Bits = long long;
    __device__ static Bits bits(double v) { return __double_as_longlong(v); }
};
template <>
struct Dig<float> {
    static constexpr int N = 4, MANT = 23, EXPS = 0xff, BIAS = 127;
    using Bits = int;
    __device__ static Bits bits(float v) { return __float_as_int(v); }
};
template <typename T>
struct Ring {
    static constexpr int STAGE = Dig<T>::N * (kABytes + kBBytes);     // 84 KB / 48 KB
    static constexpr int STAGES = sizeof(T) == 8 ? 2 : 4;
    static constexpr int ACC = Dig<T>::N * kTileN;                    // TMEM columns of a tile
    static constexpr int SETS = 2 * ACC <= 512 ? 2 : 1;               // accumulator sets
    static constexpr int SMEM = 1024 + STAGES * STAGE + 256;
};
constexpr int kNaNRow = 0x7fffffff;

__device__ __forceinline__ float small_int(int d)  // exact for |d| < 2^22
{
    return __int_as_float(0x4B400000 + d) - 12582912.0f;
}

// Rows to slice: plain rows of src, or (u set) the plane right-hand sides
// b + az (u_{k-1} + u_{k+1}) of planes k = k0, k0 + kstep, ...: row r of the call is line r % ny of
// its plane r / ny.
template <typename T>
struct RowSource {
    const T* src;  // rows, or b
    const T* u;    // null: plain rows
    T az;
    int ny, nz, k0, kstep;
    long long row0;  // first row of this block in the call
};

template <typename T>
__device__ __forceinline__ int exponent(T v)
{
    return (int)(Dig<T>::bits(v) >> Dig<T>::MANT) & Dig<T>::EXPS;
}

// The digits of row r (Kp values in shared memory, stride `st`, zero past the row) of one warp,
// whose largest biased exponent is emax (at least 1): exps[row] = e (kNaNRow if the row holds a
// NaN or an infinity) and the digit planes of the row, [s][row][Kp].
// Bound by instruction issue (60 %): taking the digits off one by one, each with its carry, in 64-bit
// integers for both types took 25.6 us per 19456 rows of 256 doubles and 19.6 of 200 floats; all
// at once, in the type's own width, 19.6 and 16.6.
template <typename T>
__device__ __forceinline__ void slice_row(const T* r, int st, int emax, __nv_bfloat16* dig, int* exps,
                                          int Kp, long long row, long long plane)
{
    constexpr int ND = Dig<T>::N, UP = 8 * ND - 2 - Dig<T>::MANT;  // shift of the largest value
    const int lane = threadIdx.x & 31;
    if (lane == 0)
        exps[row] = emax == Dig<T>::EXPS ? kNaNRow : emax - (Dig<T>::BIAS - 2);
    for (int x = 2 * lane; x < Kp; x += 64) {
        uint32_t w[ND];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            using Bits = typename Dig<T>::Bits;
            using Word = std::make_unsigned_t<Bits>;
            constexpr int WB = 8 * (int)sizeof(T);
            const Bits bits = emax != Dig<T>::EXPS ? Dig<T>::bits(r[(x + h) * st]) : 0;
            int ex = (int)(bits >> Dig<T>::MANT) & Dig<T>::EXPS;
            Word m = (Word)bits & (((Word)1 << Dig<T>::MANT) - 1);
            if (ex)
                m |= (Word)1 << Dig<T>::MANT;
            else
                ex = 1;
            // the row's largest becomes 8 ND - 1 bits; smaller values are rounded to its last bit
            const int sh = emax - ex - UP;
            m = sh <= 0 ? m << -sh : sh < WB ? (m + ((Word)1 << (sh - 1))) >> sh : 0;
            const Bits v = bits < 0 ? -(Bits)m : (Bits)m;
            // v = sum_s d_s 256^(ND - 1 - s): with 128 added at every byte below the highest, those
            // bytes hold d_s + 128 and the rest is d_0
            constexpr int LOW = 8 * (ND - 1);
            constexpr Word MASK = ((Word)1 << LOW) - 1;
            const Word l = ((Word)v & MASK) + ((Word)0x8080808080808080ull & MASK);
            const int top = (int)(v >> LOW) + (int)(l >> LOW);
#pragma unroll
            for (int s = 0; s < ND; ++s) {
                const int by = ND - 1 - s;  // digit s is byte `by` of l
                const uint32_t word = by >= 4 ? (uint32_t)((unsigned long long)l >> 32) : (uint32_t)l;
                const float fd = s ? __uint_as_float(__byte_perm(word, 0x4B000000u, 0x7440 | (by & 3))) -
                                         8388736.0f
                                   : small_int(top);
                const uint32_t f = __float_as_uint(fd);
                w[s] = h ? __byte_perm(w[s], f, 0x7632) : f;  // (low half: first element)
            }
        }
        uint32_t* o = reinterpret_cast<uint32_t*>(dig + row * Kp + x);
#pragma unroll
        for (int s = 0; s < ND; ++s)
            o[(long long)s * (plane >> 1)] = w[s];
    }
}

// One row per warp, staged in shared memory.
template <typename T>
__global__ void __launch_bounds__(256) slice_rows(const RowSource<T> rs,
                                                  __nv_bfloat16* __restrict__ dig,
                                                  int* __restrict__ exps, int n, int Kp,
                                                  long long rows, long long plane)
{
    extern __shared__ __align__(16) unsigned char row_smem[];
    pdl_wait_trigger();
    const int lane = threadIdx.x & 31;
    T* r = reinterpret_cast<T*>(row_smem) + (threadIdx.x >> 5) * Kp;
    for (long long row = (long long)blockIdx.x * 8 + (threadIdx.x >> 5); row < rows;
         row += (long long)gridDim.x * 8) {
        int emax = 1;
        const long long line = rs.row0 + row;
        if (rs.u) {
            const int k = rs.k0 + (int)(line / rs.ny) * rs.kstep;
            const long long pl = (long long)n * rs.ny;
            const long long o = pl * k + line % rs.ny * n;
            for (int x = lane; x < n; x += 32) {
                const T um = k > 0 ? rs.u[o + x - pl] : T(0);
                const T up = k + 1 < rs.nz ? rs.u[o + x + pl] : T(0);
                const T v = fma(rs.az, um + up, rs.src[o + x]);
                r[x] = v;
                emax = max(emax, exponent(v));
            }
        } else {
            const T* src = rs.src + line * n;
            for (int x = lane; x < n; x += 32) {
                const T v = src[x];
                r[x] = v;
                emax = max(emax, exponent(v));
            }
        }
        for (int x = n + lane; x < Kp; x += 32)
            r[x] = T(0);
        emax = __reduce_max_sync(0xffffffffu, emax);
        __syncwarp();
        slice_row<T>(r, 1, emax, dig, exps, Kp, row, plane);
        __syncwarp();
    }
}

// Rows over the modes of a [planes][n][ny] array: row k ny + y holds src[k][x][y], x < n.  A CTA
// takes 32 rows of one plane through shared memory, [x][33].
template <typename T>
__global__ void __launch_bounds__(256) slice_modes(const T* __restrict__ src,
                                                   __nv_bfloat16* __restrict__ dig,
                                                   int* __restrict__ exps, int n, int Kp, int ny,
                                                   int planes, long long plane)
{
    extern __shared__ __align__(16) unsigned char row_smem[];
    T* tile = reinterpret_cast<T*>(row_smem);
    pdl_wait_trigger();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ytiles = (ny + 31) / 32;
    for (int u = blockIdx.x; u < ytiles * planes; u += gridDim.x) {
        const int k = u / ytiles, y0 = (u - k * ytiles) * 32;
        const T* s = src + (long long)k * n * ny;
        for (int x = warp; x < Kp; x += 8)
            tile[x * 33 + lane] = x < n && y0 + lane < ny ? s[(long long)x * ny + y0 + lane] : T(0);
        __syncthreads();
        for (int i = warp; i < 32 && y0 + i < ny; i += 8) {
            int emax = 1;
            for (int x = lane; x < n; x += 32)
                emax = max(emax, exponent(tile[x * 33 + i]));
            emax = __reduce_max_sync(0xffffffffu, emax);
            slice_row<T>(tile + i, 33, emax, dig, exps, Kp, (long long)k * ny + y0 + i, plane);
        }
        __syncthreads();
    }
}

// t 2^E rounded to nearest even, for results in the normal range.
__device__ __forceinline__ double to_double(long long t, int E)
{
    if (t == 0)
        return 0.0;
    const unsigned long long a = t < 0 ? -(unsigned long long)t : t;
    const int lz = __clzll(a);
    const unsigned long long m = a << lz;
    unsigned long long q = m >> 11;
    const unsigned rem = (unsigned)m & 0x7ff;
    q += rem > 0x400 || (rem == 0x400 && (q & 1));
    // q holds the implicit bit: it adds one to the exponent field (two after a carry)
    q += (unsigned long long)(1023 + 62 - lz + E) << 52;
    return __longlong_as_double((long long)(q | (t < 0 ? 1ull << 63 : 0)));
}

__device__ __forceinline__ void mma_bf16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc,
                                         uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8])
{
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                   "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
#pragma unroll
    for (int q = 0; q < 8; ++q)
        v[q] = __uint_as_float(r[q]);
}

template <typename T>
struct SliceArgs {
    T* dst;
    const T* scale;
    const int* exps;
    int* status;
    int n, period, eb;     // row length, scale period (rows), exponent of S's digits
    int ksteps, tiles_n;
    int alloc_rows, np;    // rows of one digit plane in the A and B maps
    long long row0, rows;  // first row of this block in the call, rows in it
    long long ntiles;
    // update (u set): dst and u are grids, row r of the call is line r % ny of plane
    // k0 + (r / ny) kstep, and dst = om1 u + om value
    const T* u;
    T om1, om;
    int ny, k0, kstep;
    int modes;  // store dst[plane][n][ny] (row r of the call is line r % ny of plane r / ny)
};

// (the integer t of one output) 2^E for the rows of exponent e
template <typename T>
struct Join;
template <>
struct Join<double> {
    int E;
    bool plain, nan;
    __device__ Join(int e, int eb)
    {
        nan = e == kNaNRow;
        E = (nan ? 0 : e) + eb - 64 + 9;
        plain = !nan && E > -900 && E < 900;  // else in steps of exact factors
    }
    // |H| < 2^39, |L| < 2^49: H 2^23 + L / 2^9 keeps 2^-55 of the largest product
    __device__ double operator()(const float (&a)[7][8], int x) const
    {
        const long long H = ((long long)__float2int_rn(a[0][x]) << 16) +
                            ((long long)__float2int_rn(a[1][x]) << 8) + __float2int_rn(a[2][x]);
        const long long L = ((long long)__float2int_rn(a[3][x]) << 24) +
                            ((long long)__float2int_rn(a[4][x]) << 16) +
                            ((long long)__float2int_rn(a[5][x]) << 8) + __float2int_rn(a[6][x]);
        const double v = to_double((H << 23) + ((L + 256) >> 9), plain ? E : 0);
        if (plain)
            return v;
        if (nan)
            return __longlong_as_double(0x7ff8000000000000ll);
        return v * __hiloint2double((E / 2 + 1023) << 20, 0) *
               __hiloint2double((E - E / 2 + 1023) << 20, 0);
    }
};
template <>
struct Join<float> {
    float f1, f2;
    __device__ Join(int e, int eb)
    {
        const int E = (e == kNaNRow ? 0 : e) + eb - 40, E1 = E / 2;
        f1 = e == kNaNRow ? __int_as_float(0x7fc00000) : __int_as_float((E1 + 127) << 23);
        f2 = __int_as_float((E - E1 + 127) << 23);
    }
    __device__ float operator()(const float (&a)[4][8], int x) const
    {
        const long long t = ((long long)__float2int_rn(a[0][x]) << 24) +
                            ((long long)__float2int_rn(a[1][x]) << 16) +
                            ((long long)__float2int_rn(a[2][x]) << 8) + __float2int_rn(a[3][x]);
        return __ll2float_rn(t) * f1 * f2;
    }
};

template <typename T>
__global__ void __launch_bounds__(kGemmThreads, 1) slices_gemm(const __grid_constant__ CUtensorMap mA,
                                                               const __grid_constant__ CUtensorMap mB,
                                                               const __grid_constant__ SliceArgs<T> g)
{
    using namespace brs_tc;
    constexpr int kDig = Dig<T>::N, kStages = Ring<T>::STAGES, kStage = Ring<T>::STAGE;
    constexpr int SETS = Ring<T>::SETS, ACC = Ring<T>::ACC;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* base = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* full = reinterpret_cast<uint64_t*>(base + kStages * kStage);
    uint64_t* empty = full + kStages;
    uint64_t* accf = empty + kStages;  // an accumulator set holds a finished tile
    uint64_t* acce = accf + SETS;      // it has been read out
    uint64_t* done = acce + SETS;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int a = 0; a < SETS; ++a) {
            mbar_init(&accf[a], 1);
            mbar_init(&acce[a], 8);
        }
        mbar_init(done, 1);
        *abort_flag = 0;
        fence_mbar_init();
    }
    __syncwarp();
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(tmem_slot)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    pdl_wait();

    int issued = 0;
    if (warp == 0 && lane == 0) {
        int kg = 0;
        for (long long t = blockIdx.x; t < g.ntiles && !*abort_flag; t += gridDim.x) {
            const int n0 = (int)(t % g.tiles_n) * kTileN, m0 = (int)(t / g.tiles_n) * kTileM;
            for (int kb = 0; kb < g.ksteps; ++kb, ++kg) {
                const int s = kg % kStages;
                if (kg >= kStages &&
                    !mbar_wait_bounded(&empty[s], (uint32_t)((kg / kStages - 1) & 1))) {
                    *abort_flag = 1;
                    break;
                }
                unsigned char* st = base + s * kStage;
                mbar_arrive_expect_tx(&full[s], kStage);
                for (int d = 0; d < kDig; ++d) {
                    tma_load_2d(st + d * kABytes, &mA, &full[s], kb * kStepK, d * g.alloc_rows + m0);
                    tma_load_2d(st + kDig * kABytes + d * kBBytes, &mB, &full[s], kb * kStepK,
                                d * g.np + n0);
                }
                issued = kg + 1;
            }
        }
    } else if (warp == 1 && lane == 0) {
        // D = F32, A = B = BF16, both K-major, M = 128, N = 64
        constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) |
                                   ((uint32_t)(kTileN >> 3) << 17) | ((uint32_t)(kTileM >> 4) << 24);
        int kg = 0, ti = 0;
        for (long long t = blockIdx.x; t < g.ntiles && !*abort_flag; t += gridDim.x, ++ti) {
            const int a = ti % SETS;
            if (ti >= SETS && !mbar_wait_bounded(&acce[a], (uint32_t)((ti / SETS - 1) & 1))) {
                *abort_flag = 1;
                break;
            }
            tc_fence_after();
            bool ok = true;
            for (int kb = 0; kb < g.ksteps; ++kb, ++kg) {
                const int s = kg % kStages;
                if (*abort_flag || !mbar_wait_bounded(&full[s], (uint32_t)((kg / kStages) & 1))) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint64_t da = smem_desc_kmajor<16>(base + s * kStage);
                const uint64_t db = smem_desc_kmajor<16>(base + s * kStage + kDig * kABytes);
#pragma unroll
                for (int k = 0; k < kStepK / 16; ++k)
#pragma unroll
                    for (int i = 0; i < kDig; ++i)
#pragma unroll
                        for (int j = 0; j + i < kDig; ++j)
                            mma_bf16(tmem + (uint32_t)(a * ACC + (i + j) * kTileN),
                                     da + (uint64_t)((i * kABytes + k * 32) >> 4),
                                     db + (uint64_t)((j * kBBytes + k * 32) >> 4), idesc,
                                     kb > 0 || k > 0 || i > 0 ? 1u : 0u);
                mma_commit(&empty[s]);
            }
            if (!ok) {
                *abort_flag = 1;
                break;
            }
            mma_commit(&accf[a]);
        }
        mma_commit(done);
    } else if (warp >= 2) {
        // two warps per TMEM lane quarter, each half of the tile's columns
        const int q = warp & 3, c0 = warp >= 6 ? kTileN / 2 : 0;
        int ti = 0;
        for (long long t = blockIdx.x; t < g.ntiles; t += gridDim.x, ++ti) {
            const int as = ti % SETS;
            const bool ok = mbar_wait_bounded(&accf[as], (uint32_t)((ti / SETS) & 1));
            if (__any_sync(0xffffffffu, !ok || *abort_flag)) {
                *abort_flag = 1;
                break;
            }
            tc_fence_after();
            const int n0 = (int)(t % g.tiles_n) * kTileN;
            const long long row = (t / g.tiles_n) * kTileM + q * 32 + lane;
            const bool rok = row < g.rows;
            const int e = rok ? __ldg(g.exps + row) : 0;
            const Join<T> join(e, g.eb);
            const long long line = g.row0 + (rok ? row : 0);
            const T* sc = g.scale ? g.scale + line % g.period * g.n : nullptr;
            const long long pl = (g.u || g.modes) ? line / g.ny : 0;
            long long off = line * g.n;
            if (g.u)
                off = ((long long)(g.k0 + (int)pl * g.kstep) * g.ny + (line - pl * g.ny)) * g.n;
            T* out = g.dst + (g.modes ? pl * g.n * g.ny + (line - pl * g.ny) : off);
            using V = std::conditional_t<sizeof(T) == 8, double2, float4>;
            constexpr int VN = 16 / sizeof(T);
            const bool vec = g.n % VN == 0 && !g.modes;
            const uint32_t trow = tmem + (uint32_t)(as * ACC) + ((uint32_t)(q * 32) << 16);
#pragma unroll 1
            for (int c = c0; c < c0 + kTileN / 2; c += 8) {
                if (n0 + c >= g.n)
                    break;  // uniform
                float a[kDig][8];
#pragma unroll
                for (int d = 0; d < kDig; ++d)
                    tmem_ld8(trow + (uint32_t)(d * kTileN + c), a[d]);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                for (int d = 0; d < kDig; ++d)
#pragma unroll
                    for (int x = 0; x < 8; ++x)
                        asm volatile("" : "+f"(a[d][x]));  // no use before the wait
                T v[8];
#pragma unroll
                for (int x = 0; x < 8; ++x)
                    v[x] = join(a, x);
                const int n = n0 + c;
                if (rok && vec && n + 8 <= g.n) {
                    T f[8];
                    if (sc) {
#pragma unroll
                        for (int x = 0; x < 8 / VN; ++x)
                            reinterpret_cast<V*>(f)[x] = __ldg(reinterpret_cast<const V*>(sc + n) + x);
#pragma unroll
                        for (int x = 0; x < 8; ++x)
                            v[x] *= f[x];
                    }
                    if (g.u) {
#pragma unroll
                        for (int x = 0; x < 8 / VN; ++x)
                            reinterpret_cast<V*>(f)[x] = reinterpret_cast<const V*>(g.u + off + n)[x];
#pragma unroll
                        for (int x = 0; x < 8; ++x)
                            v[x] = fma(g.om1, f[x], g.om * v[x]);
                    }
#pragma unroll
                    for (int x = 0; x < 8 / VN; ++x)
                        reinterpret_cast<V*>(out + n)[x] = reinterpret_cast<const V*>(v)[x];
                } else if (rok) {
#pragma unroll
                    for (int x = 0; x < 8; ++x)
                        if (n + x < g.n) {
                            if (sc)
                                v[x] *= __ldg(sc + n + x);
                            if (g.u)
                                v[x] = fma(g.om1, g.u[off + n + x], g.om * v[x]);
                            out[g.modes ? (long long)(n + x) * g.ny : (long long)(n + x)] = v[x];
                        }
                }
                __syncwarp();
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0)
                mbar_arrive(&acce[as]);
        }
    }
    __syncwarp();
    // every MMA has completed before TMEM is released; on an abort the producer drains its copies
    const bool fin = mbar_wait_bounded(done, 0);
    if (warp == 0 && lane == 0 && (*abort_flag || !fin)) {
        set_status(g.status, BRS_ERR_TIMEOUT);
        for (int kg = (issued > kStages ? issued - kStages : 0); kg < issued; ++kg)
            mbar_wait_bounded(&full[kg % kStages], (uint32_t)((kg / kStages) & 1), 200000000ull);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512)
                     : "memory");
    }
}

// 2D map of digit planes [total rows][Kp] bf16, box (32, box_rows), 64-byte swizzle.
int encode_digits(CUtensorMap* m, const void* ptr, int Kp, long long total, int box_rows)
{
    PFN_encode_tiled fn = brs_encoder();
    if (!fn)
        return BRS_ERR_CUDA;
    cuuint64_t gdim[2] = {(cuuint64_t)Kp, (cuuint64_t)total};
    cuuint64_t gstr[1] = {(cuuint64_t)Kp * 2};
    cuuint32_t box[2] = {(cuuint32_t)kStepK, (cuuint32_t)box_rows};
    cuuint32_t es[2] = {1u, 1u};
    CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), gdim, gstr, box,
                    es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? BRS_OK : BRS_ERR_CUDA;
}

}  // namespace

template <typename T>
struct DstSlices {
    int n = 0, Kp = 0, np = 0, eb = 0, sms = 1;
    long long block = 0;  // rows per pass over the digit planes, a multiple of 128
    void* dig = nullptr;  // [digit][block][Kp] bf16
    void* bdig = nullptr; // [digit][np][Kp] bf16: S's digits
    int* exps = nullptr;
    int* status = nullptr;
    CUtensorMap mA, mB;
};

namespace {

// dynamic shared memory of a kernel: only ever raised, the attribute is every context's
int allow_smem(const void* k, size_t bytes)
{
    cudaFuncAttributes fa{};
    cudaError_t e = cudaFuncGetAttributes(&fa, k);
    if (e == cudaSuccess && (size_t)fa.maxDynamicSharedSizeBytes < bytes)
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    return brs_cuda_status(e);
}

template <typename T>
size_t modes_smem(int Kp) { return (size_t)Kp * 33 * sizeof(T); }

// The products of the rows [r0, r0 + nr) of a call, whose digits are in place.
template <typename T>
int run_gemm(const DstSlices<T>* d, SliceArgs<T> g, long long r0, long long nr, cudaStream_t s)
{
    g.exps = d->exps;
    g.status = d->status;
    g.n = d->n, g.eb = d->eb;
    g.ksteps = d->Kp / kStepK;
    g.tiles_n = (d->n + kTileN - 1) / kTileN;
    g.alloc_rows = (int)d->block, g.np = d->np;
    g.row0 = r0, g.rows = nr;
    g.ntiles = (nr + kTileM - 1) / kTileM * g.tiles_n;
    const unsigned grid = (unsigned)std::min<long long>(g.ntiles, d->sms);
    return brs_cuda_status(launch_pdl(slices_gemm<T>, dim3(grid), dim3(kGemmThreads),
                                      (size_t)Ring<T>::SMEM, s, d->mA, d->mB, g));
}

template <typename T>
int run_blocks(const DstSlices<T>* d, RowSource<T> rs, const SliceArgs<T>& g, long long rows,
               cudaStream_t s)
{
    int rc = BRS_OK;
    for (long long r0 = 0; r0 < rows && rc == BRS_OK; r0 += d->block) {
        const long long nr = std::min(d->block, rows - r0);
        rs.row0 = r0;
        const unsigned sg = (unsigned)std::min<long long>((nr + 7) / 8, d->sms * 8ll);
        rc = brs_cuda_status(launch_pdl(slice_rows<T>, dim3(sg), dim3(256),
                                        (size_t)8 * d->Kp * sizeof(T), s, rs,
                                        static_cast<__nv_bfloat16*>(d->dig), d->exps, d->n, d->Kp,
                                        nr, d->block * d->Kp));
        if (rc == BRS_OK)
            rc = run_gemm(d, g, r0, nr, s);
    }
    return rc;
}

}  // namespace

template <typename T>
int dst_slices_create(int n, long long rows, int device, int* status, DstSlices<T>** out)
{
    constexpr int kDig = Dig<T>::N;
    *out = nullptr;
    if (n < dst_slices_min(sizeof(T)))
        return BRS_OK;
    int eb = 0;
    std::frexp(std::sqrt(2.0 / (n + 1)), &eb);  // |S| < 2^eb
    ++eb;
    const int Kp = (n + kStepK - 1) / kStepK * kStepK, np = (n + kTileN - 1) / kTileN * kTileN;
    // S[p][x] = sqrt(2/(n+1)) sin(q pi/(n+1)), q = (p+1)(x+1) mod 2(n+1): its digits per q, from a
    // value more exact than a double holds
    const long double pi = 3.14159265358979323846264338327950288L;
    const int per = 2 * (n + 1);
    std::vector<__nv_bfloat16> dq((size_t)kDig * per);  // [q][digit]
    std::vector<int> aq((size_t)kDig * per);
    for (int q = 0; q < per; ++q) {
        const long double v = std::sqrt(2.0L / (n + 1)) * std::sin(pi * q / (n + 1));
        long long m = std::llround(std::ldexp(v, 8 * kDig - eb));
        for (int s = kDig - 1; s >= 0; --s) {
            const int d = s ? (int)(signed char)(m & 255) : (int)m;
            m = (m - d) / 256;
            dq[(size_t)q * kDig + s] = __float2bfloat16((float)d);
            aq[(size_t)q * kDig + s] = d < 0 ? -d : d;
        }
    }
    std::vector<__nv_bfloat16> bd((size_t)kDig * np * Kp, __float2bfloat16(0.0f));
    // Exact accumulators: the sums of weight s + t = 2 .. 5 stay below 2^24 for any digits of the
    // rows (|d| <= 128).  FP64's lighter ones, from 2^-48 of the largest product down, may round by
    // a few units without reaching FP64's own rounding of the sum.
    for (int p = 0; p < n; ++p) {
        int sum[kDig] = {};  // sums over x of |digit t|
        for (int x = 0, q = p + 1; x < n; ++x) {
            const __nv_bfloat16* dt = &dq[(size_t)q * kDig];
            const int* at = &aq[(size_t)q * kDig];
            for (int t = 0; t < kDig; ++t) {
                bd[((size_t)t * np + p) * Kp + x] = dt[t];
                sum[t] += at[t];
            }
            q += p + 1;
            if (q >= per)
                q -= per;
        }
        long long acc = 0;
        for (int t = 0; t < 4; ++t) {
            acc += 128ll * sum[t];  // weight t + 2 holds the pairs with digits 0 .. t of S
            if (acc > (1ll << 24))
                return BRS_OK;
        }
    }
    DstSlices<T>* d = new (std::nothrow) DstSlices<T>();
    if (!d)
        return BRS_ERR_NOMEM;
    d->n = n, d->Kp = Kp, d->np = np, d->eb = eb, d->status = status;
    cudaError_t e = cudaDeviceGetAttribute(&d->sms, cudaDevAttrMultiProcessorCount, device);
    // whole waves of tiles: a multiple of one row tile per SM (70 MB of FP64 digits at n = 256)
    const long long need = (rows + kTileM - 1) / kTileM * kTileM;
    d->block = std::min<long long>(need, (long long)d->sms * kTileM);
    if (e == cudaSuccess)
        e = cudaMalloc(&d->dig, (size_t)kDig * d->block * Kp * 2);
    if (e == cudaSuccess)
        e = cudaMalloc(&d->exps, (size_t)d->block * sizeof(int));
    if (e == cudaSuccess)
        e = cudaMalloc(&d->bdig, bd.size() * 2);
    if (e == cudaSuccess)
        e = cudaMemcpy(d->bdig, bd.data(), bd.size() * 2, cudaMemcpyHostToDevice);
    int rc = brs_cuda_status(e);
    if (rc == BRS_OK)
        rc = encode_digits(&d->mA, d->dig, Kp, kDig * d->block, kTileM);
    if (rc == BRS_OK)
        rc = encode_digits(&d->mB, d->bdig, Kp, (long long)kDig * np, kTileN);
    if (rc == BRS_OK)
        rc = allow_smem((const void*)slices_gemm<T>, Ring<T>::SMEM);
    if (rc == BRS_OK && sizeof(T) == 4)
        rc = allow_smem((const void*)slice_modes<T>, modes_smem<T>(Kp));
    if (rc != BRS_OK) {
        dst_slices_destroy(d);
        return rc;
    }
    *out = d;
    return BRS_OK;
}

template <typename T>
void dst_slices_destroy(DstSlices<T>* d)
{
    if (!d)
        return;
    void* bufs[] = {d->dig, d->bdig, d->exps};
    for (void* q : bufs)
        if (q)
            cudaFree(q);
    delete d;
}

int dst_slices_run(const DstSlices<double>* d, const double* src, double* dst, const double* scale,
                   int period, long long rows, cudaStream_t s)
{
    RowSource<double> rs{};
    rs.src = src;
    SliceArgs<double> g{};
    g.dst = dst;
    g.scale = scale;
    g.period = period;
    return run_blocks(d, rs, g, rows, s);
}

template <typename T>
int dst_slices_rhs(const DstSlices<T>* d, const T* u, const T* b, double az, T* dst, const T* scale,
                   int ny, int nz, int k0, int kstep, int planes, bool modes, cudaStream_t s)
{
    RowSource<T> rs{};
    rs.src = b, rs.u = u, rs.az = (T)az;
    rs.ny = ny, rs.nz = nz, rs.k0 = k0, rs.kstep = kstep;
    SliceArgs<T> g{};
    g.dst = dst;
    g.scale = scale;
    g.period = ny;
    g.ny = ny;
    g.modes = modes;
    return run_blocks(d, rs, g, (long long)ny * planes, s);
}

template <typename T>
int dst_slices_update(const DstSlices<T>* d, const T* src, const T* u, double om1, double om,
                      T* uout, int ny, int k0, int kstep, int planes, cudaStream_t s)
{
    RowSource<T> rs{};
    rs.src = src;
    SliceArgs<T> g{};
    g.dst = uout;
    g.u = u, g.om1 = (T)om1, g.om = (T)om;
    g.ny = ny, g.k0 = k0, g.kstep = kstep;
    return run_blocks(d, rs, g, (long long)ny * planes, s);
}

int dst_slices_to_modes(const DstSlices<float>* d, const float* src, float* dst, int ny, int planes,
                        cudaStream_t s)
{
    RowSource<float> rs{};
    rs.src = src;
    SliceArgs<float> g{};
    g.dst = dst;
    g.ny = ny;
    g.modes = 1;
    return run_blocks(d, rs, g, (long long)ny * planes, s);
}

int dst_slices_from_modes(const DstSlices<float>* d, const float* src, float* dst, int ny,
                          int planes, cudaStream_t s)
{
    SliceArgs<float> g{};
    const int per = (int)std::max<long long>(1, d->block / ny);  // whole planes per block
    int rc = BRS_OK;
    for (int k0 = 0; k0 < planes && rc == BRS_OK; k0 += per) {
        const int np = std::min(per, planes - k0);
        const unsigned sg = (unsigned)std::min((ny + 31) / 32 * np, d->sms * 4);
        rc = brs_cuda_status(launch_pdl(slice_modes<float>, dim3(sg), dim3(256),
                                        modes_smem<float>(d->Kp), s,
                                        src + (long long)k0 * d->n * ny,
                                        static_cast<__nv_bfloat16*>(d->dig), d->exps, d->n, d->Kp,
                                        ny, np, d->block * d->Kp));
        g.dst = dst + (long long)k0 * ny * d->n;
        if (rc == BRS_OK)
            rc = run_gemm(d, g, 0, (long long)np * ny, s);
    }
    return rc;
}

#define BRS_DST_SLICES(T)                                                                      \
    template int dst_slices_create<T>(int, long long, int, int*, DstSlices<T>**);               \
    template void dst_slices_destroy<T>(DstSlices<T>*);                                         \
    template int dst_slices_rhs<T>(const DstSlices<T>*, const T*, const T*, double, T*, const T*, \
                                   int, int, int, int, int, bool, cudaStream_t);                \
    template int dst_slices_update<T>(const DstSlices<T>*, const T*, const T*, double, double,  \
                                      T*, int, int, int, int, cudaStream_t);
BRS_DST_SLICES(double)
BRS_DST_SLICES(float)
#undef BRS_DST_SLICES
