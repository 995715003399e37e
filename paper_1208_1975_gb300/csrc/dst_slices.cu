// FP64 sine transforms along x on the tensor cores: dst = src S for rows of n doubles and the
// symmetric DST-I matrix S.
//
// GB300 retires 2 FP64 FMAs per clock per SM, 626 G/s, so the n/2 FMAs per cell of the folded
// product (plane_modes_f64.cu) take 3.6 ms per transform at 256^3, 55 % of a 50-sweep FP64 plane
// call.  Here every factor is split into 7 signed digits of 8 bits (the Ozaki scheme: K. Ozaki,
// T. Ogita, S. Oishi, S. M. Rump, "Error-free transformations of matrix multiplication by using
// fast routines of matrix multiplication and its applications", Numer. Algorithms 59, 2012):
//   x = 2^e sum_s d_s 2^(-8 s),  |d_s| <= 128,  s = 1..7   (56 bits; e from the row's largest)
// and the digit products are summed on the tensor cores in bf16 with FP32 accumulators, which hold
// integers below 2^24 exactly.  Products of equal weight, s + t = const, share an accumulator; the
// 28 pairs with s + t <= 8 reach below FP64's rounding of the row's largest product (the ones left
// out are under 2^-72 of it each).  One output is 7 exact integers, joined in 64-bit integer
// arithmetic and rounded: no FP64 instruction at all per output.
//
// Measured at 256^3, same box: 0.44 ms per transform (0.09 slicing, 0.35 products, whose digit
// tiles, 84 KB per 56 instructions, come from L2 at about 7 TB/s) against 3.6; calls of 50 FP64
// plane sweeps 20.1 -> 9.2 ms, of one 14.2 -> 1.09.  Errors against extended precision, u uniform,
// n = 48 .. 480, products on the FP64 pipe -> here: one sweep 7e-17 -> 5e-17 of the 2-norm, two
// 4.7 .. 8.4e-16 -> 1.2 .. 2.1e-16.
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

#include "dst_slices.cuh"
#include "plane_tc.cuh"

namespace {

constexpr int kDig = 7;      // digits per factor, 8 bits each
constexpr int kTileM = 128, kTileN = 64, kStepK = 32;
constexpr int kStages = 2;
constexpr int kGemmThreads = 320;  // producer warp, MMA warp, 8 epilogue warps
constexpr int kABytes = kTileM * kStepK * 2, kBBytes = kTileN * kStepK * 2;
constexpr int kStage = kDig * (kABytes + kBBytes);
constexpr int kSmem = 1024 + kStages * kStage + 128;
constexpr int kNaNRow = 0x7fffffff;
constexpr int kMinN = 48;  // below, the digits' passes cost more than n/2 FMAs per cell

__device__ __forceinline__ float small_int(int d)  // exact for |d| < 2^22
{
    return __int_as_float(0x4B400000 + d) - 12582912.0f;
}

// Rows to slice: plain rows of src, or (um set) the plane right-hand sides
// b + az (u_{k-1} + u_{k+1}) of planes k = k0, k0 + kstep, ...: row r of the call is line r % ny of
// its plane r / ny.
struct RowSource {
    const double* src;  // rows, or b
    const double* u;    // null: plain rows
    double az;
    int ny, nz, k0, kstep;
    long long row0;     // first row of this block in the call
};

// One row per warp, staged in shared memory: exps[row] = e (kNaNRow if the row holds a NaN or an
// infinity), digit planes of the row, zero in the padded columns n .. Kp.
__global__ void __launch_bounds__(256) slice_rows(const RowSource rs,
                                                  __nv_bfloat16* __restrict__ dig,
                                                  int* __restrict__ exps, int n, int Kp,
                                                  long long rows, long long plane)
{
    extern __shared__ __align__(16) double row_smem[];
    pdl_wait_trigger();
    const int lane = threadIdx.x & 31;
    double* r = row_smem + (threadIdx.x >> 5) * Kp;
    for (long long row = (long long)blockIdx.x * 8 + (threadIdx.x >> 5); row < rows;
         row += (long long)gridDim.x * 8) {
        int emax = 1;
        const long long line = rs.row0 + row;
        if (rs.u) {
            const int k = rs.k0 + (int)(line / rs.ny) * rs.kstep;
            const long long pl = (long long)n * rs.ny;
            const long long o = pl * k + line % rs.ny * n;
            for (int x = lane; x < n; x += 32) {
                const double um = k > 0 ? rs.u[o + x - pl] : 0.0;
                const double up = k + 1 < rs.nz ? rs.u[o + x + pl] : 0.0;
                const double v = fma(rs.az, um + up, rs.src[o + x]);
                r[x] = v;
                emax = max(emax, (__double2hiint(v) >> 20) & 0x7ff);
            }
        } else {
            const double* src = rs.src + line * n;
            for (int x = lane; x < n; x += 32) {
                const double v = src[x];
                r[x] = v;
                emax = max(emax, (__double2hiint(v) >> 20) & 0x7ff);
            }
        }
        for (int x = n + lane; x < Kp; x += 32)
            r[x] = 0.0;
        emax = __reduce_max_sync(0xffffffffu, emax);
        __syncwarp();
        if (lane == 0)
            exps[row] = emax == 0x7ff ? kNaNRow : emax - 1021;
        for (int x = 2 * lane; x < Kp; x += 64) {
            uint32_t w[kDig];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const long long bits = emax != 0x7ff ? __double_as_longlong(r[x + h]) : 0;
                int ex = (int)(bits >> 52) & 0x7ff;
                long long m = bits & 0xfffffffffffffll;
                if (ex)
                    m |= 1ll << 52;
                else
                    ex = 1;
                // the row's largest becomes 55 bits; smaller values are rounded to its last bit
                const int sh = emax - ex - 2;
                m = sh <= 0 ? m << -sh : sh < 62 ? (m + (1ll << (sh - 1))) >> sh : 0;
                if (bits < 0)
                    m = -m;
#pragma unroll
                for (int s = kDig - 1; s >= 0; --s) {
                    const int d = s ? (int)(signed char)(m & 255) : (int)m;
                    m = (m - d) >> 8;
                    const uint32_t f = __float_as_uint(small_int(d));
                    w[s] = h ? __byte_perm(w[s], f, 0x7632) : f;  // (low half: first element)
                }
            }
            uint32_t* o = reinterpret_cast<uint32_t*>(dig + row * Kp + x);
#pragma unroll
            for (int s = 0; s < kDig; ++s)
                o[(long long)s * (plane >> 1)] = w[s];
        }
        __syncwarp();
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

struct SliceArgs {
    double* dst;
    const double* scale;
    const int* exps;
    int* status;
    int n, period, eb;     // row length, scale period (rows), exponent of S's digits
    int ksteps, tiles_n;
    int alloc_rows, np;    // rows of one digit plane in the A and B maps
    long long row0, rows;  // first row of this block in the call, rows in it
    long long ntiles;
    // update (u set): dst and u are grids, row r of the call is line r % ny of plane
    // k0 + (r / ny) kstep, and dst = om1 u + value
    const double* u;
    double om1;
    int ny, k0, kstep;
};

__global__ void __launch_bounds__(kGemmThreads, 1) slices_gemm(const __grid_constant__ CUtensorMap mA,
                                                      const __grid_constant__ CUtensorMap mB,
                                                      const __grid_constant__ SliceArgs g)
{
    using namespace brs_tc;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* base = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* full = reinterpret_cast<uint64_t*>(base + kStages * kStage);
    uint64_t* empty = full + kStages;
    uint64_t* accf = empty + kStages;  // the accumulators hold a finished tile
    uint64_t* acce = accf + 1;         // they have been read out
    uint64_t* done = acce + 1;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(accf, 1);
        mbar_init(acce, 8);
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
            if (ti >= 1 && !mbar_wait_bounded(acce, (uint32_t)((ti - 1) & 1))) {
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
                            mma_bf16(tmem + (uint32_t)((i + j) * kTileN),
                                     da + (uint64_t)((i * kABytes + k * 32) >> 4),
                                     db + (uint64_t)((j * kBBytes + k * 32) >> 4), idesc,
                                     kb > 0 || k > 0 || i > 0 ? 1u : 0u);
                mma_commit(&empty[s]);
            }
            if (!ok) {
                *abort_flag = 1;
                break;
            }
            mma_commit(accf);
        }
        mma_commit(done);
    } else if (warp >= 2) {
        // two warps per TMEM lane quarter, each half of the tile's columns
        const int q = warp & 3, c0 = warp >= 6 ? kTileN / 2 : 0;
        int ti = 0;
        for (long long t = blockIdx.x; t < g.ntiles; t += gridDim.x, ++ti) {
            const bool ok = mbar_wait_bounded(accf, (uint32_t)(ti & 1));
            if (__any_sync(0xffffffffu, !ok || *abort_flag)) {
                *abort_flag = 1;
                break;
            }
            tc_fence_after();
            const int n0 = (int)(t % g.tiles_n) * kTileN;
            const long long row = (t / g.tiles_n) * kTileM + q * 32 + lane;
            const bool rok = row < g.rows;
            const int e = rok ? __ldg(g.exps + row) : 0;
            // value = (H 2^32 + L) 2^E
            const int E = e + g.eb - 64;
            const bool plain = E > -900 && E < 900;  // else in steps of exact factors
            const long long line = g.row0 + (rok ? row : 0);
            const double* sc = g.scale ? g.scale + line % g.period * g.n : nullptr;
            long long off = line * g.n;
            if (g.u)
                off = ((long long)(g.k0 + (int)(line / g.ny) * g.kstep) * g.ny + line % g.ny) * g.n;
            double* out = g.dst + off;
            const bool vec = (g.n & 1) == 0;
            const uint32_t trow = tmem + ((uint32_t)(q * 32) << 16);
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
                double v[8];
#pragma unroll
                for (int x = 0; x < 8; ++x) {
                    // |H| < 2^39, |L| < 2^49: H 2^23 + L / 2^9 keeps 2^-55 of the largest product
                    const long long H = ((long long)__float2int_rn(a[0][x]) << 16) +
                                        ((long long)__float2int_rn(a[1][x]) << 8) +
                                        __float2int_rn(a[2][x]);
                    const long long L = ((long long)__float2int_rn(a[3][x]) << 24) +
                                        ((long long)__float2int_rn(a[4][x]) << 16) +
                                        ((long long)__float2int_rn(a[5][x]) << 8) +
                                        __float2int_rn(a[6][x]);
                    v[x] = to_double((H << 23) + ((L + 256) >> 9), plain ? E + 9 : 0);
                }
                if (!plain) {
                    const int E1 = (E + 9) / 2;
                    const double f = __longlong_as_double(0x7ff8000000000000ll);
#pragma unroll
                    for (int x = 0; x < 8; ++x)
                        v[x] = e == kNaNRow ? f
                                            : v[x] * __hiloint2double((E1 + 1023) << 20, 0) *
                                                  __hiloint2double((E + 9 - E1 + 1023) << 20, 0);
                }
                const int n = n0 + c;
                if (rok && vec && n + 8 <= g.n) {
                    if (sc)
#pragma unroll
                        for (int x = 0; x < 8; x += 2) {
                            const double2 f = __ldg(reinterpret_cast<const double2*>(sc + n + x));
                            v[x] *= f.x;
                            v[x + 1] *= f.y;
                        }
                    if (g.u)
#pragma unroll
                        for (int x = 0; x < 8; x += 2) {
                            const double2 f = *reinterpret_cast<const double2*>(g.u + off + n + x);
                            v[x] = fma(g.om1, f.x, v[x]);
                            v[x + 1] = fma(g.om1, f.y, v[x + 1]);
                        }
#pragma unroll
                    for (int x = 0; x < 8; x += 2)
                        *reinterpret_cast<double2*>(out + n + x) = make_double2(v[x], v[x + 1]);
                } else if (rok) {
#pragma unroll
                    for (int x = 0; x < 8; ++x)
                        if (n + x < g.n) {
                            if (sc)
                                v[x] *= __ldg(sc + n + x);
                            out[n + x] = g.u ? fma(g.om1, g.u[off + n + x], v[x]) : v[x];
                        }
                }
                __syncwarp();
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0)
                mbar_arrive(acce);
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

struct DstSlices {
    int n = 0, Kp = 0, np = 0, eb = 0, sms = 1;
    long long block = 0;  // rows per pass over the digit planes, a multiple of 128
    void* dig = nullptr;  // [7][block][Kp] bf16
    void* bdig = nullptr; // [7][np][Kp] bf16: S's digits
    int* exps = nullptr;
    int* status = nullptr;
    CUtensorMap mA, mB;
};

int dst_slices_create(int n, long long rows, int device, int* status, DstSlices** out)
{
    *out = nullptr;
    if (n < kMinN)
        return BRS_OK;
    int eb = 0;
    std::frexp(std::sqrt(2.0 / (n + 1)), &eb);  // |S| < 2^eb
    ++eb;
    const int Kp = (n + kStepK - 1) / kStepK * kStepK, np = (n + kTileN - 1) / kTileN * kTileN;
    // S[p][x] = sqrt(2/(n+1)) sin(q pi/(n+1)), q = (p+1)(x+1) mod 2(n+1): its digits per q, from a
    // value more exact than a double holds
    const long double pi = 3.14159265358979323846264338327950288L;
    const int per = 2 * (n + 1);
    std::vector<__nv_bfloat16> dq((size_t)kDig * per);
    std::vector<int> aq((size_t)kDig * per);
    for (int q = 0; q < per; ++q) {
        const long double v = std::sqrt(2.0L / (n + 1)) * std::sin(pi * q / (n + 1));
        long long m = std::llround(std::ldexp(v, 56 - eb));
        for (int s = kDig - 1; s >= 0; --s) {
            const int d = s ? (int)(signed char)(m & 255) : (int)m;
            m = (m - d) / 256;
            dq[(size_t)s * per + q] = __float2bfloat16((float)d);
            aq[(size_t)s * per + q] = d < 0 ? -d : d;
        }
    }
    std::vector<__nv_bfloat16> bd((size_t)kDig * np * Kp, __float2bfloat16(0.0f));
    // Exact accumulators: the sums of weight s + t = 2 .. 5 stay below 2^24 for any digits of the
    // rows (|d| <= 128).  The lighter ones, from 2^-48 of the largest product down, may round by a
    // few units without reaching FP64's own rounding of the sum.
    for (int p = 0; p < n; ++p) {
        long long acc = 0;
        for (int t = 0; t < kDig; ++t) {
            const __nv_bfloat16* dt = &dq[(size_t)t * per];
            const int* at = &aq[(size_t)t * per];
            __nv_bfloat16* row = &bd[((size_t)t * np + p) * Kp];
            long long sum = 0;  // sum over x of |digit t|
            for (int x = 0, q = p + 1; x < n; ++x) {
                row[x] = dt[q];
                sum += at[q];
                q += p + 1;
                if (q >= per)
                    q -= per;
            }
            acc += 128 * sum;  // weight t + 2 holds the pairs with digits 0 .. t of S
            if (t < 4 && acc > (1ll << 24))
                return BRS_OK;
        }
    }
    DstSlices* d = new (std::nothrow) DstSlices();
    if (!d)
        return BRS_ERR_NOMEM;
    d->n = n, d->Kp = Kp, d->np = np, d->eb = eb, d->status = status;
    cudaError_t e = cudaDeviceGetAttribute(&d->sms, cudaDevAttrMultiProcessorCount, device);
    // whole waves of tiles: a multiple of one row tile per SM (70 MB of digits at n = 256)
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
        rc = brs_cuda_status(cudaFuncSetAttribute(
            slices_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem));
    if (rc != BRS_OK) {
        dst_slices_destroy(d);
        return rc;
    }
    *out = d;
    return BRS_OK;
}

void dst_slices_destroy(DstSlices* d)
{
    if (!d)
        return;
    for (void* q : {d->dig, d->bdig, (void*)d->exps})
        if (q)
            cudaFree(q);
    delete d;
}

namespace {

int run_blocks(const DstSlices* d, RowSource rs, SliceArgs g, long long rows, cudaStream_t s)
{
    double* dst = g.dst;
    g.exps = d->exps;
    g.status = d->status;
    g.n = d->n, g.eb = d->eb;
    g.ksteps = d->Kp / kStepK;
    g.tiles_n = (d->n + kTileN - 1) / kTileN;
    g.alloc_rows = (int)d->block, g.np = d->np;
    g.dst = dst;
    for (long long r0 = 0; r0 < rows; r0 += d->block) {
        const long long nr = std::min(d->block, rows - r0);
        rs.row0 = g.row0 = r0;
        const unsigned sg = (unsigned)std::min<long long>((nr + 7) / 8, d->sms * 8ll);
        cudaError_t e = launch_pdl(slice_rows, dim3(sg), dim3(256), (size_t)8 * d->Kp * 8, s, rs,
                                   static_cast<__nv_bfloat16*>(d->dig), d->exps, d->n, d->Kp, nr,
                                   d->block * d->Kp);
        if (e != cudaSuccess)
            return brs_cuda_status(e);
        g.rows = nr;
        g.ntiles = (nr + kTileM - 1) / kTileM * g.tiles_n;
        const unsigned grid = (unsigned)std::min<long long>(g.ntiles, d->sms);
        e = launch_pdl(slices_gemm, dim3(grid), dim3(kGemmThreads), kSmem, s, d->mA, d->mB, g);
        if (e != cudaSuccess)
            return brs_cuda_status(e);
    }
    return BRS_OK;
}

}  // namespace

int dst_slices_run(const DstSlices* d, const double* src, double* dst, const double* scale,
                   int period, long long rows, cudaStream_t s)
{
    RowSource rs{};
    rs.src = src;
    SliceArgs g{};
    g.dst = dst;
    g.scale = scale;
    g.period = period;
    return run_blocks(d, rs, g, rows, s);
}

int dst_slices_rhs(const DstSlices* d, const double* u, const double* b, double az, double* dst,
                   const double* scale, int ny, int nz, int k0, int kstep, int planes,
                   cudaStream_t s)
{
    RowSource rs{};
    rs.src = b, rs.u = u, rs.az = az;
    rs.ny = ny, rs.nz = nz, rs.k0 = k0, rs.kstep = kstep;
    SliceArgs g{};
    g.dst = dst;
    g.scale = scale;
    g.period = ny;
    return run_blocks(d, rs, g, (long long)ny * planes, s);
}

int dst_slices_update(const DstSlices* d, const double* src, const double* u, double om1,
                      double* uout, int ny, int k0, int kstep, int planes, cudaStream_t s)
{
    RowSource rs{};
    rs.src = src;
    SliceArgs g{};
    g.dst = uout;
    g.u = u, g.om1 = om1;
    g.ny = ny, g.k0 = k0, g.kstep = kstep;
    return run_blocks(d, rs, g, (long long)ny * planes, s);
}
