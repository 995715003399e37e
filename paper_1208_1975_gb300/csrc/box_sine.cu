// Box blocks in one pass: gather, exact block solve and update fused, the block inverse applied
// in the block's own sine basis.
//
// With zero values outside the box, A_b = ax Tx + ay Ty + az Tz on the box is diagonal in the
// product of the three orthonormal DST-I bases (S symmetric, S S = I; Sec. 4.3's one
// precomputed inverse, factored), so
//   Ahat r = S_x S_y S_z  diag(1 / lambda_pqr)  S_z S_y S_x r,
//   lambda_pqr = ax s_p + ay s_q + az s_r,  s_p = 2 - 2 cos((p+1) pi / (b+1)).
// A length-N transform splits by mirror symmetry (S[p][N-1-i] = (-1)^p S[p][i]) into sums and
// differences and two half-size products; for N = 2, 4, 8 the products themselves shrink, because
// the angles k pi / (N+1) are multiples of 60, 36 and 20 degrees (dst below).  An 8x8x8 box takes
// 6 x 3.75 operations per cell for the transforms and about 26 for the whole update, against 512
// for the dense inverse (64 and the folds by parity classes): FP64 is bound by its pipe (626 G
// operations/s, 24 Gcell/s; measured 19.5 at 256^3), FP32 by HBM (12 bytes per cell) and the
// trips through shared memory (320 Gcell/s, 0.57 of the measured copy, Jacobi).
//
// A CTA holds NB boxes in shared memory.  Five stages, one thread per line of cells, a line in
// registers: x rows (gather the right-hand side from global memory, transform), y lines,
// z lines (transform, divide, transform back), y lines back, x rows back with the update
// v = (1 - omega) u + omega Ahat r written to the grid.  Adjacent threads take adjacent boxes'
// rows in the x stages (contiguous grid rows), adjacent cells in the y and z stages; the plane
// and box strides in shared memory are padded so that each of those is free of bank conflicts
// for the power-of-two boxes.  FP64 CTAs have 128 threads: 96^3 8^3 Gauss-Seidel, whose passes
// have few boxes per SM, 54 us per sweep against 71 with 256; FP32 256: 52 against 61, 256^3.
//
// Taken for boxes whose sides are at most 16: a side of N costs N/2 + 1 operations per cell and
// transform, and a line of N cells has to fit a thread's registers.
#include <algorithm>
#include <cmath>
#include <new>
#include <type_traits>
#include <vector>

#include "box.cuh"

namespace {

constexpr int kMaxSide = 16;
constexpr int kHalf = kMaxSide / 2;
constexpr int kThreads = 256;

// Launch arguments.  e / o: the even / odd rows of each axis' S on its first ceil(N/2) /
// floor(N/2) columns, row stride kHalf; the kernel reads them as constant-bank operands.
template <typename T>
struct SineArgs {
    T e[3][kHalf * kHalf], o[3][kHalf * kHalf];
    int bx, by, bz, nx, ny, nz;
    int threads; // threads per CTA
    int nb;      // boxes per CTA (a power of two)
    int lognb;
    int P, Q;    // shared-memory strides of a box plane and of a box (elements)
    int mby, mbx, mbxz, mbxy;  // 2^20 / d rounded up: t / d = (t * m) >> 20 for t < 8192
    T ax, ay, az, om1;
};

// omega / lambda of a mode over the squared norms of its basis rows: FP32 as a sum of two, whose
// rounding would otherwise stay in that mode sweep after sweep (2^3 to 16x4x2 boxes: mean error 1.15
// times the dense FP32 inverse's without the second part, 1.07 with it).
template <typename T>
struct ModeScale {
    using type = T;
};
template <>
struct ModeScale<float> {
    using type = float2;
};
__device__ __forceinline__ double times(double v, double s) { return v * s; }
__device__ __forceinline__ float times(float v, float2 s) { return fma(v, s.x, v * s.y); }

struct SineState {
    void* ilam = nullptr;  // ModeScale per mode, p fastest
    SineArgs<double> a64;
    SineArgs<float> a32;
    size_t smem = 0;
    const void* kernel = nullptr;
};

// Vector of the element type for rows of N: 16 bytes where N is a whole number of them, else 8.
template <typename T, int N>
struct RowVec {
    using type = T;
};
template <int N>
struct RowVec<double, N> {
    using type = std::conditional_t<N % 2 == 0, double2, double>;
};
template <int N>
struct RowVec<float, N> {
    using type = std::conditional_t<N % 4 == 0, float4, std::conditional_t<N % 2 == 0, float2, float>>;
};
constexpr int row_vec(int es, int n)  // its length in elements
{
    return n % (16 / es) == 0 ? 16 / es : es == 4 && n % 2 == 0 ? 2 : 1;
}

// N consecutive values of global or shared memory.  Every caller's offset is a multiple of the
// vector: global rows start at multiples of N (the box side divides nx) from a 16-byte aligned
// array, and the shared-memory strides are whole vectors.
template <typename T, int N>
__device__ __forceinline__ void ld_line(T (&v)[N], const T* p)
{
    using V = typename RowVec<T, N>::type;
    constexpr int PER = row_vec(sizeof(T), N);
#pragma unroll
    for (int m = 0; m < N / PER; ++m)
        reinterpret_cast<V*>(v)[m] = reinterpret_cast<const V*>(p)[m];
}

template <typename T, int N>
__device__ __forceinline__ void st_line(T* p, const T (&v)[N])
{
    using V = typename RowVec<T, N>::type;
    constexpr int PER = row_vec(sizeof(T), N);
#pragma unroll
    for (int m = 0; m < N / PER; ++m)
        reinterpret_cast<V*>(p)[m] = reinterpret_cast<const V*>(v)[m];
}

// v <- S v / kappa (N = 2, 4, 8: kappa scales one sine of the basis to 1, which turns its
// products into sums; otherwise 1 / kappa is FP32's best_scale, or 1).  S is symmetric, so this is the
// transform back, too.
// Operations per cell: 1, 2, 3.75 for N = 2, 4, 8, and N/2 + 1 by the two half-size products.
template <typename T, int N>
__device__ __forceinline__ void dst(T (&v)[N], const T* e, const T* o)
{
    if constexpr (N > 1) {
        constexpr int H = (N + 1) / 2, L = N / 2;
        T s[H], d[L];
#pragma unroll
        for (int i = 0; i < L; ++i) {
            s[i] = v[i] + v[N - 1 - i];
            d[i] = v[i] - v[N - 1 - i];
        }
        if constexpr (N % 2)
            s[H - 1] = v[H - 1];
        if constexpr (N == 2) {  // sin(60), sin(120) scaled to 1
            v[0] = s[0];
            v[1] = d[0];
        } else if constexpr (N == 4) {  // sin(36) scaled to 1, e[0] = sin(72)
            v[0] = fma(e[0], s[1], s[0]);
            v[2] = fma(e[0], s[0], -s[1]);
            v[1] = fma(e[0], d[0], d[1]);
            v[3] = fma(-e[0], d[1], d[0]);
        } else if constexpr (N == 8) {
            // sin(60) scaled to 1, e[0], e[1] = sin(20), sin(40); sin(80) = sin(20) + sin(40)
            const T sa = s[0] + s[3], sb = s[1] + s[3], sc = s[0] - s[1];
            v[0] = fma(e[0], sa, fma(e[1], sb, s[2]));
            v[2] = (s[0] - s[3]) + s[1];
            v[4] = fma(e[0], sc, fma(e[1], sa, -s[2]));
            v[6] = fma(e[1], sc, fma(-e[0], sb, s[2]));
            const T da = d[1] + d[3], db = d[0] + d[1], dc = d[0] - d[3];
            v[1] = fma(e[0], da, fma(e[1], db, d[2]));
            v[3] = fma(e[0], db, fma(e[1], dc, -d[2]));
            v[5] = (d[0] - d[1]) + d[3];
            v[7] = fma(e[0], dc, fma(-e[1], da, d[2]));
        } else {
#pragma unroll
            for (int q = 0; q < H; ++q) {
                T acc = e[q * kHalf] * s[0];
#pragma unroll
                for (int i = 1; i < H; ++i)
                    acc = fma(e[q * kHalf + i], s[i], acc);
                v[2 * q] = acc;
            }
#pragma unroll
            for (int q = 0; q < L; ++q) {
                T acc = o[q * kHalf] * d[0];
#pragma unroll
                for (int i = 1; i < L; ++i)
                    acc = fma(o[q * kHalf + i], d[i], acc);
                v[2 * q + 1] = acc;
            }
        }
    }
}

__device__ __forceinline__ int div_m(int t, int m) { return (int)(((unsigned)t * (unsigned)m) >> 20); }

// f(integral_constant<N>) for the runtime side n <= MAXN
template <int N>
struct Side {
    static constexpr int value = N;
};
template <int MAXN, int FIX, typename F>
__device__ __forceinline__ void with_side(int n, F&& f)
{
    if constexpr (FIX > 0) {
        f(Side<FIX>());
    } else {
        switch (n) {
        case 1: f(Side<1>()); break;
        case 2: f(Side<2>()); break;
        case 3: f(Side<3>()); break;
        case 4: f(Side<4>()); break;
        case 5: if constexpr (MAXN >= 5) f(Side<5>()); break;
        case 6: if constexpr (MAXN >= 6) f(Side<6>()); break;
        case 7: if constexpr (MAXN >= 7) f(Side<7>()); break;
        case 8: if constexpr (MAXN >= 8) f(Side<8>()); break;
        case 9: if constexpr (MAXN >= 9) f(Side<9>()); break;
        case 10: if constexpr (MAXN >= 10) f(Side<10>()); break;
        case 11: if constexpr (MAXN >= 11) f(Side<11>()); break;
        case 12: if constexpr (MAXN >= 12) f(Side<12>()); break;
        case 13: if constexpr (MAXN >= 13) f(Side<13>()); break;
        case 14: if constexpr (MAXN >= 14) f(Side<14>()); break;
        case 15: if constexpr (MAXN >= 15) f(Side<15>()); break;
        default: if constexpr (MAXN >= 16) f(Side<16>()); break;
        }
    }
}

// CUBE > 0: CUBE^3 boxes (all divisions by constants); 0: any sides up to MAXN.
template <typename T, int MAXN, int CUBE>
__global__ void __launch_bounds__(kThreads) box_sine_kernel(const T* u, T* uout,
                                                            const T* __restrict__ b,
                                                            const long long* __restrict__ rows,
                                                            long long M,
                                                            const typename ModeScale<T>::type* __restrict__ ilam,
                                                            const __grid_constant__ SineArgs<T> a)
{
    extern __shared__ __align__(16) unsigned char box_smem[];
    T* sm = reinterpret_cast<T*>(box_smem);
    pdl_wait_trigger();
    const int bx = CUBE ? CUBE : a.bx, by = CUBE ? CUBE : a.by, bz = CUBE ? CUBE : a.bz;
    const int nx = a.nx, ny = a.ny, nz = a.nz, P = a.P, Q = a.Q;
    const long long plane = (long long)nx * ny;
    const long long q0 = (long long)blockIdx.x << a.lognb;
    const int have = (int)(M - q0 < a.nb ? M - q0 : a.nb);  // boxes of this CTA
    const int bxy = bx * by, bxz = bx * bz;
    const int nrow = by * bz << a.lognb;
    auto row_of = [&](int t, int* box, int* ly, int* lz) {
        const int r = t >> a.lognb;
        *box = t & (a.nb - 1);
        *lz = CUBE ? r / (CUBE ? CUBE : 1) : div_m(r, a.mby);
        *ly = r - *lz * by;
    };

    // x rows: gather and transform
    for (int t = threadIdx.x; t < nrow; t += blockDim.x) {
        int box, ly, lz;
        row_of(t, &box, &ly, &lz);
        if (box >= have)
            continue;
        const long long pk = __ldg(rows + q0 + box);
        const int i0 = (int)(pk & 0x1FFFFF) * bx;
        const int j = (int)((pk >> 21) & 0x1FFFFF) * by + ly;
        const int k = (int)(pk >> 42) * bz + lz;
        const long long cell = i0 + (long long)nx * j + plane * k;
        with_side<MAXN, CUBE>(bx, [&](auto side) {
            constexpr int N = decltype(side)::value;
            T v[N], w[N];
            ld_line<T, N>(v, b + cell);
            auto add = [&](T c, const T* p) {
                ld_line<T, N>(w, p);
#pragma unroll
                for (int m = 0; m < N; ++m)
                    v[m] = fma(c, w[m], v[m]);
            };
            // a warp holds rows of every ly: the two y faces share one add (by > 1)
            if (by > 1) {
                if ((ly == 0 && j > 0) || (ly == by - 1 && j + 1 < ny))
                    add(a.ay, u + cell + (ly == 0 ? -nx : nx));
            } else {
                if (j > 0)
                    add(a.ay, u + cell - nx);
                if (j + 1 < ny)
                    add(a.ay, u + cell + nx);
            }
            if (lz == 0 && k > 0)
                add(a.az, u + cell - plane);
            if (lz == bz - 1 && k + 1 < nz)
                add(a.az, u + cell + plane);
            if (i0 > 0)
                v[0] = fma(a.ax, u[cell - 1], v[0]);
            if (i0 + N < nx)
                v[N - 1] = fma(a.ax, u[cell + N], v[N - 1]);
            dst<T, N>(v, a.e[0], a.o[0]);
            st_line<T, N>(sm + box * Q + lz * P + ly * N, v);
        });
    }
    __syncthreads();

    // y lines: thread t -> (box, lz, lx), lx fastest
    const int nyl = have * bxz, nzl = have * bxy;
    auto y_line = [&](int t) {
        const int box = CUBE ? t / (CUBE ? CUBE * CUBE : 1) : div_m(t, a.mbxz);
        const int c = t - box * bxz;
        const int lz = CUBE ? c / (CUBE ? CUBE : 1) : div_m(c, a.mbx);
        return sm + box * Q + lz * P + (c - lz * bx);
    };
    if (by > 1) {
        for (int t = threadIdx.x; t < nyl; t += blockDim.x) {
            T* p = y_line(t);
            with_side<MAXN, CUBE>(by, [&](auto side) {
                constexpr int N = decltype(side)::value;
                T v[N];
#pragma unroll
                for (int m = 0; m < N; ++m)
                    v[m] = p[m * bx];
                dst<T, N>(v, a.e[1], a.o[1]);
#pragma unroll
                for (int m = 0; m < N; ++m)
                    p[m * bx] = v[m];
            });
        }
        __syncthreads();
    }
    // z lines there and back, with omega / lambda in between
    for (int t = threadIdx.x; t < nzl; t += blockDim.x) {
        const int box = CUBE ? t / (CUBE ? CUBE * CUBE : 1) : div_m(t, a.mbxy);
        const int c = t - box * bxy;
        T* p = sm + box * Q + c;
        with_side<MAXN, CUBE>(bz, [&](auto side) {
            constexpr int N = decltype(side)::value;
            T v[N];
#pragma unroll
            for (int m = 0; m < N; ++m)
                v[m] = p[m * P];
            dst<T, N>(v, a.e[2], a.o[2]);
#pragma unroll
            for (int m = 0; m < N; ++m)
                v[m] = times(v[m], __ldg(ilam + m * bxy + c));
            dst<T, N>(v, a.e[2], a.o[2]);
#pragma unroll
            for (int m = 0; m < N; ++m)
                p[m * P] = v[m];
        });
    }
    __syncthreads();
    if (by > 1) {
        for (int t = threadIdx.x; t < nyl; t += blockDim.x) {
            T* p = y_line(t);
            with_side<MAXN, CUBE>(by, [&](auto side) {
                constexpr int N = decltype(side)::value;
                T v[N];
#pragma unroll
                for (int m = 0; m < N; ++m)
                    v[m] = p[m * bx];
                dst<T, N>(v, a.e[1], a.o[1]);
#pragma unroll
                for (int m = 0; m < N; ++m)
                    p[m * bx] = v[m];
            });
        }
        __syncthreads();
    }
    // x rows back, update
    for (int t = threadIdx.x; t < nrow; t += blockDim.x) {
        int box, ly, lz;
        row_of(t, &box, &ly, &lz);
        if (box >= have)
            continue;
        const long long pk = __ldg(rows + q0 + box);
        const long long cell = (pk & 0x1FFFFF) * bx +
                               (long long)nx * (((pk >> 21) & 0x1FFFFF) * by + ly) +
                               plane * ((pk >> 42) * bz + lz);
        with_side<MAXN, CUBE>(bx, [&](auto side) {
            constexpr int N = decltype(side)::value;
            T v[N], w[N];
            ld_line<T, N>(w, u + cell);
            ld_line<T, N>(v, sm + box * Q + lz * P + ly * N);
            dst<T, N>(v, a.e[0], a.o[0]);
#pragma unroll
            for (int m = 0; m < N; ++m)
                v[m] = fma(a.om1, w[m], v[m]);
            st_line<T, N>(uout + cell, v);
        });
    }
}

template <typename T>
const void* sine_kernel_for(int bx, int by, int bz)
{
    const int m = bx > by ? (bx > bz ? bx : bz) : (by > bz ? by : bz);
    if (bx == by && by == bz) {
        if (m == 8)
            return (const void*)box_sine_kernel<T, 8, 8>;
        if (m == 4)
            return (const void*)box_sine_kernel<T, 4, 4>;
        if (m == 2)
            return (const void*)box_sine_kernel<T, 4, 2>;
    }
    if (m <= 4)
        return (const void*)box_sine_kernel<T, 4, 0>;
    if (m <= 8)
        return (const void*)box_sine_kernel<T, 8, 0>;
    return (const void*)box_sine_kernel<T, 16, 0>;
}

// Shared-memory wavefronts of one warp's access when lane l touches `bytes` bytes at word
// address w(l): phases of 32 banks, counting the busiest bank.
template <typename F>
int wavefronts(int bytes, F&& word)
{
    const int words = bytes / 4, lanes = 32 / words;  // lanes per phase
    int total = 0;
    for (int p = 0; p < 32; p += lanes) {
        int bank[32] = {0}, worst = 1;
        for (int l = p; l < p + lanes; ++l)
            for (int q = 0; q < words; ++q) {
                const int n = ++bank[(word(l) + q) & 31];
                worst = n > worst ? n : worst;
            }
        total += worst;
    }
    return total;
}

// Plane and box strides (elements) with the fewest wavefronts over the x-row, y-line and z-line
// accesses of a warp; both multiples of the vector that moves the rows.
void pick_strides(int es, int bx, int by, int bz, int nb, int* P, int* Q)
{
    const int step = row_vec(es, bx), w = es / 4;
    const int rowbytes = step * es;
    int best = 1 << 30;
    for (int p = 0; p <= 16; p += step)
        for (int q = 0; q <= 16; q += step) {
            const int PP = bx * by + p, QQ = PP * bz + q;
            int cost = 2 * wavefronts(rowbytes, [&](int l) {
                const int r = l / nb;  // nb is a power of two
                return w * ((l % nb) * QQ + (r / by) * PP + (r % by) * bx);
            }) * (bx * es / rowbytes);
            cost += 4 * by * wavefronts(es, [&](int l) {
                const int box = l / (bx * bz), c = l % (bx * bz);
                return w * (box * QQ + c / bx * PP + c % bx);
            });
            cost += 2 * bz * wavefronts(es, [&](int l) {
                return w * (l / (bx * by) * QQ + l % (bx * by));
            });
            cost = cost * 64 + p + q;  // the smaller padding among equals
            if (cost < best) {
                best = cost;
                *P = PP;
                *Q = QQ;
            }
        }
}

// The kernel's constants are formed in extended precision and rounded once: formed in double they
// carry a few roundings each, 1e-15 in the smallest eigenvalues by 2 - 2 cos, and that, not the
// kernel's arithmetic, was most of the error (2-norm after 5 Jacobi sweeps, a = (0.5, 1, 2): 8^3
// boxes 2.7e-15, now 3.8e-16, by the dense inverse 1.4e-15; 2^3 1.3e-15, 2.0e-16, 8.2e-16).

// Entry of the orthonormal DST-I basis of n cells whose product of indexes (from 1) is q.
long double basis(int n, int q)
{
    constexpr long double pi = 3.14159265358979323846264338327950288L;
    return std::sqrt(2.0L / (n + 1)) * std::sin(q * pi / (n + 1));
}

// An axis of the basis as the kernel has it: scaled and rounded.  The squared norms of its rows, as
// they are, go into the modes' scale: norm of row 0, and norm / (norm of row p) - 1.
struct Axis {
    long double norm = 1.0L;
    std::vector<double> off;
};

// Scale in [1, 2) at which the sines of an axis lose least to rounding to FP32: every product of the
// basis takes it, and the modes' scale takes it out.
double best_scale(int n)
{
    std::vector<double> sine;
    for (int q = 1; 2 * q <= n + 1; ++q)
        sine.push_back((double)basis(n, q));
    double best = 1.0, least = 1.0;
    for (int j = 0; j < 2048; ++j) {
        const double scale = 1.0 + j / 2048.0;
        double worst = 0.0;
        for (size_t q = 0; q < sine.size() && worst < least; ++q) {
            const double x = scale * sine[q];
            worst = std::max(worst, std::fabs((double)(float)x - x) / x);
        }
        if (worst < least)
            least = worst, best = scale;
    }
    return best;
}

// e / o of one axis of n cells (see dst for n = 2, 4, 8).
template <typename T>
Axis fill_axis(int n, T* e, T* o)
{
    Axis ax;
    ax.off.assign(n, 0.0);
    auto sq = [](long double v) { return v * v; };
    if (n == 2) {
        ax.norm = 2.0L;
    } else if (n == 4) {
        e[0] = (T)(basis(4, 2) / basis(4, 1));
        ax.norm = 2.0L * (1.0L + sq(e[0]));
    } else if (n == 8) {
        e[0] = (T)(basis(8, 1) / basis(8, 3));
        e[1] = (T)(basis(8, 2) / basis(8, 3));
        ax.norm = 2.0L * (sq(e[0]) + sq(e[1]) + sq((long double)e[0] + e[1]) + 1.0L);
        ax.off[2] = ax.off[5] = (double)(ax.norm / 6.0L - 1.0L);  // the rows of sin(60) and 0
    } else if (n > 1) {
        const int m = n + 1;
        const double scale = sizeof(T) == 4 ? best_scale(n) : 1.0;
        std::vector<T> sine(2 * m);  // basis of every product of indexes, mod its period
        for (int q = 1; 2 * q <= m; ++q) {
            sine[q] = sine[m - q] = (T)(scale * basis(n, q));
            sine[m + q] = sine[2 * m - q] = -sine[q];
        }
        std::vector<long double> norm(n, 0.0L);
        for (int q = 0; q < n; ++q)
            for (int i = 0; i < (q % 2 ? n / 2 : (n + 1) / 2); ++i) {
                const T v = sine[(q + 1) * (i + 1) % (2 * m)];
                (q % 2 ? o : e)[(q / 2) * kHalf + i] = v;
                norm[q] += sq(v) * (2 * i + 1 == n ? 1 : 2);  // once for the middle cell
            }
        ax.norm = norm[0];
        for (int q = 0; q < n; ++q)
            ax.off[q] = (double)(norm[0] / norm[q] - 1.0L);
    }
    return ax;
}

template <typename T>
void fill_args(SineArgs<T>& a, const brs_params& p, double omega, Axis (&axes)[3])
{
    const int n[3] = {p.bx, p.by, p.bz};
    for (int d = 0; d < 3; ++d)
        axes[d] = fill_axis(n[d], a.e[d], a.o[d]);
    a.bx = p.bx, a.by = p.by, a.bz = p.bz;
    a.nx = p.nx, a.ny = p.ny, a.nz = p.nz;
    // Threads and boxes per CTA: boxes until the stage with the fewest lines has one per thread
    // (longer lines mean fewer of them), at most 32 KB of shared memory.
    const int rows = p.by * p.bz, yl = p.bx * p.bz, zl = p.bx * p.by;
    const int fewest = rows < yl ? (rows < zl ? rows : zl) : (yl < zl ? yl : zl);
    a.threads = sizeof(T) == 8 ? kThreads / 2 : kThreads;
    a.nb = 1, a.lognb = 0;
    while (a.nb * 2 * fewest <= a.threads &&
           (size_t)a.nb * 2 * (p.bx * p.by + 2) * p.bz * sizeof(T) <= 32u * 1024u)
        a.nb *= 2, ++a.lognb;
    pick_strides(sizeof(T), p.bx, p.by, p.bz, a.nb, &a.P, &a.Q);
    auto magic = [](int d) { return (1 << 20) / d + 1; };
    a.mby = magic(p.by), a.mbx = magic(p.bx), a.mbxz = magic(yl), a.mbxy = magic(zl);
    a.ax = (T)p.ax, a.ay = (T)p.ay, a.az = (T)p.az;
    a.om1 = (T)(1.0 - omega);
}

// A value of extended precision as the sum of two doubles.
struct Two {
    double hi, lo;
    explicit Two(long double v) : hi((double)v), lo((double)(v - hi)) {}
};

// s / (a + b) to a rounding of the last place, in double arithmetic (extended precision runs in
// software on Arm).
double quotient(const Two& s, const Two& a, const Two& b)
{
    const double h = a.hi + b.hi, t = h - a.hi;
    const double l = ((a.hi - (h - t)) + (b.hi - t)) + (a.lo + b.lo);  // a + b = h + l
    const double q = s.hi / h;
    return q + (std::fma(-q, h, s.hi) + (s.lo - q * l)) / h;
}

// Eigenvalues 2 - 2 cos((q+1) pi / (n+1)) = 4 sin^2 of half the angle, times a.
std::vector<long double> eigenvalues(int n, double a)
{
    std::vector<long double> v(n);
    for (int q = 0; q < n; ++q) {
        const long double sine = basis(2 * n + 1, q + 1);
        v[q] = a * 4.0L * (n + 1) * sine * sine;
    }
    return v;
}

void put(std::vector<double>& v, double s) { v.push_back(s); }
void put(std::vector<float2>& v, double s)
{
    v.push_back(make_float2((float)s, (float)(s - (float)s)));
}

template <typename T>
int upload_ilam(void** dst, const brs_params& p, double omega, const Axis (&axes)[3])
{
    const std::vector<long double> x = eigenvalues(p.bx, p.ax), y = eigenvalues(p.by, p.ay),
                                   z = eigenvalues(p.bz, p.az);
    const std::vector<Two> x2(x.begin(), x.end());
    const Two scale(omega / (axes[0].norm * axes[1].norm * axes[2].norm));
    std::vector<typename ModeScale<T>::type> v;
    for (int r = 0; r < p.bz; ++r)
        for (int q = 0; q < p.by; ++q) {
            const Two yz(y[q] + z[r]);
            const double off = axes[1].off[q] + axes[2].off[r];
            for (int i = 0; i < p.bx; ++i) {
                const double s = quotient(scale, x2[i], yz);
                put(v, std::fma(s, axes[0].off[i] + off, s));
            }
        }
    const size_t bytes = v.size() * sizeof(v[0]);
    cudaError_t e = cudaMalloc(dst, bytes);
    if (e == cudaSuccess)
        e = cudaMemcpy(*dst, v.data(), bytes, cudaMemcpyHostToDevice);
    return brs_cuda_status(e);
}

template <typename T>
int launch(const SineState* S, const SineArgs<T>& a, const void* u, void* uout, const void* b,
           const long long* rows, long long M, cudaStream_t s)
{
    const T* up = static_cast<const T*>(u);
    T* op = static_cast<T*>(uout);
    const T* bp = static_cast<const T*>(b);
    const void* il = S->ilam;
    void* args[] = {&up, &op, &bp, (void*)&rows, &M, (void*)&il, (void*)&a};
    const long long ctas = (M + a.nb - 1) >> a.lognb;
    return brs_cuda_status(launch_pdl_c(S->kernel, dim3((unsigned)ctas), dim3(a.threads), S->smem,
                                        s, args));
}

}  // namespace

bool box_sine_takes(const brs_params& p)
{
    return p.bx <= kMaxSide && p.by <= kMaxSide && p.bz <= kMaxSide;
}

int box_sine_setup(const brs_params& p, double omega, void** out)
{
    SineState* S = new (std::nothrow) SineState();
    if (!S)
        return BRS_ERR_NOMEM;
    *out = S;
    int rc;
    int nb, Q;
    Axis axes[3];
    if (p.dtype == BRS_F64) {
        fill_args(S->a64, p, omega, axes);
        rc = upload_ilam<double>(&S->ilam, p, omega, axes);
        S->kernel = sine_kernel_for<double>(p.bx, p.by, p.bz);
        nb = S->a64.nb, Q = S->a64.Q;
        S->smem = (size_t)nb * Q * 8;
    } else {
        fill_args(S->a32, p, omega, axes);
        rc = upload_ilam<float>(&S->ilam, p, omega, axes);
        S->kernel = sine_kernel_for<float>(p.bx, p.by, p.bz);
        nb = S->a32.nb, Q = S->a32.Q;
        S->smem = (size_t)nb * Q * 4;
    }
    if (rc == BRS_OK && S->smem > 48u * 1024u) {
        cudaFuncAttributes fa{};
        cudaError_t e = cudaFuncGetAttributes(&fa, S->kernel);
        if (e == cudaSuccess && (size_t)fa.maxDynamicSharedSizeBytes < S->smem)
            e = cudaFuncSetAttribute(S->kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)S->smem);
        rc = brs_cuda_status(e);
    }
    return rc;
}

void box_sine_teardown(void* state)
{
    SineState* S = static_cast<SineState*>(state);
    if (!S)
        return;
    if (S->ilam)
        cudaFree(S->ilam);
    delete S;
}

int box_sine_pass(const void* state, int dtype, const void* u, void* uout, const void* b,
                  const long long* rows, long long M, cudaStream_t s)
{
    if (M == 0)
        return BRS_OK;
    const SineState* S = static_cast<const SineState*>(state);
    return dtype == BRS_F64 ? launch(S, S->a64, u, uout, b, rows, M, s)
                            : launch(S, S->a32, u, uout, b, rows, M, s);
}
