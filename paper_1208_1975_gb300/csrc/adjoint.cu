// Reverse-mode sweep of damped x-line block Jacobi (the transpose of Eq. blockiteration2).
//
// A forward sweep is u_{k+1} = u_k + omega z_k with z_k = M^{-1}(b - A u_k), i.e.
// u_{k+1} = G u_k + omega M^{-1} b with G = I - omega M^{-1} A.  A and the line block
// diagonal M are symmetric, so for a loss L(u_K) with lambda_{k+1} = dL/du_{k+1}:
//   mu_k       = M^{-1} lambda_{k+1}
//   lambda_k   = G^T lambda_{k+1} = lambda_{k+1} - omega A mu_k
//   dL/db     += omega mu_k
//   dL/da_d   += -omega mu_k . ( (dM/da_d) z_k + (dA/da_d) u_k )
// with dA/da_d = T_d (second difference along axis d, zero outside), and for x-line
// blocks dM/dax = Tx, dM/day = dM/daz = 2 I.
// One call performs these updates for one sweep; the caller supplies u_k (checkpointed
// or recomputed) and runs the calls from the last sweep to the first.
// The gradient terms only need z_k through x_k = u_k + z_k = M^{-1}(b + N u_k), the
// undamped line-Jacobi iterate (A = M - N), which the x-line sweep kernel produces in one
// pass: Tx (z + u) = Tx x, 2 z + Ty u = 2 x - Sy u, 2 z + Tz u = 2 x - Sz u, with S_d the
// sum of the two neighbours along d (T_d = 2 I - S_d).
#include "brs_internal.cuh"
#include "line_impl.cuh"
#include "line_tile.cuh"

namespace {

constexpr int kThreads = 256;

// out = M_line^{-1} in, one line group per (j,k) at a time; in-place safe (a group reads
// its whole line, and its next one, before writing it).
template <typename T, int E, int G>
__global__ void __launch_bounds__(kThreads) line_minv_kernel(const T* in, T* out,
                                                             const T* __restrict__ tab, int nx,
                                                             int ny, int nz, bool vec)
{
    // Grid-stride over lines, the next line's cells loaded before the current one is solved
    // (the load latency overlaps the solve).  Every group of a warp runs the same number of
    // iterations, because the solve shuffles across the warp; groups past the last line
    // solve zeros.
    const int groups = blockDim.x / G;
    const long long nlines = (long long)ny * nz;
    const long long stride = (long long)gridDim.x * groups;
    const int lane = threadIdx.x % G;
    const long long warp_line0 = (long long)blockIdx.x * groups + (threadIdx.x & ~31) / G;
    const long long iters = warp_line0 < nlines ? (nlines - warp_line0 + stride - 1) / stride : 0;
    brs::LineTables<T, E, G> tb;
    tb.load(tab, lane);
    constexpr int NP = G * E;
    constexpr int LG = brs::Log2<G>::value;
    const T* ptab = tab + 3 * NP + 2 * LG * G;
    // VEC: full lines (nx = E G) with 16-byte aligned rows and E a whole number of 16-byte
    // vectors: each lane moves its E cells as vectors of the element type
    using V = typename brs::Vec16<T>::type;
    constexpr int NV = (int)(E * sizeof(T) / 16);
    constexpr bool CAN_VEC = (E * sizeof(T)) % 16 == 0;
    auto load = [&](long long line, T (&r)[E]) {
        const bool active = line < nlines;
        const size_t base = (size_t)(active ? line : 0) * nx;
        if (CAN_VEC && vec) {
            const V* src = reinterpret_cast<const V*>(in + base + lane * E);
#pragma unroll
            for (int m = 0; m < NV; ++m)
                reinterpret_cast<V*>(r)[m] = active ? src[m] : V{};
        } else {
#pragma unroll
            for (int q = 0; q < E; ++q) {
                const int x = lane * E + q;
                r[q] = (active && x < nx) ? in[base + x] : T(0);
            }
        }
    };
    long long line = (long long)blockIdx.x * groups + threadIdx.x / G;
    T nxt[E];
    load(line, nxt);
    for (long long it = 0; it < iters; ++it, line += stride) {
        T r[E];
#pragma unroll
        for (int q = 0; q < E; ++q)
            r[q] = nxt[q];
        if (it + 1 < iters)
            load(line + stride, nxt);
        brs::line_solve<T, E, G>(r, tb, lane);
#pragma unroll
        for (int q = 0; q < E; ++q)
            r[q] = ptab[lane * E + q] * r[q];
        if (line < nlines) {
            const size_t base = (size_t)line * nx;
            if (CAN_VEC && vec) {
                V* dst = reinterpret_cast<V*>(out + base + lane * E);
#pragma unroll
                for (int m = 0; m < NV; ++m)
                    dst[m] = reinterpret_cast<const V*>(r)[m];
            } else {
#pragma unroll
                for (int q = 0; q < E; ++q) {
                    const int x = lane * E + q;
                    if (x < nx)
                        out[base + x] = r[q];
                }
            }
        }
    }
}

// Four consecutive cells of a row (rem = cells left in the row); VEC: 16-byte vectors.
template <typename T>
__device__ __forceinline__ void ld4(T (&v)[4], const T* p, int rem, bool vec)
{
    if (vec) {
        if constexpr (sizeof(T) == 4) {
            const float4 f = *reinterpret_cast<const float4*>(p);
            v[0] = f.x, v[1] = f.y, v[2] = f.z, v[3] = f.w;
        } else {
            const double2 f0 = reinterpret_cast<const double2*>(p)[0];
            const double2 f1 = reinterpret_cast<const double2*>(p)[1];
            v[0] = f0.x, v[1] = f0.y, v[2] = f1.x, v[3] = f1.y;
        }
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
            v[q] = q < rem ? p[q] : T(0);
    }
}

template <typename T>
__device__ __forceinline__ void st4(T* p, const T (&v)[4], int rem, bool vec)
{
    if (vec) {
        if constexpr (sizeof(T) == 4) {
            *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
        } else {
            reinterpret_cast<double2*>(p)[0] = make_double2(v[0], v[1]);
            reinterpret_cast<double2*>(p)[1] = make_double2(v[2], v[3]);
        }
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (q < rem)
                p[q] = v[q];
    }
}

// FP32 form: lambda <- lambda - omega A mu; gb += omega mu; per-CTA partial sums of the three
// coefficient-gradient terms mu.(Tx x), mu.(2x - Sy u), mu.(2x - Sz u) with x = M^{-1}(b + N u_k),
// u = u_k.  A z-march: a warp owns 128 cells of row j (four per lane)
// over a chunk of kMarchKC planes, keeps mu and u of planes k-1, k, k+1 in registers, and
// loads the next plane's inputs before computing the current one (more loads in flight per
// warp, and the z neighbours are not loaded twice).  Items (j, x-chunk, z-chunk) go to warps
// in a fixed grid-stride order, so the partial sums are reproducible.
constexpr int kMarchKC = 16;

template <int N>
__device__ __forceinline__ void zero4(float (&v)[N])
{
#pragma unroll
    for (int q = 0; q < N; ++q)
        v[q] = 0.0f;
}

struct MarchIn {  // one plane's loads for the lanes' four cells
    float mup[4], up[4], muym[4], muyp[4], uym[4], uyp[4], xc[4], lam[4], gb[4];
    float mul, mur, xl, xr;
};

__global__ void __launch_bounds__(kThreads, 2) adjoint_update_march(
    float* __restrict__ lam, const float* __restrict__ mu, const float* __restrict__ x,
    const float* __restrict__ u, float* __restrict__ gb, int nx, int ny, int nz, double ax,
    double ay, double az, double omega, double* partials, bool vec)
{
    const long long plane = (long long)nx * ny;
    const int ncx = (nx + 127) / 128, nkc = (nz + kMarchKC - 1) / kMarchKC;
    const long long nitems = (long long)ny * ncx * nkc;
    const int lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
    const float cx = (float)ax, cy = (float)ay, cz = (float)az;
    const float dg = (float)(2.0 * (ax + ay + az)), om = (float)omega;
    double g0 = 0.0, g1 = 0.0, g2 = 0.0;
    for (long long it = (long long)blockIdx.x * wpb + (threadIdx.x >> 5); it < nitems;
         it += (long long)gridDim.x * wpb) {
        const int kc = (int)(it % nkc);
        const long long rest = it / nkc;
        const int xc = (int)(rest % ncx), j = (int)(rest / ncx);
        const int i0 = xc * 128 + 4 * lane, rem = nx - i0;
        const bool act = rem > 0;
        const int k0 = kc * kMarchKC, k1 = min(nz, k0 + kMarchKC);
        const long long row = (long long)j * nx + i0;
        auto at = [&](const float* a, int k) { return a + (long long)k * plane + row; };
        // plane k's loads (zeros outside the grid or for lanes past the row)
        auto load = [&](MarchIn& P, int k) {
            zero4(P.mup), zero4(P.up), zero4(P.muym), zero4(P.muyp), zero4(P.uym), zero4(P.uyp);
            zero4(P.xc), zero4(P.lam), zero4(P.gb);
            P.mul = P.mur = P.xl = P.xr = 0.0f;
            if (!act)
                return;
            if (k + 1 < nz) {
                ld4(P.mup, at(mu, k + 1), rem, vec);
                ld4(P.up, at(u, k + 1), rem, vec);
            }
            if (j > 0) {
                ld4(P.muym, at(mu, k) - nx, rem, vec);
                ld4(P.uym, at(u, k) - nx, rem, vec);
            }
            if (j + 1 < ny) {
                ld4(P.muyp, at(mu, k) + nx, rem, vec);
                ld4(P.uyp, at(u, k) + nx, rem, vec);
            }
            const float* px = at(x, k);
            const float* pm = at(mu, k);
            ld4(P.xc, px, rem, vec);
            ld4(P.lam, at(lam, k), rem, vec);
            ld4(P.gb, at(gb, k), rem, vec);
            if (i0 > 0) {
                P.mul = pm[-1];
                P.xl = px[-1];
            }
            if (rem > 4) {
                P.mur = pm[4];
                P.xr = px[4];
            }
        };
        float mum[4], muc[4], um[4], uc[4];
        zero4(mum), zero4(muc), zero4(um), zero4(uc);
        if (act) {
            if (k0 > 0) {
                ld4(mum, at(mu, k0 - 1), rem, vec);
                ld4(um, at(u, k0 - 1), rem, vec);
            }
            ld4(muc, at(mu, k0), rem, vec);
            ld4(uc, at(u, k0), rem, vec);
        }
        MarchIn nxt;
        load(nxt, k0);
        float h0 = 0.0f, h1 = 0.0f, h2 = 0.0f;
        for (int k = k0; k < k1; ++k) {
            const MarchIn cur = nxt;
            if (k + 1 < k1)
                load(nxt, k + 1);
            float lv[4], gv[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float mq = muc[q];
                const float sxm = (q == 0 ? cur.mul : muc[q - 1]) +
                                  (q == 3 ? cur.mur : (q + 1 < rem ? muc[q + 1] : 0.0f));
                const float sym = cur.muym[q] + cur.muyp[q], szm = mum[q] + cur.mup[q];
                const float Amu = dg * mq - cx * sxm - cy * sym - cz * szm;
                lv[q] = cur.lam[q] - om * Amu;
                gv[q] = cur.gb[q] + om * mq;
                const float x2 = 2.0f * cur.xc[q];
                const float sxx = (q == 0 ? cur.xl : cur.xc[q - 1]) +
                                  (q == 3 ? cur.xr : (q + 1 < rem ? cur.xc[q + 1] : 0.0f));
                if (q < rem) {
                    h0 = fmaf(mq, x2 - sxx, h0);
                    h1 = fmaf(mq, x2 - (cur.uym[q] + cur.uyp[q]), h1);
                    h2 = fmaf(mq, x2 - (um[q] + cur.up[q]), h2);
                }
            }
            if (act) {
                st4(lam + (long long)k * plane + row, lv, rem, vec);
                st4(gb + (long long)k * plane + row, gv, rem, vec);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                mum[q] = muc[q], muc[q] = cur.mup[q];
                um[q] = uc[q], uc[q] = cur.up[q];
            }
        }
        g0 += (double)h0;
        g1 += (double)h1;
        g2 += (double)h2;
    }
    __shared__ double red[3][kThreads / 32];
    double v[3] = {g0, g1, g2};
    for (int d = 0; d < 3; ++d) {
        for (int o = 16; o > 0; o >>= 1)
            v[d] += __shfl_down_sync(0xffffffffu, v[d], o);
        if ((threadIdx.x & 31) == 0)
            red[d][threadIdx.x >> 5] = v[d];
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        for (int d = 0; d < 3; ++d) {
            double w = threadIdx.x < kThreads / 32 ? red[d][threadIdx.x] : 0.0;
            for (int o = 16; o > 0; o >>= 1)
                w += __shfl_down_sync(0xffffffffu, w, o);
            if (threadIdx.x == 0)
                partials[3 * blockIdx.x + d] = w;
        }
    }
}

// FP64 form: lanes along x, a warp marches over kc planes of 32 cells of a row with mu of planes
// k-1, k, k+1 in registers and the next plane's inputs in flight.  Bound by the FP64 pipe, so it
// counts operations, 17 per cell instead of 22: mu . Tx x = (Tx mu) . x and mu . Sd u = (Sd mu) . u,
// so the sums need the neighbours of mu only, which A mu has: (2 mu - Sx mu) x, 2 mu x - (Sy mu) u,
// 2 mu x - (Sz mu) u, differences formed cell by cell as before.  (A mu = M mu - (ay Sy + az Sz) mu
// with M mu = lambda would save two more, lambda <- (1 - omega) lambda + omega (ay Sy + az Sz) mu, but
// it carries the block solve's rounding along: grad_u0 after 8 sweeps 1.2 to 1.6 times as far from
// extended precision as with A mu itself, 40x30x20 and 33x24x25, for 4 % of a call's time.)
// The last CTA to finish adds the CTAs' sums into grad_a in a fixed order (a counter in global
// memory, left at zero for the next call).  128^3, same box: 109 -> 82 us per call.
struct StepIn {
    double mup, muym, muyp, mul, mur, lam, x, u, gb;
};

__global__ void __launch_bounds__(kThreads, 3) adjoint_update_f64(
    double* __restrict__ lam, const double* __restrict__ mu, const double* __restrict__ x,
    const double* __restrict__ u, double* __restrict__ gb, int nx, int ny, int nz, int kc, double ax,
    double ay, double az, double omega, double* partials, unsigned* counter, double* grad_a)
{
    pdl_wait_trigger();
    const long long plane = (long long)nx * ny;
    const int ncx = (nx + 31) / 32, nkc = (nz + kc - 1) / kc;
    const long long nitems = (long long)ny * ncx * nkc;
    const int lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
    const double dg = 2.0 * (ax + ay + az);
    double g0 = 0.0, g1 = 0.0, g2 = 0.0;
    for (long long it = (long long)blockIdx.x * wpb + (threadIdx.x >> 5); it < nitems;
         it += (long long)gridDim.x * wpb) {
        const long long rest = it / ncx;
        const int i = (int)(it - rest * ncx) * 32 + lane;
        const int k0 = (int)(rest / ny) * kc, j = (int)(rest % ny);
        const int k1 = min(nz, k0 + kc);
        const bool on = i < nx;
        long long o = plane * k0 + (long long)j * nx + (on ? i : 0);
        auto load = [&](StepIn& v, long long q, int k) {
            v.mup = on && k + 1 < nz ? mu[q + plane] : 0.0;
            v.muym = on && j > 0 ? mu[q - nx] : 0.0;
            v.muyp = on && j + 1 < ny ? mu[q + nx] : 0.0;
            v.mul = on && i > 0 ? mu[q - 1] : 0.0;
            v.mur = on && i + 1 < nx ? mu[q + 1] : 0.0;
            v.lam = on ? lam[q] : 0.0;
            v.x = on ? x[q] : 0.0;
            v.u = on ? u[q] : 0.0;
            v.gb = on ? gb[q] : 0.0;
        };
        double mum = on && k0 > 0 ? mu[o - plane] : 0.0;
        double muc = on ? mu[o] : 0.0;
        StepIn nxt;
        load(nxt, o, k0);
        for (int k = k0; k < k1; ++k, o += plane) {
            const StepIn c = nxt;
            if (k + 1 < k1)
                load(nxt, o + plane, k + 1);
            const double sy = c.muym + c.muyp, sz = mum + c.mup, sx = c.mul + c.mur;
            const double off = fma(ax, sx, fma(az, sz, ay * sy));
            const double lv = fma(omega, fma(-dg, muc, off), c.lam);  // lam - omega A mu
            const double gv = fma(omega, muc, c.gb);
            const double m2 = muc + muc, t = m2 * c.x;
            g0 = fma(m2 - sx, c.x, g0);
            g1 += fma(-sy, c.u, t);
            g2 += fma(-sz, c.u, t);
            if (on) {
                lam[o] = lv;
                gb[o] = gv;
            }
            mum = muc;
            muc = c.mup;
        }
    }
    __shared__ double red[3][kThreads / 32];
    __shared__ bool last;
    auto block_sum = [&](double (&v)[3]) {  // thread 0 holds the sums
        for (int d = 0; d < 3; ++d) {
            for (int q = 16; q > 0; q >>= 1)
                v[d] += __shfl_down_sync(0xffffffffu, v[d], q);
            if (lane == 0)
                red[d][threadIdx.x >> 5] = v[d];
        }
        __syncthreads();
        if (threadIdx.x == 0)
            for (int d = 0; d < 3; ++d) {
                v[d] = 0.0;
                for (int w = 0; w < kThreads / 32; ++w)
                    v[d] += red[d][w];
            }
        __syncthreads();
    };
    double v[3] = {g0, g1, g2};
    block_sum(v);
    if (threadIdx.x == 0) {
        for (int d = 0; d < 3; ++d)
            __stcg(partials + 3 * blockIdx.x + d, v[d]);
        __threadfence();
        last = atomicAdd(counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last)
        return;
    __threadfence();
    v[0] = v[1] = v[2] = 0.0;
    for (int t = threadIdx.x; t < (int)gridDim.x; t += blockDim.x)
        for (int d = 0; d < 3; ++d)
            v[d] += __ldcg(partials + 3 * t + d);
    block_sum(v);
    if (threadIdx.x == 0) {
        for (int d = 0; d < 3; ++d)
            grad_a[d] += -omega * v[d];
        *counter = 0;
    }
}

// grad_a[d] += -omega * sum of the partials, in a fixed order.
__global__ void adjoint_reduce_kernel(const double* partials, int nblocks, double omega,
                                      double* grad_a)
{
    __shared__ double red[3][kThreads / 32];
    for (int d = 0; d < 3; ++d) {
        double acc = 0.0;
        for (int t = threadIdx.x; t < nblocks; t += blockDim.x)
            acc += partials[3 * t + d];
        for (int o = 16; o > 0; o >>= 1)
            acc += __shfl_down_sync(0xffffffffu, acc, o);
        if ((threadIdx.x & 31) == 0)
            red[d][threadIdx.x >> 5] = acc;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        for (int d = 0; d < 3; ++d) {
            double w = threadIdx.x < kThreads / 32 ? red[d][threadIdx.x] : 0.0;
            for (int o = 16; o > 0; o >>= 1)
                w += __shfl_down_sync(0xffffffffu, w, o);
            if (threadIdx.x == 0)
                grad_a[d] += -omega * w;
        }
    }
}

template <typename T>
cudaError_t launch_minv(const brs_ctx* c, const T* in, T* out, cudaStream_t s)
{
    const LineCfg& L = c->lcfg;
    const int groups = kThreads / L.G;
    const long long nlines = (long long)c->p.ny * c->p.nz;
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
    const long long need = (nlines + groups - 1) / groups;
    const T* tab = static_cast<const T*>(c->line_tab);
    const int nx = c->p.nx, ny = c->p.ny, nz = c->p.nz;
    auto a16 = [](const void* q) { return (reinterpret_cast<uintptr_t>(q) & 15u) == 0; };
    const bool vec = nx == L.E * L.G && (nx * sizeof(T)) % 16 == 0 && a16(in) && a16(out);
#define BRS_MINV_CASE(EE, GG)                                                          \
    if (L.E == EE && L.G == GG) {                                                      \
        int per_sm = 1; /* one resident wave: the kernel strides over the lines */      \
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, line_minv_kernel<T, EE, GG>, \
                                                      kThreads, 0);                    \
        const long long cap = (long long)sms * (per_sm > 0 ? per_sm : 1);               \
        const unsigned blocks = (unsigned)(need < cap ? need : cap);                    \
        line_minv_kernel<T, EE, GG><<<blocks, kThreads, 0, s>>>(in, out, tab, nx, ny, nz, vec); \
        return cudaGetLastError();                                                     \
    }
    BRS_MINV_CASE(4, 4)
    BRS_MINV_CASE(4, 8)
    BRS_MINV_CASE(4, 16)
    BRS_MINV_CASE(4, 32)
    BRS_MINV_CASE(8, 32)
    BRS_MINV_CASE(12, 32)
    BRS_MINV_CASE(16, 32)
#undef BRS_MINV_CASE
    return cudaErrorInvalidConfiguration;
}

struct AdjState {
    void* mu = nullptr;
    double* partials = nullptr;
    unsigned* counter = nullptr;  // FP64 update: CTAs done
    int nblocks = 0;
    brs_ctx* xctx = nullptr;  // x-line Jacobi with omega = 1: x = M^{-1}(b + N u) in one pass
    int* xstatus = nullptr;   // xctx's own status word (its kernels report to the owner's)
    bool tile = false;        // FP64: the block solves by the elimination from both ends
};

// Which solves an FP64 step takes.  The elimination from both ends (line_tile.cu) is a serial chain
// of half a line, 32 lines at a time; the scan by lanes (line.cu, line_minv_kernel) does more
// operations in log steps.  So the chain loses on long lines while an SM has few of them, least
// where its tiles come to whole rounds: time of a step with the chain's over one with the scan's, by
// lines per SM:
//   cells     8    10    12    16    18    20    22    27    40    46
//    33    0.87  0.89  0.89  1.12  0.95  0.84  0.81  0.84  0.84  0.81
//    57    1.01  1.03  1.04  1.26  1.13  0.97  0.92  0.97  0.95  0.89
//    77    1.12  0.95  0.97  1.21  1.07  0.96  0.87  0.83  0.86  0.76
//   113    1.24  1.12  1.11  1.37  1.28  1.12  1.01  0.94  1.00  0.88
//   201    1.35  1.15  1.13  1.44  1.29  1.10  1.01  0.94  0.94  0.87
//   333    1.47  1.26  1.26  1.60  1.47  1.19  1.06  1.04  1.09  0.92
//   501    1.33  1.08  1.06  1.31  1.23  1.06  0.95  0.83  0.87  0.74
// and with rows that the scan moves as vectors (256, 384 and 512 cells) up to 1.12 from 22 lines on,
// 1.02 .. 1.11 at 40.
bool tile_solves(const brs_params& p, int sms)
{
    const long long per_sm = ((long long)p.ny * p.nz + sms - 1) / sms;
    if (p.nx <= 32 || (p.nx <= 64 && per_sm <= 12) || (p.nx <= 96 && per_sm >= 9 && per_sm <= 12))
        return true;
    return per_sm >= (p.nx <= 64 ? 20 : p.nx >= 256 && p.nx % 128 == 0 ? 41 : 22);
}

// FP64: both block solves, then the update in one pass with its reduction.
int adjoint_run_f64(brs_ctx* c, double* lam, const double* u, const double* b, double* gb,
                    double* ga, cudaStream_t s)
{
    AdjState* A = static_cast<AdjState*>(c->adjoint);
    const brs_params& p = c->p;
    double* x = static_cast<double*>(c->scratch);
    double* mu = static_cast<double*>(A->mu);
    int rc;
    if (A->tile) {
        rc = line_tile_undamped(A->xctx, u, x, b, s);
        if (rc == BRS_OK)
            rc = line_tile_solve(A->xctx, lam, mu, s);
    } else {
        rc = line_sweep_launch(A->xctx, u, x, b, s);
        if (rc == BRS_OK)
            rc = brs_cuda_status(launch_minv<double>(c, lam, mu, s));
    }
    if (rc != BRS_OK)
        return rc;
    // planes per item: the fewest plane steps (one more per item for its first loads) over whole
    // rounds of the resident warps
    const long long cols = (long long)p.ny * ((p.nx + 31) / 32), warps = A->nblocks * (kThreads / 32ll);
    int kc = 1;
    long long best = -1;
    for (int q = 1; q <= 32; ++q) {
        const long long rounds = (cols * ((p.nz + q - 1) / q) + warps - 1) / warps;
        if (best < 0 || rounds * (q + 1) < best) {
            best = rounds * (q + 1);
            kc = q;
        }
    }
    return brs_cuda_status(launch_pdl(adjoint_update_f64, dim3(A->nblocks), dim3(kThreads), 0, s,
                                      lam, (const double*)mu, (const double*)x, u, gb, p.nx, p.ny,
                                      p.nz, kc, p.ax, p.ay, p.az, c->omega,
                                      A->partials, A->counter, ga));
}

int adjoint_run_f32(brs_ctx* c, float* lam, const float* u, const float* b, float* gb, double* ga,
                    cudaStream_t s)
{
    AdjState* A = static_cast<AdjState*>(c->adjoint);
    float* x = static_cast<float*>(c->scratch);
    float* mu = static_cast<float*>(A->mu);
    // x = M^{-1}(b + N u_k): one undamped x-line Jacobi sweep from u_k
    int rc = line_sweep_launch(A->xctx, u, x, b, s);
    if (rc != BRS_OK)
        return rc;
    cudaError_t e = launch_minv<float>(c, lam, mu, s);  // mu = M^{-1} lambda
    if (e != cudaSuccess)
        return brs_cuda_status(e);
    auto a16 = [](const void* q) { return (reinterpret_cast<uintptr_t>(q) & 15u) == 0; };
    const bool vec = c->p.nx % 4 == 0 && a16(lam) && a16(mu) && a16(x) && a16(u) && a16(gb);
    adjoint_update_march<<<A->nblocks, kThreads, 0, s>>>(lam, mu, x, u, gb, c->p.nx, c->p.ny,
                                                         c->p.nz, c->p.ax, c->p.ay, c->p.az,
                                                         c->omega, A->partials, vec);
    e = cudaGetLastError();
    if (e != cudaSuccess)
        return brs_cuda_status(e);
    adjoint_reduce_kernel<<<1, kThreads, 0, s>>>(A->partials, A->nblocks, c->omega, ga);
    return brs_cuda_status(cudaGetLastError());
}

}  // namespace

void adjoint_teardown(brs_ctx* c)
{
    AdjState* A = static_cast<AdjState*>(c->adjoint);
    if (!A)
        return;
    if (A->mu)
        cudaFree(A->mu);
    if (A->partials)
        cudaFree(A->partials);
    if (A->counter)
        cudaFree(A->counter);
    if (A->xctx) {
        A->xctx->dev_status = A->xstatus;
        brsmooth_destroy(A->xctx);
    }
    delete A;
    c->adjoint = nullptr;
}

extern "C" int brsmooth_adjoint_sweep(brs_ctx* c, void* lam, const void* u_k, const void* b,
                                      void* grad_b, double* grad_a, void* stream)
{
    cudaGetLastError();  // start from a clean launch-error state
    if (!c || !lam || !u_k || !b || !grad_b || !grad_a)
        return BRS_ERR_ARG;
    if (c->batch || c->p.block != BRS_XLINE || c->p.method != BRS_JACOBI)
        return BRS_ERR_UNSUPPORTED;
    // whole elements; u_k and b from a 16-byte boundary where TMA can stage the rows (FP32 loads them
    // so; FP64 reads single elements, but takes the same arrays)
    auto misaligned = [](const void* q, size_t to) { return reinterpret_cast<uintptr_t>(q) % to != 0; };
    const size_t in = c->lcfg.tma ? 16 : c->esize;
    if (misaligned(lam, c->esize) || misaligned(grad_b, c->esize) || misaligned(u_k, in) ||
        misaligned(b, in) || misaligned(grad_a, sizeof(double)))
        return BRS_ERR_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (!c->adjoint) {
        AdjState* A = new AdjState();
        c->adjoint = A;
        int sms = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
        const long long need = ((long long)c->p.ny * c->p.nz + kThreads / 32 - 1) / (kThreads / 32);
        // FP64: one resident wave (3 CTAs per SM), shared out in items
        const long long most = (long long)sms * (c->p.dtype == BRS_F64 ? 3 : 8);
        A->nblocks = (int)(need < most ? need : most);
        if (A->nblocks < 1)
            A->nblocks = 1;
        cudaError_t e = cudaMalloc(&A->mu, (size_t)c->cells * c->esize);
        if (e == cudaSuccess)
            e = cudaMalloc(&A->partials, sizeof(double) * 3 * A->nblocks);
        if (e == cudaSuccess)
            e = cudaMalloc(&A->counter, sizeof(unsigned));
        if (e == cudaSuccess)
            e = cudaMemset(A->counter, 0, sizeof(unsigned));
        int rc = brs_cuda_status(e);
        if (rc == BRS_OK) {
            brs_params q = c->p;
            q.omega = 1.0;
            rc = brsmooth_create(&q, &A->xctx);
        }
        if (rc != BRS_OK) {
            adjoint_teardown(c);
            return rc;
        }
        // only its line kernel is used: no Jacobi buffer or line-major copies, and faults
        // land in this context
        cudaFree(A->xctx->scratch);
        A->xctx->scratch = nullptr;
        line_seq_teardown(A->xctx);
        line_tile_trim(A->xctx);
        A->tile = A->xctx->ltile && tile_solves(c->p, sms);
        A->xstatus = A->xctx->dev_status;
        A->xctx->dev_status = c->dev_status;
    }
    c->last_stream = s;
    if (c->p.dtype == BRS_F64)
        return adjoint_run_f64(c, (double*)lam, (const double*)u_k, (const double*)b,
                               (double*)grad_b, grad_a, s);
    return adjoint_run_f32(c, (float*)lam, (const float*)u_k, (const float*)b, (float*)grad_b,
                           grad_a, s);
}
