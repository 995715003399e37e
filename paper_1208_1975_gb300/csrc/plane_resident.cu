// FP32 mode-line sweeps of several sweeps per call, on chip from the first to the last.
//
// In the x-sine basis (plane_modes.cu) the x-modes of a plane call do not couple: mode p is an
// ny x nz problem of its own, y-lines with the z coupling, through all sweeps of the call.  The
// streaming sweep reads and writes every array once per sweep (12 bytes per cell, HBM-bound); here
// a cluster of C CTAs holds all of one mode in shared memory, u^ and b^ (2 MB at most: 8 CTAs of
// 227 KB), runs every sweep there and writes u^ once.  HBM carries 12 bytes per cell and call.
//
// CTA r of a cluster owns planes [r nz / C, (r+1) nz / C); a line group (G lanes, E cells each, the
// layout and the solve of the line kernels) owns a contiguous run of them:
//  * Jacobi: every group first reads the old rows just outside its run, all CTAs meet, and the
//    groups march through their runs in place, carrying the old rows k-1 and k in registers.
//  * Gauss-Seidel: the even planes, all CTAs meet, the odd planes (zebra order).
// Rows beyond a CTA's planes are read from its neighbour through distributed shared memory; two
// cluster barriers per sweep order all of it.  The operations on a cell are those of
// mode_tma_kernel, in its order, so the results are the same bit for bit.  Rows are padded to
// G E cells with zeros (zero table entries keep them zero), so any ny up to 512 does.
// Bound by the latency of a phase, two lines per warp and a cluster barrier: 34 % of the issue
// slots, most stalls on shared memory and the scans' shuffles.  Two lines are solved side by side,
// because one line's chain leaves most of its warp's issue slots empty (24 -> 20.7 us per sweep).
// Where a line takes the whole warp, a warp's share of the planes is warp-uniform and it steps
// through exactly its own lines: no masked lines, one row pointer, 137 warp instructions per
// 256-cell line instead of 165 (20.7 -> 18.5 us).  256-cell lines on 16 lanes of 16 cells, with a
// sixth fewer instructions, gained nothing here (Gauss-Seidel 20.9).
// us per sweep at 256^3, same box, streaming -> here: Jacobi 34.4 -> 18.5, Gauss-Seidel 47 -> 18.5;
// 128^3 10.3 / 13.2 -> 2.1 / 2.3; 200x190x180, which had no streaming form and ran two transforms
// per sweep, calls of 50 17.0 / 18.8 ms -> 0.81 / 0.86.
#include <algorithm>
#include <cstdlib>
#include <type_traits>

#include "line_impl.cuh"
#include "line_many.cuh"
#include "plane.cuh"
#include "row_smem.cuh"
#include "thomas_tables.h"

namespace {

struct ResArgs {
    int ny, nm, nz, C, nclusters, nsweeps, tab_len, rows;  // rows: most planes of a CTA
    float az, om1;
};

__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;"
                 ::: "memory");
}

// row_ld from the same place in another CTA of the cluster.
template <int E>
__device__ __forceinline__ void ld_remote(float (&v)[E], const float* row, int rank, int lane)
{
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(row + lane * E)), "r"(rank));
    const int h = E == 8 ? (lane >> 2) & 1 : 0;
#pragma unroll
    for (int m = 0; m < E / 4; ++m)
        asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(v[4 * m]), "=f"(v[4 * m + 1]), "=f"(v[4 * m + 2]), "=f"(v[4 * m + 3])
                     : "r"(a + 16 * (m ^ h))
                     : "memory");
}

constexpr int res_threads(int E) { return E <= 8 ? 512 : 256; }

template <int E, int G, bool GS>
__global__ void __launch_bounds__(res_threads(E), 1) mode_resident_kernel(
    const float* u, const float* __restrict__ b, float* out, const float* __restrict__ tab,
    const ResArgs a)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    constexpr int NP = E * G, NG = res_threads(E) / G;
    float* U = reinterpret_cast<float*>(smem_raw);
    float* B = U + (size_t)a.rows * NP;
    const int rank = (int)(blockIdx.x % a.C), cid = (int)(blockIdx.x / a.C);
    auto first = [&](int r) { return (int)((long long)r * a.nz / a.C); };
    const int ks = first(rank), np = first(rank + 1) - ks;
    const int below = rank > 0 ? ks - first(rank - 1) - 1 : 0;  // the lower CTA's last row
    // G = 32: the group is the warp, and so is its share of the planes
    const int g = G == 32 ? __shfl_sync(0xffffffffu, threadIdx.x / 32, 0) : threadIdx.x / G;
    const int lane = threadIdx.x % G;
    const float az = a.az, om1 = a.om1;
    const long long pstride = (long long)a.nm * a.ny;
    auto sync = [&]() {
        if (a.C == 1)
            __syncthreads();
        else
            cluster_sync();
    };
    // row i of this CTA's planes; -1 and np are the neighbours' (zero outside the grid)
    auto row = [&](float (&v)[E], int i) {
        if (i >= 0 && i < np)
            brs::row_ld<E>(v, U + (size_t)i * NP, lane);
        else if (i < 0 ? rank > 0 : rank + 1 < a.C)
            ld_remote<E>(v, U + (size_t)(i < 0 ? below : 0) * NP, i < 0 ? rank - 1 : rank + 1, lane);
        else
#pragma unroll
            for (int q = 0; q < E; ++q)
                v[q] = 0.0f;
    };
    pdl_wait();
    for (int p = cid; p < a.nm; p += a.nclusters) {
        brs::LineTables<float, E, G> tb;
        tb.load(tab + (size_t)p * a.tab_len, lane);
        __syncthreads();  // the previous mode's rows are stored
        const long long base = (long long)ks * pstride + (long long)p * a.ny;
        const bool vec = a.ny % 4 == 0;
        if (vec) {
            const int n4 = NP / 4;
            for (int t = threadIdx.x; t < np * n4; t += res_threads(E)) {
                const int i = t / n4, y = 4 * (t - i * n4);
                const bool in = y < a.ny;
                const float4 z = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                const long long o = base + i * pstride + y;
                const int q = i * NP + brs::row_pos<E>(y);
                *reinterpret_cast<float4*>(U + q) = in ? *reinterpret_cast<const float4*>(u + o) : z;
                *reinterpret_cast<float4*>(B + q) = in ? __ldg(reinterpret_cast<const float4*>(b + o)) : z;
            }
        } else {
            for (int t = threadIdx.x; t < np * NP; t += res_threads(E)) {
                const int i = t / NP, y = t - i * NP;
                const long long o = base + i * pstride + y;
                const int q = i * NP + brs::row_pos<E>(y);
                U[q] = y < a.ny ? u[o] : 0.0f;
                B[q] = y < a.ny ? __ldg(b + o) : 0.0f;
            }
        }
        sync();
        // one phase: Jacobi all planes, Gauss-Seidel those of one parity
        auto phase = [&](auto parity) {
            constexpr int PAR = decltype(parity)::value, ST = GS ? 2 : 1;
            const int f = GS ? (ks + PAR) & 1 : 0;     // first own plane of the phase
            const int cnt = (np - f + ST - 1) / ST;    // how many
            const int j0 = g * cnt / NG, j1 = (g + 1) * cnt / NG, n = j1 - j0;
            // um: the plane before the next line (Jacobi: its old values); hi: the one after the run
            float um[E], hi[E];
            const int i0 = n > 0 ? f + ST * j0 : 0;  // groups without a line look at row 0
            row(um, n > 0 ? i0 - 1 : 0);
            row(hi, n > 0 ? f + ST * (j1 - 1) + 1 : 0);
            if constexpr (!GS)
                sync();
            float* own = U + (size_t)i0 * NP;
            const float* brow = B + (size_t)i0 * NP;
            // the next M lines of every group, s of its n done before; groups of a warp that have
            // fewer (MASK) work on their first rows and store nothing
            auto step = [&](auto many, auto mask, int s) {
                constexpr int M = decltype(many)::value;
                constexpr bool MASK = decltype(mask)::value;
                float r[M][E];
#pragma unroll
                for (int m = 0; m < M; ++m) {
                    const bool on = !MASK || s + m < n;
                    const int o = on ? m * ST * NP : 0;
                    float up[E], bb[E];
                    if (s + m + 1 < n)
                        brs::row_ld<E>(up, own + o + NP, lane);
                    else
#pragma unroll
                        for (int q = 0; q < E; ++q)
                            up[q] = hi[q];
                    brs::row_ld<E>(bb, brow + o, lane);
#pragma unroll
                    for (int q = 0; q < E; ++q)
                        r[m][q] = PAR ? fma(az, up[q], fma(az, um[q], bb[q]))
                                      : fma(az, um[q] + up[q], bb[q]);
                    // the next line's lower neighbour: its old own row (Jacobi), or the row
                    // above this line (the other parity)
                    if constexpr (GS) {
#pragma unroll
                        for (int q = 0; q < E; ++q)
                            um[q] = up[q];
                    } else
                        brs::row_ld<E>(um, own + o, lane);
                }
                brs::line_solve_many<E, G, M>(r, tb, lane);
#pragma unroll
                for (int m = 0; m < M; ++m) {
                    const bool on = !MASK || s + m < n;
                    float uc[E];
                    brs::row_ld<E>(uc, own + (on ? m * ST * NP : 0), lane);
#pragma unroll
                    for (int q = 0; q < E; ++q)
                        r[m][q] = fma(tb.wp[q], r[m][q], om1 * uc[q]);
                    if (on)
                        brs::row_st<E>(own + m * ST * NP, r[m], lane);
                }
                if (!MASK || s + M < n) {
                    own += M * ST * NP;
                    brow += M * ST * NP;
                }
            };
            using One = std::integral_constant<int, 1>;
            using Two = std::integral_constant<int, 2>;
            int s = 0;
            if constexpr (G == 32) {
#pragma unroll 1
                for (; s + 1 < n; s += 2)
                    step(Two(), std::false_type(), s);
                if (s < n)
                    step(One(), std::false_type(), s);
            } else {
                // the groups of a warp step together, as often as the longest run of the CTA
                const int most = (cnt + NG - 1) / NG;
#pragma unroll 1
                for (; s + 1 < most && __any_sync(0xffffffffu, s < n); s += 2)
                    step(Two(), std::true_type(), s);
                if (s < most && __any_sync(0xffffffffu, s < n))
                    step(One(), std::true_type(), s);
            }
            sync();
        };
        for (int it = 0; it < a.nsweeps; ++it) {
            phase(std::integral_constant<int, 0>());
            if constexpr (GS)
                phase(std::integral_constant<int, 1>());
        }
        if (vec) {
            const int n4 = NP / 4;
            for (int t = threadIdx.x; t < np * n4; t += res_threads(E)) {
                const int i = t / n4, y = 4 * (t - i * n4);
                if (y < a.ny)
                    *reinterpret_cast<float4*>(out + base + i * pstride + y) =
                        *reinterpret_cast<const float4*>(U + i * NP + brs::row_pos<E>(y));
            }
        } else {
            for (int t = threadIdx.x; t < np * NP; t += res_threads(E)) {
                const int i = t / NP, y = t - i * NP;
                if (y < a.ny)
                    out[base + i * pstride + y] = U[i * NP + brs::row_pos<E>(y)];
            }
        }
    }
}

template <bool GS>
const void* res_kernel(int E, int G)
{
    if (E == 4)
        return G == 4    ? (const void*)mode_resident_kernel<4, 4, GS>
               : G == 8  ? (const void*)mode_resident_kernel<4, 8, GS>
               : G == 16 ? (const void*)mode_resident_kernel<4, 16, GS>
                         : (const void*)mode_resident_kernel<4, 32, GS>;
    return E == 8    ? (const void*)mode_resident_kernel<8, 32, GS>
           : E == 12 ? (const void*)mode_resident_kernel<12, 32, GS>
                     : (const void*)mode_resident_kernel<16, 32, GS>;
}

size_t res_smem(int rows, int E, int G) { return (size_t)2 * rows * E * G * sizeof(float); }

cudaLaunchConfig_t res_launch(const ModeResident& m, int C, int rows, int clusters,
                              cudaLaunchAttribute* at, cudaStream_t s)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(clusters * C));
    cfg.blockDim = dim3(res_threads(m.E));
    cfg.dynamicSmemBytes = res_smem(rows, m.E, m.G);
    cfg.stream = s;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)C;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    return cfg;
}

}  // namespace

int mode_resident_config(int ny, int nm, int nz, bool gs, ModeResident* out)
{
    ModeResident m;
    if (!scan_lanes(ny, &m.E, &m.G))
        return BRS_ERR_UNSUPPORTED;
    m.ny = ny, m.nm = nm, m.nz = nz;
    const void* k = gs ? res_kernel<true>(m.E, m.G) : res_kernel<false>(m.E, m.G);
    const int cap = (int)(220u * 1024u / res_smem(1, m.E, m.G));  // planes a CTA can hold
    cudaFuncAttributes fa{};
    cudaError_t e = cudaFuncGetAttributes(&fa, k);
    const int most = (int)res_smem(cap, m.E, m.G);
    if (e == cudaSuccess && fa.maxDynamicSharedSizeBytes < most)
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    // Cluster size: the least clocks per sweep over all rounds of modes.  A phase takes about 400
    // clocks, 600 more where CTAs meet, and 1000 per line of a group (256-cell lines, 16 warps)
    const int groups = res_threads(m.E) / m.G;
    double best = 1e300;
    for (int C = 1; C <= 8 && C <= nz && e == cudaSuccess; ++C) {
        const int rows = (nz + C - 1) / C;
        if (rows > cap)
            continue;
        cudaLaunchAttribute at[2];
        cudaLaunchConfig_t cfg = res_launch(m, C, rows, 1, at, nullptr);
        int nc = 0;
        e = cudaOccupancyMaxActiveClusters(&nc, k, &cfg);
        if (e != cudaSuccess || nc < 1)
            continue;
        const int rounds = (nm + nc - 1) / nc;
        const int lines = gs ? (rows + 1) / 2 : rows;
        const double cost = (double)rounds * (gs ? 2 : 1) *
                            (400.0 + (C > 1 ? 600.0 : 0.0) + 1000.0 * ((lines + groups - 1) / groups));
        if (cost < best) {
            best = cost;
            m.C = C;
            m.rows = rows;
            m.clusters = std::min(nc, nm);
        }
    }
    if (e != cudaSuccess)
        return brs_cuda_status(e);
    if (m.C == 0)
        return BRS_ERR_UNSUPPORTED;
    *out = m;
    return BRS_OK;
}

int mode_resident_launch(const ModeResident& m, const float* u, const float* b, float* out,
                         const float* tab, double az, double omega, bool gs, int nsweeps,
                         cudaStream_t s)
{
    ResArgs a{};
    a.ny = m.ny, a.nm = m.nm, a.nz = m.nz;
    a.C = m.C, a.nclusters = m.clusters, a.nsweeps = nsweeps;
    a.tab_len = scan_table_len(m.E, m.G, false);
    a.rows = m.rows;
    a.az = (float)az;
    a.om1 = (float)(1.0 - omega);
    const void* k = gs ? res_kernel<true>(m.E, m.G) : res_kernel<false>(m.E, m.G);
    cudaLaunchAttribute at[2];
    cudaLaunchConfig_t cfg = res_launch(m, m.C, m.rows, m.clusters, at, s);
    void* args[] = {&u, &b, &out, &tab, &a};
    return brs_cuda_status(cudaLaunchKernelExC(&cfg, k, args));
}
