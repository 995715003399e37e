// Batched x-line block sweeps over many independent patches of different sizes
// (Sec. 1.1 / Sec. 4.2: an AMR level holds many patches; the GPU processes their blocks
// as one stream of work, with no synchronisation between patches).
//
// Work items are (patch, y-block of R lines, z-chunk of KC planes).  A persistent grid
// of warps pulls items from an atomic counter (load balance across uneven patches);
// each warp marches its R lines in +z: u(j,k-1), u(j,k), u(j,k+1) stay in registers,
// the y neighbours inside the warp come by shuffle (FP32 patches with aligned rows: from the
// ring that stages them) and only the two halo lines of the y-block are loaded.  Lines are solved exactly with the shared-pivot Thomas scan of the
// single-grid path (the factor of M_line depends only on nx and the coefficients, so one
// table per distinct nx is built once).  One launch per sweep; the sweep sequence of a
// call is captured once into a CUDA graph and replayed as a single graph launch.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdlib>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "batched.cuh"
#include "line_impl.cuh"
#include "thomas_tables.h"

namespace {

struct PatchDesc {
    int nx, ny, nz;
    int cls;          // lanes per line G = 4 << cls (E = 4 cells per lane)
    long long off;    // element offset of the patch in the packed arrays
    int item0;        // first work item of the patch
    int njb;          // y-blocks (R = 32 / G lines each)
    int nkc;          // z-chunks
    int tab;          // element offset of the patch's line tables
    int vec;          // rows and patch start are 16-byte aligned
    int bchunk0;      // level: first 256-element chunk of the patch's ghost block
    long long g0;     // level: start of the patch's ghost block
};

struct Graph {
    const void* u;
    const void* b;
    int nsweeps;
    int mode;  // level ghost chaining at capture: bit 0 on, bit 1 ghosts valid, bit 2 parity
    cudaGraphExec_t exec;
};

struct BatchState {
    int npatch = 0;
    std::vector<int> dims;      // 3 * npatch
    long long total = 0;        // cells
    int KC = 8;                 // z-chunk
    int warps = 8;              // warps per CTA
    int grid = 0;               // persistent CTAs
    int ctas_per_sm = 1;
    int nitems = 0;
    PatchDesc* d_desc = nullptr;
    int* d_item_patch = nullptr;
    void* d_tab = nullptr;
    int* d_counters = nullptr;  // one per sweep of a call
    int ncounters = 0;
    std::vector<PatchDesc> h_desc;
    std::vector<int> h_item_patch;
    cudaStream_t cap = nullptr; // private capture stream
    std::vector<Graph> graphs;
    bool async = false;         // cp.async kernel (every patch row is 16-byte aligned)
    // level of patches (ghost values from the face neighbours, refreshed after every step)
    bool level = false;
    int* d_nbr = nullptr;        // 6 per patch: -x, +x, -y, +y, -z, +z neighbour or -1
    int* d_chunk_patch = nullptr; // boundary-cell chunk -> patch
    int nchunks = 0;
    void* ghost = nullptr;       // ghost blocks of every patch (neighbours' face layers)
    void* ghost2 = nullptr;      // the second ghost buffer (written during a step, read by the next)
    long long* d_push = nullptr; // 6 per patch: where each face goes in a ghost buffer, or -1
    bool push = true;            // steps after a call's first write their faces themselves
    // ghosts kept across calls (brsmooth_level_keep_ghosts): the last step of a call also
    // writes its faces, and the next call's first step reads them instead of gathering;
    // gpar is the ghost buffer the next step reads (0: ghost, 1: ghost2)
    bool keep = false;
    bool gvalid = false;
    int gpar = 0;
    int stages = 4;             // its ring depth (slots per warp)
};

BatchState* bs(brs_ctx* c)
{
    return static_cast<BatchState*>(c->batch);
}

constexpr int kE = 4;
// cp.async ring (FP32): a slot's rows of u (at most 96 16-byte pieces), then b
constexpr int kSlotB = 96 * 16;
constexpr int kSlotBytes = kSlotB + 32 * 16;
// x ghosts of one work item of a level, staged per warp: 2 faces x z-steps x lines
constexpr int kMaxKC = 32;
constexpr size_t kXgBytes = (size_t)2 * kMaxKC * 8 * sizeof(float);
// bytes of one warp's cp.async area: the ring, plus the staged x ghosts of a level
constexpr size_t async_ring_bytes(int stages, bool level)
{
    return (size_t)stages * kSlotBytes + (level ? kXgBytes : 0);
}

// Ghost block of a patch of a level (the face neighbours' adjacent layers as they were before
// the step; zero on the physical boundary), at g0 in a ghost array: the z- and z+ faces
// ([j][i], nx*ny each), the y- and y+ faces ([k][i], nx*nz), the x- and x+ faces ([k][j],
// ny*nz), each face starting on a multiple of 4 elements.
__host__ __device__ __forceinline__ long long round4(long long v) { return (v + 3) & ~3ll; }
__host__ __device__ __forceinline__ long long ghost_block(int nx, int ny, int nz)
{
    return 2 * (round4((long long)nx * ny) + round4((long long)nx * nz) +
                round4((long long)ny * nz));
}

// Row (jj, kk) just outside the patch across a z or y face: its x = 0 element in the
// ghost block, or null (no ghosts, or not a face row).
template <typename T>
__device__ __forceinline__ const T* outside_row(const PatchDesc& d, const T* ghost, int jj, int kk)
{
    if (!ghost)
        return nullptr;
    const long long A = round4((long long)d.nx * d.ny), Bz = round4((long long)d.nx * d.nz);
    const T* g = ghost + d.g0;
    if (jj >= 0 && jj < d.ny) {
        if (kk == -1)
            return g + (long long)jj * d.nx;
        if (kk == d.nz)
            return g + A + (long long)jj * d.nx;
    } else if (kk >= 0 && kk < d.nz) {
        if (jj == -1)
            return g + 2 * A + (long long)kk * d.nx;
        if (jj == d.ny)
            return g + 2 * A + Bz + (long long)kk * d.nx;
    }
    return nullptr;
}

// x- face ghost of line (j, k); the x+ ghost is ghost_x(...) + round4(ny * nz).
template <typename T>
__device__ __forceinline__ const T* ghost_x(const PatchDesc& d, const T* ghost, int j, int k)
{
    const long long A = round4((long long)d.nx * d.ny), Bz = round4((long long)d.nx * d.nz);
    return ghost + d.g0 + 2 * A + 2 * Bz + j + (long long)d.ny * k;
}

// Level contexts, steps after the first of a call: once a work item's lines are stored, the
// warp copies the item's cells that lie on a patch face into the ghost block of the face
// neighbour, in the ghost buffer that the next step reads (the current step reads the other
// one, so every patch still sees its neighbours' values of the previous step).  Every cell
// is written once per step, so the values are final; they are re-read from the output (just
// written by this warp, L2-resident).  push[f] is the offset of the destination face in that
// buffer, -1 where face f has no neighbour; destination layouts: z faces [j][i], y faces
// [k][i], x faces [k][j].  With yz_done (the cp.async kernel) the step loop has stored the
// y- and z-face rows itself, from registers, and only the x faces (and the y faces of a
// one-line patch) are copied here.  Not inlined and kept small: the step loop keeps its
// registers; the item is re-read here.
template <typename T>
__device__ __noinline__ void push_item(const PatchDesc* __restrict__ desc,
                                       const long long* __restrict__ push_all, T* gnext,
                                       const T* uout, int pq, int item, int KC, bool yz_done)
{
    __syncwarp();  // the item's stores by every lane of the warp are visible to all lanes
    const PatchDesc d = desc[pq];
    const long long* push = push_all + 6 * pq;
    const int local = item - d.item0;
    const int R = 32 / (4 << d.cls);
    const int j0 = (local % d.njb) * R, k0 = (local / d.njb) * KC;
    const int k1 = min(d.nz, k0 + KC);
    const T* uo = uout + d.off;
    const int lane = threadIdx.x & 31;
    const int nx = d.nx, ny = d.ny, nz = d.nz;
    const long long plane = (long long)nx * ny;
    const int nj = min(R, ny - j0), nk = k1 - k0;
    for (int f = 0; f < 2; ++f) {  // x faces: the item's cells at x = 0 and x = nx - 1
        const long long o = __ldg(push + f);
        if (o < 0)
            continue;
        const int xi = f ? nx - 1 : 0;
        const int lgR = 3 - d.cls;  // R = 8 >> cls
        for (int t = lane; t < nj * nk; t += 32) {
            const int kk = nj == R ? t >> lgR : t / nj;
            const int jl = t - kk * nj;
            const int j = j0 + jl, k = k0 + kk;
            gnext[o + j + (long long)ny * k] = uo[k * plane + (long long)j * nx + xi];
        }
    }
    for (int f = 2; f < 4; ++f) {  // y faces: line 0 or ny - 1, when the item holds it
        if (yz_done && ny > 1)
            break;  // written by the step loop
        const int j = f == 2 ? 0 : ny - 1;
        if (j < j0 || j >= j0 + nj)
            continue;
        const long long o = __ldg(push + f);
        if (o < 0)
            continue;
        for (int t = lane; t < nk * nx; t += 32) {
            const int kk = t / nx, i = t - kk * nx;
            const int k = k0 + kk;
            gnext[o + (long long)k * nx + i] = uo[k * plane + (long long)j * nx + i];
        }
    }
    for (int f = 4; f < 6 && !yz_done; ++f) {  // z faces: plane 0 or nz - 1, when held
        const int k = f == 4 ? 0 : nz - 1;
        if (k < k0 || k >= k1)
            continue;
        const long long o = __ldg(push + f);
        if (o < 0)
            continue;
        for (int t = lane; t < nj * nx; t += 32) {
            const int jl = t / nx, i = t - jl * nx;
            const int j = j0 + jl;
            gnext[o + (long long)j * nx + i] = uo[k * plane + (long long)j * nx + i];
        }
    }
}

template <typename T, int G, bool GS, bool LV>
__device__ __forceinline__ void batched_item(const PatchDesc& d, int jb, int kc, int KC,
                                             const T* uin, T* uout, const T* __restrict__ b,
                                             const T* __restrict__ tab, T ax, T ay, T az,
                                             T om1, const T* ghost)
{
    constexpr int R = 32 / G;
    const int lanew = threadIdx.x & 31;
    const int g = lanew / G, l = lanew % G;
    const int nx = d.nx, ny = d.ny, nz = d.nz;
    const int j = jb * R + g;
    const bool jin = j < ny;
    const int x0 = l * kE;
    const bool xin = x0 < nx;
    const long long plane = (long long)nx * ny;
    const T* ub = uin + d.off;
    T* uo = uout + d.off;
    const T* bb = b + d.off;
    brs::LineTables<T, kE, G> tb;
    tb.load(tab + d.tab, l);
    const int k0 = kc * KC;
    const int k1 = min(nz, k0 + KC);

    // load E cells of line (jj, kk) of `src`; outside the patch the ghost row (u only,
    // level contexts) or zero
    auto ld = [&](const T* src, int jj, int kk, T (&v)[kE]) {
        const bool in = jj >= 0 && jj < ny && kk >= 0 && kk < nz;
        const T* row = in ? src + (long long)kk * plane + (long long)jj * nx
                          : ((LV && src == ub) ? outside_row(d, ghost, jj, kk) : nullptr);
        if (xin && row) {
            const T* p = row + x0;
            if (d.vec) {
                if (sizeof(T) == 4) {
                    float4 f = *reinterpret_cast<const float4*>(p);
                    v[0] = (T)f.x; v[1] = (T)f.y; v[2] = (T)f.z; v[3] = (T)f.w;
                } else {
                    const double2* q = reinterpret_cast<const double2*>(p);
                    double2 f0 = q[0], f1 = q[1];
                    v[0] = (T)f0.x; v[1] = (T)f0.y; v[2] = (T)f1.x; v[3] = (T)f1.y;
                }
            } else {
#pragma unroll
                for (int q = 0; q < kE; ++q)
                    v[q] = (x0 + q < nx) ? p[q] : T(0);
            }
        } else {
#pragma unroll
            for (int q = 0; q < kE; ++q)
                v[q] = T(0);
        }
    };

    T um[kE], uc[kE], up[kE], r[kE], bv[kE], un[kE], us[kE];
    // next step's u(k+2), b(k+1) and halo lines (y-block edges), loaded one step ahead
    T upn[kE], bvn[kE], hnn[kE], hsn[kE];
    // x ghosts of the line (level contexts): the lane holding x = 0 and the one holding
    // x = nx - 1 add ax times the neighbour's value, loaded one step ahead
    const bool xlo = LV && xin && jin && x0 == 0;
    const bool xhi = LV && xin && jin && x0 <= nx - 1 && nx - 1 < x0 + kE;
    const long long xpo = round4((long long)ny * nz);
    T gxm = T(0), gxp = T(0), gxmn = T(0), gxpn = T(0);
    if (xlo)
        gxmn = *ghost_x(d, ghost, j, k0);
    if (xhi)
        gxpn = ghost_x(d, ghost, j, k0)[xpo];
    ld(ub, j, k0 - 1, um);
    ld(ub, j, k0, uc);
    ld(ub, j, k0 + 1, upn);
    ld(bb, j, k0, bvn);
    ld(ub, g == 0 ? j - 1 : -2, k0, hnn);
    ld(ub, g == R - 1 ? j + 1 : -2, k0, hsn);
    for (int k = k0; k < k1; ++k) {
        T hn[kE], hs[kE];
#pragma unroll
        for (int q = 0; q < kE; ++q) {
            up[q] = upn[q];
            bv[q] = bvn[q];
            hn[q] = hnn[q];
            hs[q] = hsn[q];
        }
        gxm = gxmn;
        gxp = gxpn;
        if (k + 1 < k1) {
            ld(ub, j, k + 2, upn);
            ld(bb, j, k + 1, bvn);
            // y neighbours at the block edges come from memory (row -1 reads as zero)
            ld(ub, g == 0 ? j - 1 : -2, k + 1, hnn);
            ld(ub, g == R - 1 ? j + 1 : -2, k + 1, hsn);
            if (xlo)
                gxmn = *ghost_x(d, ghost, j, k + 1);
            if (xhi)
                gxpn = ghost_x(d, ghost, j, k + 1)[xpo];
        }
#pragma unroll
        for (int q = 0; q < kE; ++q) {
            T a = __shfl_up_sync(0xffffffffu, uc[q], G);
            T c = __shfl_down_sync(0xffffffffu, uc[q], G);
            un[q] = (g == 0) ? hn[q] : a;
            us[q] = (g == R - 1) ? hs[q] : c;
        }
#pragma unroll
        for (int q = 0; q < kE; ++q)
            r[q] = (xin && jin) ? fma(az, um[q] + up[q], fma(ay, un[q] + us[q], bv[q])) : T(0);
        if (xlo)
            r[0] = fma(ax, gxm, r[0]);
        if (xhi) {
#pragma unroll
            for (int q = 0; q < kE; ++q)
                if (x0 + q == nx - 1)
                    r[q] = fma(ax, gxp, r[q]);
        }
        brs::line_solve<T, kE, G>(r, tb, l);
        T v[kE];
#pragma unroll
        for (int q = 0; q < kE; ++q)
            v[q] = fma(tb.wp[q], r[q], om1 * uc[q]);
        if (xin && jin) {
            T* p = uo + (long long)k * plane + (long long)j * nx + x0;
            if (d.vec && sizeof(T) == 4) {
                *reinterpret_cast<float4*>(p) = make_float4((float)v[0], (float)v[1],
                                                            (float)v[2], (float)v[3]);
            } else {
#pragma unroll
                for (int q = 0; q < kE; ++q)
                    if (x0 + q < nx)
                        p[q] = v[q];
            }
        }
#pragma unroll
        for (int q = 0; q < kE; ++q) {
            um[q] = GS ? ((xin && jin) ? v[q] : T(0)) : uc[q];
            uc[q] = up[q];
        }
    }
}

// 16-byte asynchronous copy global -> shared (per thread); src_bytes = 0 writes zeros
// without reading global memory (rows and planes outside the patch).
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t src_bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src),
                 "r"(src_bytes)
                 : "memory");
}
// 4-byte variant (through L1), for the staged x ghosts of a level
__device__ __forceinline__ void cp_async4(uint32_t dst, const void* src, uint32_t src_bytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src),
                 "r"(src_bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Same work item as batched_item in FP32, with the per-step inputs staged by cp.async through a
// per-warp ring of D slots in shared memory.  The slot of step k holds b(k) of the warp's R lines
// and plane k + 1 of u for them and one more line on each side, as R + 2 rows of G 16-byte pieces:
// a lane's own piece, and those of the lines before and after it, lie G pieces apart.  Step k takes
// u(k+1) and b(k) from its slot and the y neighbours from the slot before, which it then refills.
// Every patch row is a multiple of 16 bytes (checked on the host).
// Bound by the latency of a step's chain until enough warps are resident, then by DRAM: 600 patches
// of 16 to 64 cells a side (36 M cells), us per sweep: with the y neighbours by shuffle and select,
// and every row's address formed anew per step, 87 in 118 registers (16 warps per SM, 54 % of the
// issue slots, DRAM 57 %); so, 82 with 16 warps and 76 with the 20 that 96 registers allow, 0.84
// of the copy rate.  24 warps in 80 registers: 78.
template <int G, bool GS, int D, bool LV>
__device__ __forceinline__ void batched_item_async(const PatchDesc& d, int jb, int kc, int KC,
                                                   const float* uin, float* uout,
                                                   const float* __restrict__ b,
                                                   const float* __restrict__ tab, float ax,
                                                   float ay, float az, float om1,
                                                   const float* ghost, unsigned char* ring,
                                                   float* gnext, const long long* pp)
{
    constexpr int R = 32 / G;
    const int lanew = threadIdx.x & 31;
    const int g = lanew / G, l = lanew % G;
    const int nx = d.nx, ny = d.ny, nz = d.nz;
    const int j = jb * R + g;
    const bool jin = j < ny;
    const int x0 = l * kE;
    const bool xin = x0 < nx;
    const long long plane = (long long)nx * ny;
    const float* ub = uin + d.off;
    brs::LineTables<float, kE, G> tb;
    tb.load(tab + d.tab, l);
    const int k0 = kc * KC;
    const int k1 = min(nz, k0 + KC);
    const uint32_t ring0 = (uint32_t)__cvta_generic_to_shared(ring);
    // A row of u as the steps walk along z: its piece at x0 in the next plane, and the stride to
    // the one after.  Rows outside the patch are the ghost rows of a level's y faces, or zero.
    struct Row {
        const float* p;
        int step;
        bool ok;
    };
    auto row_at = [&](int jj) -> Row {
        Row r{ub, 0, false};
        if (jj >= 0 && jj < ny)
            r = {ub + (long long)k0 * plane + (long long)jj * nx + x0, nx * ny, xin};
        else if (LV && (jj == -1 || jj == ny)) {
            const float* gy = outside_row(d, ghost, jj, 0);
            if (gy)
                r = {gy + (long long)k0 * nx + x0, nx, xin};
        }
        return r;
    };
    Row own = row_at(j);
    // the lines before and after the warp's: lanes 0 .. G-1 and G .. 2G-1 (G = 32: both)
    Row edge = row_at(G == 32 || lanew < G ? jb * R - 1 : lanew < 2 * G ? jb * R + R : -2);
    Row edge2 = row_at(G == 32 ? jb * R + R : -2);
    const uint32_t edge_at = (uint32_t)((G == 32 || lanew < G ? lanew : 32 + lanew) * 16);
    const float* pb = b + d.off + (long long)k0 * plane + (long long)j * nx + x0;
    const bool ok_b = xin && jin;
    const float* gzp = LV && jin ? outside_row(d, ghost, j, nz) : nullptr;
    auto copy = [&](uint32_t dst, const Row& r) {
        cp_async16(dst, r.ok ? r.p : ub, r.ok ? 16u : 0u);
    };
    // plane kk of u and, unless first, b(kk - 1)
    auto issue = [&](int kk, uint32_t slot, bool first) {
        if (kk == nz) {
            own.p = LV && gzp ? gzp + x0 : ub;
            own.ok = LV && gzp && xin;
        }
        copy(slot + (uint32_t)(lanew + G) * 16, own);
        own.p += own.step;
        if (kk < nz) {  // the y neighbours of plane nz are not used
            if (G == 32 || lanew < 2 * G)
                copy(slot + edge_at, edge);
            edge.p += edge.step;
            if constexpr (G == 32) {
                copy(slot + (uint32_t)(lanew + 2 * G) * 16, edge2);
                edge2.p += edge2.step;
            }
        }
        if (!first) {
            cp_async16(slot + kSlotB + lanew * 16, ok_b ? pb : ub, ok_b ? 16u : 0u);
            pb += plane;
        }
    };
    // x ghosts of the line (level contexts): the lanes holding x = 0 and x = nx - 1
    const bool xlo = LV && xin && jin && x0 == 0;
    const bool xhi = LV && xin && jin && x0 <= nx - 1 && nx - 1 < x0 + kE;
    // a level step that writes the next step's ghosts (gnext set): the y- and z-face rows
    // its lines feed are stored as the steps produce them, from registers (row k of a y face
    // at o + k nx, row j of a z face at o + j nx; pp: the patch's six push offsets).  Lines
    // 0 and ny - 1 are distinct when ny > 1; a one-line patch leaves its y faces to push_item.
    long long gy = -1;  // this lane's piece of the y-face row of plane k, or -1
    if (LV && gnext && xin && ny > 1 && (j == 0 || j == ny - 1)) {
        const long long o = __ldg(pp + (j == 0 ? 2 : 3));
        if (o >= 0)
            gy = o + (long long)k0 * nx + x0;
    }
    // the item's x ghosts, staged once: xg[face][k - k0][line in the warp], copied
    // asynchronously with the first plane (zero beyond the last line)
    float* xg = reinterpret_cast<float*>(ring + (size_t)D * kSlotBytes);
    if (LV) {
        // x faces are [k][j] in the ghost block: element (kk, jl) of the item at
        // xb + face * xpo + kk * ny + jl (R a power of two: no divisions)
        const long long xpo = round4((long long)ny * nz);
        const int nk = k1 - k0;
        const uint32_t xg0 = (uint32_t)__cvta_generic_to_shared(xg);
        const float* xb = ghost_x(d, ghost, jb * R, k0);
        for (int face = 0; face < 2; ++face)
            for (int idx = lanew; idx < nk * R; idx += 32) {
                const int kk = idx / R, jl = idx % R;
                const bool ok = jb * R + jl < ny;
                const float* src = ok ? xb + (face ? xpo : 0) + (long long)kk * ny + jl : ghost;
                cp_async4(xg0 + (uint32_t)(((face * kMaxKC + kk) * 8 + jl) * sizeof(float)), src,
                          ok ? 4u : 0u);
            }
    }
    auto ld4 = [](float (&v)[kE], const float* p) {
        *reinterpret_cast<float4*>(v) = *reinterpret_cast<const float4*>(p);
    };
    const float* mine = reinterpret_cast<const float*>(ring) + lanew * kE;  // in slot 0
    constexpr int SW = kSlotBytes / 4;

    float um[kE] = {0.0f, 0.0f, 0.0f, 0.0f}, uc[kE], up[kE], r[kE], bv[kE], un[kE], us[kE];
    if (ok_b) {
        const float* pm = k0 > 0 ? ub + (long long)(k0 - 1) * plane + (long long)j * nx
                                 : LV ? outside_row(d, ghost, j, -1) : nullptr;
        if (pm)
            ld4(um, pm + x0);
    }
#pragma unroll
    for (int i = 0; i < D; ++i) {
        if (k0 + i <= k1)
            issue(k0 + i, ring0 + i * kSlotBytes, i == 0);
        cp_async_commit();
    }
    cp_async_wait<D - 1>();
    __syncwarp();  // plane k0 and the x ghosts have landed and every lane sees them
    ld4(uc, mine + G * kE);
    int prv = 0, cur = 1;  // slots of step k - 1 (plane k) and step k
    float* po = uout + d.off + (long long)k0 * plane + (long long)j * nx + x0;
    for (int k = k0; k < k1; ++k) {
        cp_async_wait<D - 2>();  // the group of step k is complete
        __syncwarp();
        const float *sp = mine + prv * SW, *sc = mine + cur * SW;
        ld4(un, sp);
        ld4(us, sp + 2 * G * kE);
        ld4(up, sc + G * kE);
        ld4(bv, sc + kSlotB / 4);
        float gxm = 0.0f, gxp = 0.0f;
        if (LV) {
            if (xlo)
                gxm = xg[(k - k0) * 8 + g];
            if (xhi)
                gxp = xg[(kMaxKC + k - k0) * 8 + g];
        }
        __syncwarp();  // every lane has read the slot before: refill it
        if (k + D <= k1)
            issue(k + D, ring0 + prv * kSlotBytes, false);
        cp_async_commit();
        prv = cur;
        cur = cur + 1 == D ? 0 : cur + 1;
        // zero beyond the row; lines beyond the patch compute values that nothing reads
#pragma unroll
        for (int q = 0; q < kE; ++q)
            r[q] = fma(az, um[q] + up[q], fma(ay, un[q] + us[q], bv[q]));
        if (xlo)
            r[0] = fma(ax, gxm, r[0]);
        if (xhi) {
#pragma unroll
            for (int q = 0; q < kE; ++q)
                if (x0 + q == nx - 1)
                    r[q] = fma(ax, gxp, r[q]);
        }
        brs::line_solve<float, kE, G>(r, tb, l);
        float v[kE];
#pragma unroll
        for (int q = 0; q < kE; ++q)
            v[q] = fma(tb.wp[q], r[q], om1 * uc[q]);
        if (ok_b)
            *reinterpret_cast<float4*>(po) = *reinterpret_cast<const float4*>(v);
        po += plane;
        if constexpr (LV) {
            if (gy >= 0) {
                *reinterpret_cast<float4*>(gnext + gy) = *reinterpret_cast<const float4*>(v);
                gy += nx;
            }
            if (gnext && (k == 0 || k == nz - 1) && xin && jin) {  // k is the same for the warp
#pragma unroll
                for (int f = 4; f < 6; ++f) {
                    const long long o = (f == 4 ? k == 0 : k == nz - 1) ? __ldg(pp + f) : -1;
                    if (o >= 0)
                        *reinterpret_cast<float4*>(gnext + o + (long long)j * nx + x0) =
                            *reinterpret_cast<const float4*>(v);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < kE; ++q) {
            um[q] = GS ? (ok_b ? v[q] : 0.0f) : uc[q];
            uc[q] = up[q];
        }
    }
    cp_async_wait<0>();  // only empty groups remain
    __syncwarp();        // and every lane has read its last slot and ghosts: the ring is free
}

constexpr int kAsyncThreads = 256;

template <bool GS, int D, bool LV>
__global__ void __launch_bounds__(kAsyncThreads, 2) batched_async_kernel(const PatchDesc* __restrict__ desc,
                                                            const int* __restrict__ item_patch,
                                                            int nitems, int* counter, int KC,
                                                            const float* uin, float* uout,
                                                            const float* __restrict__ b,
                                                            const float* __restrict__ tab,
                                                            double ax, double ay, double az,
                                                            double om1, const float* ghost,
                                                            float* gnext,
                                                            const long long* __restrict__ push)
{
    extern __shared__ __align__(16) unsigned char async_smem[];
    pdl_wait_trigger();
    const int lanew = threadIdx.x & 31;
    unsigned char* ring =
        async_smem + (size_t)(threadIdx.x >> 5) * async_ring_bytes(D, LV);
    while (true) {
        int item = 0;
        if (lanew == 0)
            item = atomicAdd(counter, 1);
        item = __shfl_sync(0xffffffffu, item, 0);
        if (item >= nitems)
            return;
        const int pq = item_patch[item];
        const PatchDesc d = desc[pq];
        const int local = item - d.item0;
        const int jb = local % d.njb, kc = local / d.njb;
        const long long* pp = push ? push + 6 * pq : nullptr;
        switch (d.cls) {
        case 0: batched_item_async<4, GS, D, LV>(d, jb, kc, KC, uin, uout, b, tab, (float)ax, (float)ay, (float)az, (float)om1, ghost, ring, gnext, pp); break;
        case 1: batched_item_async<8, GS, D, LV>(d, jb, kc, KC, uin, uout, b, tab, (float)ax, (float)ay, (float)az, (float)om1, ghost, ring, gnext, pp); break;
        case 2: batched_item_async<16, GS, D, LV>(d, jb, kc, KC, uin, uout, b, tab, (float)ax, (float)ay, (float)az, (float)om1, ghost, ring, gnext, pp); break;
        default: batched_item_async<32, GS, D, LV>(d, jb, kc, KC, uin, uout, b, tab, (float)ax, (float)ay, (float)az, (float)om1, ghost, ring, gnext, pp); break;
        }
        if (LV && gnext)
            push_item<float>(desc, push, gnext, uout, item_patch[item], item, KC, true);
    }
}

// Ghost exchange of a level (Sec. 2: ghost cells updated in a Jacobi fashion after each
// complete smoothing step): every patch's ghost block receives its face neighbours' adjacent
// layers of u (zero where a face is the physical boundary).  One thread per ghost element,
// chunks of 256 elements per patch; the sweep that follows reads these values wherever its
// stencil leaves the patch.
template <typename T>
__global__ void __launch_bounds__(256) level_exchange_kernel(const PatchDesc* __restrict__ desc,
                                                             const int* __restrict__ chunk_patch,
                                                             const int* __restrict__ nbr,
                                                             const T* u, T* __restrict__ ghost)
{
    pdl_wait_trigger();
    const int p = __ldg(chunk_patch + blockIdx.x);
    const int nx = __ldg(&desc[p].nx), ny = __ldg(&desc[p].ny), nz = __ldg(&desc[p].nz);
    const int t = (int)(blockIdx.x - __ldg(&desc[p].bchunk0)) * (int)blockDim.x + threadIdx.x;
    const int A = (int)round4((long long)nx * ny), Bz = (int)round4((long long)nx * nz);
    const int C = (int)round4((long long)ny * nz);
    if (t >= 2 * (A + Bz + C))
        return;
    auto at = [&](int q, int ii, int jj, int kk) -> T {
        const int qx = __ldg(&desc[q].nx), qy = __ldg(&desc[q].ny);
        return u[__ldg(&desc[q].off) + ii + (long long)qx * (jj + (long long)qy * kk)];
    };
    const int* nb = nbr + 6 * p;
    T v = T(0);
    if (t < 2 * A) {  // z faces, [j][i]
        const bool hi = t >= A;
        const int r = hi ? t - A : t;
        if (r >= nx * ny)
            return;  // padding
        const int j = r / nx, i = r - j * nx;
        const int q = __ldg(nb + (hi ? 5 : 4));
        if (q >= 0)
            v = at(q, i, j, hi ? 0 : __ldg(&desc[q].nz) - 1);
    } else if (t < 2 * A + 2 * Bz) {  // y faces, [k][i]
        const int t2 = t - 2 * A;
        const bool hi = t2 >= Bz;
        const int r = hi ? t2 - Bz : t2;
        if (r >= nx * nz)
            return;
        const int k = r / nx, i = r - k * nx;
        const int q = __ldg(nb + (hi ? 3 : 2));
        if (q >= 0)
            v = at(q, i, hi ? 0 : __ldg(&desc[q].ny) - 1, k);
    } else {  // x faces, [k][j]
        const int t3 = t - 2 * A - 2 * Bz;
        const bool hi = t3 >= C;
        const int r = hi ? t3 - C : t3;
        if (r >= ny * nz)
            return;
        const int k = r / ny, j = r - k * ny;
        const int q = __ldg(nb + (hi ? 1 : 0));
        if (q >= 0)
            v = at(q, hi ? 0 : __ldg(&desc[q].nx) - 1, j, k);
    }
    ghost[__ldg(&desc[p].g0) + t] = v;
}

template <typename T, bool GS, bool LV>
__global__ void __launch_bounds__(512) batched_line_kernel(const PatchDesc* __restrict__ desc,
                                                           const int* __restrict__ item_patch,
                                                           int nitems, int* counter, int KC,
                                                           const T* uin, T* uout,
                                                           const T* __restrict__ b,
                                                           const T* __restrict__ tab,
                                                           double ax, double ay, double az,
                                                           double om1, const T* ghost,
                                                           T* gnext,
                                                           const long long* __restrict__ push)
{
    pdl_wait_trigger();
    const int lanew = threadIdx.x & 31;
    while (true) {
        int item = 0;
        if (lanew == 0)
            item = atomicAdd(counter, 1);
        item = __shfl_sync(0xffffffffu, item, 0);
        if (item >= nitems)
            return;
        const int pq = item_patch[item];
        const PatchDesc d = desc[pq];
        const int local = item - d.item0;
        const int jb = local % d.njb, kc = local / d.njb;
        switch (d.cls) {
        case 0: batched_item<T, 4, GS, LV>(d, jb, kc, KC, uin, uout, b, tab, (T)ax, (T)ay, (T)az, (T)om1, ghost); break;
        case 1: batched_item<T, 8, GS, LV>(d, jb, kc, KC, uin, uout, b, tab, (T)ax, (T)ay, (T)az, (T)om1, ghost); break;
        case 2: batched_item<T, 16, GS, LV>(d, jb, kc, KC, uin, uout, b, tab, (T)ax, (T)ay, (T)az, (T)om1, ghost); break;
        default: batched_item<T, 32, GS, LV>(d, jb, kc, KC, uin, uout, b, tab, (T)ax, (T)ay, (T)az, (T)om1, ghost); break;
        }
        if (LV && gnext)
            push_item<T>(desc, push, gnext, uout, item_patch[item], item, KC, false);
    }
}

// FP32 only (the FP64 item does not fit the register budget with its ring addressing)
template <bool LV>
const void* async_kernel_lv(bool gs, int stages)
{
    if (stages >= 8)
        return gs ? (const void*)batched_async_kernel<true, 8, LV>
                  : (const void*)batched_async_kernel<false, 8, LV>;
    if (stages >= 6)
        return gs ? (const void*)batched_async_kernel<true, 6, LV>
                  : (const void*)batched_async_kernel<false, 6, LV>;
    return gs ? (const void*)batched_async_kernel<true, 4, LV>
              : (const void*)batched_async_kernel<false, 4, LV>;
}

const void* async_kernel_for(bool gs, int stages, bool level)
{
    return level ? async_kernel_lv<true>(gs, stages) : async_kernel_lv<false>(gs, stages);
}

template <bool LV>
const void* kernel_lv(int dtype, bool gs)
{
    if (dtype == BRS_F64)
        return gs ? (const void*)batched_line_kernel<double, true, LV>
                  : (const void*)batched_line_kernel<double, false, LV>;
    return gs ? (const void*)batched_line_kernel<float, true, LV>
              : (const void*)batched_line_kernel<float, false, LV>;
}

const void* kernel_for(int dtype, bool gs, bool level)
{
    return level ? kernel_lv<true>(dtype, gs) : kernel_lv<false>(dtype, gs);
}

// Line tables of one nx for E = 4 and G lanes (same layout and recurrences as the
// single-grid line path).
std::vector<double> tables_for(int nx, int G, const brs_params& p, double omega)
{
    return scan_thomas_tables<double>(nx, p.ax, 2.0 * (p.ax + p.ay + p.az), omega, kE, G, false);
}

int build_items(brs_ctx* c, int KC)
{
    BatchState* B = bs(c);
    B->h_item_patch.clear();
    int item = 0;
    for (int q = 0; q < B->npatch; ++q) {
        PatchDesc& d = B->h_desc[q];
        const int G = 4 << d.cls, R = 32 / G;
        d.njb = (d.ny + R - 1) / R;
        d.nkc = (d.nz + KC - 1) / KC;
        d.item0 = item;
        const int n = d.njb * d.nkc;
        for (int t = 0; t < n; ++t)
            B->h_item_patch.push_back(q);
        item += n;
    }
    B->nitems = item;
    B->KC = KC;
    if (B->d_desc)
        cudaFree(B->d_desc);
    if (B->d_item_patch)
        cudaFree(B->d_item_patch);
    B->d_desc = nullptr;
    B->d_item_patch = nullptr;
    cudaError_t e = cudaMalloc(&B->d_desc, sizeof(PatchDesc) * B->npatch);
    if (e == cudaSuccess)
        e = cudaMemcpy(B->d_desc, B->h_desc.data(), sizeof(PatchDesc) * B->npatch,
                       cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMalloc(&B->d_item_patch, sizeof(int) * std::max(1, item));
    if (e == cudaSuccess && item > 0)
        e = cudaMemcpy(B->d_item_patch, B->h_item_patch.data(), sizeof(int) * item,
                       cudaMemcpyHostToDevice);
    return brs_cuda_status(e);
}

int ensure_counters(BatchState* B, int n)
{
    if (B->ncounters >= n)
        return BRS_OK;
    if (B->d_counters)
        cudaFree(B->d_counters);
    B->d_counters = nullptr;
    B->ncounters = 0;
    cudaError_t e = cudaMalloc(&B->d_counters, sizeof(int) * n);
    if (e != cudaSuccess)
        return brs_cuda_status(e);
    B->ncounters = n;
    return BRS_OK;
}

int launch_one(brs_ctx* c, const void* uin, void* uout, const void* b, int* counter,
               cudaStream_t s, const void* ghost = nullptr, void* gnext = nullptr)
{
    BatchState* B = bs(c);
    const bool gs = c->p.method == BRS_CHAOTIC_GS;
    const void* k = B->async ? async_kernel_for(gs, B->stages, B->level)
                             : kernel_for(c->p.dtype, gs, B->level);
    const size_t smem =
        B->async ? (size_t)B->warps * async_ring_bytes(B->stages, B->level) : 0;
    const PatchDesc* desc = B->d_desc;
    const int* ip = B->d_item_patch;
    int nitems = B->nitems, KC = B->KC;
    const void* tab = B->d_tab;
    double ax = c->p.ax, ay = c->p.ay, az = c->p.az, om1 = 1.0 - c->omega;
    // ghost: the buffer this step reads (null unless the context is a level); gnext: the
    // one its face pushes go to (null: no pushes)
    const long long* push = B->d_push;
    void* args[] = {(void*)&desc, (void*)&ip, &nitems, &counter, &KC, (void*)&uin, &uout,
                    (void*)&b, (void*)&tab, &ax, &ay, &az, &om1, (void*)&ghost, &gnext,
                    (void*)&push};
    return brs_cuda_status(launch_pdl_c(k, dim3(B->grid), dim3(B->warps * 32), smem, s, args));
}

int level_exchange(brs_ctx* c, const void* u, void* ghost, cudaStream_t s)
{
    BatchState* B = bs(c);
    const PatchDesc* desc = B->d_desc;
    const int* cp = B->d_chunk_patch;
    const int* nb = B->d_nbr;
    cudaError_t e;
    if (c->p.dtype == BRS_F64)
        e = launch_pdl(level_exchange_kernel<double>, dim3(B->nchunks), dim3(256), 0, s, desc, cp,
                       nb, static_cast<const double*>(u), static_cast<double*>(ghost));
    else
        e = launch_pdl(level_exchange_kernel<float>, dim3(B->nchunks), dim3(256), 0, s, desc, cp,
                       nb, static_cast<const float*>(u), static_cast<float*>(ghost));
    return brs_cuda_status(e);
}

// Enqueue one call's sweeps (counter reset + one launch per sweep) on stream s.
int enqueue_sweeps(brs_ctx* c, void* u, const void* b, int nsweeps, cudaStream_t s)
{
    BatchState* B = bs(c);
    cudaError_t e = cudaMemsetAsync(B->d_counters, 0, sizeof(int) * nsweeps, s);
    if (e != cudaSuccess)
        return brs_cuda_status(e);
    const bool gs = c->p.method == BRS_CHAOTIC_GS;
    void* cur = u;
    void* nxt = gs ? u : c->scratch;
    int rc = BRS_OK;
    const bool chain = B->level && B->push && B->keep;
    const int par0 = chain ? B->gpar : 0;
    for (int k = 0; k < nsweeps && rc == BRS_OK; ++k) {
        void* gcur = nullptr;
        void* gnext = nullptr;
        if (B->level) {
            // the call's first step gathers its ghost layer from the iterate (unless the
            // previous call left it, ghosts kept across calls); every step but the last (every
            // step, when kept) then writes the next step's ghosts as it computes its faces
            // (two buffers, alternating)
            const int idx = (par0 + k) & 1;
            gcur = (B->push && idx) ? B->ghost2 : B->ghost;
            if (!B->push || (k == 0 && !(chain && B->gvalid)))
                rc = level_exchange(c, cur, gcur, s);
            if (B->push && (k + 1 < nsweeps || chain))
                gnext = idx ? B->ghost : B->ghost2;
        }
        if (rc == BRS_OK)
            rc = launch_one(c, cur, nxt, b, B->d_counters + k, s, gcur, gnext);
        if (!gs)
            std::swap(cur, nxt);
    }
    if (rc == BRS_OK && cur != u)
        rc = brs_cuda_status(cudaMemcpyAsync(u, cur, (size_t)B->total * c->esize,
                                             cudaMemcpyDeviceToDevice, s));
    return rc;
}

int env_int(const char* name, int dflt)
{
    const char* v = std::getenv(name);
    return (v && *v) ? std::atoi(v) : dflt;
}

// z-chunk fixed by the environment (0: none); a level stages at most kMaxKC z-steps of x ghosts.
int fixed_chunk() { return std::min(std::max(env_int("BRSMOOTH_BATCH_KC", 0), 0), kMaxKC); }

// The cp.async rings of every resident warp fit one SM.
bool async_fits(const BatchState* B, int warps, int ctas_per_sm, bool level)
{
    return (size_t)warps * ctas_per_sm * async_ring_bytes(B->stages, level) <= 220u * 1024u;
}

void set_shape(brs_ctx* c, int warps, int ctas_per_sm)
{
    BatchState* B = bs(c);
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
    B->warps = warps;
    B->ctas_per_sm = ctas_per_sm;
    B->grid = std::max(1, sms * ctas_per_sm);
}

// Autotuner: time each candidate (z-chunk, warps per CTA, CTAs per SM) on scratch
// arrays of the real patch set and keep the fastest.  Results are cached per process, keyed by
// all that decides which candidates there are and how fast they run: the device, the patch set,
// dtype, method, the kernel and its ring, and a chunk length fixed by BRSMOOTH_BATCH_KC.  The cp.async
// kernel of a level is timed itself: the plain kernel's shapes cut to the 16 warps per SM that its
// registers allow took nine 48x43x48 patches 187 us for 20 steps (8 warps, chunks of 8) against 178
// before and 155 now, two of 72^3 214 against 201 and 187.  The arrays are zero, so its ghosts stay so.
struct TuneKey {
    std::vector<int> dims;
    int device, dtype, method;
    bool level;  // a level's cp.async kernel
    int stages;  // cp.async ring slots; 0: direct loads
    int kc;      // fixed z-chunk; 0: any
    bool operator<(const TuneKey& o) const
    {
        return std::tie(device, dtype, method, level, stages, kc, dims) <
               std::tie(o.device, o.dtype, o.method, o.level, o.stages, o.kc, o.dims);
    }
};
struct TuneVal {
    int KC, warps, cps;
};
std::map<TuneKey, TuneVal> g_tune_cache;
std::mutex g_tune_mutex;

int autotune(brs_ctx* c)
{
    BatchState* B = bs(c);
    const int fixed_kc = fixed_chunk();
    const bool level = B->async && B->level;
    TuneKey key{B->dims, c->device, c->p.dtype, c->p.method, level, B->async ? B->stages : 0, fixed_kc};
    {
        std::lock_guard<std::mutex> lk(g_tune_mutex);
        auto it = g_tune_cache.find(key);
        if (it != g_tune_cache.end()) {
            set_shape(c, it->second.warps, it->second.cps);
            return build_items(c, it->second.KC);
        }
    }
    std::vector<TuneVal> cands;
    for (int kc : fixed_kc ? std::vector<int>{fixed_kc} : std::vector<int>{4, 8, 16, 32})
        for (int w : {4, 8, 16})
            for (int cps : {2, 4, 5, 8}) {
                if (w * cps > 64 || (!B->async && cps == 5))
                    continue;
                // cp.async kernel: 8 or 20 warps per SM in CTAs of 4 warps, 16 in CTAs of 8; a level: 8
                // or 16 in CTAs of 4, 16 in CTAs of 8
                if (B->async && (w * 32 > kAsyncThreads || cps == (level ? 5 : 4) ||
                                 (level && w * cps > 16) || !async_fits(B, w, cps, level)))
                    continue;
                cands.push_back({kc, w, cps});
            }
    const size_t bytes = (size_t)B->total * c->esize;
    void *tu = nullptr, *tb = nullptr;
    cudaError_t e = cudaMalloc(&tu, bytes);
    if (e == cudaSuccess)
        e = cudaMalloc(&tb, bytes);
    if (e == cudaSuccess)
        e = cudaMemset(tu, 0, bytes);
    if (e == cudaSuccess)
        e = cudaMemset(tb, 0, bytes);
    int rc = brs_cuda_status(e);
    if (rc == BRS_OK)
        rc = ensure_counters(B, 8);  // the timed calls run up to 5 sweeps
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (rc == BRS_OK) {
        cudaEventCreate(&e0);
        cudaEventCreate(&e1);
    }
    TuneVal best = cands[0];
    float best_ms = 1e30f;
    for (const TuneVal& v : cands) {
        if (rc != BRS_OK)
            break;
        set_shape(c, v.warps, v.cps);
        rc = build_items(c, v.KC);
        if (rc != BRS_OK)
            break;
        rc = enqueue_sweeps(c, tu, tb, 1, nullptr);  // warm
        // best of two 5-sweep timings: one short timing picked shapes 8 % apart run to run (four of
        // sweeps under 12 us, where launches scatter)
        float ms = 1e30f;
        for (int rep = 0; rep < (ms < 0.06f ? 4 : 2) && rc == BRS_OK; ++rep) {
            cudaEventRecord(e0, nullptr);
            rc = enqueue_sweeps(c, tu, tb, 5, nullptr);
            cudaEventRecord(e1, nullptr);
            if (cudaEventSynchronize(e1) != cudaSuccess && rc == BRS_OK)
                rc = BRS_ERR_CUDA;
            float t = 0.f;
            cudaEventElapsedTime(&t, e0, e1);
            ms = t < ms ? t : ms;
        }
        // plain cp.async kernel: fewer warps where more gain nothing
        if (rc == BRS_OK && ms < (B->async && !level ? 0.98f : 1.0f) * best_ms) {
            best_ms = ms;
            best = v;
        }
    }
    if (e0)
        cudaEventDestroy(e0);
    if (e1)
        cudaEventDestroy(e1);
    if (tu)
        cudaFree(tu);
    if (tb)
        cudaFree(tb);
    if (rc != BRS_OK)
        return rc;
    {
        std::lock_guard<std::mutex> lk(g_tune_mutex);
        g_tune_cache[key] = best;
    }
    set_shape(c, best.warps, best.cps);
    return build_items(c, best.KC);
}

}  // namespace

int batched_setup(brs_ctx* c, int npatch, const int* dims, bool level)
{
    BatchState* B = new BatchState();
    c->batch = B;
    B->npatch = npatch;
    B->dims.assign(dims, dims + 3 * npatch);
    std::map<int, int> tab_off;  // nx -> table offset
    std::vector<double> tabs;
    long long off = 0;
    const long long align = 16 / (long long)c->esize;
    for (int q = 0; q < npatch; ++q) {
        PatchDesc d{};
        d.nx = dims[3 * q];
        d.ny = dims[3 * q + 1];
        d.nz = dims[3 * q + 2];
        d.cls = d.nx <= 16 ? 0 : d.nx <= 32 ? 1 : d.nx <= 64 ? 2 : 3;
        d.off = off;
        d.vec = (d.nx % 4 == 0) && (off % align == 0) && (d.nx * (long long)c->esize) % 16 == 0;
        const int G = 4 << d.cls;
        const int key = d.nx;
        if (!tab_off.count(key)) {
            tab_off[key] = (int)tabs.size();
            auto t = tables_for(d.nx, G, c->p, c->omega);
            tabs.insert(tabs.end(), t.begin(), t.end());
        }
        d.tab = tab_off[key];
        B->h_desc.push_back(d);
        off += (long long)d.nx * d.ny * d.nz;
    }
    B->total = off;
    c->cells = off;
    cudaError_t e;
    if (c->p.dtype == BRS_F64) {
        e = cudaMalloc(&B->d_tab, tabs.size() * sizeof(double));
        if (e == cudaSuccess)
            e = cudaMemcpy(B->d_tab, tabs.data(), tabs.size() * sizeof(double),
                           cudaMemcpyHostToDevice);
    } else {
        std::vector<float> tf(tabs.begin(), tabs.end());
        e = cudaMalloc(&B->d_tab, tf.size() * sizeof(float));
        if (e == cudaSuccess)
            e = cudaMemcpy(B->d_tab, tf.data(), tf.size() * sizeof(float),
                           cudaMemcpyHostToDevice);
    }
    if (e != cudaSuccess)
        return brs_cuda_status(e);
    e = cudaStreamCreateWithFlags(&B->cap, cudaStreamNonBlocking);
    if (e != cudaSuccess)
        return brs_cuda_status(e);
    if (c->p.method == BRS_JACOBI) {
        e = cudaMalloc(&c->scratch, (size_t)B->total * c->esize);
        if (e != cudaSuccess)
            return brs_cuda_status(e);
    }
    // cp.async kernel when every patch row is a whole number of aligned 16-byte pieces
    B->async = c->p.dtype == BRS_F32 && env_int("BRSMOOTH_BATCH_ASYNC", 1) != 0;
    for (const PatchDesc& d : B->h_desc)
        B->async = B->async && d.vec;
    B->stages = env_int("BRSMOOTH_BATCH_STAGES", 4);
    B->stages = B->stages >= 8 ? 8 : B->stages >= 6 ? 6 : 4;
    if (B->async) {
        // both the plain and the level kernel (a level is set up after the tuner ran)
        for (bool lv : {false, true}) {
            const size_t want =
                std::min<size_t>(227u * 1024u, 16 * async_ring_bytes(B->stages, lv));
            const void* k = async_kernel_for(c->p.method == BRS_CHAOTIC_GS, B->stages, lv);
            cudaFuncAttributes fa{};
            e = cudaFuncGetAttributes(&fa, k);
            if (e == cudaSuccess && (size_t)fa.maxDynamicSharedSizeBytes < want)
                e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)want);
            if (e != cudaSuccess)
                return brs_cuda_status(e);
        }
    }
    if (env_int("BRSMOOTH_BATCH_NOTUNE", 0)) {
        const int kc = fixed_chunk();
        set_shape(c, 8, B->async ? 2 : 4);
        return build_items(c, kc ? kc : 8);
    }
    return level && B->async ? BRS_OK : autotune(c);
}

int level_setup(brs_ctx* c, const int* nbr)
{
    BatchState* B = bs(c);
    B->level = true;
    // boundary-cell chunks per patch (every dim >= 2, checked by the caller)
    std::vector<int> chunk_patch;
    long long gtotal = 0;
    for (int q = 0; q < B->npatch; ++q) {
        PatchDesc& d = B->h_desc[q];
        const long long gb = ghost_block(d.nx, d.ny, d.nz);
        if (gb >= (1ll << 31))
            return BRS_ERR_UNSUPPORTED;  // the exchange kernel numbers ghosts in 32 bits
        d.g0 = gtotal;
        gtotal += gb;
        d.bchunk0 = (int)chunk_patch.size();
        for (long long t = 0; t < (gb + 255) / 256; ++t)
            chunk_patch.push_back(q);
    }
    B->nchunks = (int)chunk_patch.size();
    const bool tuned = B->d_desc;  // direct loads, or BRSMOOTH_BATCH_NOTUNE
    // a level's rings also hold its x ghosts
    while (tuned && B->async && B->ctas_per_sm > 1 &&
           !async_fits(B, B->warps, B->ctas_per_sm, true))
        set_shape(c, B->warps, B->ctas_per_sm - 1);
    cudaError_t e = cudaSuccess;
    if (tuned)
        e = cudaMemcpy(B->d_desc, B->h_desc.data(), sizeof(PatchDesc) * B->npatch,
                       cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMalloc(&B->d_chunk_patch, sizeof(int) * chunk_patch.size());
    if (e == cudaSuccess)
        e = cudaMemcpy(B->d_chunk_patch, chunk_patch.data(), sizeof(int) * chunk_patch.size(),
                       cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMalloc(&B->d_nbr, sizeof(int) * 6 * B->npatch);
    if (e == cudaSuccess)
        e = cudaMemcpy(B->d_nbr, nbr, sizeof(int) * 6 * B->npatch, cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMalloc(&B->ghost, (size_t)gtotal * c->esize);
    if (e == cudaSuccess)
        e = cudaMemset(B->ghost, 0, (size_t)gtotal * c->esize);
    // face pushes: patch p's face f lands in the opposite ghost face of neighbour q
    // (x- -> q's x+, x+ -> q's x-, and so on); physical-boundary ghosts stay zero in both
    // buffers because nothing writes them
    B->push = env_int("BRSMOOTH_LEVEL_PUSH", 1) != 0;
    if (B->push) {
        std::vector<long long> push(6 * (size_t)B->npatch, -1);
        for (int p = 0; p < B->npatch; ++p)
            for (int f = 0; f < 6; ++f) {
                const int q = nbr[6 * p + f];
                if (q < 0)
                    continue;
                const PatchDesc& d = B->h_desc[q];
                const long long A = round4((long long)d.nx * d.ny);
                const long long Bz = round4((long long)d.nx * d.nz);
                const long long C = round4((long long)d.ny * d.nz);
                const long long face[6] = {2 * A + 2 * Bz + C, 2 * A + 2 * Bz, 2 * A + Bz,
                                           2 * A, A, 0};
                push[6 * (size_t)p + f] = d.g0 + face[f];
            }
        if (e == cudaSuccess)
            e = cudaMalloc(&B->ghost2, (size_t)gtotal * c->esize);
        if (e == cudaSuccess)
            e = cudaMemset(B->ghost2, 0, (size_t)gtotal * c->esize);
        if (e == cudaSuccess)
            e = cudaMalloc(&B->d_push, sizeof(long long) * push.size());
        if (e == cudaSuccess)
            e = cudaMemcpy(B->d_push, push.data(), sizeof(long long) * push.size(),
                           cudaMemcpyHostToDevice);
    }
    return e != cudaSuccess || tuned ? brs_cuda_status(e) : autotune(c);
}

void batched_teardown(brs_ctx* c)
{
    BatchState* B = bs(c);
    if (!B)
        return;
    for (auto& g : B->graphs)
        cudaGraphExecDestroy(g.exec);
    for (void* q : {(void*)B->d_desc, (void*)B->d_item_patch, B->d_tab, (void*)B->d_counters,
                    (void*)B->d_nbr, (void*)B->d_chunk_patch, B->ghost, B->ghost2,
                    (void*)B->d_push})
        if (q)
            cudaFree(q);
    if (B->cap)
        cudaStreamDestroy(B->cap);
    delete B;
    c->batch = nullptr;
}

int batched_sweep(brs_ctx* c, void* u, const void* b, int nsweeps, cudaStream_t s)
{
    BatchState* B = bs(c);
    if (nsweeps == 0)
        return BRS_OK;
    int rc = ensure_counters(B, nsweeps);
    if (rc != BRS_OK)
        return rc;
    const bool chain = B->level && B->push && B->keep;
    const int mode = chain ? (1 | (B->gvalid ? 2 : 0) | (B->gpar << 2)) : 0;
    // after this call the kept ghosts are valid and sit in the buffer its next step would read
    auto advance = [&]() {
        if (chain) {
            B->gpar = (B->gpar + nsweeps) & 1;
            B->gvalid = true;
        }
    };
    for (auto& g : B->graphs)
        if (g.u == u && g.b == b && g.nsweeps == nsweeps && g.mode == mode) {
            advance();
            return brs_cuda_status(cudaGraphLaunch(g.exec, s));
        }
    // capture this call's sweep sequence once on the private stream, replay on `s`
    cudaGraph_t graph = nullptr;
    cudaError_t e = cudaStreamBeginCapture(B->cap, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess)
        return brs_cuda_status(e);
    rc = enqueue_sweeps(c, u, b, nsweeps, B->cap);
    e = cudaStreamEndCapture(B->cap, &graph);
    if (rc != BRS_OK || e != cudaSuccess) {
        if (graph)
            cudaGraphDestroy(graph);
        return rc != BRS_OK ? rc : brs_cuda_status(e);
    }
    cudaGraphExec_t exec = nullptr;
    e = cudaGraphInstantiate(&exec, graph, 0);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess)
        return brs_cuda_status(e);
    if (B->graphs.size() >= 8) {
        cudaGraphExecDestroy(B->graphs.front().exec);
        B->graphs.erase(B->graphs.begin());
    }
    B->graphs.push_back({u, b, nsweeps, mode, exec});
    advance();
    return brs_cuda_status(cudaGraphLaunch(exec, s));
}

int level_keep_ghosts(brs_ctx* c, int on)
{
    BatchState* B = bs(c);
    if (!B || !B->level)
        return BRS_ERR_ARG;
    B->keep = on != 0 && B->push;
    B->gvalid = false;
    B->gpar = 0;
    return BRS_OK;
}

void batched_describe(const brs_ctx* c, int* kc, int* warps, int* grid, int* nitems)
{
    const BatchState* B = static_cast<const BatchState*>(c->batch);
    *kc = B->KC;
    *warps = B->warps;
    *grid = B->grid;
    *nitems = B->nitems;
}
