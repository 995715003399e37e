// FP64 x-line sweeps on the caller's layout (Sec. 2, Alg. 1 / Alg. 2 with full x-line blocks,
// Thomas elimination from both ends of the line).
//
// The operations are those of line_seq.cu (7 FP64 operations per cell; GB300's FP64 pipe retires
// 2 per clock per SM), in its order, so the results are the same; only the data path differs.
// A CTA takes a task of up to 16 lines in three phases around a shared-memory tile:
//   1. all warps form the scaled right-hand sides, lanes along x (coalesced loads of the caller's
//      arrays, 20 of them in flight per lane);
//   2. one warp, two threads per line, eliminates from both ends and substitutes back, reading
//      and writing the tile (odd line stride: no bank conflicts), its next 8 cells in flight;
//   3. all warps update, lanes along x.
// No copies into a line-major layout (48 bytes per cell and call) and no trips of the
// elimination values through L2; and a grid of a few lines per SM spreads its loads and updates
// over all warps, where two threads per line alone would wait on memory latency.  An FP64 warp
// instruction occupies its SM quarter for 64 clocks, so the chain warp's place rotates with the
// CTA.  Calls of few sweeps, and grids of few lines per SM (line_seq_min_sweeps),
// run fastest on it (us per sweep, same box, line-major -> tile): 32^3 Jacobi 12.3 -> 4.4 in calls of
// 30, 64^3 22.6 -> 9.0, 96^3 32.6 -> 17.5, 128^3 44.7 -> 35.7; Gauss-Seidel 96x88x72 60.1 -> 21.7;
// 256^3 one-sweep calls 400 -> 325, but 223 -> 250 in calls of 30.  What bounds it at 256^3 is the
// balance of the chain against the other warps (FP64 pipe 75 % busy); at 32^3 latency: launch,
// loads, and 32 dependent FMAs.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <new>
#include <vector>

#include "brs_internal.cuh"
#include "line_tile.cuh"

namespace {

constexpr int kLines = 16;        // most lines per task: a warp's two threads per line
constexpr int kMaxSteps = 256; // lines of at most 512 cells, 256 steps per side
constexpr int kChain = 8;         // chain steps whose shared-memory reads are in flight

struct TileArgs {
    int nx, ny, nz, m;    // grid, twist cell
    int nl, pitch;        // lines per task, shared-memory stride of a line (odd)
    int colour;           // -1: all lines; 0 / 1: lines with (j + k) % 2 == colour
    int early;            // let the next launch start at once (it fits beside this one)
    long long nlines;     // lines to update
    double om1, gm;       // 1 - omega; ax g_m
    const double* tab;    // [3][nx]: omega pv_i, omega pv_i ay, omega pv_i az
    double fm[kMaxSteps + kChain];  // step s: ax p_s
};

struct Shape {
    int nl = kLines, threads = 32;
    int lpu = 4;   // lines a warp gathers or updates at once: 1, 2 or 4
    bool early = false, pdl = true;
};

struct TileState {
    double* tab = nullptr;
    double* bs = nullptr;     // omega pv_i b_i (calls of several sweeps)
    bool own_bs = false;
    TileArgs a{};
    Shape sh;                 // of a sweep, or of one colour's launch
};

TileState* st(brs_ctx* c) { return static_cast<TileState*>(c->ltile); }

enum { B_PLAIN = 0, B_SCALED = 1, SOLVE_ONLY = 2 };

__device__ __forceinline__ double ld_if(const double* p, bool ok) { return ok ? *p : 0.0; }

template <bool OMEGA1, int MODE, int LPU>
__global__ void __launch_bounds__(256, 4) xline_tile_kernel(const double* u, double* out,
                                                         const double* __restrict__ b,
                                                         const __grid_constant__ TileArgs a)
{
    extern __shared__ __align__(16) double Z[];
    __shared__ long long base[kLines];  // first cell of each line
    __shared__ int flags[kLines];       // 1: j > 0, 2: j + 1 < ny, 4: k > 0, 8: k + 1 < nz, 16: active
    const int nx = a.nx, nl = a.nl, pitch = a.pitch;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    if (threadIdx.x < nl) {
        const long long q = (long long)blockIdx.x * nl + threadIdx.x;
        int j = 0, k = 0, f = 0;
        if (q < a.nlines) {
            if (a.colour < 0) {
                k = (int)(q / a.ny);
                j = (int)(q - (long long)k * a.ny);
            } else {
                // two rows hold ny lines of one colour, the even row (ny + 1 - colour) / 2
                const long long pr = q / a.ny;
                const int rem = (int)(q - pr * a.ny), n0 = (a.ny + 1 - a.colour) >> 1;
                const int odd = rem >= n0;
                k = (int)(2 * pr) + odd;
                j = 2 * (rem - (odd ? n0 : 0)) + (a.colour ^ odd);
            }
            f = (j > 0) | (j + 1 < a.ny ? 2 : 0) | (k > 0 ? 4 : 0) | (k + 1 < a.nz ? 8 : 0) | 16;
        }
        base[threadIdx.x] = ((long long)k * a.ny + j) * nx;
        flags[threadIdx.x] = f;
    }
    __syncthreads();
    pdl_wait();
    if (a.early)
        pdl_trigger();
    const long long plane = (long long)nx * a.ny;
    const int chunks = (nx + 31) >> 5, groups = (nl + LPU - 1) / LPU;

    // right-hand sides, LPU lines by 32 cells at a time
    for (int unit = warp; unit < chunks * groups; unit += nwarp) {
        const int ch = unit / groups, g = unit - ch * groups;
        const int i = ch * 32 + lane;
        const bool act = i < nx;
        const int ic = act ? i : nx - 1;
        double bb[LPU], yn[LPU], yp[LPU], zn[LPU], zp[LPU];
#pragma unroll
        for (int h = 0; h < LPU; ++h) {
            const int l = g * LPU + h;
            const int f = l < nl && act ? flags[l < nl ? l : 0] : 0;
            const long long p = base[l < nl ? l : 0] + ic;
            bb[h] = ld_if(b + p, f & 16);
            if (MODE != SOLVE_ONLY) {
                yn[h] = ld_if(u + p - nx, f & 1);
                yp[h] = ld_if(u + p + nx, f & 2);
                zn[h] = ld_if(u + p - plane, f & 4);
                zp[h] = ld_if(u + p + plane, f & 8);
            }
        }
        double sb = 1.0, fa = 0.0, fb = 0.0;
        if (MODE != B_SCALED)
            sb = __ldg(a.tab + ic);
        if (MODE != SOLVE_ONLY) {
            fa = __ldg(a.tab + nx + ic);
            fb = __ldg(a.tab + 2 * nx + ic);
        }
#pragma unroll
        for (int h = 0; h < LPU; ++h) {
            const int l = g * LPU + h;
            double r = MODE == B_SCALED ? bb[h] : __dmul_rn(sb, bb[h]);
            if (MODE != SOLVE_ONLY)
                r = fma(fb, zn[h] + zp[h], fma(fa, yn[h] + yp[h], r));
            if (l < nl && act)
                Z[l * pitch + i] = r;
        }
    }
    __syncthreads();

    // elimination from both ends, twist cell, back substitution outwards
    if (warp == (int)(blockIdx.x % nwarp)) {
        const bool right = lane >= 16;
        const int l = lane & 15, m = a.m;
        const int Rc = nx - 1 - m;
        const int cnt = l < nl ? (right ? Rc : m) : 0;
        const int dir = right ? -1 : 1;
        double* p = Z + (l < nl ? l : 0) * pitch + (right ? nx - 1 : 0);
        double z = 0.0, v[kChain], w[kChain];
#pragma unroll
        for (int h = 0; h < kChain; ++h)
            v[h] = h < cnt ? p[dir * h] : 0.0;
#pragma unroll 1
        for (int s = 0; s < Rc; s += kChain) {
#pragma unroll
            for (int h = 0; h < kChain; ++h)
                w[h] = s + kChain + h < cnt ? p[dir * (s + kChain + h)] : 0.0;
#pragma unroll
            for (int h = 0; h < kChain; ++h)
                if (s + h < cnt) {
                    z = fma(a.fm[s + h], z, v[h]);
                    p[dir * (s + h)] = z;
                }
#pragma unroll
            for (int h = 0; h < kChain; ++h)
                v[h] = w[h];
        }
        const double zr = __shfl_xor_sync(0xffffffffu, z, 16);
        double y = 0.0;
        if (!right && l < nl) {
            y = fma(a.gm, z + zr, p[m]);
            p[m] = y;
        }
        const double yo = __shfl_xor_sync(0xffffffffu, y, 16);
        if (right)
            y = yo;
        // cells t from the end, t = Rc-1 .. 0: the pivot index is the same on both sides
#pragma unroll
        for (int h = 0; h < kChain; ++h) {
            const int t = Rc - 1 - h;
            v[h] = t >= 0 && t < cnt ? p[dir * t] : 0.0;
        }
#pragma unroll 1
        for (int s = 0; s < Rc; s += kChain) {
#pragma unroll
            for (int h = 0; h < kChain; ++h) {
                const int t = Rc - 1 - kChain - s - h;
                w[h] = t >= 0 && t < cnt ? p[dir * t] : 0.0;
            }
#pragma unroll
            for (int h = 0; h < kChain; ++h) {
                const int t = Rc - 1 - s - h;
                if (t >= 0 && t < cnt) {
                    y = fma(a.fm[t], y, v[h]);
                    p[dir * t] = y;
                }
            }
#pragma unroll
            for (int h = 0; h < kChain; ++h)
                v[h] = w[h];
        }
    }
    __syncthreads();
    if (!a.early)
        pdl_trigger();

    // update
    for (int unit = warp; unit < chunks * groups; unit += nwarp) {
        const int ch = unit / groups, g = unit - ch * groups;
        const int i = ch * 32 + lane;
        double own[LPU];
#pragma unroll
        for (int h = 0; h < LPU; ++h) {
            const int l = g * LPU + h;
            const bool on = l < nl && i < nx && (flags[l < nl ? l : 0] & 16);
            own[h] = !OMEGA1 && on ? u[base[l] + i] : 0.0;
        }
#pragma unroll
        for (int h = 0; h < LPU; ++h) {
            const int l = g * LPU + h;
            if (l < nl && i < nx && (flags[l] & 16)) {
                const double y = Z[l * pitch + i];
                out[base[l] + i] = OMEGA1 ? y : fma(a.om1, own[h], y);
            }
        }
    }
}

// dst = scale[i] * src, rows of nx
__global__ void __launch_bounds__(256) scale_rows_kernel(const double* __restrict__ src,
                                                         double* __restrict__ dst,
                                                         const double* __restrict__ scale, int nx,
                                                         long long n)
{
    pdl_wait_trigger();
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += stride)
        dst[q] = __dmul_rn(__ldg(scale + (int)(q % nx)), src[q]);
}

int env_int(const char* name, int dflt)
{
    const char* v = std::getenv(name);
    return (v && *v) ? std::atoi(v) : dflt;
}

size_t tile_smem(const TileArgs& a, int nl) { return (size_t)nl * a.pitch * sizeof(double); }

template <int MODE, int LPU>
const void* tile_kernel(bool om1)
{
    if constexpr (MODE != SOLVE_ONLY)  // a block solve has no own value to keep
        if (!om1)
            return (const void*)xline_tile_kernel<false, MODE, LPU>;
    return (const void*)xline_tile_kernel<true, MODE, LPU>;
}

const void* tile_kernel(int mode, int lpu, bool om1)
{
    if (mode == B_PLAIN)
        return lpu == 1 ? tile_kernel<B_PLAIN, 1>(om1)
             : lpu == 2 ? tile_kernel<B_PLAIN, 2>(om1) : tile_kernel<B_PLAIN, 4>(om1);
    if (mode == B_SCALED)
        return lpu == 1 ? tile_kernel<B_SCALED, 1>(om1)
             : lpu == 2 ? tile_kernel<B_SCALED, 2>(om1) : tile_kernel<B_SCALED, 4>(om1);
    return lpu == 1 ? tile_kernel<SOLVE_ONLY, 1>(om1)
         : lpu == 2 ? tile_kernel<SOLVE_ONLY, 2>(om1) : tile_kernel<SOLVE_ONLY, 4>(om1);
}

int launch_tile(brs_ctx* c, int mode, bool om1, int colour, const Shape& sh, const double* u,
                double* out, const double* b, cudaStream_t s)
{
    TileState* S = st(c);
    TileArgs a = S->a;
    const long long lines = (long long)c->p.ny * c->p.nz;
    a.colour = colour;
    a.nlines = colour < 0 ? lines : (lines + 1 - colour) / 2;
    a.nl = sh.nl;
    if (a.nlines == 0)
        return BRS_OK;
    a.early = sh.early;
    const void* k = tile_kernel(mode, sh.lpu, om1);
    const dim3 grid((unsigned)((a.nlines + sh.nl - 1) / sh.nl));
    void* args[] = {&u, &out, &b, &a};
    cudaError_t e;
    if (sh.pdl)
        e = launch_pdl_c(k, grid, dim3(sh.threads), tile_smem(a, sh.nl), s, args);
    else
        e = cudaLaunchKernel(k, grid, dim3(sh.threads), args, tile_smem(a, sh.nl), s);
    return brs_cuda_status(e);
}

// Lines per task and threads per CTA.  A task's pipe time goes with 6 nl + 32 (the chain costs a
// warp's two instructions per step whatever the lines); a wave of r resident tasks per SM takes
// about (r + 2) of them (a task alone is latency-bound).  Same box, us per Jacobi sweep in calls
// of 30, 16 / 12 / 8 lines: 256^3 250 / 257 / 293, 384x200x100 174 / 134 / 160, 64^3 10.5 / 10.8
// / 9.3.  Up to four resident tasks per SM get 256 threads (96^3: 17.5 us against 21.6), more
// 128 (256^3: 250 against 270).
Shape pick_shape(const TileArgs& a, long long lines, int sms)
{
    Shape sh;
    double best = 1e300, res = 1.0;
    for (int nl = kLines; nl >= 4; nl -= 4) {
        const double tps = (double)((lines + nl - 1) / nl) / sms;  // tasks per SM
        const double r = std::max(1.0, std::min(8.0, std::floor(220.0 * 1024.0 / tile_smem(a, nl))));
        const double full = std::floor(tps / r), rest = std::ceil(tps - full * r);
        const double cost = (6 * nl + 32) * (full * (r + 2) + (rest > 0.0 ? rest + 2 : 0.0));
        if (cost < best) {
            best = cost;
            res = std::min(r, tps);
            sh.nl = nl;
        }
    }
    sh.threads = res <= 4.5 ? 256 : 128;
    // as few lines per warp and trip as keep every warp at one trip: an FP64 warp instruction
    // holds its SM quarter for 64 clocks, so a trip of 4 lines takes 1300
    const int chunks = (a.nx + 31) / 32, nw = sh.threads / 32;
    sh.lpu = chunks * sh.nl <= nw ? 1 : chunks * ((sh.nl + 1) / 2) <= nw ? 2 : 4;
    sh.early = (lines + sh.nl - 1) / sh.nl <= 2ll * sms;
    sh.pdl = env_int("BRSMOOTH_LINE_PDL", 1) != 0;
    return sh;
}

}  // namespace

int line_tile_setup(brs_ctx* c)
{
    const brs_params& p = c->p;
    if (p.nx > 2 * kMaxSteps)
        return BRS_ERR_UNSUPPORTED;
    TileState* S = new (std::nothrow) TileState();
    if (!S)
        return BRS_ERR_NOMEM;
    c->ltile = S;
    const std::vector<double> pv = seq_line_pivots(p.nx, p.ax, p.ay, p.az);
    std::vector<double> tab(3 * (size_t)p.nx);
    for (int i = 0; i < p.nx; ++i) {
        tab[i] = c->omega * pv[i];
        tab[p.nx + i] = c->omega * pv[i] * p.ay;
        tab[2 * (size_t)p.nx + i] = c->omega * pv[i] * p.az;
    }
    TileArgs& a = S->a;
    a.nx = p.nx, a.ny = p.ny, a.nz = p.nz;
    a.m = (p.nx - 1) / 2;
    a.pitch = p.nx | 1;
    a.om1 = 1.0 - c->omega;
    a.gm = p.ax * pv[a.m];
    for (int q = 0; q < p.nx - 1 - a.m; ++q)
        a.fm[q] = p.ax * pv[p.nx - 1 - q];  // = p_q on the left side
    cudaError_t e = cudaMalloc(&S->tab, tab.size() * sizeof(double));
    if (e == cudaSuccess)
        e = cudaMemcpy(S->tab, tab.data(), tab.size() * sizeof(double), cudaMemcpyHostToDevice);
    // calls of 4 or more sweeps scale b into bs (the line-major form's, where the context has that)
    if (e == cudaSuccess && line_seq_min_sweeps(c) == 0) {
        e = cudaMalloc(&S->bs, (size_t)c->cells * sizeof(double));
        S->own_bs = true;
    }
    a.tab = S->tab;
    const size_t smem = tile_smem(a, kLines);
    for (int q = 0; q < 18 && smem > 48u * 1024u && e == cudaSuccess; ++q) {
        const void* k = tile_kernel(q % 3, 1 << (q / 6), q / 3 % 2 != 0);
        cudaFuncAttributes fa{};
        e = cudaFuncGetAttributes(&fa, k);
        if (e == cudaSuccess && (size_t)fa.maxDynamicSharedSizeBytes < smem)
            e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    }
    if (e != cudaSuccess)
        return brs_cuda_status(e);
    const long long lines = (long long)p.ny * p.nz;
    int sms = 0;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
    if (e != cudaSuccess)
        return brs_cuda_status(e);
    S->sh = pick_shape(a, p.method == BRS_JACOBI ? lines : (lines + 1) / 2, sms);
    return BRS_OK;
}

void line_tile_teardown(brs_ctx* c)
{
    TileState* S = st(c);
    if (!S)
        return;
    if (S->tab)
        cudaFree(S->tab);
    line_tile_trim(c);
    delete S;
    c->ltile = nullptr;
}

int line_tile_sweep(brs_ctx* c, void* u, const void* b, int nsweeps, cudaStream_t s)
{
    if (nsweeps == 0)
        return BRS_OK;
    TileState* S = st(c);
    const brs_params& p = c->p;
    const bool om1 = S->a.om1 == 0.0;
    const double* bp = static_cast<const double*>(b);
    int mode = B_PLAIN, rc = BRS_OK;
    // b scaled once where that pays: 24 bytes per cell and a launch (2 us) against one FP64
    // operation per cell and sweep (626 G/s).  The results are the same bit for bit.
    if (S->bs && nsweeps >= 4 && (double)(nsweeps - 4) * c->cells > 1.25e6) {
        const long long need = (c->cells + 255) / 256;
        const unsigned grid = (unsigned)std::min<long long>(need, 152 * 16);
        rc = brs_cuda_status(launch_pdl(scale_rows_kernel, dim3(grid), dim3(256), 0, s, bp, S->bs,
                                        (const double*)S->tab, p.nx, c->cells));
        bp = S->bs;
        mode = B_SCALED;
    }
    double* cur = static_cast<double*>(u);
    if (p.method == BRS_CHAOTIC_GS) {
        for (int q = 0; q < nsweeps && rc == BRS_OK; ++q)
            for (int col = 0; col < 2 && rc == BRS_OK; ++col)
                rc = launch_tile(c, mode, om1, col, S->sh, cur, cur, bp, s);
        return rc;
    }
    double* nxt = static_cast<double*>(c->scratch);
    for (int q = 0; q < nsweeps && rc == BRS_OK; ++q) {
        rc = launch_tile(c, mode, om1, -1, S->sh, cur, nxt, bp, s);
        std::swap(cur, nxt);
    }
    if (rc == BRS_OK && cur != u)
        rc = brs_cuda_status(cudaMemcpyAsync(u, cur, (size_t)c->cells * sizeof(double),
                                             cudaMemcpyDeviceToDevice, s));
    return rc;
}

int line_tile_undamped(brs_ctx* c, const double* u, double* out, const double* b, cudaStream_t s)
{
    return launch_tile(c, B_PLAIN, true, -1, st(c)->sh, u, out, b, s);
}

int line_tile_solve(brs_ctx* c, const double* r, double* out, cudaStream_t s)
{
    return launch_tile(c, SOLVE_ONLY, true, -1, st(c)->sh, nullptr, out, r, s);
}

void line_tile_trim(brs_ctx* c)
{
    TileState* S = st(c);
    if (!S)
        return;
    if (S->own_bs)
        cudaFree(S->bs);
    S->own_bs = false;
    S->bs = nullptr;
}

void line_tile_borrow(brs_ctx* c, double* bs)
{
    st(c)->bs = bs;
}
