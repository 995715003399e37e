// FP32 x-line block Jacobi, two sweeps per pass over the grid (Sec. 2, Alg. 2 with full x-line
// blocks).
//
// The one-sweep kernel (line_impl.cuh) moves 12 bytes per cell and sweep and is bound by HBM.  Here
// a CTA marches in +z over a tile of lines and forms, at step s, the first sweep's values of plane
// k = kb - 1 + s for the tile's lines and one more line on each side, and the second sweep's values
// of plane k - 2 from those of planes k - 3 .. k - 1: 12 bytes per cell for two sweeps, and 16 line
// solves for every 14 of the first sweep.
//  * 16 warps, one line each (lines j0-1 .. j0+14).  The two solves of a step do not depend on each
//    other and run side by side (line_solve_many): their lane scans, the longest chain of a step,
//    overlap.  The second sweep's y neighbours were published in shared memory two steps before, its
//    own z neighbours are in registers.  One CTA barrier per step.  (Solving plane k - 1 instead,
//    one solve after the other, took 32.3 us where this takes 29.9; two CTAs of 8 warps 34.9.)
//  * u rows j0-2 .. j0+15 and b rows j0-1 .. j0+14 of the planes ahead come through a TMA ring, as in
//    the one-sweep kernel: rows and planes outside the grid read as zero, which is the Dirichlet
//    boundary; first-sweep values outside the grid are set to zero.
//  * The planes are shared out as there (contiguous runs of (y tile, plane)); a run of n planes takes
//    n + 3 steps.
// The operations on a cell are those of the one-sweep kernel, in its order: bit-identical results.
//
// Measured, us per sweep in calls of 50 (one-sweep kernel -> this): 256^3 37.6 -> 29.8,
// 256x256x512 70.0 -> 55.2, 128x512x512 99.7 -> 69.5, 72x300x300 37.4 -> 27.0, 256x40x2000 44.6 ->
// 38.0.  A pass
// is bound by its steps, not by HBM (about 3.4 TB/s at 256^3): 53 % of the issue slots, with 16 warps
// per SM in 128 registers the lane scans' shuffles are the largest stall.
#include <algorithm>
#include <cstdlib>

#include "line_impl.cuh"
#include "line_many.cuh"
#include "line_two.cuh"
#include "row_smem.cuh"

namespace {

constexpr int kWarps = 16, kOut = kWarps - 2;  // lines solved / written per tile
constexpr int kURows = kWarps + 2;

struct TwoArgs {
    int nx, ny, nz, NS;
    long long total;  // y tiles * nz
    float ay, az, om1;
    int* status;
};

template <int E>
__global__ void __launch_bounds__(kWarps * 32, 1) line_two_kernel(
    const __grid_constant__ CUtensorMap tm_u, const __grid_constant__ CUtensorMap tm_b,
    float* __restrict__ out, const float* __restrict__ tab, const TwoArgs a)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    constexpr int G = 32, NP = 32 * E;
    const int NS = a.NS, nx = a.nx;
    // every TMA box lands on a 128-byte boundary
    const uint32_t ubox = ((uint32_t)(kURows * nx * 4) + 127u) & ~127u;
    const uint32_t bbox = ((uint32_t)(kWarps * nx * 4) + 127u) & ~127u;
    const uint32_t ubytes = (uint32_t)(kURows * nx * 4), bbytes = (uint32_t)(kWarps * nx * 4);
    const uint32_t slot_bytes = ubox + bbox;
    float* v1 = reinterpret_cast<float*>(smem_raw + (size_t)NS * slot_bytes);  // [3][kWarps][NP]
    uint64_t* full = reinterpret_cast<uint64_t*>(v1 + 3 * kWarps * NP);

    const int tid = threadIdx.x, g = tid >> 5, lane = tid & 31;
    const int x0 = lane * E;
    const bool xin = x0 < nx;  // nx % E == 0: a lane's cells are all in the row or none
    brs::LineTables<float, E, G> tb;
    tb.load(tab, lane);
    if (tid == 0) {
        for (int s = 0; s < NS; ++s)
            mbar_init(&full[s], 1);
        fence_mbar_init();
    }
    __syncthreads();

    const long long L0 = (long long)blockIdx.x * a.total / gridDim.x;
    const long long L1 = (long long)(blockIdx.x + 1) * a.total / gridDim.x;
    auto inc = [&](int slot) { return slot + 1 == NS ? 0 : slot + 1; };
    // producer (thread 0): stage t of a run holds u plane kb-2+t and, from t = 2 on, b plane kb-3+t
    brs::SegIter pit{L0, L1, a.nz, 0, 0, 0};
    int p_next = 0, p_slot = 0, p_seg_base = 0, p_end = 0;
    bool p_has = false;
    auto issue = [&](int limit) {
        while (true) {
            if (!p_has || p_next >= p_end) {
                if (p_has)
                    p_seg_base = p_end;
                p_has = pit.next();
                if (!p_has)
                    return;
                p_end = p_seg_base + pit.n + 4;
            }
            if (p_next >= limit)
                return;
            const int t = p_next - p_seg_base;
            unsigned char* dst = smem_raw + (uint32_t)p_slot * slot_bytes;
            uint64_t* bar = &full[p_slot];
            const bool with_b = t >= 2;
            mbar_arrive_expect_tx(bar, ubytes + (with_b ? bbytes : 0u));
            const int j0 = pit.jt * kOut, ku = pit.kb - 2 + t;
            tma_load_3d(dst, &tm_u, bar, 0, j0 - 2, ku);
            if (with_b)
                tma_load_3d(dst + ubox, &tm_b, bar, 0, j0 - 1, ku - 1);
            ++p_next;
            p_slot = inc(p_slot);
        }
    };
    pdl_wait_trigger();
    if (tid == 0)
        issue(NS);

    brs::SegIter cit{L0, L1, a.nz, 0, 0, 0};
    int c_base = 0, cs_slot = 0;
    int waited = 0, w_slot = 0;
    uint32_t w_phase = 0;
    bool failed = false;
    const float ay = a.ay, az = a.az, om1 = a.om1;
    // A lane's cells of a ring row, for E = 8 with the two 16-byte halves in the order that is free of
    // bank conflicts (halves traded when lane / 4 is odd).  Sums and products of such rows need no
    // order; turn() puts the halves right (or back) where a line solve wants them.
    const int h = E == 8 ? (lane >> 2) & 1 : 0;
    auto ld = [&](float (&v)[E], const float* p) {
#pragma unroll
        for (int m = 0; m < E / 4; ++m) {
            const float4 t = reinterpret_cast<const float4*>(p)[m ^ h];
            v[4 * m] = t.x, v[4 * m + 1] = t.y, v[4 * m + 2] = t.z, v[4 * m + 3] = t.w;
        }
    };
    auto turn = [&](float (&v)[E]) {
        if constexpr (E == 8) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float lo = h ? v[q + 4] : v[q], hi = h ? v[q] : v[q + 4];
                v[q] = lo, v[q + 4] = hi;
            }
        }
    };
    auto stage = [&](int slot) {
        return reinterpret_cast<const float*>(smem_raw + (uint32_t)slot * slot_bytes) + x0;
    };
    const uint32_t boff = ubox / 4 + g * nx;
    auto zero = [&](float (&v)[E]) {
#pragma unroll
        for (int q = 0; q < E; ++q)
            v[q] = 0.0f;
    };
    // first-sweep values of the own line, planes k-3, k-2, k-1 (the steps rotate their names)
    float w0[E], w1[E], w2[E];
    zero(w0);
    zero(w1);
    zero(w2);
    int vs = 0;  // v1 slot of plane k
    while (cit.next()) {
        const int j = cit.jt * kOut - 1 + g;
        const bool jin = j >= 0 && j < a.ny;
        const bool mine = jin && g >= 1 && g <= kOut && xin;
        const size_t plane = (size_t)a.ny * nx;
        float* outp = out + ((size_t)cit.kb * a.ny + (jin ? j : 0)) * nx + x0;
        const int last = cit.n + 2;  // steps 0 .. last
        // false: the last step, or a wait that ran out
        auto step = [&](int s, float (&va)[E], float (&vb)[E], float (&vc)[E]) -> bool {
            const int need = c_base + (s + 3 < cit.n + 4 ? s + 3 : cit.n + 4);
            bool ok = true;
            while (waited < need && ok) {
                ok = mbar_wait_bounded(&full[w_slot], w_phase);
                if (ok) {
                    ++waited;
                    w_slot = inc(w_slot);
                    if (w_slot == 0)
                        w_phase ^= 1u;
                }
            }
            ok = __all_sync(0xffffffffu, ok);
            const int s1 = inc(cs_slot), s2 = inc(s1);
            if (ok) {
                const int k = cit.kb - 1 + s;
                const float *st0 = stage(cs_slot), *st1 = stage(s1), *st2 = stage(s2);
                float r[2][E];
                {  // r[0]: first sweep, plane k; r[1]: second sweep, plane k - 2
                    float a0[E], a1[E];
                    if (xin && s < last) {
                        ld(r[0], st2 + boff);
                        ld(a0, st1 + g * nx);
                        ld(a1, st1 + (g + 2) * nx);
#pragma unroll
                        for (int q = 0; q < E; ++q)
                            r[0][q] = fma(ay, a0[q] + a1[q], r[0][q]);
                        ld(a0, st0 + (g + 1) * nx);
                        ld(a1, st2 + (g + 1) * nx);
#pragma unroll
                        for (int q = 0; q < E; ++q)
                            r[0][q] = fma(az, a0[q] + a1[q], r[0][q]);
                    } else
                        zero(r[0]);
                    if (xin && s >= 3)
                        ld(r[1], st0 + boff);
                    else
                        zero(r[1]);
                    turn(r[0]);
                    turn(r[1]);
                    const int pv = vs == 0 ? 1 : vs == 1 ? 2 : 0;  // slot of plane k - 2
                    const float* prev = v1 + (pv * kWarps + g) * NP;
                    brs::row_ld<E>(a0, g > 0 ? prev - NP : prev, lane);
                    brs::row_ld<E>(a1, g + 1 < kWarps ? prev + NP : prev, lane);
#pragma unroll
                    for (int q = 0; q < E; ++q)
                        r[1][q] = fma(az, va[q] + vc[q], fma(ay, a0[q] + a1[q], r[1][q]));
                }
                brs::line_solve_many<E, G, 2>(r, tb, lane);
                if (jin && k >= 0 && k < a.nz && s < last) {  // warp-uniform
                    if (xin)
                        ld(va, st1 + (g + 1) * nx);
                    else
                        zero(va);
                    turn(va);
#pragma unroll
                    for (int q = 0; q < E; ++q)
                        va[q] = fma(tb.wp[q], r[0][q], om1 * va[q]);
                } else
                    zero(va);
                brs::row_st<E>(v1 + (vs * kWarps + g) * NP, va, lane);
                if (s >= 3 && mine) {
#pragma unroll
                    for (int q = 0; q < E; ++q)
                        r[1][q] = fma(tb.wp[q], r[1][q], om1 * vb[q]);
                    brs::st_global_vec<float, E>(outp, r[1]);
                }
            }
            if (s >= 3)
                outp += plane;
            vs = vs == 2 ? 0 : vs + 1;
            cs_slot = s1;
            failed = __syncthreads_or(!ok) != 0;
            if (failed)
                return false;
            if (tid == 0)
                // stages below the first one the next step needs are free
                issue((s < last ? c_base + s + 1 : c_base + cit.n + 4) + NS);
            return s < last;
        };
#pragma unroll 1
        for (int s = 0;; s += 3) {
            if (!step(s, w0, w1, w2) || !step(s + 1, w1, w2, w0) || !step(s + 2, w2, w0, w1))
                break;
        }
        if (failed)
            break;
        c_base += cit.n + 4;
        cs_slot = inc(cs_slot);  // skip the run's last stage
    }
    if (failed && tid == 0) {
        set_status(a.status, BRS_ERR_TIMEOUT);
        // drain copies still in flight before the CTA's shared memory is released
        for (int q = waited; q < p_next; ++q) {
            mbar_wait_bounded(&full[w_slot], w_phase, 200000000ull);
            w_slot = inc(w_slot);
            if (w_slot == 0)
                w_phase ^= 1u;
        }
    }
}

size_t stage_bytes(int nx)
{
    return (((size_t)kURows * nx * 4 + 127) & ~size_t(127)) +
           (((size_t)kWarps * nx * 4 + 127) & ~size_t(127));
}

size_t two_smem(int nx, int E, int NS)
{
    return (size_t)NS * stage_bytes(nx) + (size_t)3 * kWarps * 32 * E * 4 + (size_t)NS * 8;
}

long long tiles(const brs_params& p)
{
    return (p.ny + kOut - 1) / kOut;
}

const void* two_kernel(int E)
{
    return E == 4 ? (const void*)line_two_kernel<4> : (const void*)line_two_kernel<8>;
}

}  // namespace

// Fewest planes per CTA of the two-sweep form.  A run's three steps of start-up, and the lines that
// the tiles' edges solve twice, cost more than the saved traffic below it: at 8.4 planes per CTA
// 256x128x128 took 13.1 us per sweep (one-sweep form 12.0) and 128^3 8.9 (9.1), at 12.6 160^3 16.2
// (17.1), at 16 256x257x128 16.9 (21.1) and 256x128x256 19.5 (20.5).
constexpr int kMinPlanes = 12;

int line_two_setup(brs_ctx* c)
{
    const brs_params& p = c->p;
    const LineCfg& L = c->lcfg;
    c->two_stages = 0;
    const char* ev = std::getenv("BRSMOOTH_LINE_TWO");
    if (p.dtype != BRS_F32 || p.method != BRS_JACOBI || !L.tma || L.G != 32 || L.E > 8 ||
        L.pieces != 1 || (ev && ev[0] == '0'))
        return BRS_OK;
    int sms = 0;
    cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
    if (e != cudaSuccess)
        return brs_cuda_status(e);
    if (tiles(p) * p.nz < (long long)kMinPlanes * sms && !(ev && ev[0] == '2'))
        return BRS_OK;
    int NS = 8;
    while (NS > 4 && two_smem(p.nx, L.E, NS) > 220u * 1024u)
        --NS;
    const void* k = two_kernel(L.E);
    const size_t smem = two_smem(p.nx, L.E, NS);
    cudaFuncAttributes fa{};
    e = cudaFuncGetAttributes(&fa, k);
    if (e == cudaSuccess && (size_t)fa.maxDynamicSharedSizeBytes < smem)
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess)
        return brs_cuda_status(e);
    c->two_stages = NS;
    return BRS_OK;
}

// A pass goes from one vector to the other, and an odd number of passes ends with a copy back to the
// caller's (20 us at 256^3); two one-sweep passes in place of one pair cost 15 us.
int line_two_pairs(const brs_ctx* c, int nsweeps)
{
    if (!c->two_stages)
        return 0;
    const int pairs = nsweeps / 2;
    return (nsweeps - pairs) % 2 && pairs > 0 ? pairs - 1 : pairs;
}

int line_two_launch(brs_ctx* c, const void* uin, void* uout, const void* b, cudaStream_t s)
{
    const brs_params& p = c->p;
    const LineCfg& L = c->lcfg;
    CUtensorMap tu, tbm;
    int rc = brs_tmap(c, uin, kURows, &tu);
    if (rc == BRS_OK)
        rc = brs_tmap(c, b, kWarps, &tbm);
    if (rc != BRS_OK)
        return rc;
    TwoArgs a{};
    a.nx = p.nx, a.ny = p.ny, a.nz = p.nz;
    a.NS = c->two_stages;
    a.total = tiles(p) * p.nz;
    a.ay = (float)p.ay, a.az = (float)p.az, a.om1 = (float)(1.0 - c->omega);
    a.status = c->dev_status;
    int sms = 0;
    cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
    if (e != cudaSuccess)
        return brs_cuda_status(e);
    const unsigned grid = (unsigned)std::min<long long>(a.total, sms);
    float* out = static_cast<float*>(uout);
    const float* tab = static_cast<const float*>(c->line_tab);
    void* args[] = {&tu, &tbm, &out, &tab, &a};
    return brs_cuda_status(launch_pdl_c(two_kernel(L.E), dim3(grid), dim3(kWarps * 32),
                                        two_smem(p.nx, L.E, a.NS), s, args));
}
