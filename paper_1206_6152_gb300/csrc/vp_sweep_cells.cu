// vp_sweep_cells.cu -- FP64 sweeps of grids with few lines, one thread per cell
// (the one-dimensional problems run on degenerate six-dimensional grids, and
// other small boxes).
//
// With one thread per line a 128-cell line is a serial chain of 128 x 7 FP64
// instructions of 64 pipe cycles and their latencies, on as many quadrants as there are
// warps of lines: 128 lines of 128 kept four of the GPU's 608 quadrants busy for 84 us.
// Here the lines are staged in shared memory, every thread computes the flux of
// its own cells (pfc_flux, bit for bit the line routines' arithmetic), and the
// update reads its neighbour's flux from shared memory.  Any whole-cell shift.
//
// It pays while the lines do not fill the GPU's quadrants with a warp each (32
// lanes x 4 quadrants x SMs = 19456 lines) and are long (the rules are below); else the
// other kernels do less work per cell.  128 x 128 cells (1D1V): x drift 88 -> 5 us, fused kick 140 ->
// 10 us, and with the sweeps along periodic axes of one cell passed over a step
// 254 -> 44 us.
#include <cuda_runtime.h>
#include <math.h>

#include "vp_device.cuh"
#include "vp_fast_line.cuh"
#include "vp_internal.cuh"

using namespace vpline;

int vp_sm_count();

namespace {

// Adds the CTA's losses to *lost_out.  Most cells lose nothing: warps whose lanes have
// only zeros pass the merge over (25 FP64 instructions), and the warps' sums are merged
// by as many steps as there are warps (x drift with outflow of 16^2 x 4 of 12 x 8 x 10
// cells 104 us with every warp's merge).
__device__ __forceinline__ void add_lost(double lost, double *lost_out, Acc<double> *red)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    Acc<double> a;
    if (__any_sync(0xffffffffu, __double_as_longlong(lost) << 1 != 0)) {
        a.add(lost);
        for (int d = 16; d > 0; d >>= 1) a.shfl_merge(d);
    }
    if (lane == 0) red[warp] = a;
    __syncthreads();
    if (warp != 0) return;
    a = lane < nw ? red[lane] : Acc<double>();
    if (!__any_sync(0xffffffffu, __double_as_longlong(a.s) << 1 != 0)) return;
    for (int d = 16; d > 0; d >>= 1)
        if (d < nw) a.shfl_merge(d);
    if (lane == 0) atomicAdd(lost_out, a.value());
}

// maxima (at least 0) of L lines in shared memory, line u at first(u), n cells
// at stride st, one warp per line; the caller synchronises
template <class F>
__device__ __forceinline__ void line_maxima(const double *f, int L, int n, int st, F first, double *fmx)
{
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int u = threadIdx.x >> 5; u < L; u += nw) {
        const double *p = f + first(u);
        double m = 0.0;
        for (int j = lane; j < n; j += 32) m = vmax(m, p[j * st]);
        for (int d = 16; d > 0; d >>= 1) m = vmax(m, __shfl_xor_sync(0xffffffffu, m, d));
        if (lane == 0) fmx[u] = m;
    }
}

// drift along a spatial axis: a CTA takes C neighbouring velocity cells' lines
// of one outer index
template <bool PERIODIC>
__global__ void __launch_bounds__(512) k_drift_cells(const double *f,
                                                    const LineCoef<double> *__restrict__ coef, int n,
                                                    int C, long long cell_stride, int od, long long m1,
                                                    long long m2, int nvc, int va_stride, int va_n,
                                                    double *lost_out, double *fo)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ Acc<double> red[32];
    double *tile = reinterpret_cast<double *>(smem_raw);     // [n][C], upwind order
    double *phi = tile + n * C, *fmx = phi + n * C;
    const int v0 = blockIdx.x * C, nb = nvc - v0 < C ? nvc - v0 : C, NT = blockDim.x;
    const long long o = blockIdx.y, st = cell_stride * nvc;
    const long long base = ((o / od) * m1 + (o % od) * m2) * nvc + v0;
    auto line = [&](int b) { return coef[((v0 + b) / va_stride) % va_n]; };
    for (int e = threadIdx.x; e < n * nb; e += NT) {
        const int p = e / nb, b = e - p * nb, j = line(b).code & 1 ? n - 1 - p : p;
        tile[j * C + b] = f[base + p * st + b];
    }
    __syncthreads();
    line_maxima(tile, nb, n, C, [](int u) { return u; }, fmx);
    __syncthreads();
    double lost = 0.0;
    for (int e = threadIdx.x; e < n * nb; e += NT) {
        const int j = e / nb, b = e - j * nb;
        const LineCoef<double> c = line(b);
        const double *L = tile + b;
        const double f0 = L[j * C];
        const double fm = j ? L[(j - 1) * C] : (PERIODIC ? L[(n - 1) * C] : 0.0);
        const double fp = j + 1 < n ? L[(j + 1) * C] : (PERIODIC ? L[0] : 0.0);
        const double ph = pfc_flux(fm, f0, fp, fmx[b], c.c0, c.c1, c.c2);
        phi[j * C + b] = ph;
        if (!PERIODIC) {
            const int s = c.code >> 1;
            if (j >= n - s) lost += f0;
            if (j == n - 1 - s) lost += ph;
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < n * nb; e += NT) {
        const int p = e / nb, b = e - p * nb;
        const LineCoef<double> c = line(b);
        const int i = c.code & 1 ? n - 1 - p : p, s = c.code >> 1;
        // upwind position i receives cell j = i - s and the flux of the cell before it
        int j = PERIODIC ? i - s % n : (s > i ? -1 : i - s);
        if (PERIODIC && j < 0) j += n;
        double out = 0.0;
        if (j >= 0) {
            const double phm = j ? phi[(j - 1) * C + b] : (PERIODIC ? phi[(n - 1) * C + b] : 0.0);
            out = (tile[j * C + b] - phi[j * C + b]) + phm;
        }
        fo[base + p * st + b] = out;
    }
    if (!PERIODIC) add_lost(lost, lost_out, red);
}

// nsweeps velocity sweeps of whole cubes, one CTA per cube at a time; a sweep
// whose shift is exactly zero leaves the cube as it is and is passed over, one
// that moves whole cells takes the serial line routine
__global__ void __launch_bounds__(512) k_kick_cells(const double *src, double *dst,
                                                   const LineCoef<double> *__restrict__ ca,
                                                   const LineCoef<double> *__restrict__ cb, int nsweeps,
                                                   int first_axis, int nx, int ny, int nz, long long np,
                                                   double *lost_out)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ Acc<double> red[32];
    const int nvc = nx * ny * nz, NT = blockDim.x, t = threadIdx.x;
    double *cube = reinterpret_cast<double *>(smem_raw), *phi = cube + nvc, *fmx = phi + nvc;
    double lost = 0.0;
    for (long long cell = blockIdx.x; cell < np; cell += gridDim.x) {
        for (int e = t; e < nvc; e += NT) cube[e] = src[cell * nvc + e];
        __syncthreads();
        for (int sw = 0; sw < nsweeps; ++sw) {
            const int va = (first_axis + sw) % 3;
            const LineCoef<double> c = (sw < 3 ? ca : cb)[cell * 3 + va];
            const int n = va == 0 ? nx : (va == 1 ? ny : nz), L = nvc / n;
            const int st = va == 0 ? ny * nz : (va == 1 ? nz : 1), neg = c.code & 1;
            if ((c.code >> 1) == 0 && c.c0 == 0.0) continue;
            auto first = [&](int u) {
                return va == 0 ? u : (va == 1 ? (u / nz) * ny * nz + u % nz : u * nz);
            };
            if ((c.code >> 1) != 0) {
                for (int u = t; u < L; u += NT) lost += kick_line_shifted(cube + first(u), st, n, c);
                __syncthreads();
                continue;
            }
            line_maxima(cube, L, n, st, first, fmx);
            __syncthreads();
            const int dn = neg ? -st : st;              // the downwind neighbour
            // element e: line u, position p in memory, j in upwind order
            auto where = [&](int e, int &u, int &j) {
                int p;
                if (va == 0) { p = e / st; u = e - p * st; }
                else if (va == 1) { const int i = e / (ny * nz), r = e - i * ny * nz; p = r / nz; u = i * nz + r - p * nz; }
                else { u = e / nz; p = e - u * nz; }
                j = neg ? n - 1 - p : p;
            };
            for (int e = t; e < nvc; e += NT) {
                int u, j;
                where(e, u, j);
                const double ph = pfc_flux(j ? cube[e - dn] : 0.0, cube[e], j + 1 < n ? cube[e + dn] : 0.0,
                                           fmx[u], c.c0, c.c1, c.c2);
                phi[e] = ph;
                if (j == n - 1) lost += ph;
            }
            __syncthreads();
            for (int e = t; e < nvc; e += NT) {
                int u, j;
                where(e, u, j);
                cube[e] = (cube[e] - phi[e]) + (j ? phi[e - dn] : 0.0);
            }
            __syncthreads();
        }
        for (int e = t; e < nvc; e += NT) dst[cell * nvc + e] = cube[e];
        __syncthreads();
    }
    add_lost(lost, lost_out, red);
}

int threads_for(long long cells)
{
    const long long t = (cells + 31) / 32 * 32;
    return (int)(t > 512 ? 512 : t);
}

// The rules below compare estimates of the time a call takes, in units of 39 ns (an FP64
// instruction of a quadrant's warp, 64 cycles or 33 ns, with the gaps that these kernels
// leave): a constant per launch or sweep and the FP64 instructions of the busiest quadrant.  Rounds of n warps' lanes over the
// SMs' quadrants (32 lanes x 4 quadrants each):
double rounds_of(long long n)
{
    const long long round = 128LL * vp_sm_count();
    return (double)((n + round - 1) / round);
}

// lines per CTA of k_drift_cells: one while that gives at most four CTAs per
// SM, and at most 4096 cells (64 KB of shared memory)
int cells_lines(const vp_ctx *c, int n)
{
    const long long lines = c->ncells / n;
    int C = 1;
    while (C < 32 && lines / C > 4LL * vp_sm_count() && 2 * C * n <= 4096) C *= 2;
    return C;
}

}  // namespace

// One thread per cell where that is the cheaper one.  Fitted to every drift of 27
// boxes of 3^3 to 128 positions with 10 velocity grids each, both boundary rules: the
// choice takes 0.3 % more than the better of the two on average.  Lines of 64: 16 against 35 us (4^2 x 64 of
// 6^3 cells), but 43 against 34 us with 12 x 8 x 10 velocity cells; lines below 8 cells
// gain nothing.  Lines above 64 cells have only the shared-memory kernel beside it.
int vp_drift_cells_ok(const vp_ctx *c, int axis)
{
    const int n = c->n[axis];
    if (!c->isdouble || n < 8) return 0;
    const double cells = 170 + 16 * rounds_of(c->ncells) + (c->periodic_space ? 0 : 40);
    const double lines = n <= 64 ? 165 + 7.3 * n * rounds_of(c->ncells / n) + (c->periodic_space ? 0 : 60)
                                 : 200 + 13.0 * n * rounds_of(c->ncells / n);
    return cells < lines;
}

cudaError_t launch_drift_cells(vp_ctx *c, const void *f, int axis, const void *coef, void *fo)
{
    const int n = c->n[axis], C = cells_lines(c, n);
    long long cs = (long long)c->n[1] * c->n[2], m1 = 1, m2 = 0;
    int od = 1;
    if (axis == 1) { cs = c->n[2]; od = c->n[2]; m1 = (long long)c->n[1] * c->n[2]; m2 = 1; }
    else if (axis == 2) { cs = 1; m1 = c->n[2]; }
    const int vs = axis == 0 ? c->nv[1] * c->nv[2] : (axis == 1 ? c->nv[2] : 1);
    const size_t smem = (size_t)(2 * n * C + C) * sizeof(double);
    auto kern = c->periodic_space ? k_drift_cells<true> : k_drift_cells<false>;
    if (smem + 1024 > 48 * 1024) {      // (with the static part)
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
        if (e != cudaSuccess) return e;
    }
    const dim3 grid((unsigned)((c->nvc + C - 1) / C), (unsigned)(c->np / n));
    kern<<<grid, threads_for((long long)n * C), smem, c->stream>>>(
        (const double *)f, (const LineCoef<double> *)coef + (size_t)axis * c->maxnv, n, C, cs, od, m1, m2,
        (int)c->nvc, vs, c->nv[axis], &c->sc->lost, (double *)fo);
    return cudaGetLastError();
}

// Which kernel sweeps FP64 cubes.  Lines (one launch per sweep, no axis above 64) are the
// cheapest where there are enough of them; with few cubes their launches weigh more
// than the sweeps, and one CTA per cube with all sweeps in one launch is better: one
// thread per line where lines are short (k_kick; a chain of n cells, or the FP64
// instructions of a cube's warps of lines over four quadrants), one thread per cell
// where they are not (its two buffers and line maxima in 96 KB).  Fitted to single
// sweeps, half kicks and fused kicks of the same boxes: none takes more than 1.07 times
// the whole-cube kernel (150 x 2 of 12^3, not among them, 1.14), and 0.4 % more than the
// best of the three on average.
// Fused kick of 4^3 cubes of 6 x 7 x 8: whole cubes 45, lines 62, cells 43 us; 4^3 of 9 x
// 10 x 11: 57, 74, 66; 8^3 of 6 x 7 x 8: 64, 78, 76; 8^3 of 9 x 10 x 11: 125, 114, 181;
// 128 cubes of 64 x 1 x 1: 92, 105, 69.
KickF64 vp_kick_f64_route(const vp_ctx *c, int nsweeps, int first_axis)
{
    const double sms = vp_sm_count(), np = (double)c->np;
    int nmin = c->nv[0];
    for (int a = 1; a < 3; ++a)
        if (c->nv[a] < nmin) nmin = c->nv[a];
    double cubes = 250, cells = 250, lines = 0;
    for (int k = 0; k < nsweeps; ++k) {
        const int n = c->nv[(first_axis + k) % 3];
        const double warps = (double)((c->nvc / n + 31) / 32);
        cubes += 40 + n * fmax(10.0, (10 + 0.75 * warps) * fmax(np / sms, 1.0) * warps / 4);
        cells += 40 + 20 * ceil(np / sms) * (double)((c->nvc + 127) / 128);
        lines += 200 + 8 * n * rounds_of(c->ncells / n);
    }
    if ((2 * c->nvc + c->nvc / nmin) * sizeof(double) > 96 * 1024) cells = INFINITY;
    if (c->maxnv > 64) lines = INFINITY;
    else if (!vp_kick_cube_ok(c)) cubes = INFINITY;
    if (cells < cubes && cells < lines) return KICK_CELLS;
    return lines < cubes ? KICK_LINES : KICK_CUBES;
}

cudaError_t launch_kick_cells(vp_ctx *c, const void *f, const void *ca, const void *cb, int nsweeps,
                              int first_axis, void *fo)
{
    int nmin = c->nv[0];
    for (int a = 1; a < 3; ++a)
        if (c->nv[a] < nmin) nmin = c->nv[a];
    const size_t smem = (size_t)(2 * c->nvc + c->nvc / nmin) * sizeof(double);
    if (smem + 1024 > 48 * 1024) {      // (with the static part)
        const cudaError_t e = cudaFuncSetAttribute(k_kick_cells, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   96 * 1024);
        if (e != cudaSuccess) return e;
    }
    const long long cap = 8LL * vp_sm_count();
    k_kick_cells<<<(unsigned)(c->np < cap ? c->np : cap), threads_for(c->nvc), smem, c->stream>>>(
        (const double *)f, (double *)fo, (const LineCoef<double> *)ca, (const LineCoef<double> *)cb, nsweeps,
        first_axis, c->nv[0], c->nv[1], c->nv[2], c->np, &c->sc->lost);
    return cudaGetLastError();
}
