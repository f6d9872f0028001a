// vp_sweep_lines.cu -- sweeps along lines of any length up to 64 cells, one
// line per thread in registers (zero whole-cell shift; vp_clamp_line.cuh).
// These serve every grid whose lengths have no kernel of their own; the
// shared-memory kernels of vp_sweep.cu remain for longer lines and for shifts
// of one cell or more.
//
//  * k_drift_lines: lines along a spatial axis straight from global memory to
//    registers and back (a warp reads 32 neighbouring velocity cells per
//    load).  Scalar lines, not packed pairs, so that each lane reads its own
//    direction.  FP32: bound by HBM; 20 x 18 x 22 positions of 24 x 28 x 26
//    velocity cells 0.30 -> 0.21 ms a sweep (5.3 TB/s) against the shared-memory
//    kernel.  FP64: at the FP64 pipe's rate (7.3 instructions per cell counted,
//    74 cycles each per quadrant's warp); 20 x 18 x 22 of the same 1.48 -> 0.86
//    ms, and FP64 lines of 16 and 32 go through here as well: the saturating
//    form takes 9 FP64 instructions and a reciprocal per line, and the z drift
//    ran both directions' code in every warp (16^6: 0.59 -> 0.25 ms).
//  * k_kick_lines: one velocity sweep of every cube, the same way (vx and vy
//    lines: a warp reads neighbouring cells; vz: each thread its own row, whose
//    32-byte sectors it uses up over consecutive loads).  A line with a
//    whole-cell shift takes the generic in-place routine.  FP64 cubes go
//    through it one launch per sweep: at 16 bytes per cell the sweep is bound by
//    the FP64 pipe alone.
#include <cuda_runtime.h>

#include "vp_clamp_line.cuh"
#include "vp_device.cuh"
#include "vp_fast_line.cuh"
#include "vp_internal.cuh"

using namespace vpline;

int vp_sm_count();

namespace {

// What a thread's lines lose through the outflow ends, over all of its lines:
// merging a CTA's threads takes about 50 FP64 instructions a warp, so it is
// done once per CTA of a grid that just fills the SMs, not once per line.
template <typename T>
struct Lost;
template <>
struct Lost<float> {
    Acc<float> a;
    __device__ __forceinline__ void add(float v) { a.add(v); }
    __device__ __forceinline__ double value() const { return a.value(); }
};
template <>
struct Lost<double> {
    double a = 0.0;
    __device__ __forceinline__ void add(double v) { a += v; }
    __device__ __forceinline__ double value() const { return a; }
};

template <typename T>
__device__ __forceinline__ void add_lost(const Lost<T> &lost, double *lost_out)
{
    __shared__ Acc<double> red[32];
    Acc<double> a;
    a.add(lost.value());
    a = block_merge(a, red);
    if (threadIdx.x == 0 && a.value() != 0.0) atomicAdd(lost_out, a.value());
}

struct LinesGeom {
    int n;                     // cells per line
    long long cell_stride;     // spatial-cell stride along the line
    int od;                    // outer index o -> first cell: (o / od) m1 + (o % od) m2
    long long m1, m2;
    int nvc;                   // velocity cells per spatial cell
    int va_stride, va_n;       // velocity index along the axis: (v / va_stride) % va_n
    long long lines;           // outer indices times nvc
};

// FP32 drifts without losses are faster as one line per thread, the next
// CTA's loads starting as a CTA ends (lines of 64: 0.24 ms against 0.28)
template <typename T, bool PERIODIC>
__host__ __device__ constexpr bool drift_persistent() { return !PERIODIC || sizeof(T) == 8; }

template <typename T, int NMAX, bool PERIODIC>
__global__ void __launch_bounds__(128) k_drift_lines(const T *f, const LineCoef<T> *__restrict__ coef,
                                                    LinesGeom g, double *lost_out, T *fo)
{
    const int n = g.n;
    const long long step = g.cell_stride * g.nvc;
    Lost<T> lost;
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < g.lines;
         q += (long long)gridDim.x * blockDim.x) {
        const int o = (int)(q / g.nvc), v = (int)(q - (long long)o * g.nvc);
        const LineCoef<T> cf = coef[(v / g.va_stride) % g.va_n];
        const bool neg = cf.code & 1;
        const long long off = ((o / g.od) * g.m1 + (o % g.od) * g.m2) * g.nvc + v +
                              (neg ? (n - 1) * step : 0);
        const long long st = neg ? -step : step;
        T x[NMAX + 1];
        const T *p = f + off;
        x[0] = *p;
#pragma unroll
        for (int j = 1; j <= NMAX; ++j) {
            p += st;
            x[j] = j < n ? *p : (PERIODIC ? x[0] : T(0));
        }
        T fm1 = T(0), fm2 = T(0);
        if (PERIODIC) {
            fm1 = f[off + (n - 1) * st];
            fm2 = f[off + (n > 1 ? n - 2 : 0) * st];
        }
        T *w = fo + off;
        const T out = clamp_line<T, NMAX, PERIODIC>(x, n, fm1, fm2, cf.c0, cf.c1, cf.c2, [&](int, T u) {
            *w = u;
            w += st;
        });
        if (!PERIODIC) lost.add(out);
        if (!drift_persistent<T, PERIODIC>()) break;
    }
    if (!PERIODIC) add_lost(lost, lost_out);
}

template <typename T, int NMAX>
__global__ void __launch_bounds__(128) k_kick_lines(const T *src, T *dst,
                                                   const LineCoef<T> *__restrict__ coef, int va,
                                                   int nx, int ny, int nz, long long np,
                                                   double *lost_out)
{
    const int n = va == 0 ? nx : (va == 1 ? ny : nz);
    const int nvc = nx * ny * nz, lines = nvc / n;
    Lost<T> lost;
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < np * lines;
         q += (long long)gridDim.x * blockDim.x) {
        const long long cell = q / lines;
        const int u = (int)(q - cell * lines);
        // line u of the cube: (vy, vz) = (u / nz, u % nz), (vx, vz) likewise, or row u
        int base, step;
        if (va == 0) { base = u; step = ny * nz; }
        else if (va == 1) { base = (u / nz) * ny * nz + u % nz; step = nz; }
        else { base = u * nz; step = 1; }
        const LineCoef<T> cf = coef[cell * 3 + va];
        const long long off = cell * nvc + base;
        if ((cf.code >> 1) != 0) {
            if (src != dst)
                for (int j = 0; j < n; ++j) dst[off + (long long)j * step] = src[off + (long long)j * step];
            lost.add(kick_line_shifted(dst + off, step, n, cf));
            continue;
        }
        const bool neg = cf.code & 1;
        const int st = neg ? -step : step;
        const T *p = src + off + (neg ? (n - 1) * step : 0);
        T *w = dst + off + (neg ? (n - 1) * step : 0);
        T x[NMAX + 1];
        x[0] = *p;
#pragma unroll
        for (int j = 1; j <= NMAX; ++j) {
            p += st;
            x[j] = j < n ? *p : T(0);
        }
        lost.add(clamp_line<T, NMAX, false>(x, n, T(0), T(0), cf.c0, cf.c1, cf.c2, [&](int, T v) {
            *w = v;
            w += st;
        }));
    }
    add_lost(lost, lost_out);
}

// CTAs of 128 threads, one line per thread at a time: as many as there are
// lines for, or with persistent only those that fit on the GPU at once.  The
// persistent grid pays where every CTA ends with a merge of its losses (FP64
// kicks of 20 x 18 x 22 cubes 1.14 -> 0.83 ms).
template <class K>
cudaError_t lines_grid(K kernel, long long lines, bool persistent, unsigned &grid)
{
    const long long g = (lines + 127) / 128;
    if (!persistent && g <= 0x7fffffffLL) {
        grid = (unsigned)g;
        return cudaSuccess;
    }
    int per_sm = 0;
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 128, 0);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    const long long cap = (long long)per_sm * vp_sm_count();
    grid = (unsigned)(g < cap ? g : cap);
    return cudaSuccess;
}

template <typename T>
cudaError_t kick_lines_t(vp_ctx *c, const T *src, T *dst, const LineCoef<T> *coef, int va)
{
    const int n = c->nv[va];
    auto kern = n <= 16 ? k_kick_lines<T, 16> : (n <= 32 ? k_kick_lines<T, 32> : k_kick_lines<T, 64>);
    unsigned grid;
    const cudaError_t e = lines_grid(kern, c->np * (c->nvc / n), true, grid);
    if (e != cudaSuccess) return e;
    kern<<<grid, 128, 0, c->stream>>>(src, dst, coef, va, c->nv[0], c->nv[1], c->nv[2], c->np,
                                      &c->sc->lost);
    return cudaGetLastError();
}

template <typename T, bool PERIODIC>
cudaError_t drift_lines_p(vp_ctx *c, const T *f, const LineCoef<T> *coef, const LinesGeom &g, T *fo)
{
    auto kern = g.n <= 16 ? k_drift_lines<T, 16, PERIODIC>
                          : (g.n <= 32 ? k_drift_lines<T, 32, PERIODIC> : k_drift_lines<T, 64, PERIODIC>);
    unsigned grid;
    const cudaError_t e = lines_grid(kern, g.lines, drift_persistent<T, PERIODIC>(), grid);
    if (e != cudaSuccess) return e;
    kern<<<grid, 128, 0, c->stream>>>(f, coef, g, &c->sc->lost, fo);
    return cudaGetLastError();
}

template <typename T>
cudaError_t drift_lines_t(vp_ctx *c, const T *f, int axis, const LineCoef<T> *coef, T *fo)
{
    LinesGeom g;
    g.n = c->n[axis];
    if (axis == 0) {
        g.cell_stride = (long long)c->n[1] * c->n[2];
        g.od = 1; g.m1 = 1; g.m2 = 0;
    } else if (axis == 1) {
        g.cell_stride = c->n[2];
        g.od = c->n[2]; g.m1 = (long long)c->n[1] * c->n[2]; g.m2 = 1;
    } else {
        g.cell_stride = 1;
        g.od = 1; g.m1 = c->n[2]; g.m2 = 0;
    }
    g.nvc = (int)c->nvc;
    g.va_stride = axis == 0 ? c->nv[1] * c->nv[2] : (axis == 1 ? c->nv[2] : 1);
    g.va_n = c->nv[axis];
    g.lines = c->np / g.n * c->nvc;
    const LineCoef<T> *cf = coef + (size_t)axis * c->maxnv;
    return c->periodic_space ? drift_lines_p<T, true>(c, f, cf, g, fo)
                             : drift_lines_p<T, false>(c, f, cf, g, fo);
}

}  // namespace

// lines of at most 64 cells (the caller checks that no shift reaches a cell)
int vp_drift_lines_ok(const vp_ctx *c, int axis) { return c->n[axis] <= 64; }

cudaError_t launch_drift_lines(vp_ctx *c, const void *f, int axis, const void *coef, void *fo)
{
    if (c->isdouble)
        return drift_lines_t<double>(c, (const double *)f, axis, (const LineCoef<double> *)coef,
                                     (double *)fo);
    return drift_lines_t<float>(c, (const float *)f, axis, (const LineCoef<float> *)coef, (float *)fo);
}

// FP64 cubes with no axis longer than 64, one launch per sweep
int vp_kick_lines_ok(const vp_ctx *c)
{
    return c->isdouble && c->maxnv <= 64;
}

cudaError_t launch_kick_lines(vp_ctx *c, const void *f, const void *ca, const void *cb, int nsweeps,
                              int first_axis, void *fo)
{
    const double *src = (const double *)f;
    double *dst = (double *)fo;
    for (int sw = 0; sw < nsweeps; ++sw) {
        const LineCoef<double> *cf = (const LineCoef<double> *)(sw < 3 ? ca : cb);
        // the first sweep reads f, the rest fo
        const cudaError_t e = kick_lines_t<double>(c, sw ? dst : src, dst, cf, (first_axis + sw) % 3);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}
