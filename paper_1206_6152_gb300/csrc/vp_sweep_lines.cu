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
#include <cuda_runtime.h>

#include "vp_clamp_line.cuh"
#include "vp_device.cuh"
#include "vp_internal.cuh"

using namespace vpline;

namespace {

struct LinesGeom {
    int n;                     // cells per line
    long long cell_stride;     // spatial-cell stride along the line
    int od;                    // outer index o -> first cell: (o / od) m1 + (o % od) m2
    long long m1, m2;
    long long nvc;             // velocity cells per spatial cell
    int va_stride, va_n;       // velocity index along the axis: (v / va_stride) % va_n
};

template <typename T, int NMAX, bool PERIODIC>
__global__ void __launch_bounds__(128) k_drift_lines(const T *f, const LineCoef<T> *__restrict__ coef,
                                                    LinesGeom g, double *lost_out, T *fo)
{
    __shared__ Acc<double> red[32];
    const long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int n = g.n;
    T lost = T(0);
    if (v < g.nvc) {
        const LineCoef<T> cf = coef[(int)((v / g.va_stride) % g.va_n)];
        const bool neg = cf.code & 1;
        const long long o = blockIdx.y;
        const long long step = g.cell_stride * g.nvc;
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
        T *q = fo + off;
        const T out = clamp_line<T, NMAX, PERIODIC>(x, n, fm1, fm2, cf.c0, cf.c1, cf.c2, [&](int, T u) {
            *q = u;
            q += st;
        });
        if (!PERIODIC) lost = out;
    }
    if (!PERIODIC) {
        Acc<double> a;
        a.add((double)lost);
        a = block_merge(a, red);
        if (threadIdx.x == 0 && a.value() != 0.0) atomicAdd(lost_out, a.value());
    }
}

template <typename T, int NMAX>
cudaError_t drift_lines_n(vp_ctx *c, const T *f, const LineCoef<T> *coef, const LinesGeom &g,
                          long long outer, T *fo)
{
    const dim3 grid((unsigned)((c->nvc + 127) / 128), (unsigned)outer);
    if (c->periodic_space)
        k_drift_lines<T, NMAX, true><<<grid, 128, 0, c->stream>>>(f, coef, g, &c->sc->lost, fo);
    else
        k_drift_lines<T, NMAX, false><<<grid, 128, 0, c->stream>>>(f, coef, g, &c->sc->lost, fo);
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
    g.nvc = c->nvc;
    g.va_stride = axis == 0 ? c->nv[1] * c->nv[2] : (axis == 1 ? c->nv[2] : 1);
    g.va_n = c->nv[axis];
    const LineCoef<T> *cf = coef + (size_t)axis * c->maxnv;
    const long long outer = c->np / g.n;
    if (g.n <= 16) return drift_lines_n<T, 16>(c, f, cf, g, outer, fo);
    if (g.n <= 32) return drift_lines_n<T, 32>(c, f, cf, g, outer, fo);
    return drift_lines_n<T, 64>(c, f, cf, g, outer, fo);
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
