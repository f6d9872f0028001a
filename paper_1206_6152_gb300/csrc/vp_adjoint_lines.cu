// vp_adjoint_lines.cu -- adjoint sweeps of lines of any length from 3 to 64,
// one line per thread: the transpose of one sweep with
// the limiter arms of vp_adjoint.cu's line_adjoint, each sum formed in its
// order, so that the results are those of that routine bit for bit.
//
// A thread holds its line of the state in registers and streams the cotangent
// from shared memory, where asynchronous copies put it; lines are held in upwind
// order (u < 0: read and written from the far end), so a warp runs one code path.
// Of cell j the frozen-arm terms are l0 (to cell j), lp (to j + 1) and lm (to
// j - 1); the input cotangent of a cell is complete one cell later:
//   li_j = ((lp_{j-1} + l_j) + l0_j) + lm_{j+1},
// for periodic lines with the wrapped terms where the routine adds them (lm_0
// first in cell n - 1, lp_{n-1} last in cell 0).  A whole-cell shift s only moves the
// cotangent: cell j meets entries j + s and j + s + 1, wrapped or zero past the end.
// Lines along x, y, z, vx and vy are copied element by element into the thread's
// own slots (a warp copies neighbouring cells); vz rows go through a tile, rows
// at odd pitch, with the CTA's contiguous rows copied in and out coalesced.
//
// What bounds it: FP32 issue and HBM, 12 bytes per cell; FP64 the FP64 pipe (64
// cycles per warp instruction): comparisons, doublings and selections of FP64 run
// on the integer pipes, which leaves 13 FP64 instructions per cell, 17 with the
// beta derivative.  Measured, one sweep: FP32 20 x 18 x 22 of 24 x 28 x 26 cells
// (1.66 GB, 245 us at 6.8 TB/s) 365-410 us, vz 534 us, where the shared-memory
// kernel of vp_adjoint.cu took 1140-1710 us, shifted by whole cells or not; FP64 16^6 440 us (drifts) and 577-595 us
// (kicks), where lines of all FP64 instructions in registers took 1120 us and, with
// both directions in a warp, 2200 us; FP64 12 x 10 x 14 of 16 x 18 x 20 260-411 us,
// shared memory 770-890 us.
#include <cuda_runtime.h>

#include "vp_clamp_line.cuh"
#include "vp_device.cuh"
#include "vp_internal.cuh"

using namespace vpline;

int vp_sm_count();

namespace {

__device__ __forceinline__ bool less(float a, float b) { return a < b; }
__device__ __forceinline__ bool nan64(double a)
{
    return (unsigned long long)__double_as_longlong(a) << 1 > 0xffe0000000000000ULL;
}
// (for operands one of which is not 0: the key orders -0 below +0)
__device__ __forceinline__ bool less(double a, double b)
{
    return dkey(a) < dkey(b) && !nan64(a) && !nan64(b);
}
// below 0 (-0 is not)
__device__ __forceinline__ bool negative(float a) { return a < 0.f; }
__device__ __forceinline__ bool negative(double a)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(a);
    return b > 0x8000000000000000ULL && b <= 0xfff0000000000000ULL;
}
__device__ __forceinline__ bool nonzero(float a) { return a != 0.f; }
__device__ __forceinline__ bool nonzero(double a) { return __double_as_longlong(a) << 1 != 0; }
__device__ __forceinline__ float fused(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fused(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float pick(bool p, float a, float b) { return p ? a : b; }
__device__ __forceinline__ double pick(bool p, double a, double b)
{
    return __hiloint2double(p ? __double2hiint(a) : __double2hiint(b),
                            p ? __double2loint(a) : __double2loint(b));
}

template <typename T>
__device__ __forceinline__ void copy_async(T *smem, const T *gmem)
{
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    if constexpr (sizeof(T) == 8)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(sa), "l"(gmem) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// the adjoint of the line x (upwind order) of n cells; lo(j): output cotangent,
// put(j, v): input cotangent without the line maximum's part, which is lfinf to
// position arg; DB: the beta derivative (in the frame of travel) in db
template <typename T, int NMAX, bool PERIODIC, bool DB, class L, class P>
__device__ __forceinline__ void adjoint_line(const T (&x)[NMAX + 1], int n, T fm1, const LineCoef<T> &cf,
                                             L lo, P put, int &arg, T &lfinf, T &db)
{
    const T c0 = cf.c0, c1 = cf.c1, c2 = cf.c2, beta = c0;
    const T dc1 = (T(2) - T(6) * beta + T(3) * beta * beta) / T(6);
    const T dc2 = (T(1) - T(3) * beta * beta) / T(6);
    T finf = T(0);
    arg = 0;
#pragma unroll
    for (int j = 0; j < NMAX; ++j) {
        if (j >= n) break;
        const bool up = less(finf, x[j]);
        finf = pick(up, x[j], finf);
        arg = up ? j : arg;
    }
    const T k1 = twice(c1), k2 = twice(c2), nc1 = negate(c1), nc2 = negate(c2), nk1 = negate(k1),
            nk2 = negate(k2);
    lfinf = T(0);
    db = T(0);
    const T l0first = lo(0);
    T l1 = l0first, dm = PERIODIC ? x[0] - fm1 : x[0];
    T lp = T(0), open = T(0), lmfirst = T(0), first = T(0);
#pragma unroll
    for (int j = 0; j < NMAX; ++j) {
        if (j >= n) break;
        const T l2 = j + 1 < n ? lo(j + 1) : (PERIODIC ? l0first : T(0));
        const T mu = l2 - l1, f0 = x[j], dp = x[j + 1] - f0;
        const T up = twice(f0), gap = twice(finf - f0), nup = negate(up), ngap = negate(gap);
        const bool dpos = less(T(0), dp), dneg = negative(dp);
        const bool mpos = less(T(0), dm), mneg = negative(dm);
        const bool pu = dpos && less(up, dp), pl = dneg && less(dp, ngap);
        const bool mh = mpos && less(gap, dm), ml = mneg && less(dm, nup);
        const bool plim = pu || pl, mlim = mh || ml;
        T l0 = c0 * mu;
        l0 = fused(pick(plim, k1, nc1), mu, l0);
        l0 = fused(pick(mlim, nk2, c2), mu, l0);
        // (the arms at the line maximum are rare: a branch over their terms)
        if (pl) lfinf = fused(nk1, mu, lfinf);
        if (mh) lfinf = fused(k2, mu, lfinf);
        const T lm = pick(mlim, T(0), nc2 * mu);
        if (DB) {
            const T ep = pick(pu, up, pick(pl, ngap, dp)), em = pick(mh, gap, pick(ml, nup, dm));
            if (nonzero(mu)) db = fused(mu, fused(dc2, em, fused(dc1, ep, f0)), db);
        }
        // cell j - 1 is complete with lm
        if (j == 0) {
            lmfirst = lm;
        } else {
            const T done = open + lm;
            if (PERIODIC && j == 1) first = done;
            else put(j - 1, done);
        }
        if (PERIODIC && j == n - 1) lp = lmfirst + lp;
        open = (lp + l1) + l0;
        lp = pick(plim, T(0), c1 * mu);
        l1 = l2;
        dm = dp;
    }
    put(n - 1, open);
    if (PERIODIC) put(0, first + lp);
}

struct AdjLines {
    int n, axis;
    long long stride;          // element stride along the line
    long long nvc;
    int inner;                 // lines per outer index (drift) or per cube (kick)
    int od;                    // drift: outer index o -> first cell (o / od) m1 + (o % od) m2
    long long m1, m2;
    int va_stride, va_n;       // drift: velocity index (v / va_stride) % va_n
    int ny, nz;                // kick
};

// grid: x the chunk of lines and y the outer index (drift), or x the cube and y
// the chunk (kick).  ROWS: lines of stride 1.
template <typename T, int NMAX, bool PERIODIC, bool DB, bool ROWS>
__global__ void __launch_bounds__(128) k_adjoint_lines(const T *__restrict__ fin, T *lam,
                                                      const LineCoef<T> *__restrict__ coef, AdjLines g,
                                                      double *lam_g, double scale)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red[32];
    T *S = reinterpret_cast<T *>(smem_raw);
    const int t = threadIdx.x, NT = blockDim.x, n = g.n, P = n | 1;
    const bool kick = g.axis >= 3;
    const int u0 = (kick ? blockIdx.y : blockIdx.x) * NT, u = u0 + t;
    const bool active = u < g.inner;
    long long off = 0;
    LineCoef<T> cf;
    cf.code = 0;
    if (kick) {
        const long long base = (long long)blockIdx.x * g.nvc;
        cf = coef[(long long)blockIdx.x * 3 + g.axis - 3];
        if (g.axis == 3) off = base + u;
        else if (g.axis == 4) off = base + (long long)(u / g.nz) * g.ny * g.nz + u % g.nz;
        else off = base + (long long)u * n;
    } else {
        const long long o = blockIdx.y;
        off = ((o / g.od) * g.m1 + (o % g.od) * g.m2) * g.nvc + u;
        if (active) cf = coef[(u / g.va_stride) % g.va_n];
    }
    const bool neg = cf.code & 1;
    // entries of the output cotangent before the wrap (periodic) or the end
    const int shift = PERIODIC ? (cf.code >> 1) % n : (cf.code >> 1 < n ? cf.code >> 1 : n), nb = n - shift;
    const long long st = neg ? -g.stride : g.stride, o0 = off + (neg ? (n - 1) * g.stride : 0);
    T x[NMAX + 1], fm1 = T(0);
    int cnt = 0;
    if constexpr (ROWS) {
        // the CTA's rows through the tile, the state first, then the cotangent (read at
        // or past the cell that is written)
        cnt = (g.inner - u0 < NT ? g.inner - u0 : NT) * n;
        const T *src = fin + (off - (long long)t * n);
        const int dr = NT / n, dk = NT - dr * n;
        const int r0 = t / n, c0 = t - r0 * n;
        auto each = [&](auto f) {
            int r = r0, k = c0;
#pragma unroll 4
            for (int e = t; e < cnt; e += NT) {
                f(e, r * P + k);
                r += dr;
                k += dk;
                if (k >= n) { k -= n; ++r; }
            }
        };
        each([&](int e, int q) { copy_async(S + q, src + e); });
        copy_wait();
        __syncthreads();
        const T *row = S + t * P + (neg ? n - 1 : 0);
        const int rs = neg ? -1 : 1;
        if (active) load_line<T, NMAX, false, 1>(x, n, [&]() { const T v = *row; row += rs; return v; });
        __syncthreads();
        T *dst = lam + (off - (long long)t * n);
        each([&](int e, int q) { copy_async(S + q, (const T *)dst + e); });
        copy_wait();
        __syncthreads();
        double da = 0.0;
        if (active) {
            T *l = S + t * P + (neg ? n - 1 : 0);
            int arg;
            T lfinf, db;
            adjoint_line<T, NMAX, false, DB>(
                x, n, T(0), cf, [&](int j) { return j < nb ? l[(j + shift) * rs] : T(0); },
                [&](int j, T v) { l[j * rs] = v; }, arg,
                lfinf, db);
            l[arg * rs] += lfinf;
            da = neg ? -(double)db : (double)db;
        }
        __syncthreads();
        each([&](int e, int q) { dst[e] = S[q]; });
        if (DB) {
            da = block_sum(da, red);
            if (t == 0 && da != 0.0) atomicAdd(lam_g + blockIdx.x, da * scale);
        }
        return;
    }
    double da = 0.0;
    if (active) {
        T *l = S + t;
        {
            const T *p = lam + o0;
            for (int j = 0; j < n; ++j) {
                copy_async(l + j * NT, p);
                p += st;
            }
        }
        const T *p = fin + o0;
        load_line<T, NMAX, PERIODIC, 1>(x, n, [&]() { const T v = *p; p += st; return v; });
        if (PERIODIC) fm1 = fin[o0 + (n - 1) * st];
        copy_wait();
        int arg;
        T lfinf, db;
        adjoint_line<T, NMAX, PERIODIC, DB>(
            x, n, fm1, cf,
            [&](int j) {
                if (!PERIODIC) return j < nb ? l[(j + shift) * NT] : T(0);
                return l[(j < nb ? j + shift : j - nb) * NT];
            },
            [&](int j, T v) { lam[o0 + j * st] = v; }, arg,
            lfinf, db);
        lam[o0 + arg * st] += lfinf;
        da = neg ? -(double)db : (double)db;
    }
    if (DB) {
        da = block_sum(da, red);
        if (t == 0 && da != 0.0) atomicAdd(lam_g + blockIdx.x, da * scale);
    }
}

template <typename T, int NMAX, bool PERIODIC, bool DB, bool ROWS>
cudaError_t go(vp_ctx *c, const T *fin, T *lam, const LineCoef<T> *coef, const AdjLines &g, dim3 grid, int NT,
               double *lam_g, double scale)
{
    const size_t smem = (size_t)NT * (ROWS ? (g.n | 1) : g.n) * sizeof(T);
    auto kern = k_adjoint_lines<T, NMAX, PERIODIC, DB, ROWS>;
    if (smem + 1024 > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 72 * 1024);
        if (e != cudaSuccess) return e;
    }
    kern<<<grid, NT, smem, c->stream>>>(fin, lam, coef, g, lam_g, scale);
    return cudaGetLastError();
}

template <typename T, int NMAX>
cudaError_t lines_n(vp_ctx *c, const T *fin, T *lam, const LineCoef<T> *coef, const AdjLines &g, dim3 grid,
                    int NT, double *lam_g, double scale)
{
    if (g.axis < 3)
        return c->periodic_space ? go<T, NMAX, true, false, false>(c, fin, lam, coef, g, grid, NT, nullptr, 0.0)
                                 : go<T, NMAX, false, false, false>(c, fin, lam, coef, g, grid, NT, nullptr, 0.0);
    if (g.axis == 5)
        return lam_g ? go<T, NMAX, false, true, true>(c, fin, lam, coef, g, grid, NT, lam_g, scale)
                     : go<T, NMAX, false, false, true>(c, fin, lam, coef, g, grid, NT, nullptr, 0.0);
    return lam_g ? go<T, NMAX, false, true, false>(c, fin, lam, coef, g, grid, NT, lam_g, scale)
                 : go<T, NMAX, false, false, false>(c, fin, lam, coef, g, grid, NT, nullptr, 0.0);
}

template <typename T>
cudaError_t lines_t(vp_ctx *c, const T *fin, T *lam, int axis, const LineCoef<T> *coef, double *lam_g,
                    double scale)
{
    AdjLines g{};
    g.axis = axis;
    g.nvc = c->nvc;
    g.ny = c->nv[1];
    g.nz = c->nv[2];
    int NT = 128;
    dim3 grid;
    if (axis < 3) {
        g.n = c->n[axis];
        long long cs = (long long)c->n[1] * c->n[2];
        g.od = 1; g.m1 = 1; g.m2 = 0;
        if (axis == 1) { cs = c->n[2]; g.od = c->n[2]; g.m1 = (long long)c->n[1] * c->n[2]; g.m2 = 1; }
        else if (axis == 2) { cs = 1; g.m1 = c->n[2]; }
        g.stride = cs * c->nvc;
        g.inner = (int)c->nvc;
        g.va_stride = axis == 0 ? c->nv[1] * c->nv[2] : (axis == 1 ? c->nv[2] : 1);
        g.va_n = c->nv[axis];
        coef += (size_t)axis * c->maxnv;
    } else {
        g.n = c->nv[axis - 3];
        g.stride = axis == 3 ? (long long)g.ny * g.nz : (axis == 4 ? g.nz : 1);
        g.inner = (int)(c->nvc / g.n);
        lam_g = lam_g ? lam_g + (size_t)(axis - 3) * c->np : nullptr;
    }
    if (g.inner < NT) NT = (g.inner + 31) / 32 * 32;
    const unsigned chunks = (unsigned)((g.inner + NT - 1) / NT);
    grid = axis < 3 ? dim3(chunks, (unsigned)(c->np / g.n)) : dim3((unsigned)c->np, chunks);
    if (g.n <= 16) return lines_n<T, 16>(c, fin, lam, coef, g, grid, NT, lam_g, scale);
    if (g.n <= 32) return lines_n<T, 32>(c, fin, lam, coef, g, grid, NT, lam_g, scale);
    return lines_n<T, 64>(c, fin, lam, coef, g, grid, NT, lam_g, scale);
}

}  // namespace

int vp_adjoint_lines_ok(const vp_ctx *c, int axis)
{
    const int n = axis < 3 ? c->n[axis] : c->nv[axis - 3];
    // (the grid's y dimension: outer indices for the position axes, chunks of 128
    // lines for the velocity axes; the lines of one outer index count in an int)
    return n >= 3 && n <= 64 && c->nvc <= (1LL << 30) &&
           (axis < 3 ? c->np / n <= 65535 : c->nvc / n <= 65535LL * 128);
}

cudaError_t launch_adjoint_lines(vp_ctx *c, const void *fin, void *lam, int axis, const void *coef,
                                 double *lam_g, double scale)
{
    if (c->isdouble)
        return lines_t<double>(c, (const double *)fin, (double *)lam, axis, (const LineCoef<double> *)coef,
                               lam_g, scale);
    return lines_t<float>(c, (const float *)fin, (float *)lam, axis, (const LineCoef<float> *)coef, lam_g,
                          scale);
}
