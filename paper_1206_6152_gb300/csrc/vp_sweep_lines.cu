// vp_sweep_lines.cu -- sweeps along lines of any length up to 64 cells, one
// line per thread in registers (vp_clamp_line.cuh).  These serve every grid whose
// lengths have no kernel of their own; the shared-memory kernels of vp_sweep.cu
// remain for longer lines and for drifts by one cell or more.
//
//  * k_drift_lines: lines along a spatial axis straight from global memory to
//    registers and back (a warp reads 32 neighbouring velocity cells per
//    load).  Scalar lines, not packed pairs, so that each lane reads its own
//    direction.  FP32: bound by HBM; 20 x 18 x 22 positions of 24 x 28 x 26
//    velocity cells 0.30 -> 0.21 ms a sweep (5.3 TB/s) against the shared-memory
//    kernel.  Indices by multiplication (FastDiv): with 64-bit divisions, about a
//    hundred instructions each, lines of 4 to 20 cells were bound by issue (x drift
//    of 4 x 64^2 of 32^3 cells 1.65 -> 1.36 ms, 8 x 8 x 4 of 48^3, z 95 -> 80, x 60 ->
//    53 us).  FP64: at the FP64 pipe's rate (7.3 instructions per cell counted,
//    64 cycles each per quadrant's warp); 20 x 18 x 22 of the same 1.48 -> 0.86
//    ms, and FP64 lines of 16 and 32 go through here as well: the saturating
//    form takes 9 FP64 instructions and a reciprocal per line, and the z drift
//    ran both directions' code in every warp (16^6: 0.59 -> 0.25 ms).
//  * k_kick_lines: one velocity sweep of every cube, the same way (vx and vy
//    lines: a warp reads neighbouring cells; vz: each thread its own row, whose
//    32-byte sectors it uses up over consecutive loads).  FP64 cubes go through it
//    one launch per sweep: at 16 bytes per cell the sweep is bound by the FP64 pipe
//    alone.  A line that moves by whole cells is held in registers as well
//    (shifted_line): in place in global memory, sweeps of 24 x 28 x 26 cubes by 1.5
//    cells took 420 us where one by 0.4 of a cell takes 250, now 285.
//  * k_kick_blocks: FP32 cubes in blocks of vx planes in shared memory: whole
//    cubes, all sweeps of a kick in one pass, where they fit (220 KB); larger
//    ones as one pass per vx sweep (k_kick_lines) and one per run of vy and vz
//    sweeps (both inside a vx plane).  Bound by issue (about 30 instructions per
//    cell and sweep, 15 of them the flux and update), so the line loops go in
//    whole groups of four cells where NMAX fits the lines, and the tile is
//    addressed as shared memory.  Fused six-sweep kick against the shared-memory
//    lines of vp_sweep.cu: 24 x 28 x 26 cubes (553 MB of f) 1.83 -> 0.89 ms, 24^3
//    (764 MB) 2.77 -> 1.15 ms.
//  * k_kick_planes: the vy and vz sweeps of cubes too large for that whose vx planes are
//    40^2, 48^2, 56^2 or 64^2, at compile-time length.  With k_kick_lines along vx, fused
//    kick: 40^3 (1.05 GB) 5.2 -> 1.76 ms, 64^3 (537 MB) 2.53 -> 0.84 ms.
#include <cuda_runtime.h>

#include "vp_clamp_line.cuh"
#include "vp_device.cuh"
#include "vp_fast_line.cuh"
#include "vp_internal.cuh"
#include "vp_line.cuh"

using namespace vpline;

int vp_sm_count();

namespace {

// What a thread's lines lose through the outflow ends, over all of its lines.
// FP32 sums are kept and merged as double-floats on the FP32 pipe, one FP64
// addition per warp at the end.  FP64: merging a CTA's threads takes about 50
// FP64 instructions a warp, so it is done once per CTA of a grid that just
// fills the SMs, not once per line.  Both merges shuffle whole warps: a CTA has a
// multiple of 32 threads (a lane that does not exist has no defined value).
template <typename T>
struct Lost;
template <>
struct Lost<float> {
    Acc<float> a;
    __device__ __forceinline__ void add(float v) { a.add(v); }
};
template <>
struct Lost<double> {
    double a = 0.0;
    __device__ __forceinline__ void add(double v) { a += v; }
};

__device__ __forceinline__ void add_lost(Lost<float> lost, double *lost_out)
{
    __shared__ double red[32];
    for (int d = 16; d > 0; d >>= 1) lost.a.shfl_merge(d);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = lost.a.value();
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x + 31) / 32; ++w) s += red[w];
        if (s != 0.0) atomicAdd(lost_out, s);
    }
}

__device__ __forceinline__ void add_lost(const Lost<double> &lost, double *lost_out)
{
    __shared__ Acc<double> red[32];
    Acc<double> a;
    a.add(lost.a);
    a = block_merge(a, red);
    if (threadIdx.x == 0 && a.value() != 0.0) atomicAdd(lost_out, a.value());
}

// *p, and p stepped on through an opaque register (the compiler would
// otherwise keep every address of a line live from its loads to its stores)
template <typename T, typename S>
__device__ __forceinline__ T next(const T *&p, S st)
{
    const T v = *p;
    p += st;
    asm volatile("" : "+l"(p));
    return v;
}

struct LinesGeom {
    int n;                     // cells per line
    long long cell_stride;     // spatial-cell stride along the line
    int od;                    // outer index o -> first cell: (o / od) m1 + (o % od) m2
    long long m1, m2;
    int nvc;                   // velocity cells per spatial cell
    FastDiv by_nvc, by_od;
    VelIndex vel;              // velocity index along the axis
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
        const int o = q < (1LL << 31) ? (int)g.by_nvc((unsigned)q) : (int)(q / g.nvc);
        const int v = (int)(q - (long long)o * g.nvc), oh = (int)g.by_od((unsigned)o);
        const LineCoef<T> cf = coef[g.vel(v)];
        const bool neg = cf.code & 1;
        const long long off = (oh * g.m1 + (o - oh * g.od) * g.m2) * g.nvc + v +
                              (neg ? (n - 1) * step : 0);
        const long long st = neg ? -step : step;
        T x[NMAX + 1];
        const T *p = f + off;
        load_line<T, NMAX, PERIODIC, 1>(x, n, [&]() { return next(p, st); });
        T fm1 = T(0), fm2 = T(0);
        if (PERIODIC) {
            fm1 = f[off + (n - 1) * st];
            fm2 = f[off + (n > 1 ? n - 2 : 0) * st];
        }
        T *w = fo + off;
        const T out = clamp_line<T, NMAX, PERIODIC, 1>(x, n, fm1, fm2, cf.c0, cf.c1, cf.c2, [&](int, T u) {
            *w = u;
            w += st;
            asm volatile("" : "+l"(w));
        });
        if (!PERIODIC) lost.add(out);
        if (!drift_persistent<T, PERIODIC>()) break;
    }
    if (!PERIODIC) add_lost(lost, lost_out);
}

// CTAs per SM that the sub-cell code alone leaves room for (the function for lines that
// move by whole cells would take registers of its own beyond that)
template <typename T, int NMAX>
constexpr int kick_lines_ctas()
{
    if (sizeof(T) == 8) return NMAX <= 16 ? 7 : (NMAX <= 32 ? 4 : 3);
    return NMAX <= 16 ? 10 : (NMAX <= 32 ? 8 : (NMAX <= 48 ? 6 : 5));
}

template <typename T, int NMAX>
__global__ void __launch_bounds__(128, kick_lines_ctas<T, NMAX>()) k_kick_lines(const T *src, T *dst,
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
        const bool neg = cf.code & 1;
        const int st = neg ? -step : step;
        const T *p = src + off + (neg ? (n - 1) * step : 0);
        T *w = dst + off + (neg ? (n - 1) * step : 0);
        if ((cf.code >> 1) != 0) {
            lost.add(shifted_line<T, NMAX>(p, st, w, st, n, cf));
            continue;
        }
        T x[NMAX + 1];
        load_line<T, NMAX, false, 1>(x, n, [&]() { return next(p, st); });
        lost.add(clamp_line<T, NMAX, false, 1>(x, n, T(0), T(0), cf.c0, cf.c1, cf.c2, [&](int, T v) {
            *w = v;
            w += st;
            asm volatile("" : "+l"(w));
        }));
    }
    add_lost(lost, lost_out);
}

// A block of G vx planes of a velocity cube (all of them: the whole cube) in
// shared memory, rows at pitch nz | 1 (rows and columns free of bank
// conflicts), one line per thread at a time.
struct Block {
    int g, ny, nz;         // planes, rows, cells per row
    // the lines along axis va: how many, their length, line u's first cell and
    // its step in an array of row pitch P
    __device__ __forceinline__ int lines(int va) const { return va == 0 ? ny * nz : (va == 1 ? g * nz : g * ny); }
    __device__ __forceinline__ int len(int va) const { return va == 0 ? g : (va == 1 ? ny : nz); }
    __device__ __forceinline__ int step(int va, int P) const { return va == 0 ? ny * P : (va == 1 ? P : 1); }
    __device__ __forceinline__ int first(int va, int u, int P) const
    {
        if (va == 2) return u * P;
        const int r = u / nz, k = u - r * nz;
        return (va == 0 ? r : r * ny) * P + k;
    }
};

// f(e, tile offset) for every element e of rows of nz cells; element e lies in
// row r at tile offset e + r (P - nz), r stepped along instead of divided out
// (a division per element took longer than the sweeps: vz alone of 64^3
// cubes, 537 MB of traffic, 1.06 -> 0.45 ms)
template <class F>
__device__ __forceinline__ void each_element(int count, int nz, F f)
{
    const int NT = blockDim.x, pad = (nz | 1) - nz, dr = NT / nz, dk = NT - dr * nz;
    int r = threadIdx.x / nz, k = threadIdx.x - r * nz;
#pragma unroll 4
    for (int e = threadIdx.x; e < count; e += NT) {
        f(e, e + r * pad);
        r += dr;
        k += dk;
        if (k >= nz) { k -= nz; ++r; }
    }
}

// one sweep of the block's lines along va, from src (IN) or the tile, into dst
// (OUT) or the tile; which one it is is known at compile time, so that the tile
// is addressed as shared memory (with one generic pointer for both a cell took
// 35 instructions and the 24 x 28 x 26 kick 1.14 ms).  SHIFT: lines that move by
// whole cells, in the tile
template <int NMAX, bool IN, bool OUT, bool SHIFT = false>
__device__ __forceinline__ void sweep_lines(const Block &B, int va, const float *src, float *dst, float *tile,
                            const LineCoef<float> &c, Lost<float> &lost)
{
    constexpr int GR = NMAX <= 32 ? 4 : 1;
    const int nz = B.nz, P = nz | 1, n = B.len(va), L = B.lines(va), neg = c.code & 1;
    const int sp = neg ? -B.step(va, P) : B.step(va, P), sg = neg ? -B.step(va, nz) : B.step(va, nz);
    for (int u = threadIdx.x; u < L; u += blockDim.x) {
        const int a = B.first(va, u, P) + (neg ? (1 - n) * sp : 0);
        const int g = IN || OUT ? B.first(va, u, nz) + (neg ? (1 - n) * sg : 0) : 0;
        if constexpr (SHIFT && NMAX > 32) {
            lost.add(shifted_line<float, NMAX>(tile + a, sp, tile + a, sp, n, c));
            continue;
        }
        float x[NMAX + 1];
        if constexpr (IN) {
            const float *p = src + g;
            load_line<float, NMAX, false, GR>(x, n, [&]() { return next(p, sg); });
        } else {
            int q = 4 * a;
            load_line<float, NMAX, false, GR>(x, n, [&]() {
                const float v = *reinterpret_cast<const float *>(reinterpret_cast<const char *>(tile) + q);
                q += 4 * sp;
                asm volatile("" : "+r"(q));
                return v;
            });
        }
        if constexpr (SHIFT) {
            const int s = c.code >> 1 < n ? c.code >> 1 : n;
            for (int j = 0; j < s; ++j) tile[a + j * sp] = 0.f;
            int q = 4 * (a + s * sp);
            lost.add(clamp_line_shifted<float, NMAX>(x, n, s, c.c0, c.c1, c.c2, [&](float v) {
                *reinterpret_cast<float *>(reinterpret_cast<char *>(tile) + q) = v;
                q += 4 * sp;
                asm volatile("" : "+r"(q));
            }));
            continue;
        }
        float *w = dst + g;
        int r = 4 * a;
        lost.add(clamp_line<float, NMAX, false, GR>(x, n, 0.f, 0.f, c.c0, c.c1, c.c2, [&](int, float v) {
            if constexpr (OUT) {
                *w = v;
                w += sg;
                asm volatile("" : "+l"(w));
            } else {
                *reinterpret_cast<float *>(reinterpret_cast<char *>(tile) + r) = v;
                r += 4 * sp;
                asm volatile("" : "+r"(r));
            }
        }));
    }
}

// nsweeps consecutive sweeps first_axis, first_axis + 1, ... (mod 3) of a
// block, from src (global, pitch nz) into dst.  The first sweep reads vx or vy
// lines, and the last one writes them, straight from and to global memory
// (coalesced along vz); vz rows, and sweeps that move by whole cells, go
// through the tile.  Starts and ends with the tile free.
template <int NMAX>
__device__ __forceinline__ void sweep_block(const Block &B, const float *src, float *dst, float *tile,
                                            const LineCoef<float> *cf, int nsweeps, int first_axis,
                                            Lost<float> &lost)
{
    const int nz = B.nz, rows = B.g * B.ny;
    auto whole = [&](int sw) { return (cf[sw].code >> 1) != 0; };
    const bool in = first_axis < 2 && !whole(0);
    if (!in) {
        each_element(rows * nz, nz, [&](int e, int q) { tile[q] = src[e]; });
        __syncthreads();
    }
    bool out = false;
    for (int sw = 0; sw < nsweeps; ++sw) {
        const int va = (first_axis + sw) % 3;
        const LineCoef<float> c = cf[sw];
        out = sw == nsweeps - 1 && va < 2 && !whole(sw);
        if (whole(sw)) {
            sweep_lines<NMAX, false, false, true>(B, va, src, dst, tile, c, lost);
        } else if (sw == 0 && in) {
            if (out) sweep_lines<NMAX, true, true>(B, va, src, dst, tile, c, lost);
            else sweep_lines<NMAX, true, false>(B, va, src, dst, tile, c, lost);
        } else if (out) {
            sweep_lines<NMAX, false, true>(B, va, src, dst, tile, c, lost);
        } else {
            sweep_lines<NMAX, false, false>(B, va, src, dst, tile, c, lost);
        }
        __syncthreads();
    }
    if (!out) {
        each_element(rows * nz, nz, [&](int e, int q) { dst[e] = tile[q]; });
        __syncthreads();
    }
}

// FP32 cubes in blocks of G vx planes (G = nx: whole cubes), nsweeps <= 6
// sweeps per block; tables ca for the first three sweeps of the kick, cb after
// (k0: how many sweeps of the kick came before)
template <int NMAX>
__global__ void __launch_bounds__(512) k_kick_blocks(const float *src, float *dst,
                                                    const LineCoef<float> *__restrict__ ca,
                                                    const LineCoef<float> *__restrict__ cb, int k0,
                                                    int nsweeps, int first_axis, int nx, int ny, int nz,
                                                    int G, long long np, double *lost_out)
{
    extern __shared__ float tile[];
    __shared__ LineCoef<float> scf[6];
    const int per = (nx + G - 1) / G;
    Lost<float> lost;
    for (long long u = blockIdx.x; u < np * per; u += gridDim.x) {
        const long long cell = u / per;
        const int i0 = (int)(u - cell * per) * G;
        if (threadIdx.x < nsweeps)
            scf[threadIdx.x] = (k0 + (int)threadIdx.x < 3 ? ca : cb)[cell * 3 + (first_axis + threadIdx.x) % 3];
        __syncthreads();
        const Block B{nx - i0 < G ? nx - i0 : G, ny, nz};
        const long long off = (cell * nx + i0) * ny * (long long)nz;
        sweep_block<NMAX>(B, src + off, dst + off, tile, scf, nsweeps, first_axis, lost);
    }
    add_lost(lost, lost_out);
}

// The vy (do1) and vz (do2) sweeps of FP32 cubes whose vx planes are N x N, N
// known at compile time (no test and no address arithmetic per cell: 18
// instructions instead of 30), persistent CTAs of two planes at a time: vy lines
// from global memory (coalesced along vz), through the tile (row pitch N + 4: 16
// bytes aligned, rows free of bank conflicts) to vz rows read and written 16
// bytes at a time, and out of it with coalesced 16-byte stores; the CTA's next
// planes are fetched into L2 meanwhile.  CTAs of whole warps, as add_lost's merge
// needs: two planes of 40 or 56 lines leave 16 threads that take no line and join the
// barriers and the merge only.
template <int N>
struct Planes {
    static constexpr int G = 2, NT = (G * N + 31) / 32 * 32, P = N + 4;
    static constexpr size_t SMEM = (size_t)G * N * P * sizeof(float);
    static constexpr int CTAS = N <= 40 ? 9 : (N <= 48 ? 8 : (N <= 56 ? 6 : 4));   // as kick_lines_ctas
};

template <int N>
__device__ __forceinline__ float sweep_exact(float (&x)[N], const LineCoef<float> &c)
{
    const float finf = line_max(x);
    return c.code & 1 ? clamp_exact<N, true>(x, finf, c.c0, c.c1, c.c2)
                      : clamp_exact<N, false>(x, finf, c.c0, c.c1, c.c2);
}

template <int N>
__global__ void __launch_bounds__(Planes<N>::NT, Planes<N>::CTAS) k_kick_planes(const float *src, float *dst,
                                                               const LineCoef<float> *__restrict__ coef,
                                                               int do1, int do2, int nx, long long np,
                                                               double *lost_out)
{
    typedef Planes<N> B;
    static_assert(B::NT % 32 == 0, "add_lost merges whole warps");
    constexpr int P = B::P, NN = N * N, Q = N / 4;
    extern __shared__ __align__(16) float tile[];
    const int t = threadIdx.x, g = t / N, m = t % N, per = (nx + B::G - 1) / B::G;
    Lost<float> lost;
    for (long long u = blockIdx.x; u < np * per; u += gridDim.x) {
        const long long cell = u / per;
        const int i0 = (int)(u - cell * per) * B::G, planes = nx - i0 < B::G ? nx - i0 : B::G;
        const LineCoef<float> c1 = coef[cell * 3 + 1], c2 = coef[cell * 3 + 2];
        const long long off = (cell * nx + i0) * NN, un = u + gridDim.x;
        const float *s = src + off;
        float *d = dst + off;
        // (uniform over the CTA) a sweep that moves by whole cells: lines in upwind order
        const bool shifted = (do1 && (c1.code >> 1) != 0) || (do2 && (c2.code >> 1) != 0);
        float x[N];
        if (g < planes && !shifted) {
            // vy line (plane g, vz = m)
#pragma unroll
            for (int j = 0; j < N; ++j) x[j] = s[g * NN + j * N + m];
            if (do1) lost.add(sweep_exact<N>(x, c1));
#pragma unroll
            for (int j = 0; j < N; ++j) tile[(g * N + j) * P + m] = x[j];
        } else if (g < planes) {
            const int j0 = c1.code & 1 ? N - 1 : 0, d1 = c1.code & 1 ? -1 : 1;
            const float *p = s + (g * N + j0) * N + m;
            float *q = tile + (g * N + j0) * P + m;
            if (do1) lost.add(shifted_line<float, N>(p, d1 * N, q, d1 * P, N, c1));
            else
                for (int j = 0; j < N; ++j) q[j * d1 * P] = p[j * d1 * N];
        }
        if (t == 0 && un < np * per) {
            const long long cn = un / per;
            const int in = (int)(un - cn * per) * B::G;
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src + (cn * nx + in) * NN),
                         "r"((nx - in < B::G ? nx - in : B::G) * NN * 4)
                         : "memory");
        }
        __syncthreads();
        if (do2 && g < planes && !shifted) {
            // vz row (plane g, vy = m)
            float4 *r = reinterpret_cast<float4 *>(tile + (g * N + m) * P);
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const float4 v = r[q];
                x[4 * q] = v.x; x[4 * q + 1] = v.y; x[4 * q + 2] = v.z; x[4 * q + 3] = v.w;
            }
            lost.add(sweep_exact<N>(x, c2));
#pragma unroll
            for (int q = 0; q < Q; ++q)
                r[q] = make_float4(x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]);
        } else if (do2 && g < planes) {
            const int d2 = c2.code & 1 ? -1 : 1;
            float *r = tile + (g * N + m) * P + (c2.code & 1 ? N - 1 : 0);
            lost.add(shifted_line<float, N>(r, d2, r, d2, N, c2));
        }
        __syncthreads();
#pragma unroll 4
        for (int e = t; e < planes * N * Q; e += B::NT) {
            const int row = e / Q, q = e - row * Q;
            reinterpret_cast<float4 *>(d)[e] = *reinterpret_cast<const float4 *>(tile + row * P + 4 * q);
        }
        __syncthreads();
    }
    add_lost(lost, lost_out);
}

// CTAs of 128 threads, one line per thread at a time: as many as there are
// lines for, or with persistent only those that fit on the GPU at once.  The
// persistent grid pays where every CTA ends with a merge of its losses (FP64
// kicks of 20 x 18 x 22 cubes 1.14 -> 0.83 ms).  More CTAs than a grid holds (over a
// terabyte of f) are an error: kernels launched without persistent take one line each.
template <class K>
cudaError_t lines_grid(K kernel, long long lines, bool persistent, unsigned &grid)
{
    const long long g = (lines + 127) / 128;
    if (!persistent) {
        grid = (unsigned)g;
        return g <= 0x7fffffffLL ? cudaSuccess : cudaErrorInvalidConfiguration;
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
    auto kern = k_kick_lines<T, 64>;
    if (n <= 16) kern = k_kick_lines<T, 16>;
    else if (n <= 32) kern = k_kick_lines<T, 32>;
    else if (n <= 48) kern = k_kick_lines<T, 48>;
    unsigned grid;
    const cudaError_t e = lines_grid(kern, c->np * (c->nvc / n), true, grid);
    if (e != cudaSuccess) return e;
    kern<<<grid, 128, 0, c->stream>>>(src, dst, coef, va, c->nv[0], c->nv[1], c->nv[2], c->np,
                                      &c->sc->lost);
    return cudaGetLastError();
}

cudaError_t kick_blocks(vp_ctx *c, const float *src, float *dst, const LineCoef<float> *ca,
                        const LineCoef<float> *cb, int k0, int nsweeps, int first_axis, int G)
{
    const int nx = c->nv[0], ny = c->nv[1], nz = c->nv[2];
    const size_t smem = (size_t)G * ny * (nz | 1) * sizeof(float);
    int lmax = G * (ny > nz ? ny : nz);              // most lines of one sweep
    if (G == nx && ny * nz > lmax) lmax = ny * nz;
    // a CTA alone on its SM gets 16 warps, CTAs that share one 8 at most
    int threads = (lmax + 31) / 32 * 32;
    const int cap = smem > 110 * 1024 ? 512 : 256;
    if (threads > cap) threads = cap;
    auto kern = k_kick_blocks<64>;
    if (c->maxnv <= 16) kern = k_kick_blocks<16>;
    else if (c->maxnv <= 24) kern = k_kick_blocks<24>;
    else if (c->maxnv <= 32) kern = k_kick_blocks<32>;
    else if (c->maxnv <= 48) kern = k_kick_blocks<48>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    long long grid = (long long)per_sm * vp_sm_count();
    const long long units = c->np * ((nx + G - 1) / G);
    if (grid > units) grid = units;
    kern<<<(unsigned)grid, threads, smem, c->stream>>>(src, dst, ca, cb, k0, nsweeps, first_axis, nx, ny,
                                                       nz, G, c->np, &c->sc->lost);
    return cudaGetLastError();
}

template <int N>
cudaError_t kick_planes(vp_ctx *c, const float *src, float *dst, const LineCoef<float> *coef, int do1, int do2)
{
    typedef Planes<N> B;
    cudaError_t e = cudaFuncSetAttribute(k_kick_planes<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)B::SMEM);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_kick_planes<N>, B::NT, B::SMEM);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    long long grid = (long long)per_sm * vp_sm_count();
    const long long units = c->np * ((c->nv[0] + B::G - 1) / B::G);
    if (grid > units) grid = units;
    k_kick_planes<N><<<(unsigned)grid, B::NT, B::SMEM, c->stream>>>(src, dst, coef, do1, do2, c->nv[0], c->np,
                                                                    &c->sc->lost);
    return cudaGetLastError();
}

// 1 for vx planes of 40^2, 48^2, 56^2 or 64^2 cells (multiples of 8 whose cubes
// do not fit in shared memory) in 16-byte aligned arrays
int planes_ok(const vp_ctx *c, const void *src, const void *dst)
{
    const int n = c->nv[1];
    return n == c->nv[2] && (n == 40 || n == 48 || n == 56 || n == 64) &&
           (((uintptr_t)src | (uintptr_t)dst) & 15) == 0;
}

// FP32: whole cubes in one pass where they fit in shared memory; else one
// pass per vx sweep (register lines) and one per run of vy and vz sweeps (both
// inside a vx plane; blocks of enough planes for four warps of lines)
cudaError_t kick_lines_f32(vp_ctx *c, const float *src, float *dst, const LineCoef<float> *ca,
                           const LineCoef<float> *cb, int nsweeps, int first_axis)
{
    const int nx = c->nv[0], ny = c->nv[1], nz = c->nv[2];
    if ((size_t)nx * ny * (nz | 1) * sizeof(float) <= 220 * 1024)
        return kick_blocks(c, src, dst, ca, cb, 0, nsweeps, first_axis, nx);
    int G = 128 / (ny < nz ? ny : nz);
    if (G < 1) G = 1;
    if (G > nx) G = nx;
    for (int sw = 0; sw < nsweeps;) {
        const int va = (first_axis + sw) % 3;
        int run = 1;
        cudaError_t e;
        if (va == 0) {
            e = kick_lines_t<float>(c, src, dst, sw < 3 ? ca : cb, 0);
        } else {
            if (va == 1 && sw + 1 < nsweeps) run = 2;
            const LineCoef<float> *cf = sw < 3 ? ca : cb;   // (a run belongs to one half kick)
            const int do1 = va == 1, do2 = va == 2 || run == 2;
            if (!planes_ok(c, src, dst)) e = kick_blocks(c, src, dst, ca, cb, sw, run, va, G);
            else if (nz == 40) e = kick_planes<40>(c, src, dst, cf, do1, do2);
            else if (nz == 48) e = kick_planes<48>(c, src, dst, cf, do1, do2);
            else if (nz == 56) e = kick_planes<56>(c, src, dst, cf, do1, do2);
            else e = kick_planes<64>(c, src, dst, cf, do1, do2);
        }
        if (e != cudaSuccess) return e;
        src = dst;              // the first pass reads src, the rest dst
        sw += run;
    }
    return cudaSuccess;
}

template <typename T, bool PERIODIC>
cudaError_t drift_lines_p(vp_ctx *c, const T *f, const LineCoef<T> *coef, const LinesGeom &g, T *fo)
{
    auto kern = k_drift_lines<T, 64, PERIODIC>;
    if (g.n <= 16) kern = k_drift_lines<T, 16, PERIODIC>;
    else if (g.n <= 32) kern = k_drift_lines<T, 32, PERIODIC>;
    else if (g.n <= 48) kern = k_drift_lines<T, 48, PERIODIC>;
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
    g.by_nvc = FastDiv(g.nvc);
    g.by_od = FastDiv(g.od);
    g.vel = VelIndex(axis == 0 ? c->nv[1] * c->nv[2] : (axis == 1 ? c->nv[2] : 1), c->nv[axis]);
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

// velocity cubes with no axis longer than 64
int vp_kick_lines_ok(const vp_ctx *c) { return c->maxnv <= 64; }

cudaError_t launch_kick_lines(vp_ctx *c, const void *f, const void *ca, const void *cb, int nsweeps,
                              int first_axis, void *fo)
{
    if (!c->isdouble)
        return kick_lines_f32(c, (const float *)f, (float *)fo, (const LineCoef<float> *)ca,
                              (const LineCoef<float> *)cb, nsweeps, first_axis);
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
