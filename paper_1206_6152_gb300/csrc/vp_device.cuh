// vp_device.cuh -- device helpers: the PFC flux of one cell, compensated
// accumulators and block reductions.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include "vp_internal.cuh"

// ---------------------------------------------------------------------------
// FP64 minimum and maximum on the integer pipes: an FP64 instruction takes 64 cycles of
// a quadrant's FP64 pipe per warp, however few lanes are active (measured with the SM's
// clock counter: 64.0 with one to four warps per quadrant), and a comparison of
// two doubles is exact on a key of their bits that orders every non-NaN
// double as its value (-0 below +0).  vmin/vmax: these for double, the FP32
// instructions for float.
// ---------------------------------------------------------------------------
__device__ __forceinline__ long long dkey(double x)
{
    const long long b = __double_as_longlong(x);
    return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ double vmin(double a, double b) { return dkey(b) < dkey(a) ? b : a; }
__device__ __forceinline__ double vmax(double a, double b) { return dkey(b) > dkey(a) ? b : a; }
__device__ __forceinline__ float vmin(float a, float b) { return fminf(a, b); }
__device__ __forceinline__ float vmax(float a, float b) { return fmaxf(a, b); }

// ---------------------------------------------------------------------------
// n / d for 0 <= n < 2^31 by a divisor known on the host (Granlund & Montgomery,
// "Division by invariant integers using multiplication", 1994): a multiplication,
// an addition and a shift, where a 64-bit division takes about a hundred
// instructions, as many as four to eight cells of a sweep.
// ---------------------------------------------------------------------------
struct FastDiv {
    unsigned m = 1, s = 0;      // (d = 1)
    FastDiv() = default;
    explicit FastDiv(unsigned d)
    {
        while ((1ull << s) < d) ++s;
        m = (unsigned)(((1ull << 32) * ((1ull << s) - d)) / d + 1);
    }
    __device__ __forceinline__ unsigned operator()(unsigned n) const { return (__umulhi(m, n) + n) >> s; }
};

// index along an axis of velocity cell v: (v / stride) % n
struct VelIndex {
    FastDiv by_stride, by_n;
    int stride = 1, n = 1;
    VelIndex() = default;
    VelIndex(int stride_, int n_) : by_stride(stride_), by_n(n_), stride(stride_), n(n_) {}
    __device__ __forceinline__ int operator()(long long v) const
    {
        if (v >= (1LL << 31)) return (int)((v / stride) % n);
        const unsigned a = by_stride((unsigned)v);
        return (int)(a - by_n(a) * (unsigned)n);
    }
};

// Blocks of the fused y and z drifts: block b = (x plane, chunk of vc velocity cells of one
// vz row), chunks fastest.
struct YZBlocks {
    long long nvb = 1;          // chunks per x plane (below 2^31)
    FastDiv by_nvb, by_row, by_nvy;
    int row = 1, nvy = 1;       // chunks per vz row
    YZBlocks(long long nvc, int nvy_, int nvz, int vc)
        : nvb(nvc / vc), by_nvb((unsigned)(nvc / vc)), by_row(nvz / vc), by_nvy(nvy_), row(nvz / vc), nvy(nvy_)
    {
    }
    __device__ __forceinline__ void split(long long b, long long &x, unsigned &chunk) const
    {
        x = b < (1LL << 31) ? by_nvb((unsigned)b) : b / nvb;
        chunk = (unsigned)(b - x * nvb);
    }
    // vy index of a chunk and its first vz index in units of chunks
    __device__ __forceinline__ void velocity(unsigned chunk, int &vy, int &vzc) const
    {
        const unsigned r = by_row(chunk);
        vzc = (int)(chunk - r * (unsigned)row);
        vy = (int)(r - by_nvy(r) * (unsigned)nvy);
    }
};

// ---------------------------------------------------------------------------
// PFC partial flux of cell j (Sec. 2.1): the integral of the third-order
// reconstruction over the fraction beta of cell j that crosses its downwind
// face, in units of the cell average.  The slope corrector of Filbet,
// Sonnendruecker & Bertrand (2001) is written as clamps of the one-sided
// differences:
//   E+ = clamp(f_{j+1} - f_j, -2 (finf - f_j), 2 f_j)
//   E- = clamp(f_j - f_{j-1}, -2 f_j, 2 (finf - f_j))
//   phi_j = c0 f_j + c1 E+ + c2 E-,
// with finf the maximum of f over the line.  In exact arithmetic 0 <= phi_j
// <= f_j; the final clamp only removes rounding excursions, so that the
// update (f_j - phi_j) + phi_{j-1} is never negative.
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ T pfc_flux(T fm, T f0, T fp, T finf, T c0, T c1, T c2)
{
    const T a = f0 + f0;
    const T b = (finf - f0) * T(2);
    const T ep = vmin(vmax(fp - f0, -b), a);
    const T em = vmin(vmax(f0 - fm, -a), b);
    T phi = c0 * f0 + c1 * ep + c2 * em;
    return vmin(vmax(phi, T(0)), f0);
}

// ---------------------------------------------------------------------------
// compensated accumulation.  float: a double-float pair (s, e) built with
// Knuth's TwoSum; the inputs are exact floats, so the pair carries about 48
// bits.  double: Neumaier's compensated sum.
// ---------------------------------------------------------------------------
template <typename T>
struct Acc;

template <>
struct Acc<float> {
    float s = 0.f, e = 0.f;
    __device__ __forceinline__ void add(float x)
    {
        const float t = s + x;
        const float bb = t - s;
        const float err = (s - (t - bb)) + (x - bb);
        s = t;
        e += err;
    }
    __device__ __forceinline__ void merge(const Acc<float> &o)
    {
        const float t = s + o.s;
        const float bb = t - s;
        const float err = (s - (t - bb)) + (o.s - bb);
        s = t;
        e += o.e + err;
    }
    __device__ __forceinline__ double value() const { return (double)s + (double)e; }
    __device__ __forceinline__ void shfl_merge(int delta)
    {
        Acc<float> o;
        o.s = __shfl_xor_sync(0xffffffffu, s, delta);
        o.e = __shfl_xor_sync(0xffffffffu, e, delta);
        merge(o);
    }
};

template <>
struct Acc<double> {
    double s = 0.0, c = 0.0;
    // Neumaier's sum with the larger operand chosen by its exponent (that is
    // all the error term needs to be exact) on the integer pipes: four FP64
    // instructions of 64 pipe cycles each; comparing and subtracting in both
    // orders took eight
    __device__ __forceinline__ void add(double x)
    {
        const double t = s + x;
        const int sh = __double2hiint(s), sl = __double2loint(s);
        const int xh = __double2hiint(x), xl = __double2loint(x);
        const bool ge = (sh & 0x7fffffff) >= (xh & 0x7fffffff);
        const double big = __hiloint2double(ge ? sh : xh, ge ? sl : xl);
        const double small = __hiloint2double(ge ? xh : sh, ge ? xl : sl);
        c += (big - t) + small;
        s = t;
    }
    __device__ __forceinline__ void merge(const Acc<double> &o)
    {
        add(o.s);
        c += o.c;
    }
    __device__ __forceinline__ double value() const { return s + c; }
    __device__ __forceinline__ void shfl_merge(int delta)
    {
        Acc<double> o;
        o.s = __shfl_xor_sync(0xffffffffu, s, delta);
        o.c = __shfl_xor_sync(0xffffffffu, c, delta);
        merge(o);
    }
};

// Block-wide merge of Acc values; the result is valid in thread 0.
// `scratch` must hold 32 entries of Acc<T>.
template <typename T>
__device__ __forceinline__ Acc<T> block_merge(Acc<T> a, Acc<T> *scratch)
{
    for (int d = 16; d > 0; d >>= 1) a.shfl_merge(d);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nwarps = (blockDim.x + 31) >> 5;
    __syncthreads();
    if (lane == 0) scratch[warp] = a;
    __syncthreads();
    if (warp == 0) {
        Acc<T> b;
        if (lane < nwarps) b = scratch[lane];
        for (int d = 16; d > 0; d >>= 1) b.shfl_merge(d);
        a = b;
    }
    return a;
}

// Block-wide sum of a double (result in thread 0).  scratch: 32 doubles.
__device__ __forceinline__ double block_sum(double v, double *scratch)
{
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nwarps = (blockDim.x + 31) >> 5;
    __syncthreads();
    if (lane == 0) scratch[warp] = v;
    __syncthreads();
    if (warp == 0) {
        v = lane < nwarps ? scratch[lane] : 0.0;
        for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    }
    return v;
}

__device__ __forceinline__ double block_max(double v, double *scratch)
{
    for (int d = 16; d > 0; d >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, d));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nwarps = (blockDim.x + 31) >> 5;
    __syncthreads();
    if (lane == 0) scratch[warp] = v;
    __syncthreads();
    if (warp == 0) {
        v = lane < nwarps ? scratch[lane] : 0.0;
        for (int d = 16; d > 0; d >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, d));
    }
    return v;
}

// x / 6, correctly rounded for normal x and quotient: the quotient by the
// rounded reciprocal and one residual correction (Brisebarre, Muller & Raina,
// "Accelerating correctly rounded floating-point division when the divisor is
// known in advance", 2004).  Three FP64 instructions, 64 cycles of the FP64
// pipe each per warp, where a division takes about three times as many.
__device__ __forceinline__ double div6(double x)
{
    const double z = 1.0 / 6.0, q = x * z;
    return fma(fma(-6.0, q, x), z, q);
}

// Shift alpha = u tau / h as LineCoef (FP64 in, the storage type out).
template <typename T>
__device__ __forceinline__ LineCoef<T> make_line_coef(double alpha)
{
    LineCoef<T> c;
    const int neg = alpha < 0.0;
    double a = fabs(alpha);
    if (!(a < 1.0e8)) a = 1.0e8;          // also catches NaN: no motion past this
    const double s = floor(a);
    const double b = a - s;
    c.code = 2 * (int)s + neg;
    c.c0 = (T)b;
    c.c1 = (T)div6(b * (1.0 - b) * (2.0 - b));
    c.c2 = (T)div6(b * (1.0 - b) * (1.0 + b));
    return c;
}
