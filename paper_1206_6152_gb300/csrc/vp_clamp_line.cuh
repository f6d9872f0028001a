// vp_clamp_line.cuh -- the PFC update of one line of run-time length held in
// registers, in the clamp form of the slope corrector (pfc_flux of
// vp_device.cuh, bit for bit), for lines of any length up to a compile-time
// NMAX.
//
// The line is held in upwind order: a line with u < 0 is read and written from
// its far end with a negative stride, so that the lanes of a warp run one code
// path whatever their directions (a z drift has both signs of v_z in every
// warp).  x[n .. NMAX] hold what lies beyond the line's end: its first cell
// (periodic) or 0 (outflow).
#pragma once

#include <cuda_runtime.h>

#include "vp_device.cuh"

namespace vpline {

// 2 a and -a.  FP64: on the integer pipes (an FP64 instruction, a negation or
// one that is predicated off included, takes 64 cycles of a quadrant's FP64
// pipe): 2 a is the exponent plus one, for zeros and subnormals the mantissa
// shifted, for infinities and NaN a itself, infinity where it overflows.
__device__ __forceinline__ float twice(float a) { return a + a; }
__device__ __forceinline__ double twice(double a)
{
    const unsigned hi = (unsigned)__double2hiint(a), lo = (unsigned)__double2loint(a);
    const unsigned e = hi & 0x7ff00000u, s = hi & 0x80000000u;
    unsigned h2 = e ? hi + 0x00100000u : s | (((hi << 1) | (lo >> 31)) & 0x7fffffffu);
    unsigned l2 = e ? lo : lo << 1;
    if (e >= 0x7fe00000u) {
        h2 = e == 0x7ff00000u ? hi : (s | 0x7ff00000u);
        l2 = e == 0x7ff00000u ? lo : 0u;
    }
    return __hiloint2double((int)h2, (int)l2);
}
__device__ __forceinline__ float negate(float a) { return -a; }
__device__ __forceinline__ double negate(double a)
{
    return __hiloint2double(__double2hiint(a) ^ (int)0x80000000, __double2loint(a));
}

// pfc_flux with the differences dp = fp - f0 and dm = f0 - fm (each cell's dp
// is the next one's dm).  FP64: with the difference and the two additions of
// the update 7 FP64 instructions per cell.
template <typename T>
__device__ __forceinline__ T clamp_flux(T dm, T f0, T dp, T finf, T c0, T c1, T c2)
{
    const T a = twice(f0), b = twice(finf - f0);
    const T ep = vmin(vmax(dp, negate(b)), a);
    const T em = vmin(vmax(dm, negate(a)), b);
    const T phi = c0 * f0 + c1 * ep + c2 * em;
    return vmin(vmax(phi, T(0)), f0);
}

// Loops over the cells go in groups of GR, unrolled: whole groups without any
// test per cell, then one partial group.  GR = 1 (a branch out after the last
// cell) is what FP64 needs, as instructions of cells past the end would take FP64
// pipe slots even where predicated off, and what serves FP32 lines best that are
// bound by HBM or much shorter than NMAX; GR = 4 serves the issue-bound kicks.

// cells 0 .. n - 1 of a line by get() in turn, and what lies behind them (the
// first cell, or 0)
template <typename T, int NMAX, bool PERIODIC, int GR, class G>
__device__ __forceinline__ void load_line(T (&x)[NMAX + 1], int n, G get)
{
    if constexpr (GR == 1) {
        x[0] = get();
#pragma unroll
        for (int j = 1; j <= NMAX; ++j) x[j] = j < n ? get() : (PERIODIC ? x[0] : T(0));
    } else {
#pragma unroll
        for (int j = 0; j < NMAX; j += GR) {
            if (j + GR <= n) {
#pragma unroll
                for (int i = 0; i < GR; ++i) x[j + i] = get();
            } else {
                // (every x is set on every path: registers left undefined
                // past the end would be held over from the line before)
#pragma unroll
                for (int i = 0; i < GR; ++i) {
                    x[j + i] = PERIODIC && j + i ? x[0] : T(0);
                    if (j + i < n) x[j + i] = get();
                }
            }
        }
        x[NMAX] = PERIODIC ? x[0] : T(0);
    }
}

// maximum of the line and 0
template <typename T, int NMAX, int GR>
__device__ __forceinline__ T clamp_line_max(const T (&x)[NMAX + 1], int n)
{
    T m = T(0);
#pragma unroll
    for (int j = 0; j < NMAX; j += GR) {
        if (GR == 1 && j >= n) break;
        if (j < n) {                    // (a partial group's pads are 0 or x[0])
#pragma unroll
            for (int i = 0; i < GR; ++i) m = vmax(m, x[j + i]);
        }
    }
    return m;
}

// the zero-shift update of the line x; put(j, v) takes cell j's new value, in
// increasing j, after every cell of the line has been read.  PERIODIC: fm1,
// fm2 are the line's last and last but one cells.  Returns the last cell's
// flux (what leaves an outflow line).
template <typename T, int NMAX, bool PERIODIC, int GR, class P>
__device__ __forceinline__ T clamp_line(const T (&x)[NMAX + 1], int n, T fm1, T fm2, T c0, T c1, T c2,
                                        P put)
{
    const T finf = clamp_line_max<T, NMAX, GR>(x, n);
    T dm = x[0], phm = T(0);                    // outflow: f_{-1} = 0
    if (PERIODIC) {
        dm = x[0] - fm1;
        phm = clamp_flux(fm1 - fm2, fm1, dm, finf, c0, c1, c2);
    }
    auto cell = [&](int i) {
        const T dp = x[i + 1] - x[i];
        const T ph = clamp_flux(dm, x[i], dp, finf, c0, c1, c2);
        put(i, (x[i] - ph) + phm);
        phm = ph;
        dm = dp;
    };
#pragma unroll
    for (int j = 0; j < NMAX; j += GR) {
        if constexpr (GR == 1) {
            if (j >= n) break;
            cell(j);
        } else if (j + GR <= n) {
#pragma unroll
            for (int i = 0; i < GR; ++i) cell(j + i);
        } else if (j < n) {
#pragma unroll
            for (int i = 0; i < GR; ++i)
                if (j + i < n) cell(j + i);
        }
    }
    return phm;
}

// the update of the outflow line x moved on by s whole cells as well (0 <= s <= n),
// in the arithmetic and the order of sums of kick_line_shifted (vp_fast_line.cuh): cell
// j and the flux before it go to position j + s, cells that would pass the end are
// lost, positions below s are empty (the caller's to write).  put(v) takes the new
// values of positions s, s + 1, ... in turn.  Returns what leaves.  Only the fluxes of
// cells that stay are computed, so a sweep by several cells takes about as long as one
// by a part of one; line by line in place in global memory, two reads per cell and no
// more than one under way, the vz sweep of 8^3 cubes of 64^3 took 1440 us (now 190-270).
template <typename T, int NMAX, class P>
__device__ __forceinline__ T clamp_line_shifted(const T (&x)[NMAX + 1], int n, int s, T c0, T c1, T c2,
                                                P put)
{
    const T finf = clamp_line_max<T, NMAX, 1>(x, n);
    T dm = x[0], phm = T(0), lost = T(0);
    const int stay = n - s;
#pragma unroll
    for (int j = 0; j < NMAX; ++j) {
        if (j >= n) break;
        if (j < stay) {
            const T dp = x[j + 1] - x[j];
            const T ph = clamp_flux(dm, x[j], dp, finf, c0, c1, c2);
            put((x[j] - ph) + phm);
            phm = ph;
            dm = dp;
        } else {
            lost += x[j];
        }
    }
    return lost + phm;
}

// The same from p (step sp) to w (step sw; p may be w), both at the upwind end, shared or
// global memory.  A call: inlined beside the sub-cell code of lines in global memory, of
// planes and of blocks of lines above 32 cells it took registers and instruction fetches
// that made the sub-cell sweeps 2 to 5 % slower.
template <typename T, int NMAX>
__device__ __noinline__ T shifted_line(const T *p, int sp, T *w, int sw, int n, const LineCoef<T> cf)
{
    const int s = cf.code >> 1 < n ? cf.code >> 1 : n;
    T x[NMAX + 1];
    load_line<T, NMAX, false, 1>(x, n, [&]() {
        const T v = *p;
        p += sp;
        asm volatile("" : "+l"(p));
        return v;
    });
    for (int j = 0; j < s; ++j, w += sw) *w = T(0);
    return clamp_line_shifted<T, NMAX>(x, n, s, cf.c0, cf.c1, cf.c2, [&](T v) {
        *w = v;
        w += sw;
        asm volatile("" : "+l"(w));
    });
}

// clamp_line for FP32 lines of N cells known at compile time, in array order and
// in place (outflow)
template <int N, bool NEG>
__device__ __forceinline__ float clamp_exact(float (&x)[N], float finf, float c0, float c1, float c2)
{
#define AT(j) x[NEG ? N - 1 - (j) : (j)]
    float dm = AT(0), phm = 0.f;
#pragma unroll
    for (int j = 0; j < N; ++j) {
        const float f = AT(j), dp = (j + 1 < N ? AT(j + 1 < N ? j + 1 : 0) : 0.f) - f;
        const float ph = clamp_flux(dm, f, dp, finf, c0, c1, c2);
        AT(j) = (f - ph) + phm;
        phm = ph;
        dm = dp;
    }
#undef AT
    return phm;
}

}  // namespace vpline
