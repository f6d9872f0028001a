// vp_energy.cu -- the sums behind the diagnostics M, K and U (Sec. 3.1, 3.2 of
// Yoshikawa, Yoshida & Umemura 2013).
//
//  * k_energy_partials: per spatial cell sum f and sum f |v|^2, one read of f,
//    and the density with them.  A thread owns columns (vy, vz) and runs along
//    vx: with M_c = sum_i f and W_c = sum_i f vx_i^2 of a column,
//    sum f |v|^2 = sum_c W_c + (vy^2 + vz^2)_c M_c.
//    FP32 f: an FP64 instruction takes 74 cycles of its quadrant's pipe, so the
//    two sums of a column are kept as double-floats on the FP32 pipe (TwoSum,
//    and TwoProd with vx^2 in three floats: 19 FP32 instructions per cell, close
//    to what HBM takes) and added to FP64 totals once per column.
//    32^3 x 32^3 cells: 39.8 ms with two FP64 compensated sums per cell, 0.81 ms
//    now.  The weights are taken in units of a power of two near the largest |v|^2, so
//    that no unit of velocity brings the products near the ends of the FP32 range.  A
//    cell whose sums are so small or large that low parts could underflow or a sum
//    overflow is summed in FP64 instead.
//  * k_energy_sums: the compensated sums over the spatial cells, of these and of
//    rho phi (or the density misfit), by as many CTAs as pay; the last to arrive
//    adds the CTAs' sums in order.
#include <cuda_runtime.h>
#include <math.h>

#include "vp_device.cuh"
#include "vp_internal.cuh"

namespace {

constexpr int SUM_CTAS = 256;      // most CTAs of k_energy_sums (their sums: 3 each)

// a double-float: value s + e
struct FF {
    float s = 0.f, e = 0.f;
    __device__ __forceinline__ void add(float x, float low)
    {
        const float t = s + x, bb = t - s;
        e += ((s - (t - bb)) + (x - bb)) + low;
        s = t;
    }
};

// v as the sum of three floats (x, y, z), all 53 bits: with two, the error of a
// weight is the same in every cell and does not average out
__device__ __forceinline__ float4 split(double v)
{
    const float h = (float)v, m = (float)(v - (double)h);
    return make_float4(h, m, (float)(v - (double)h - (double)m), 0.f);
}

__device__ __forceinline__ float2 two_sum(float a, float b)
{
    const float t = a + b, bb = t - a;
    return make_float2(t, (a - (t - bb)) + (b - bb));
}

// the sum of two such weights
__device__ __forceinline__ float4 add3(float4 a, float4 b)
{
    const float2 h = two_sum(a.x, b.x), m = two_sum(a.y, b.y), n = two_sum(h.y, m.x);
    return make_float4(h.x, n.x, (n.y + m.y) + (a.z + b.z), 0.f);
}

template <int VEC>
__device__ __forceinline__ void load(float (&x)[VEC], const float *p)
{
    if constexpr (VEC == 4) {
        const float4 v = *reinterpret_cast<const float4 *>(p);
        x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
    } else {
        x[0] = *p;
    }
}

// the cell's columns g, g + G, ... (VEC adjacent ones at a time) of an FP32
// cube; v2: vx^2, vy^2, vz^2 in three floats each
template <int VEC>
__device__ void cell_sums(const float *q, int nx, int ny, int nz, const float4 *v2, int g, int G, double &M, double &Q)
{
    const int plane = ny * nz;
    const float4 *x2 = v2, *y2 = v2 + nx, *z2 = y2 + ny;
    for (int c = g * VEC; c < plane; c += G * VEC) {
        FF m[VEC], w;
        const float *p = q + c;
#pragma unroll 8
        for (int i = 0; i < nx; ++i) {
            float x[VEC];
            load<VEC>(x, p + (long long)i * plane);
            const float4 a = x2[i];
#pragma unroll
            for (int k = 0; k < VEC; ++k) {
                m[k].add(x[k], 0.f);
                const float t = __fmul_rn(x[k], a.x);
                w.add(t, __fmaf_rn(x[k], a.z, __fmaf_rn(x[k], a.y, __fmaf_rn(x[k], a.x, -t))));
            }
        }
        const int j = c / nz, k0 = c - j * nz;
        const float4 b = y2[j];
        FF tot;
#pragma unroll
        for (int k = 0; k < VEC; ++k) {
            const float4 wt = add3(b, z2[k0 + k]);          // vy^2 + vz^2
            const float t = __fmul_rn(m[k].s, wt.x);
            // (smallest terms first: added to a rounded larger one they would be
            // lost, always to the same side)
            const float low = __fmaf_rn(m[k].s, wt.y,
                                        __fmaf_rn(m[k].e, wt.x, __fmaf_rn(m[k].s, wt.z, m[k].e * wt.y)));
            w.add(t, __fmaf_rn(m[k].s, wt.x, -t) + low);
            tot.add(m[k].s, m[k].e);
        }
        M += (double)tot.s + (double)tot.e;
        Q += (double)w.s + (double)w.e;
    }
}

// the same in FP64, for any T
template <typename T>
__device__ void cell_sums_f64(const T *q, int nx, int ny, int nz, const double *v, int g, int G,
                              double &M, double &Q)
{
    const int plane = ny * nz;
    const double *vx = v, *vy = v + nx, *vz = vy + ny;
    Acc<double> am, aq;
    for (int c = g; c < plane; c += G) {
        const double y = vy[c / nz], z = vz[c % nz], yz = y * y + z * z;
#pragma unroll 4
        for (int i = 0; i < nx; ++i) {
            const double x = (double)q[c + (long long)i * plane];
            am.add(x);
            aq.add(x * (vx[i] * vx[i] + yz));
        }
    }
    M = am.value();
    Q = aq.value();
}

// G threads of a CTA of 256 per cell: 32 where there are cells enough to fill
// the SMs with one warp each, else the whole CTA.  v: the cell centres along vx,
// vy, vz, one after the other; v2exp: exponent of the largest |v|^2.
template <typename T, int VEC, int G>
__global__ void __launch_bounds__(256) k_energy_partials(const T *__restrict__ f, long long np, int nx,
                                                        int ny, int nz, const double *vcx,
                                                        const double *vcy, const double *vcz,
                                                        int v2exp, double *__restrict__ partials,
                                                        double dvol, double *__restrict__ rho)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red[2][8];
    float4 *v2 = reinterpret_cast<float4 *>(smem_raw);
    double *v = reinterpret_cast<double *>(v2 + nx + ny + nz);
    const int t = threadIdx.x, nt = nx + ny + nz;
    for (int e = t; e < nt; e += 256) {
        const double u = e < nx ? vcx[e] : (e < nx + ny ? vcy[e - nx] : vcz[e - nx - ny]);
        v[e] = u;
        v2[e] = split(scalbn(u * u, -v2exp));
    }
    __syncthreads();
    const int nvc = nx * ny * nz, g = t % G;
    auto merge = [&](double &M, double &Q) {
        for (int d = 16; d > 0; d >>= 1) {
            M += __shfl_xor_sync(0xffffffffu, M, d);
            Q += __shfl_xor_sync(0xffffffffu, Q, d);
        }
        if (G > 32) {
            __syncthreads();
            if ((t & 31) == 0) { red[0][t >> 5] = M; red[1][t >> 5] = Q; }
            __syncthreads();
            M = Q = 0.0;
            for (int w = 0; w < G / 32; ++w) { M += red[0][w]; Q += red[1][w]; }
        }
    };
    for (long long cell = (long long)blockIdx.x * (256 / G) + t / G; cell < np;
         cell += (long long)gridDim.x * (256 / G)) {
        const T *q = f + cell * nvc;
        double M = 0.0, Q = 0.0;
        if constexpr (sizeof(T) == 4) {
            cell_sums<VEC>(q, nx, ny, nz, v2, g, G, M, Q);
            merge(M, Q);
            // (low parts below 2^-126 are flushed: at most a few times that per cell of f,
            // and as much of each weight)
            const double a = fabs(M), b = fabs(Q), lo = nvc * 0x1p-70;
            Q = scalbn(Q, v2exp);
            if (!((a == 0.0 && b == 0.0) || (a > lo && a < 1e30 && b > lo && b > a * 0x1p-70 && b < 1e30))) {
                cell_sums_f64(q, nx, ny, nz, v, g, G, M, Q);
                merge(M, Q);
            }
        } else {
            cell_sums_f64(q, nx, ny, nz, v, g, G, M, Q);
            merge(M, Q);
        }
        if (g == 0) {
            partials[2 * cell] = M;
            partials[2 * cell + 1] = Q;
            rho[cell] = M * dvol;
        }
    }
}

// out[0], out[1] = sums of pm's interleaved pairs (pm may be null); out[2] = sum
// of rho phi over the box, or with target of (rho - target)^2
__global__ void __launch_bounds__(128) k_energy_sums(const double *__restrict__ pm,
                                                     const double *__restrict__ rho,
                                                     const double *__restrict__ phi,
                                                     const double *__restrict__ target, int n1, int n2,
                                                     int f1, int f2, long long np, double *scratch,
                                                     DevScalars *sc, double *out)
{
    __shared__ Acc<double> red[32];
    __shared__ bool last;
    Acc<double> a[3];
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < np;
         t += (long long)gridDim.x * blockDim.x) {
        if (pm) {
            a[0].add(pm[2 * t]);
            a[1].add(pm[2 * t + 1]);
        }
        if (target) {
            const double r = rho[t] - target[t];
            a[2].add(r * r);
        } else {
            const int k = (int)(t % n2);
            const int j = (int)((t / n2) % n1);
            const int i = (int)(t / ((long long)n1 * n2));
            a[2].add(rho[t] * phi[((long long)i * f1 + j) * f2 + k]);
        }
    }
    for (int q = pm ? 0 : 2; q < 3; ++q) {
        a[q] = block_merge(a[q], red);
        if (threadIdx.x == 0) scratch[3 * blockIdx.x + q] = a[q].value();
    }
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(&sc->arrived, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    if (threadIdx.x == 0) sc->arrived = 0;
    for (int q = pm ? 0 : 2; q < 3; ++q) {
        Acc<double> b;
        for (int w = threadIdx.x; w < (int)gridDim.x; w += blockDim.x) b.add(scratch[3 * w + q]);
        b = block_merge(b, red);
        if (threadIdx.x == 0) out[q] = b.value();
    }
}

template <typename T, int VEC>
cudaError_t partials_t(vp_ctx *c, const T *f, double *partials, double *rho)
{
    const int nt = c->nv[0] + c->nv[1] + c->nv[2];
    const size_t smem = (size_t)nt * (sizeof(double) + sizeof(float4));
    const bool warp = c->np >= 16LL * vp_sm_count();
    auto kern = warp ? k_energy_partials<T, VEC, 32> : k_energy_partials<T, VEC, 256>;
    long long grid = warp ? (c->np + 7) / 8 : c->np;
    if (grid > 8LL * vp_sm_count()) grid = 8LL * vp_sm_count();
    double v2 = 0.0;
    for (int a = 0; a < 3; ++a) {
        const double v = fmax(fabs(c->cfg.vlo[a] + 0.5 * c->dv[a]), fabs(c->cfg.vhi[a] - 0.5 * c->dv[a]));
        v2 += v * v;
    }
    const int v2exp = v2 > 0.0 && isfinite(v2) ? ilogb(v2) : 0;
    kern<<<(unsigned)grid, 256, smem, c->stream>>>(f, c->np, c->nv[0], c->nv[1], c->nv[2], c->vc[0],
                                                   c->vc[1], c->vc[2], v2exp, partials, c->dvol_v, rho);
    return cudaGetLastError();
}

}  // namespace

size_t vp_energy_scratch(long long np) { return 2 * (size_t)np + 3 + 3 * SUM_CTAS; }

cudaError_t launch_energy_partials(vp_ctx *c, const void *f, double *partials, double *rho)
{
    if (c->isdouble) return partials_t<double, 1>(c, (const double *)f, partials, rho);
    if (c->nv[2] % 4 == 0) return partials_t<float, 4>(c, (const float *)f, partials, rho);
    return partials_t<float, 1>(c, (const float *)f, partials, rho);
}

cudaError_t launch_energy_sums(vp_ctx *c, const double *partials, const double *rho,
                               const double *target, double *out)
{
    long long grid = (c->np + 127) / 128;
    if (grid > SUM_CTAS) grid = SUM_CTAS;
    k_energy_sums<<<(unsigned)grid, 128, 0, c->stream>>>(partials, rho, c->phi, target, c->n[1], c->n[2],
                                                         c->fn[1], c->fn[2], c->np, c->red + 2 * c->np + 3,
                                                         c->sc, out);
    return cudaGetLastError();
}
