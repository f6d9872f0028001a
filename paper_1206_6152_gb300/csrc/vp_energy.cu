// vp_energy.cu -- the sums behind the diagnostics M, K and U (Sec. 3.1, 3.2 of
// Yoshikawa, Yoshida & Umemura 2013).
//
//  * k_energy_partials: per spatial cell sum f and sum f |v|^2, one read of f,
//    and the density with them.  A thread owns columns (vy, vz) and runs along
//    vx: with M_c = sum_i f and W_c = sum_i f vx_i^2 of a column,
//    sum f |v|^2 = sum_c W_c + (vy^2 + vz^2)_c M_c.
//    FP32 f: an FP64 instruction takes 64 cycles of its quadrant's pipe, so the sums
//    are kept on the FP32 pipe as three floats each (TwoSum; products by TwoProd, with
//    weights of three floats: about 27 FP32 instructions per cell), whose roundings lie
//    below those of FP64 compensated sums, and turned into FP64 once per cube.  Bound by
//    FP32 issue.  32^3 x 32^3 cells: 39.8 ms with two FP64 compensated sums per cell,
//    1.1 ms now; 0.81 ms with two floats per sum, which lost up to 5e-14 of K where
//    columns are few.  The weights are taken in units of a power of two near the largest
//    |v|^2, so that no unit of velocity brings the products near the ends of the FP32
//    range.  A cell whose sums are so small or large that low parts could underflow or a
//    sum overflow is summed in FP64 instead.  All merges of threads, warps and CTAs keep
//    the compensation.
//  * k_energy_sums: the compensated sums over the spatial cells, of these and of
//    rho phi (or the density misfit), by as many CTAs as pay; the last to arrive
//    adds the CTAs' sums (both words) in order.
#include <cuda_runtime.h>
#include <math.h>

#include "vp_device.cuh"
#include "vp_internal.cuh"

namespace {

constexpr int SUM_CTAS = 256;      // most CTAs of k_energy_sums (their sums: 3 of two words each)

// A sum as three floats s + e + g: what s loses is added to e, what e loses to g, so
// that the roundings left are 2^-48 of g's.  (As two floats, the additions into e alone
// cost 1e-14 of a column of 64 cells, 5e-14 of a one-dimensional problem's K, against the
// 1e-16 of FP64 compensated sums.)
struct Sum3 {
    float s = 0.f, e = 0.f, g = 0.f;
    __device__ __forceinline__ void low(float v)
    {
        const float t = e + v, bb = t - e;
        g += (e - (t - bb)) + (v - bb);
        e = t;
    }
    __device__ __forceinline__ void add(float x)
    {
        const float t = s + x, bb = t - s;
        low((s - (t - bb)) + (x - bb));
        s = t;
    }
    __device__ __forceinline__ void merge(const Sum3 &o)
    {
        add(o.s);
        low(o.e);
        g += o.g;
    }
    __device__ __forceinline__ double value() const { return ((double)g + (double)e) + (double)s; }
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

// The FP32 cube q in groups of four columns (vy, vz), adjacent ones read 16 bytes at a
// time (VEC), or G apart: group g's, g + G's, ... sums of f and of f |v|^2.  vx^2 is
// common to a group, so its four cells are added first: their sum as two floats (three
// TwoSums, 5 instructions per cell), its product with vx^2 and the additions (8 per
// cell); each column's own sum takes 13.  v2: vx^2, vy^2, vz^2 in three floats each
template <bool VEC>
__device__ void cell_sums(const float *q, int nx, int ny, int nz, const float4 *v2, int g, int G, Sum3 &M, Sum3 &Q)
{
    const int plane = ny * nz, step = VEC ? 1 : G;
    const float4 *x2 = v2, *y2 = v2 + nx, *z2 = y2 + ny;
    for (int c = VEC ? 4 * g : g; c < plane; c += 4 * G) {
        Sum3 m[4];
        const float *p = q + c;
        const int have = VEC ? 4 : (plane - c + G - 1) / G;         // columns of the group
#pragma unroll 4
        for (int i = 0; i < nx; ++i) {
            float x[4];
            if constexpr (VEC) {
                const float4 v = *reinterpret_cast<const float4 *>(p + (long long)i * plane);
                x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k) x[k] = k < have ? p[(long long)i * plane + k * step] : 0.f;
            }
            const float4 a = x2[i];
#pragma unroll
            for (int k = 0; k < 4; ++k) m[k].add(x[k]);
            const float2 u = two_sum(x[0], x[1]), v = two_sum(x[2], x[3]), h = two_sum(u.x, v.x);
            const float l = (u.y + v.y) + h.y, t = __fmul_rn(h.x, a.x);
            Q.add(t);
            Q.low(__fmaf_rn(h.x, a.x, -t));
            Q.low(__fmaf_rn(h.x, a.y, __fmaf_rn(l, a.x, __fmul_rn(h.x, a.z))));
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (k < have) {
                const int col = c + k * step, j = col / nz;
                const float4 w = add3(y2[j], z2[col - j * nz]);      // vy^2 + vz^2
                const float t = __fmul_rn(m[k].s, w.x), u = __fmul_rn(m[k].s, w.y), v = __fmul_rn(m[k].e, w.x);
                Q.add(t);
                Q.low(__fmaf_rn(m[k].s, w.x, -t));
                Q.low(u);
                Q.low(v);
                Q.g += (__fmaf_rn(m[k].s, w.y, -u) + __fmaf_rn(m[k].e, w.x, -v)) +
                       __fmaf_rn(m[k].s, w.z, __fmaf_rn(m[k].e, w.y, m[k].g * w.x));
                M.merge(m[k]);
            }
        }
    }
}

// the same in FP64, for any T
template <typename T>
__device__ void cell_sums_f64(const T *q, int nx, int ny, int nz, const double *v, int g, int G,
                              Acc<double> &am, Acc<double> &aq)
{
    const int plane = ny * nz;
    const double *vx = v, *vy = v + nx, *vz = vy + ny;
    for (int c = g; c < plane; c += G) {
        const double y = vy[c / nz], z = vz[c % nz], yz = y * y + z * z;
#pragma unroll 4
        for (int i = 0; i < nx; ++i) {
            const double x = (double)q[c + (long long)i * plane];
            am.add(x);
            aq.add(x * (vx[i] * vx[i] + yz));
        }
    }
}

// a as held by the lane `lane` ^ d
__device__ __forceinline__ Sum3 from_lane(const Sum3 &a, int d)
{
    Sum3 o;
    o.s = __shfl_xor_sync(0xffffffffu, a.s, d);
    o.e = __shfl_xor_sync(0xffffffffu, a.e, d);
    o.g = __shfl_xor_sync(0xffffffffu, a.g, d);
    return o;
}
__device__ __forceinline__ Acc<double> from_lane(const Acc<double> &a, int d)
{
    Acc<double> o;
    o.s = __shfl_xor_sync(0xffffffffu, a.s, d);
    o.c = __shfl_xor_sync(0xffffffffu, a.c, d);
    return o;
}

// M and Q over the G threads of a cell (32 or the CTA's 256), on return in all of them
// (FP64 sums, whose merges take the FP64 pipe: in the first warp).  Lanes below 16 merge
// M and the others Q, half the merges of doing both in every lane.  scratch: 8 pairs
template <int G, class A>
__device__ __forceinline__ void merge_cell(const A &M, const A &Q, A (&scratch)[8][2], double &m, double &q)
{
    const int lane = threadIdx.x & 31, half = lane >> 4;
    A a = half ? Q : M;
    const A o = from_lane(half ? M : Q, 16);
    a.merge(o);
#pragma unroll
    for (int d = 8; d > 0; d >>= 1) a.merge(from_lane(a, d));
    if (G > 32) {
        __syncthreads();                    // the last cell's are read
        if ((lane & 15) == 0) scratch[threadIdx.x >> 5][half] = a;
        __syncthreads();
        if (sizeof(a.s) == 8 && threadIdx.x >= 32) return;
        a = scratch[lane & 7][half];        // the eight warps' sums
#pragma unroll
        for (int d = 4; d > 0; d >>= 1) a.merge(from_lane(a, d));
    }
    const double v = a.value();
    m = __shfl_sync(0xffffffffu, v, 0);
    q = __shfl_sync(0xffffffffu, v, 16);
}

// G threads of a CTA of 256 per cell: 32 where there are cells enough to fill
// the SMs with one warp each, else the whole CTA.  v: the cell centres along vx,
// vy, vz, one after the other; v2exp: exponent of the largest |v|^2.
template <typename T, bool VEC, int G>
__global__ void __launch_bounds__(256) k_energy_partials(const T *__restrict__ f, long long np, int nx,
                                                        int ny, int nz, const double *vcx,
                                                        const double *vcy, const double *vcz,
                                                        int v2exp, double *__restrict__ partials,
                                                        double dvol, double *__restrict__ rho)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ Sum3 red3[8][2];
    __shared__ Acc<double> red[8][2];
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
    for (long long cell = (long long)blockIdx.x * (256 / G) + t / G; cell < np;
         cell += (long long)gridDim.x * (256 / G)) {
        const T *q = f + cell * nvc;
        double M = 0.0, Q = 0.0;
        bool done = false;
        if constexpr (sizeof(T) == 4) {
            Sum3 m, w;
            cell_sums<VEC>(q, nx, ny, nz, v2, g, G, m, w);
            merge_cell<G>(m, w, red3, M, Q);
            // (low parts below 2^-126 are flushed: at most a few times that per cell of f,
            // and as much of each weight)
            const double a = fabs(M), b = fabs(Q), lo = nvc * 0x1p-70;
            done = (a == 0.0 && b == 0.0) || (a > lo && a < 1e30 && b > lo && b > a * 0x1p-70 && b < 1e30);
            Q = scalbn(Q, v2exp);
        }
        if (!done) {
            Acc<double> am, aq;
            cell_sums_f64(q, nx, ny, nz, v, g, G, am, aq);
            merge_cell<G>(am, aq, red, M, Q);
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
                                                     int f1, int f2, long long np, Acc<double> *scratch,
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
        if (threadIdx.x == 0) scratch[3 * blockIdx.x + q] = a[q];
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
        for (int w = threadIdx.x; w < (int)gridDim.x; w += blockDim.x) b.merge(scratch[3 * w + q]);
        b = block_merge(b, red);
        if (threadIdx.x == 0) out[q] = b.value();
    }
}

template <typename T, bool VEC>
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

size_t vp_energy_scratch(long long np) { return 2 * (size_t)np + 3 + 6 * SUM_CTAS; }

cudaError_t launch_energy_partials(vp_ctx *c, const void *f, double *partials, double *rho)
{
    if (c->isdouble) return partials_t<double, false>(c, (const double *)f, partials, rho);
    if (c->nv[2] % 4 == 0) return partials_t<float, true>(c, (const float *)f, partials, rho);
    return partials_t<float, false>(c, (const float *)f, partials, rho);
}

cudaError_t launch_energy_sums(vp_ctx *c, const double *partials, const double *rho,
                               const double *target, double *out)
{
    long long grid = (c->np + 127) / 128;
    if (grid > SUM_CTAS) grid = SUM_CTAS;
    k_energy_sums<<<(unsigned)grid, 128, 0, c->stream>>>(partials, rho, c->phi, target, c->n[1], c->n[2],
                                                         c->fn[1], c->fn[2], c->np,
                                                         reinterpret_cast<Acc<double> *>(c->red + 2 * c->np + 3),
                                                         c->sc, out);
    return cudaGetLastError();
}
