// vp_field.cu -- density -> potential -> acceleration (Sec. 2.2 of Yoshikawa,
// Yoshida & Umemura 2013) in FP64 on sm_103a.
//
//  * periodic Poisson: phi = IFFT( G(k) FFT(rho) ), G(k) the Green's function
//    of the 7-point discrete Laplacian, -pi G / sum_l sin^2(k_l D_l/2)/D_l^2
//    (equal to -pi G D^2 / sum sin^2(k_l D/2) for equal spacings), G(0) = 0.
//  * isolated Poisson: Hockney's doubling; rho zero-padded to 2N per axis,
//    kernel -G/r on 0..N mirrored to N+1..2N-1, its r = 0 value the mean of
//    -G/r over one cubic cell, -G (3 ln(2 + sqrt 3) - pi/2) / D.
//  * force: g = -(phi_{i+1} - phi_{i-1}) / (2 D) per axis; for the isolated
//    case the neighbours outside the box come from the doubled grid.
//
// The convolution runs in five launches: z forward (reading the real data), y
// forward, x forward times G and back in the same CTA, y back, z back (writing
// the real potential).  Rows and planes that are zero (the padding) are
// neither read nor transformed, and only the planes the force needs (the box
// and one layer around it) are transformed back.
//
// What bounds it: the solve is a chain of small dependent launches (a 32^3
// grid is 0.5 MB), so its time is launches and the FP64 pipe, which takes 64
// cycles per warp instruction however few lanes are active.  A stage therefore
// gives every output element a thread of its own (one butterfly per thread
// left 3/4 of the lanes idle and put four times the FP64 instructions in a
// row), a warp's threads compute the same output p of their butterflies (p = 0
// needs additions only), each element is multiplied by its twiddle once, as it
// is stored, and lines are dealt to enough CTAs to keep every SM busy.
// Measured (events around the launches: potential, force and all tables of a
// step), against one launch per transform, copy and table and one butterfly
// per thread: 16^3 127 -> 61 us, 32^3 256 -> 91 us, 48^3 566 -> 172 us,
// isolated 64 x 32 x 32 765 -> 333 us.
#include <cuda_runtime.h>
#include <math.h>

#include "vp_device.cuh"
#include "vp_internal.cuh"

int vp_sm_count();

namespace {

// a b with its roundings spelled out (which product is rounded by itself), so
// that the transform's last bits do not hang on what the compiler contracts;
// x_first: the imaginary part as fma(a.x, b.y, a.y b.x), else the other way
__device__ __forceinline__ double2 cmul(double2 a, double2 b, bool x_first)
{
    const double u = x_first ? a.x : a.y, v = x_first ? b.y : b.x;
    const double r = x_first ? __dmul_rn(a.y, b.x) : __dmul_rn(a.x, b.y);
    return make_double2(__fma_rn(a.x, b.x, -__dmul_rn(a.y, b.y)), __fma_rn(u, v, r));
}

// output p of the DFT of R values at stride nr: sum_q W_R^{pq} v_q with
// W_R^m = tw[m nr] (W_R^0 = 1 is not multiplied by where the threads of a warp
// share p; every sum is rounded as in the plain sum over q)
template <int R>
__device__ __forceinline__ double2 dft_out(const double2 *v, int nr, int p,
                                           const double2 *__restrict__ tw, int inverse)
{
    double2 a = v[0];
    if (p == 0) {
#pragma unroll
        for (int q = 1; q < R; ++q) {
            a.x += v[q * nr].x;
            a.y += v[q * nr].y;
        }
        return a;
    }
#pragma unroll
    for (int q = 1; q < R; ++q) {
        const int m = q * p % R;
        double2 t = v[q * nr];
        if (m) {
            double2 w = tw[m * nr];
            if (inverse) w.y = -w.y;
            t = cmul(t, w, !inverse);
        }
        a.x += t.x;
        a.y += t.y;
    }
    return a;
}

struct FFTPlan {
    int n, nrad;
    int rad[24];
    const double2 *tw;
};

// nb lines of P.n (pitch n + 1: lines start on different banks), from src
// through the Stockham stages; src and dst are used in turn.  Starts after a
// barrier and ends with one; returns the buffer that holds the result.
__device__ double2 *fft_lines(const FFTPlan &P, double2 *src, double2 *dst, int nb, int inverse)
{
    const int n = P.n, pitch = n + 1;
    int Ns = 1;
    for (int st = 0; st < P.nrad; ++st) {
        const int R = P.rad[st], nr = n / R, per = nb * nr, Nn = Ns * R;
        // radix and twiddle step of the next stage
        const int R2 = st + 1 < P.nrad ? P.rad[st + 1] : 1, nr2 = n / R2, step2 = nr2 / Nn;
        for (int t = threadIdx.x; t < nb * n; t += blockDim.x) {
            const int p = t / per, u = t - p * per, b = u / nr, j = u - b * nr;
            const double2 *s = src + b * pitch + j;
            double2 x;
            switch (R) {
            case 2: x = dft_out<2>(s, nr, p, P.tw, inverse); break;
            case 3: x = dft_out<3>(s, nr, p, P.tw, inverse); break;
            case 4: x = dft_out<4>(s, nr, p, P.tw, inverse); break;
            case 5: x = dft_out<5>(s, nr, p, P.tw, inverse); break;
            case 7: x = dft_out<7>(s, nr, p, P.tw, inverse); break;
            case 11: x = dft_out<11>(s, nr, p, P.tw, inverse); break;
            default: x = dft_out<13>(s, nr, p, P.tw, inverse); break;
            }
            const int o = (j / Ns) * Nn + p * Ns + j % Ns;
            if (R2 > 1) {
                const int r2 = o / nr2, m = r2 * ((o - r2 * nr2) % Nn) * step2;      // < n
                if (m) {
                    double2 w = P.tw[m];
                    if (inverse) w.y = -w.y;
                    x = cmul(x, w, false);
                }
            }
            dst[b * pitch + o] = x;
        }
        __syncthreads();
        double2 *t = src; src = dst; dst = t;
        Ns = Nn;
    }
    return src;
}

// the convolution's geometry: FFT grid f; real data with rows of the in box
// (the rest of the FFT grid is zero) and, on the way back, m0 x m1 rows
struct Conv {
    int f0, f1, f2;
    int i0, i1, i2;         // input box
    int m0, m1;             // output rows: planes 0 .. m0 - 2 and f0 - 1 (all if m0 == f0)
    int B;                  // lines per CTA
};

// plane index of output slot i of m: the box, one layer above, the last layer
__device__ __forceinline__ int out_plane(int i, int m, int f) { return i == m - 1 ? f - 1 : i; }

// z forward: real rows r = i i1 + j of the input
__global__ void __launch_bounds__(256) k_conv_z(const double *__restrict__ in,
                                                double2 *__restrict__ spec, Conv C, FFTPlan P)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = C.f2, pitch = n + 1, rows = C.i0 * C.i1;
    double2 *b0 = reinterpret_cast<double2 *>(smem_raw), *b1 = b0 + C.B * pitch;
    const int r0 = blockIdx.x * C.B, nb = min(C.B, rows - r0);
    for (int e = threadIdx.x; e < nb * n; e += blockDim.x) {
        const int b = e / n, k = e - b * n;
        b0[b * pitch + k] = make_double2(k < C.i2 ? in[(long long)(r0 + b) * C.i2 + k] : 0.0, 0.0);
    }
    __syncthreads();
    const double2 *X = fft_lines(P, b0, b1, nb, 0);
    for (int e = threadIdx.x; e < nb * n; e += blockDim.x) {
        const int b = e / n, k = e - b * n, r = r0 + b;
        spec[((long long)(r / C.i1) * C.f1 + r % C.i1) * n + k] = X[b * pitch + k];
    }
}

// y lines of plane blockIdx.y (back: of output plane blockIdx.y), forward
// from the i1 rows of the input or back to the m1 rows of the output
__global__ void __launch_bounds__(256) k_conv_y(double2 *__restrict__ spec, Conv C, FFTPlan P,
                                                int inverse)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = C.f1, pitch = n + 1;
    double2 *b0 = reinterpret_cast<double2 *>(smem_raw), *b1 = b0 + C.B * pitch;
    const int k0 = blockIdx.x * C.B, nb = min(C.B, C.f2 - k0);
    const int i = inverse ? out_plane(blockIdx.y, C.m0, C.f0) : blockIdx.y;
    double2 *g = spec + (long long)i * n * C.f2 + k0;
    const int nin = inverse ? n : C.i1;
    for (int e = threadIdx.x; e < nb * n; e += blockDim.x) {
        const int j = e / nb, b = e - j * nb;
        b0[b * pitch + j] = j < nin ? g[(long long)j * C.f2 + b] : make_double2(0.0, 0.0);
    }
    __syncthreads();
    const double2 *X = fft_lines(P, b0, b1, nb, inverse);
    const int nout = inverse ? C.m1 : n;
    for (int e = threadIdx.x; e < nb * nout; e += blockDim.x) {
        const int s = e / nb, b = e - s * nb;
        const int j = inverse ? out_plane(s, C.m1, n) : s;
        g[(long long)j * C.f2 + b] = X[b * pitch + j];
    }
}

// x lines of row blockIdx.y: forward, times the Green's function, back
__global__ void __launch_bounds__(256) k_conv_x(double2 *__restrict__ spec,
                                                const double *__restrict__ ghat, Conv C, FFTPlan P)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = C.f0, pitch = n + 1;
    double2 *b0 = reinterpret_cast<double2 *>(smem_raw), *b1 = b0 + C.B * pitch;
    const int k0 = blockIdx.x * C.B, nb = min(C.B, C.f2 - k0), j = blockIdx.y;
    double2 *g = spec + (long long)j * C.f2 + k0;
    const double *gh = ghat + (long long)j * C.f2 + k0;
    const long long pi = (long long)C.f1 * C.f2;
    for (int e = threadIdx.x; e < nb * n; e += blockDim.x) {
        const int i = e / nb, b = e - i * nb;
        b0[b * pitch + i] = i < C.i0 ? g[i * pi + b] : make_double2(0.0, 0.0);
    }
    __syncthreads();
    double2 *X = fft_lines(P, b0, b1, nb, 0);
    for (int e = threadIdx.x; e < nb * n; e += blockDim.x) {
        const int i = e / nb, b = e - i * nb;
        const double w = gh[i * pi + b];
        double2 v = X[b * pitch + i];
        v.x *= w;
        v.y *= w;
        X[b * pitch + i] = v;
    }
    __syncthreads();
    X = fft_lines(P, X, X == b0 ? b1 : b0, nb, 1);
    for (int e = threadIdx.x; e < nb * C.m0; e += blockDim.x) {
        const int s = e / nb, b = e - s * nb, i = out_plane(s, C.m0, n);
        g[i * pi + b] = X[b * pitch + i];
    }
}

// z back: the real part of the output's rows
__global__ void __launch_bounds__(256) k_conv_z_back(const double2 *__restrict__ spec,
                                                     double *__restrict__ out, Conv C, FFTPlan P)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = C.f2, pitch = n + 1, rows = C.m0 * C.m1;
    double2 *b0 = reinterpret_cast<double2 *>(smem_raw), *b1 = b0 + C.B * pitch;
    const int r0 = blockIdx.x * C.B, nb = min(C.B, rows - r0);
    auto row = [&](int r) {
        return (long long)out_plane(r / C.m1, C.m0, C.f0) * C.f1 + out_plane(r % C.m1, C.m1, C.f1);
    };
    for (int e = threadIdx.x; e < nb * n; e += blockDim.x) {
        const int b = e / n, k = e - b * n;
        b0[b * pitch + k] = spec[row(r0 + b) * n + k];
    }
    __syncthreads();
    const double2 *X = fft_lines(P, b0, b1, nb, 1);
    for (int e = threadIdx.x; e < nb * n; e += blockDim.x) {
        const int b = e / n, k = e - b * n;
        out[row(r0 + b) * n + k] = X[b * pitch + k].x;
    }
}

// complex lines of the whole FFT grid along one axis (set-up of the isolated
// Green's function)
struct Lines {
    long long so, si, sp;   // strides of outer index, line, position
    int ni, B;
};
__global__ void __launch_bounds__(256) k_fft(double2 *__restrict__ data, Lines L, FFTPlan P)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = P.n, pitch = n + 1;
    double2 *b0 = reinterpret_cast<double2 *>(smem_raw), *b1 = b0 + L.B * pitch;
    const int l0 = blockIdx.x * L.B, nb = min(L.B, L.ni - l0);
    double2 *g = data + blockIdx.y * L.so + l0 * L.si;
    for (int e = threadIdx.x; e < nb * n; e += blockDim.x) {
        const int p = e / nb, b = e - p * nb;
        b0[b * pitch + p] = g[b * L.si + p * L.sp];
    }
    __syncthreads();
    const double2 *X = fft_lines(P, b0, b1, nb, 0);
    for (int e = threadIdx.x; e < nb * n; e += blockDim.x) {
        const int p = e / nb, b = e - p * nb;
        g[b * L.si + p * L.sp] = X[b * pitch + p];
    }
}

struct ForceGeom {
    int n0, n1, n2, f0, f1, f2;
    double idx0, idx1, idx2;
};

// g_a = -(phi(i+1) - phi(i-1)) / (2 dx_a) of cell t, neighbours wrapped on the FFT grid
__device__ __forceinline__ double force_cell(const double *__restrict__ phi, const ForceGeom &F,
                                             long long t, int a)
{
    const int k = (int)(t % F.n2);
    const int j = (int)((t / F.n2) % F.n1);
    const int i = (int)(t / ((long long)F.n1 * F.n2));
    const int x = a == 0 ? i : (a == 1 ? j : k), f = a == 0 ? F.f0 : (a == 1 ? F.f1 : F.f2);
    const long long s = a == 0 ? (long long)F.f1 * F.f2 : (a == 1 ? F.f2 : 1);
    const double *p = phi + ((long long)i * F.f1 + j) * F.f2 + k - x * s;
    const double idx = a == 0 ? F.idx0 : (a == 1 ? F.idx1 : F.idx2);
    return -(p[(x + 1 == f ? 0 : x + 1) * s] - p[(x == 0 ? f - 1 : x - 1) * s]) * 0.5 * idx;
}

__global__ void __launch_bounds__(64) k_force(const double *__restrict__ phi, double *__restrict__ g,
                                              ForceGeom F)
{
    const long long np = (long long)F.n0 * F.n1 * F.n2;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < 3 * np) g[t] = force_cell(phi, F, t % np, (int)(t / np));
}

// The last CTA of the grid to arrive takes the grid's maximum (sc->amax_bits,
// a non-negative double ordered as its bits) and sets dt = C min(dt_p, dt_v)
// of Sec. 2.4, or the fixed dt; it leaves the accumulators zero for the next
// launch.
__device__ void grid_max_to_dt(DevScalars *sc, double m, double *red, const DtParams &D)
{
    m = block_max(m, red);
    if (threadIdx.x != 0) return;
    if (m > 0.0) atomicMax(&sc->amax_bits, (unsigned long long)__double_as_longlong(m));
    __threadfence();
    if (atomicAdd(&sc->arrived, 1u) != gridDim.x - 1) return;
    __threadfence();
    const double a = __longlong_as_double((long long)atomicExch(&sc->amax_bits, 0ULL));
    sc->arrived = 0;
    sc->amax = a;
    if (D.advance) sc->t += sc->dt;
    if (D.dt_fixed > 0.0) {
        sc->dt = D.dt_fixed;
    } else {
        const double dtv = a > 0.0 ? 1.0 / a : INFINITY;
        sc->dt = D.courant * fmin(D.dtp, dtv);
    }
}

// force, the half-kick table of this g with the step's dt, the end of the
// step (t += dt) and, with next, the dt of the next step from this g.  One
// thread per component and cell in small CTAs: a component's table entry
// takes about 30 FP64 instructions of 64 pipe cycles each, so what counts is
// that every SM quadrant gets its share of the warps (16^3 cells: one thread
// per cell in CTAs of 256 took 13 us, 32^3 cells 13.6 us).
template <typename T>
__global__ void __launch_bounds__(64) k_force_step(const double *__restrict__ phi,
                                                   double *__restrict__ g, ForceGeom F,
                                                   LineCoef<T> *__restrict__ kick, double dv0,
                                                   double dv1, double dv2, DevScalars *sc, DtParams D,
                                                   int next)
{
    __shared__ double red[32];
    const long long np = (long long)F.n0 * F.n1 * F.n2;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    double m = 0.0;
    if (t < 3 * np) {
        const int a = (int)(t / np);
        const long long cell = t - a * np;
        const double tau = sc->dt * 0.5, ga = force_cell(phi, F, cell, a);
        g[t] = ga;
        kick[3 * cell + a] = make_line_coef<T>(ga * tau / (a == 0 ? dv0 : (a == 1 ? dv1 : dv2)));
        m = fmax(m, fabs(ga) * (a == 0 ? D.idv0 : (a == 1 ? D.idv1 : D.idv2)));
    }
    if (next) grid_max_to_dt(sc, m, red, D);
    else if (t == 0) sc->t += sc->dt;
}

__global__ void __launch_bounds__(256) k_dt(DevScalars *sc, const double *__restrict__ g,
                                            long long np, DtParams D)
{
    __shared__ double red[32];
    double m = 0.0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < np;
         i += (long long)gridDim.x * blockDim.x) {
        m = fmax(m, fabs(g[i]) * D.idv0);
        m = fmax(m, fabs(g[np + i]) * D.idv1);
        m = fmax(m, fabs(g[2 * np + i]) * D.idv2);
    }
    grid_max_to_dt(sc, m, red, D);
}

__global__ void k_copy_box(const double *__restrict__ src, double *__restrict__ dst, int n0,
                           int n1, int n2, int f1, int f2)
{
    const long long np = (long long)n0 * n1 * n2;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= np) return;
    const int k = (int)(t % n2);
    const int j = (int)((t / n2) % n1);
    const int i = (int)(t / ((long long)n1 * n2));
    dst[t] = src[((long long)i * f1 + j) * f2 + k];
}

inline unsigned blocks_for(long long n, int threads) { return (unsigned)((n + threads - 1) / threads); }

FFTPlan plan_of(const FFTAxis &A)
{
    FFTPlan P;
    P.n = A.n;
    P.nrad = A.nrad;
    for (int i = 0; i < A.nrad; ++i) P.rad[i] = A.rad[i];
    P.tw = A.tw;
    return P;
}

// lines per CTA: 8 (128 bytes of neighbouring lines per access), fewer where
// that would leave SMs short of CTAs or the two buffers exceed 96 KB
int lines_per_cta(long long lines, int n)
{
    int B = 8;
    while (B > 2 && (lines + B - 1) / B < 2 * vp_sm_count()) B /= 2;
    while (B > 1 && (size_t)2 * B * (n + 1) * sizeof(double2) > 96 * 1024) B /= 2;
    return B;
}

// threads of a CTA of B lines of n: one per element, at most 256
unsigned line_threads(int B, int n)
{
    const int t = (B * n + 31) / 32 * 32;
    return (unsigned)(t > 256 ? 256 : t);
}

// two line buffers of B lines of n; the attribute is set to the largest such
// size once a launch needs more than the default 48 KB, never lowered
template <class K>
cudaError_t line_smem(K kernel, int B, int n, size_t &smem)
{
    smem = (size_t)2 * B * (n + 1) * sizeof(double2);
    if (smem + 1024 <= 48 * 1024) return cudaSuccess;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
}

ForceGeom force_geom(const vp_ctx *c)
{
    return ForceGeom{c->n[0], c->n[1], c->n[2], c->fn[0], c->fn[1], c->fn[2],
                     1.0 / c->dx[0], 1.0 / c->dx[1], 1.0 / c->dx[2]};
}

DtParams dt_params(const vp_ctx *c)
{
    DtParams D;
    D.dtp = INFINITY;
    for (int a = 0; a < 3; ++a) {
        const double vmax = fmax(fabs(c->cfg.vlo[a]), fabs(c->cfg.vhi[a]));
        if (vmax > 0) D.dtp = fmin(D.dtp, c->dx[a] / vmax);
    }
    D.idv0 = 1.0 / c->dv[0];
    D.idv1 = 1.0 / c->dv[1];
    D.idv2 = 1.0 / c->dv[2];
    D.courant = c->cfg.courant;
    D.dt_fixed = c->cfg.dt_fixed;
    D.advance = 0;
    return D;
}

}  // namespace

// radix plan for one axis: 4s first, then 2, 3, 5, 7, 11, 13
int vp_fft_plan_axis(FFTAxis *a, int n)
{
    a->n = n;
    a->nrad = 0;
    int m = n;
    for (int r : {4, 2, 3, 5, 7, 11, 13}) {
        while (m % r == 0) {
            if (a->nrad >= 24) return VP_ERR_UNSUPPORTED;
            a->rad[a->nrad++] = r;
            m /= r;
        }
    }
    if (m != 1) return VP_ERR_UNSUPPORTED;
    return VP_OK;
}

cudaError_t launch_fft(vp_ctx *c, double2 *data, int axis)
{
    const FFTPlan P = plan_of(c->ax[axis]);
    const long long f0 = c->fn[0], f1 = c->fn[1], f2 = c->fn[2];
    Lines L;
    long long nouter;
    if (axis == 2) { L.so = f1 * f2; L.si = f2; L.sp = 1; L.ni = (int)f1; nouter = f0; }
    else if (axis == 1) { L.so = f1 * f2; L.si = 1; L.sp = f2; L.ni = (int)f2; nouter = f0; }
    else { L.so = f2; L.si = 1; L.sp = f1 * f2; L.ni = (int)f2; nouter = f1; }
    L.B = lines_per_cta(L.ni * nouter, P.n);
    size_t smem;
    cudaError_t e = line_smem(k_fft, L.B, P.n, smem);
    if (e != cudaSuccess) return e;
    k_fft<<<dim3(blocks_for(L.ni, L.B), (unsigned)nouter), line_threads(L.B, P.n), smem, c->stream>>>(data, L, P);
    return cudaGetLastError();
}

// out (real, FFT grid) = G * in (real): in holds the box (whole = 0: N^p
// values) or the whole FFT grid; out receives the box and the layer of cells
// around it (all of a periodic grid).  in and out may be the same array.
cudaError_t launch_convolve(vp_ctx *c, const double *in, int whole, double *out)
{
    Conv C;
    C.f0 = c->fn[0]; C.f1 = c->fn[1]; C.f2 = c->fn[2];
    C.i0 = whole ? C.f0 : c->n[0];
    C.i1 = whole ? C.f1 : c->n[1];
    C.i2 = whole ? C.f2 : c->n[2];
    C.m0 = C.f0 < c->n[0] + 2 ? C.f0 : c->n[0] + 2;
    C.m1 = C.f1 < c->n[1] + 2 ? C.f1 : c->n[1] + 2;
    const FFTPlan P0 = plan_of(c->ax[0]), P1 = plan_of(c->ax[1]), P2 = plan_of(c->ax[2]);
    cudaError_t e;
    size_t smem;
    double2 *spec = c->cbuf;
    const long long rin = (long long)C.i0 * C.i1, rout = (long long)C.m0 * C.m1;
    C.B = lines_per_cta(rin, C.f2);
    if ((e = line_smem(k_conv_z, C.B, C.f2, smem)) != cudaSuccess) return e;
    k_conv_z<<<blocks_for(rin, C.B), line_threads(C.B, C.f2), smem, c->stream>>>(in, spec, C, P2);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // (lines of one cell are their own transform)
    if (C.f1 > 1) {
        C.B = lines_per_cta((long long)C.i0 * C.f2, C.f1);
        if ((e = line_smem(k_conv_y, C.B, C.f1, smem)) != cudaSuccess) return e;
        k_conv_y<<<dim3(blocks_for(C.f2, C.B), C.i0), line_threads(C.B, C.f1), smem, c->stream>>>(
            spec, C, P1, 0);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    C.B = lines_per_cta((long long)C.f1 * C.f2, C.f0);
    if ((e = line_smem(k_conv_x, C.B, C.f0, smem)) != cudaSuccess) return e;
    k_conv_x<<<dim3(blocks_for(C.f2, C.B), C.f1), line_threads(C.B, C.f0), smem, c->stream>>>(
        spec, c->ghat, C, P0);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (C.f1 > 1) {
        C.B = lines_per_cta((long long)C.m0 * C.f2, C.f1);
        if ((e = line_smem(k_conv_y, C.B, C.f1, smem)) != cudaSuccess) return e;
        k_conv_y<<<dim3(blocks_for(C.f2, C.B), C.m0), line_threads(C.B, C.f1), smem, c->stream>>>(
            spec, C, P1, 1);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    C.B = lines_per_cta(rout, C.f2);
    if ((e = line_smem(k_conv_z_back, C.B, C.f2, smem)) != cudaSuccess) return e;
    k_conv_z_back<<<blocks_for(rout, C.B), line_threads(C.B, C.f2), smem, c->stream>>>(spec, out, C, P2);
    return cudaGetLastError();
}

cudaError_t launch_field_solve(vp_ctx *c, const double *rho, double *g_out)
{
    cudaError_t e = launch_convolve(c, rho, 0, c->phi);
    if (e != cudaSuccess || !g_out) return e;
    k_force<<<blocks_for(3 * c->np, 64), 64, 0, c->stream>>>(c->phi, g_out, force_geom(c));
    return cudaGetLastError();
}

// the field of the step: phi and g = c->g of rho, the table of the second half
// kick, t += dt and, with next, the dt of the next step
cudaError_t launch_field_step(vp_ctx *c, const double *rho, void *kick, int next)
{
    cudaError_t e = launch_convolve(c, rho, 0, c->phi);
    if (e != cudaSuccess) return e;
    DtParams D = dt_params(c);
    D.advance = 1;
    const unsigned grid = blocks_for(3 * c->np, 64);
    if (c->isdouble)
        k_force_step<double><<<grid, 64, 0, c->stream>>>(c->phi, c->g, force_geom(c),
                                                          (LineCoef<double> *)kick, c->dv[0], c->dv[1],
                                                          c->dv[2], c->sc, D, next);
    else
        k_force_step<float><<<grid, 64, 0, c->stream>>>(c->phi, c->g, force_geom(c),
                                                         (LineCoef<float> *)kick, c->dv[0], c->dv[1],
                                                         c->dv[2], c->sc, D, next);
    return cudaGetLastError();
}

cudaError_t launch_dt(vp_ctx *c, const double *g)
{
    unsigned grid = blocks_for(c->np, 256);
    if (grid > 2u * vp_sm_count()) grid = 2u * vp_sm_count();
    k_dt<<<grid, 256, 0, c->stream>>>(c->sc, g, c->np, dt_params(c));
    return cudaGetLastError();
}

cudaError_t launch_copy_phi_box(vp_ctx *c, double *dst)
{
    k_copy_box<<<blocks_for(c->np, 256), 256, 0, c->stream>>>(c->phi, dst, c->n[0], c->n[1],
                                                              c->n[2], c->fn[1], c->fn[2]);
    return cudaGetLastError();
}
