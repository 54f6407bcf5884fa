// Auxiliary kernels: twiddle tables, FP64 propagators, layout conversion between the public
// centred FP64 field and the internal transform-order field, and an FMA throughput probe.
#include <cuda_runtime.h>
#include <math.h>

#include "cme_internal.h"

namespace cme {

namespace {

// A complex factor of modulus <= 1, one + re + i im, times 2^62 as balanced limbs (cme_fixed.cuh).
// one = 1: re as expm1 gives it, without the rounding of 1 + re to FP64.
__device__ int4 factor_limbs(double re, double im, int one = 0)
{
    const long long C = __double2ll_rn(re * 4611686018427387904.0) + ((long long)one << 62);
    const long long S = __double2ll_rn(im * 4611686018427387904.0);
    return make_int4((int)((unsigned)(C >> 32) + ((unsigned)C >> 31)), (int)C,
                     (int)((unsigned)(S >> 32) + ((unsigned)S >> 31)), (int)S);
}

__global__ void twiddle_kernel(int N, int prec, void* out)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= N)
        return;
    double s, c;
    sincospi(2.0 * (double)k / (double)N, &s, &c);   // exp(2 pi i k/N) in FP64
    if (prec == PREC_FP64) {
        reinterpret_cast<int4*>(out)[k] = factor_limbs(c, s);
    } else
        reinterpret_cast<float2*>(out)[k] = make_float2((float)c, (float)s);
}

// expm1 of a complex argument z = x + iy without cancellation:
//   e^z - 1 = (expm1(x) cos y - 2 sin^2(y/2)) + i e^x sin y.
__device__ double2 cexpm1(double x, double y)
{
    double sy, cy, sh, ch;
    sincos(y, &sy, &cy);
    sincos(0.5 * y, &sh, &ch);
    const double em = expm1(x);
    return make_double2(em * cy - 2.0 * sh * sh, (em + 1.0) * sy);
}

template <typename V>
__device__ void put(void* p, int m, double2 v)
{
    if constexpr (sizeof(V) == 16) {
        reinterpret_cast<double2*>(p)[m] = v;
    } else {
        reinterpret_cast<float2*>(p)[m] = make_float2((float)v.x, (float)v.y);
    }
}

// Per mode: L = -kappa/2 + i(omega - omega_0 - sigma);  E = exp(L h/2), e1 = expm1(L h/2),
// e2 = expm1(L h), all in FP64, stored in the batch precision.
template <typename V>
__global__ void prop_kernel(PropArgs a)
{
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= a.total)
        return;
    const int i = a.mode_inst[m];
    const double Lr = -0.5 * a.kappa[m];
    const double Li = a.omega[m] - a.sigma[i];
    const double hh = 0.5 * a.h;
    const double2 e1 = cexpm1(Lr * hh, Li * hh);
    double2 e2 = cexpm1(Lr * a.h, Li * a.h);
    // The fixed-point stages take |E| <= 1 (loss); their bounds have room for a gain of 1.2.  A
    // larger one would overflow without a trace, so that the mode becomes NaN instead.
    if (a.Ef && Lr * hh > 0.1823)   // log 1.2
        e2.x = e2.y = __longlong_as_double(0x7ff8000000000000LL);
    put<V>(a.E, m, make_double2(e1.x + 1.0, e1.y));
    if (a.e1)
        put<V>(a.e1, m, e1);
    // The fixed-point stages apply E to the state itself, the same E in every step: it keeps the bits
    // that expm1 gives it, where 1 + expm1 rounded to FP64 is off by up to 2^-54.
    if (a.Ef)
        reinterpret_cast<int4*>(a.Ef)[m] = factor_limbs(e1.x, e1.y, 1);
    put<V>(a.e2, m, e2);
    // Strang pump increment over h/2 on the pumped mode (transform position 0):
    //   c = (exp(L_0 h/2) - 1) / L_0 * pump   (h/2 * pump when L_0 = 0)
    if (m == a.inst_off[i]) {
        const double2 p = a.pump[i];
        double2 c;
        const double den = Lr * Lr + Li * Li;
        if (den == 0.0) {
            c = make_double2(hh * p.x, hh * p.y);
        } else {
            // q = e1 / L
            const double qr = (e1.x * Lr + e1.y * Li) / den;
            const double qi = (e1.y * Lr - e1.x * Li) / den;
            c = make_double2(qr * p.x - qi * p.y, qr * p.y + qi * p.x);
        }
        a.cpump[i] = c;
        if (a.cpump2) {
            // over h: (exp(L_0 h) - 1) / L_0 * pump   (h * pump when L_0 = 0)
            double2 c2;
            if (den == 0.0) {
                c2 = make_double2(a.h * p.x, a.h * p.y);
            } else {
                const double qr = (e2.x * Lr + e2.y * Li) / den;
                const double qi = (e2.y * Lr - e2.x * Li) / den;
                c2 = make_double2(qr * p.x - qi * p.y, qr * p.y + qi * p.x);
            }
            a.cpump2[i] = c2;
        }
        if (a.cphi) {
            // phi(L) = (exp(L hh) - 1)/L and phi'(L) = (hh exp(L hh) - phi(L))/L; for small
            // |z| = |L hh| the series phi'(L) = hh^2 sum_{k>=1} k z^(k-1)/(k+1)! (12 terms,
            // truncation below 1e-20 at |z| < 0.1) avoids the cancellation of the quotient
            const double zr = Lr * hh, zi = Li * hh;
            double2 phi, dphi;
            if (den == 0.0)
                phi = make_double2(hh, 0.0);
            else
                phi = make_double2((e1.x * Lr + e1.y * Li) / den, (e1.y * Lr - e1.x * Li) / den);
            if (zr * zr + zi * zi < 0.01) {
                double sr = 0.0, si = 0.0;   // Horner in z over k = 12 .. 1
                double fact = 1.0;           // (k+1)! for k = 12
                for (int k = 2; k <= 13; ++k)
                    fact *= k;
                for (int k = 12; k >= 1; --k) {
                    const double ck = (double)k / fact;
                    const double tr = sr * zr - si * zi + ck, ti = sr * zi + si * zr;
                    sr = tr;
                    si = ti;
                    fact /= (double)(k + 1);
                }
                dphi = make_double2(hh * hh * sr, hh * hh * si);
            } else {
                const double nr = hh * (e1.x + 1.0) - phi.x, ni = hh * e1.y - phi.y;
                dphi = make_double2((nr * Lr + ni * Li) / den, (ni * Lr - nr * Li) / den);
            }
            a.cphi[2 * i] = phi;
            a.cphi[2 * i + 1] = dphi;
        }
    }
}

// Centred public index of the mode stored at internal position q of an instance of size N.
// Up to N = 4096 the internal order is the transform order m = mu mod N; above, the four-step
// groups store mode m = m1 N2 + m2 column-major at q = m2 N1 + m1 (N1 = 2^ceil(log2 N / 2)),
// so that their column kernels read the per-mode state contiguously.
__device__ __forceinline__ int centred_of(int q, int N)
{
    int pm = q;
    if (N > 4096) {
        const int l = 31 - __clz(N);
        const int l1 = (l + 1) / 2;
        pm = ((q & ((1 << l1) - 1)) << (l - l1)) + (q >> l1);
    }
    return (pm + N / 2) & (N - 1);
}

// inst_M (may be null): per-instance physical mode count; padding modes are set to zero.
__global__ void import_kernel(int prec, int total, const int* mode_inst, const int* inst_N,
                              const long long* inst_off, const int* inst_M, const double2* src,
                              void* hi, void* lo)
{
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= total)
        return;
    const int i = mode_inst[m];
    const int N = inst_N[i];
    const long long off = inst_off[i];
    const int c = centred_of((int)(m - off), N);
    double2 v = src[off + c];
    if (inst_M) {
        const int M = inst_M[i], first = N / 2 - M / 2;
        if (c < first || c >= first + M)
            v = make_double2(0.0, 0.0);
    }
    if (prec == PREC_FP64) {
        reinterpret_cast<double2*>(hi)[m] = v;
    } else {
        const float hr = (float)v.x, hi_ = (float)v.y;
        reinterpret_cast<float2*>(hi)[m] = make_float2(hr, hi_);
        reinterpret_cast<float2*>(lo)[m] =
            make_float2((float)(v.x - (double)hr), (float)(v.y - (double)hi_));
    }
}

// what: 0 power (|D|^2 into a double array), 1 rotating-frame field, 2 Eq. 1 frame field.
__global__ void export_kernel(int prec, int total, const int* mode_inst, const int* inst_N,
                              const long long* inst_off, const void* hi, const void* lo,
                              double2* dst, int what, const double* omega, const double* sigma,
                              double tau)
{
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= total)
        return;
    const int i = mode_inst[m];
    const int N = inst_N[i];
    const long long off = inst_off[i];
    double2 v;
    if (prec == PREC_FP64) {
        v = reinterpret_cast<const double2*>(hi)[m];
    } else {
        const float2 a = reinterpret_cast<const float2*>(hi)[m];
        const float2 b = reinterpret_cast<const float2*>(lo)[m];
        v = make_double2((double)a.x + (double)b.x, (double)a.y + (double)b.y);
    }
    const long long c = off + centred_of((int)(m - off), N);
    if (what == 0) {
        reinterpret_cast<double*>(dst)[c] = v.x * v.x + v.y * v.y;
    } else if (what == 1) {
        dst[c] = v;
    } else {
        // A = D exp(-i (omega_mu - omega_0 - sigma) tau), phase in FP64
        double s, co;
        sincos(-(omega[m] - sigma[i]) * tau, &s, &co);
        dst[c] = make_double2(v.x * co - v.y * s, v.x * s + v.y * co);
    }
}

// Copy a transform-order array (diagnostics output) to FP64, optionally centring the order.
__global__ void export_plain_kernel(int prec, int total, const int* mode_inst, const int* inst_N,
                                    const long long* inst_off, const void* src, double2* dst,
                                    int reorder_centred)
{
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= total)
        return;
    double2 v;
    if (prec == PREC_FP64) {
        v = reinterpret_cast<const double2*>(src)[m];
    } else {
        const float2 a = reinterpret_cast<const float2*>(src)[m];
        v = make_double2(a.x, a.y);
    }
    long long c = m;
    if (reorder_centred) {
        const int i = mode_inst[m];
        const long long off = inst_off[i];
        c = off + centred_of((int)(m - off), inst_N[i]);
    }
    dst[c] = v;
}

// Independent FMA chains: 8 per thread, `iters` rounds.
template <typename T>
__global__ void fma_kernel(T* out, int iters, T a, T b)
{
    T x0 = threadIdx.x, x1 = x0 + 1, x2 = x0 + 2, x3 = x0 + 3, x4 = x0 + 4, x5 = x0 + 5,
      x6 = x0 + 6, x7 = x0 + 7;
    for (int k = 0; k < iters; ++k) {
#pragma unroll
        for (int u = 0; u < 16; ++u) {
            x0 = x0 * a + b;
            x1 = x1 * a + b;
            x2 = x2 * a + b;
            x3 = x3 * a + b;
            x4 = x4 * a + b;
            x5 = x5 * a + b;
            x6 = x6 * a + b;
            x7 = x7 * a + b;
        }
    }
    const T s = x0 + x1 + x2 + x3 + x4 + x5 + x6 + x7;
    if (s == (T)-1.2345)  // practically never: keeps the chains alive
        out[blockIdx.x * blockDim.x + threadIdx.x] = s;
}

__global__ void loss_seed_kernel(int prec, int total, const int* mode_inst, const int* inst_N,
                                 const long long* inst_off, const void* hi, const void* lo,
                                 const double* target, double eps, double* loss, void* dbar)
{
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= total)
        return;
    const int i = mode_inst[m];
    const int N = inst_N[i];
    const long long off = inst_off[i];
    double2 v;
    if (prec == PREC_FP64) {
        v = reinterpret_cast<const double2*>(hi)[m];
    } else {
        const float2 a = reinterpret_cast<const float2*>(hi)[m];
        const float2 b = reinterpret_cast<const float2*>(lo)[m];
        v = make_double2((double)a.x + (double)b.x, (double)a.y + (double)b.y);
    }
    const double P = v.x * v.x + v.y * v.y;
    const double r = log10(P + eps) - target[off + centred_of((int)(m - off), N)];
    loss[m] = r * r;   // per mode; summed per instance in a fixed order by grad_reduce
    const double g = 4.0 * r / ((P + eps) * 2.302585092994045684);  // 2 dL/dP, d|D|^2 = 2 Re(conj D dD)
    if (prec == PREC_FP64)
        reinterpret_cast<double2*>(dbar)[m] = make_double2(g * v.x, g * v.y);
    else
        reinterpret_cast<float2*>(dbar)[m] = make_float2((float)(g * v.x), (float)(g * v.y));
}

__global__ void strang_pump_grad_kernel(int count, const long long* inst_off,
                                        const double2* cphi, const double2* pump, double2* pbar,
                                        double2* gL)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count)
        return;
    const double2 cb = pbar[i], phi = cphi[2 * i], dphi = cphi[2 * i + 1], p = pump[i];
    // conj(phi) cbar
    pbar[i] = make_double2(phi.x * cb.x + phi.y * cb.y, phi.x * cb.y - phi.y * cb.x);
    // conj(p phi') cbar, added at the pumped mode (transform position 0 of the instance)
    const double qr = p.x * dphi.x - p.y * dphi.y, qi = p.x * dphi.y + p.y * dphi.x;
    double2 g = gL[inst_off[i]];
    g.x += qr * cb.x + qi * cb.y;
    g.y += qr * cb.y - qi * cb.x;
    gL[inst_off[i]] = g;
}

__global__ void grad_reduce_kernel(const int* inst_N, const long long* inst_off, const double2* gL,
                                   const double* loss_modes, double* red)
{
    const int i = blockIdx.x;
    const int N = inst_N[i];
    const long long off = inst_off[i];
    double s0 = 0, s2 = 0, s3 = 0, sl = 0;
    for (int pm = threadIdx.x; pm < N; pm += blockDim.x) {
        const double mu = pm < N / 2 ? pm : pm - N;   // transform position -> mode number
        const double g = gL[off + pm].y;
        s0 += g;
        s2 += g * mu * mu * 0.5;
        s3 += g * mu * mu * mu / 6.0;
        sl += loss_modes[off + pm];
    }
    __shared__ double sh[4][256];
    sh[0][threadIdx.x] = s0;
    sh[1][threadIdx.x] = s2;
    sh[2][threadIdx.x] = s3;
    sh[3][threadIdx.x] = sl;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w)
            for (int k = 0; k < 4; ++k)
                sh[k][threadIdx.x] += sh[k][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        red[4 * i + 0] = sh[0][0];
        red[4 * i + 1] = sh[1][0];
        red[4 * i + 2] = sh[2][0];
        red[4 * i + 3] = sh[3][0];
    }
}

__global__ void grad_export_kernel(int prec, int total, const int* mode_inst, const int* inst_N,
                                   const long long* inst_off, const void* dbar,
                                   const double2* gL, const double* red, double2* dD0,
                                   double* domega, double* dkappa)
{
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= total)
        return;
    const int i = mode_inst[m];
    const int N = inst_N[i];
    const long long off = inst_off[i];
    const long long c = off + centred_of((int)(m - off), N);
    double2 d;
    if (prec == PREC_FP64) {
        d = reinterpret_cast<const double2*>(dbar)[m];
    } else {
        const float2 a = reinterpret_cast<const float2*>(dbar)[m];
        d = make_double2(a.x, a.y);
    }
    if (dD0)
        dD0[c] = d;
    if (domega)
        domega[c] = gL[m].y - (m == off ? red[4 * i] : 0.0);
    if (dkappa)
        dkappa[c] = -0.5 * gL[m].x;
}

inline int nblocks(long long n, int t) { return (int)((n + t - 1) / t); }

}  // namespace

cudaError_t launch_twiddles(int N, int prec, void* out, cudaStream_t s)
{
    twiddle_kernel<<<nblocks(N, 256), 256, 0, s>>>(N, prec, out);
    return cudaGetLastError();
}

cudaError_t launch_propagators(const PropArgs& a, cudaStream_t s)
{
    if (a.prec == PREC_FP64)
        prop_kernel<double2><<<nblocks(a.total, 256), 256, 0, s>>>(a);
    else
        prop_kernel<float2><<<nblocks(a.total, 256), 256, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_import(int prec, int total, const int* mode_inst, const int* inst_N,
                          const long long* inst_off, const int* inst_M, const double2* src,
                          void* hi, void* lo, cudaStream_t s)
{
    import_kernel<<<nblocks(total, 256), 256, 0, s>>>(prec, total, mode_inst, inst_N, inst_off,
                                                       inst_M, src, hi, lo);
    return cudaGetLastError();
}

cudaError_t launch_export(int prec, int total, const int* mode_inst, const int* inst_N,
                          const long long* inst_off, const void* hi, const void* lo,
                          double2* dst, int what, const double* omega, const double* sigma,
                          double tau, cudaStream_t s)
{
    export_kernel<<<nblocks(total, 256), 256, 0, s>>>(prec, total, mode_inst, inst_N, inst_off,
                                                       hi, lo, dst, what, omega, sigma, tau);
    return cudaGetLastError();
}

cudaError_t launch_export_plain(int prec, int total, const int* mode_inst, const int* inst_N,
                                const long long* inst_off, const void* src, double2* dst,
                                int reorder_centred, cudaStream_t s)
{
    export_plain_kernel<<<nblocks(total, 256), 256, 0, s>>>(prec, total, mode_inst, inst_N,
                                                             inst_off, src, dst,
                                                             reorder_centred);
    return cudaGetLastError();
}

cudaError_t launch_loss_seed(int prec, int total, const int* mode_inst, const int* inst_N,
                             const long long* inst_off, const void* hi, const void* lo,
                             const double* target, double eps, double* loss, void* dbar,
                             cudaStream_t s)
{
    loss_seed_kernel<<<nblocks(total, 256), 256, 0, s>>>(prec, total, mode_inst, inst_N, inst_off,
                                                          hi, lo, target, eps, loss, dbar);
    return cudaGetLastError();
}

cudaError_t launch_strang_pump_grad(int count, const long long* inst_off, const double2* cphi,
                                    const double2* pump, double2* pbar, double2* gL,
                                    cudaStream_t s)
{
    strang_pump_grad_kernel<<<nblocks(count, 128), 128, 0, s>>>(count, inst_off, cphi, pump,
                                                                 pbar, gL);
    return cudaGetLastError();
}

cudaError_t launch_grad_reduce(int count, const int* inst_N, const long long* inst_off,
                               const double2* gL, const double* loss_modes, double* red,
                               cudaStream_t s)
{
    grad_reduce_kernel<<<count, 256, 0, s>>>(inst_N, inst_off, gL, loss_modes, red);
    return cudaGetLastError();
}

cudaError_t launch_grad_export(int prec, int total, const int* mode_inst, const int* inst_N,
                               const long long* inst_off, const void* dbar, const double2* gL,
                               const double* red, double2* dD0, double* domega, double* dkappa,
                               cudaStream_t s)
{
    grad_export_kernel<<<nblocks(total, 256), 256, 0, s>>>(prec, total, mode_inst, inst_N,
                                                            inst_off, dbar, gL, red, dD0, domega,
                                                            dkappa);
    return cudaGetLastError();
}

// Copies within a buffer pair that stays resident in L2, `reps` passes per launch (float4 per
// thread, grid-stride; pass r reads at a rotated offset, and the accesses are volatile PTX, so
// no pass is merged with another).  For the L2 bandwidth the large-N kernels are measured
// against.
__device__ __forceinline__ float4 ld_v4(const float4* p)
{
    float4 v;
    asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_v4(float4* p, float4 v)
{
    asm volatile("st.global.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v.x), "f"(v.y),
                 "f"(v.z), "f"(v.w) : "memory");
}
__global__ void l2_copy_kernel(const float4* src, float4* dst, long long n, int reps)
{
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (int r = 0; r < reps; ++r)
        for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
            st_v4(dst + i, ld_v4(src + ((i + 4099LL * r) & (n - 1))));
}

cudaError_t run_l2_peak(size_t bytes, double* bytes_per_s)
{
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess)
        e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess)
        return e;
    size_t n = 1;   // float4 elements per buffer: the largest power of two that fits
    while (n * 2 * 16 <= bytes)
        n *= 2;
    void* buf = nullptr;
    e = cudaMalloc(&buf, 2 * n * 16);
    if (e != cudaSuccess)
        return e;
    cudaMemset(buf, 0, 2 * n * 16);
    const float4* src = reinterpret_cast<const float4*>(buf);
    float4* dst = reinterpret_cast<float4*>(buf) + n;
    cudaEvent_t a, b;
    cudaEventCreate(&a);
    cudaEventCreate(&b);
    float best = 1e30f;
    const int reps = 32;
    for (int rep = 0; rep < 5; ++rep) {
        cudaEventRecord(a);
        l2_copy_kernel<<<sms * 4, 512>>>(src, dst, (long long)n, reps);
        cudaEventRecord(b);
        cudaEventSynchronize(b);
        float ms = 0;
        cudaEventElapsedTime(&ms, a, b);
        if (rep > 0 && ms < best)   // the first launch brings the buffers into L2
            best = ms;
    }
    e = cudaGetLastError();
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    cudaFree(buf);
    *bytes_per_s = 2.0 * (double)n * 16.0 * reps / (best * 1e-3);
    return e;
}

cudaError_t run_fma_peak(int prec, double* flops)
{
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess)
        return e;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess)
        return e;
    void* out = nullptr;
    e = cudaMalloc(&out, 1 << 24);
    if (e != cudaSuccess)
        return e;
    cudaEvent_t a, b;
    cudaEventCreate(&a);
    cudaEventCreate(&b);
    const int threads = 512, blocks = sms * 4;
    const int iters = prec == PREC_FP64 ? 64 : 2048;
    float best = 1e30f;
    for (int rep = 0; rep < 4; ++rep) {
        cudaEventRecord(a);
        if (prec == PREC_FP64)
            fma_kernel<double><<<blocks, threads>>>((double*)out, iters, 0.999999, 1e-7);
        else
            fma_kernel<float><<<blocks, threads>>>((float*)out, iters, 0.999999f, 1e-7f);
        cudaEventRecord(b);
        cudaEventSynchronize(b);
        float ms = 0;
        cudaEventElapsedTime(&ms, a, b);
        if (rep > 0 && ms < best)
            best = ms;
    }
    e = cudaGetLastError();
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    cudaFree(out);
    const double fmas = (double)blocks * threads * iters * 16.0 * 8.0;
    *flops = 2.0 * fmas / (best * 1e-3);
    return e;
}

}  // namespace cme
