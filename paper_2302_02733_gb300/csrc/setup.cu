// Set-up and reduction kernels: the FMKS inverse table and the image statistics.
#include "transfer.cuh"

namespace prt {

// Table of X2(w, theta) for the FMKS map theta = theta_G(X2) + w (theta_J(X2) - theta_G(X2)),
// w in [0, 1] (64 rows), theta in [0, pi] (1024 columns), by bisection to the last bit. The
// transfer kernels start Newton's method from a bilinear read of this table.
__global__ void x2_table_kernel(GridModel g, double *tab, float *tabf) {
    int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= kX2TabW * kX2TabT) return;
    int iw = idx / kX2TabT, it = idx % kX2TabT;
    double w = (double)iw / (kX2TabW - 1);
    double th = kPi * (double)it / (kX2TabT - 1);
    double lo = 0.0, hi = 1.0;
    for (int k = 0; k < 70; k++) {
        double mid = 0.5 * (lo + hi);
        if (fmks_theta_w<double>(g, w, mid, nullptr, nullptr) < th)
            lo = mid;
        else
            hi = mid;
    }
    tab[idx] = 0.5 * (lo + hi);
    tabf[idx] = (float)(0.5 * (lo + hi));
}

void launch_x2_table(const GridModel &g, double *table, float *table_f, cudaStream_t s) {
    int n = kX2TabW * kX2TabT;
    x2_table_kernel<<<(n + 255) / 256, 256, 0, s>>>(g, table, table_f);
}

// The FP64 tables of ThermTab: on each segment the functions at the D + 1 Chebyshev nodes (one thread
// each), their Chebyshev coefficients (one a thread), and from those the powers of u (one thread a function).
__device__ void bessel_ratio_values(double Te, double v[2]) {
    // K_n(z) e^z = int_0^inf e^{-2 z sinh^2(t/2)} cosh(n t) dt by the trapezoid rule
    const double z = 1.0 / Te, h = 0.125 * fmin(1.0, rsqrt(z));
    double s0 = 0.5, s1 = 0.5, s2 = 0.5;
    for (int k = 1; k < 100000; k++) {
        const double t = k * h, sh = sinh(0.5 * t), e = 2.0 * z * sh * sh;
        if (e > 2.0 * t + 60.0) break;
        const double w = exp(-e), c = cosh(t);
        s0 += w;
        s1 += w * c;
        s2 += w * (2.0 * c * c - 1.0);
    }
    v[0] = s0 / s2;
    v[1] = s1 / s2;
}
__device__ void shcherbakov_values(double X, double v[2]) {
    v[0] = shcherbakov_fX(X);
    v[1] = 1.0 - 0.11 * log1p(0.035 * X);
}

constexpr int kThermPerBlock = 16;
template <int D, void (*fn)(double, double *)>
__global__ void therm_table_kernel(double *tab, int bits, int e0) {
    __shared__ double f[2][kThermPerBlock][D + 1], ch[2][kThermPerBlock][D + 1];
    const int li = threadIdx.x / (D + 1), j = threadIdx.x % (D + 1), i = blockIdx.x * kThermPerBlock + li;
    double v[2];
    fn(ThermTab::at(i, bits, e0, cospi((j + 0.5) / (D + 1))), v);
    f[0][li][j] = v[0];
    f[1][li][j] = v[1];
    __syncthreads();
    for (int m = 0; m < 2; m++) ch[m][li][j] = therm_chebyshev<D>(f[m][li], j);
    __syncthreads();
    if (j >= 2) return;
    double p[D + 1];
    therm_powers<D>(ch[j][li], p);
    for (int q = 0; q <= D; q++) tab[(2 * i + j) * (D + 1) + q] = p[q];
}

int launch_thermal_tables(double *buf, cudaStream_t s) {
    typedef ThermTab T;
    constexpr int B = kThermPerBlock;
    static_assert(T::nb % B == 0 && T::ns % B == 0 && T::nf % B == 0, "whole blocks");
    therm_table_kernel<T::db, bessel_ratio_values><<<T::nb / B, B * (T::db + 1), 0, s>>>(buf + T::bes, 4, T::eb);
    therm_table_kernel<T::ds, shcherbakov_values><<<T::ns / B, B * (T::ds + 1), 0, s>>>(buf + T::shc, 4, T::es);
    therm_table_kernel<T::ds, shcherbakov_values>
        <<<T::nf / B, B * (T::ds + 1), 0, s>>>(buf + T::shc + T::ns * 2 * (T::ds + 1), 6, T::ef);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// Image statistics in two deterministic passes: each block takes a fixed contiguous range of
// pixels, sums it with Kahan compensation per thread and a pairwise tree in shared memory, and
// writes its partial sums; one block then adds the partials in block order. The epilogue forms
// the flux sum(I) dOmega 1e23 [Jy] and the net polarization fractions.
constexpr int kStatThreads = 256;

template <typename T, int NC>  // NC components per pixel: 4 (IQUV) or 1 (I)
__global__ void __launch_bounds__(kStatThreads) image_partial_kernel(const T *img, long long npix, double *part) {
    __shared__ double sh[4][kStatThreads];
    long long per = (npix + gridDim.x - 1) / gridDim.x;
    long long p0 = (long long)blockIdx.x * per, p1 = min(npix, p0 + per);
    double s[4] = {0, 0, 0, 0}, cmp[4] = {0, 0, 0, 0};
    for (long long p = p0 + threadIdx.x; p < p1; p += kStatThreads) {
#pragma unroll
        for (int k = 0; k < NC; k++) {
            double y = (double)img[NC * p + k] - cmp[k];
            double t = s[k] + y;
            cmp[k] = (t - s[k]) - y;
            s[k] = t;
        }
    }
#pragma unroll
    for (int k = 0; k < 4; k++) sh[k][threadIdx.x] = s[k];
    __syncthreads();
    for (int w = kStatThreads / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w)
#pragma unroll
            for (int k = 0; k < 4; k++) sh[k][threadIdx.x] += sh[k][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x < 4) part[4 * blockIdx.x + threadIdx.x] = sh[threadIdx.x][0];
}

__global__ void image_final_kernel(const double *part, int nblocks, double domega, double *out) {
    if (threadIdx.x != 0) return;
    double s[4] = {0, 0, 0, 0}, cmp[4] = {0, 0, 0, 0};
    for (int b = 0; b < nblocks; b++)
        for (int k = 0; k < 4; k++) {
            double y = part[4 * b + k] - cmp[k];
            double t = s[k] + y;
            cmp[k] = (t - s[k]) - y;
            s[k] = t;
        }
    double I = s[0], Q = s[1], U = s[2], V = s[3];
    out[0] = I;
    out[1] = Q;
    out[2] = U;
    out[3] = V;
    out[4] = I * domega * 1e23;
    out[5] = sqrt(Q * Q + U * U) / I;
    out[6] = V / I;
}

// out must hold 8 + 4 * kStatBlocks doubles (the partials live after the 7 results).
void launch_image_sums(const void *img, int form, long long npix, double domega, double *out, cudaStream_t s) {
    double *part = out + 8;
    if (form == 0)
        image_partial_kernel<double, 4><<<kStatBlocks, kStatThreads, 0, s>>>((const double *)img, npix, part);
    else if (form == 1)
        image_partial_kernel<float, 4><<<kStatBlocks, kStatThreads, 0, s>>>((const float *)img, npix, part);
    else
        image_partial_kernel<float, 1><<<kStatBlocks, kStatThreads, 0, s>>>((const float *)img, npix, part);
    image_final_kernel<<<1, 32, 0, s>>>(part, kStatBlocks, domega, out);
}

}  // namespace prt
