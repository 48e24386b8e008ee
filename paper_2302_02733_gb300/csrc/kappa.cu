// Kappa-distribution coefficients by quadrature: the synchrotron-kernel tables and the batch
// kernel behind rt_kappa_coeffs (one thread per point).
#include "kappa.cuh"
#include "rt_kernels.cuh"

namespace prt {

// Polynomials of K(x) e^x x^(-1/3) in t = -1 .. 1 on each interval of ln x: the values at the 8
// Chebyshev nodes (one thread each, 16 intervals a block), their Chebyshev coefficients, and from
// those the powers of t (the series falls off fast enough for the powers to lose nothing).
constexpr int kSynPerBlock = 16;
__global__ void __launch_bounds__(8 * kSynPerBlock) synch_poly_kernel(double *kern) {
    __shared__ double f[3][kSynPerBlock][8], ch[3][kSynPerBlock][8];
    const int li = threadIdx.x >> 3, j = threadIdx.x & 7, i = blockIdx.x * kSynPerBlock + li;
    const double t = cospi((j + 0.5) * 0.125), lx = kSynLo + (i + 0.5 + 0.5 * t) * 0.125, x = exp(lx);
    double k[3];
    synch_kernels_scaled(x, k);
    for (int m = 0; m < 3; m++) f[m][li][j] = k[m] * exp(-lx * (1.0 / 3.0));
    __syncthreads();
    for (int m = 0; m < 3; m++) {
        double s = 0.0;
        for (int n = 0; n < 8; n++) s += f[m][li][n] * cospi(j * (n + 0.5) * 0.125);
        ch[m][li][j] = s * (j == 0 ? 0.125 : 0.25);
    }
    __syncthreads();
    if (i >= kSynN || j >= 3) return;
    double p[8] = {0}, a[8] = {1, 0, 0, 0, 0, 0, 0, 0}, b[8] = {0, 1, 0, 0, 0, 0, 0, 0};  // T_n, T_n+1
    for (int n = 0; n < 8; n++) {
        double c[8];
        for (int q = 0; q < 8; q++) {
            p[q] += ch[j][li][n] * a[q];
            c[q] = (q > 0 ? 2.0 * b[q - 1] : 0.0) - a[q];
        }
        for (int q = 0; q < 8; q++) a[q] = b[q], b[q] = c[q];
    }
    for (int q = 0; q < 8; q++) kern[(3 * i + j) * 8 + q] = p[q];
}

__global__ void kap_node_kernel(KapNode *node) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < kKapN) node[k] = kap_node(kKapLo + k * kKapH);
}

__global__ void kappa_quad_kernel(KappaTables T, const double *in, double *out, long long n) {
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
        const double *v = in + 6 * q;
        double o[8];
        kappa_coeffs_quad(T, v[0], v[1], v[2], v[3], v[4], v[5], o);
#pragma unroll
        for (int k = 0; k < 8; k++) out[8 * q + k] = o[k];
    }
}

KappaTables kappa_tables(const double *buf) {
    return KappaTables{buf, reinterpret_cast<const KapNode *>(buf + 24 * kSynN)};
}

static_assert(kKapTabBytes == sizeof(double) * 24 * kSynN + sizeof(KapNode) * kKapN, "kappa tables' size");

int launch_kappa_tables(double *buf, cudaStream_t s) {
    synch_poly_kernel<<<(kSynN + kSynPerBlock - 1) / kSynPerBlock, 8 * kSynPerBlock, 0, s>>>(buf);
    kap_node_kernel<<<(kKapN + 127) / 128, 128, 0, s>>>(reinterpret_cast<KapNode *>(buf + 24 * kSynN));
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

void launch_kappa_quad(const KappaTables &T, const double *in, double *out, long long n, int grid, cudaStream_t s) {
    kappa_quad_kernel<<<grid, 128, 0, s>>>(T, in, out, n);
}

}  // namespace prt
