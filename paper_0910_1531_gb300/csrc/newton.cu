// Newton-Krylov solver of the fixed point rho = G(rho) (Sec. "Nonlinear solver" mentions
// Newton-GMRES as the alternative it tried): F(u) = u - log G(e^u) on the accessible voxels
// (u = log rho), Jacobian-vector products by finite differences of F (each one G evaluation),
// restarted GMRES with modified Gram-Schmidt and Givens rotations on the host, and a
// backtracking line search on |F|.  Elementwise kernels over the S N field here; G comes from
// the plan's Picard map.
#include <cmath>
#include <vector>

#include "common.cuh"
#include "newton.h"

namespace {

constexpr int kNkThreads = 256;

template <typename Real>
__global__ void k_nk_residual(const Real* __restrict__ rho, const Real* __restrict__ g, const Real* __restrict__ V,
                              Real* __restrict__ F, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const Real v = V[i];
        F[i] = (isinf(v) && v > Real(0)) ? Real(0) : log(rho[i]) - log(g[i]);
    }
}

// out = rho exp(s d) on accessible voxels, 0 elsewhere
template <typename Real>
__global__ void k_nk_step(const Real* __restrict__ rho, const Real* __restrict__ d, Real s, const Real* __restrict__ V,
                          Real* __restrict__ out, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const Real v = V[i];
        out[i] = (isinf(v) && v > Real(0)) ? Real(0) : rho[i] * exp(s * d[i]);
    }
}

// out = ((log rho_p - log g_p) - F) / eps on accessible voxels
template <typename Real>
__global__ void k_nk_jv(const Real* __restrict__ rho_p, const Real* __restrict__ g_p, const Real* __restrict__ F,
                        const Real* __restrict__ V, Real inv_eps, Real* __restrict__ out, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const Real v = V[i];
        out[i] = (isinf(v) && v > Real(0)) ? Real(0) : ((log(rho_p[i]) - log(g_p[i])) - F[i]) * inv_eps;
    }
}

// per-block partial sums of a * b, accumulated in FP64
template <typename Real>
__global__ void __launch_bounds__(kNkThreads) k_nk_dot(const Real* __restrict__ a, const Real* __restrict__ b,
                                                       long long n, double* __restrict__ partial) {
    __shared__ double sh[kNkThreads / 32];
    double s = 0.0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        s += double(a[i]) * double(b[i]);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kNkThreads / 32; ++w) t += sh[w];
        partial[blockIdx.x] = t;
    }
}

// One step of modified Gram-Schmidt: w -= h v_prev, with h the sum of the previous step's nparts
// partials (stored at h_out), and this step's partials of w . v_next (v_next NULL: w . w).  v_prev NULL: no
// subtraction (the first step).  Every block sums the partials itself, so that a product's steps follow
// one another without the host: bound by launch latency on small grids (4 x 4 x 512: 2.3 us for a dot and
// 1.5 for its update as kernels of their own, and some 15 for the host to read each dot; the whole solve
// 31.6 -> 25.0 ms).
template <typename Real>
__global__ void __launch_bounds__(kNkThreads) k_nk_mgs(const Real* __restrict__ v_prev, const Real* __restrict__ v_next,
                                                       Real* __restrict__ w, long long n,
                                                       const double* __restrict__ part_in, int nparts,
                                                       double* __restrict__ h_out, double* __restrict__ part_out) {
    __shared__ double sh[kNkThreads / 32];
    auto block_sum = [&](double s) {        // of all threads, to every thread
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
        __syncthreads();
        double t = 0.0;
        for (int k = 0; k < kNkThreads / 32; ++k) t += sh[k];
        __syncthreads();
        return t;
    };
    Real mh = Real(0);
    if (v_prev) {
        double s = 0.0;
        for (int k = threadIdx.x; k < nparts; k += kNkThreads) s += part_in[k];
        const double h = block_sum(s);
        if (blockIdx.x == 0 && threadIdx.x == 0) *h_out = h;
        mh = Real(-h);
    }
    double s = 0.0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        Real wi = w[i];
        if (v_prev) w[i] = wi = mh * v_prev[i] + wi;
        s += double(wi) * double(v_next ? v_next[i] : wi);
    }
    s = block_sum(s);
    if (threadIdx.x == 0) part_out[blockIdx.x] = s;
}

// y = alpha x + beta y
template <typename Real>
__global__ void k_nk_axpby(Real alpha, const Real* __restrict__ x, Real beta, Real* __restrict__ y, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        y[i] = alpha * x[i] + beta * y[i];
}

}  // namespace

template <typename Real>
NkVec<Real>::NkVec(cudaStream_t st, long long n, int grid) : st_(st), n_(n), grid_(grid) {}

template <typename Real>
cudaError_t NkVec<Real>::residual(const Real* rho, const Real* g, const Real* V, Real* F) const {
    k_nk_residual<Real><<<grid_, kNkThreads, 0, st_>>>(rho, g, V, F, n_);
    return cudaGetLastError();
}

template <typename Real>
cudaError_t NkVec<Real>::step(const Real* rho, const Real* d, double s, const Real* V, Real* out) const {
    k_nk_step<Real><<<grid_, kNkThreads, 0, st_>>>(rho, d, Real(s), V, out, n_);
    return cudaGetLastError();
}

template <typename Real>
cudaError_t NkVec<Real>::jv(const Real* rho_p, const Real* g_p, const Real* F, const Real* V, double eps, Real* out) const {
    k_nk_jv<Real><<<grid_, kNkThreads, 0, st_>>>(rho_p, g_p, F, V, Real(1.0 / eps), out, n_);
    return cudaGetLastError();
}

template <typename Real>
cudaError_t NkVec<Real>::axpby(double alpha, const Real* x, double beta, Real* y) const {
    k_nk_axpby<Real><<<grid_, kNkThreads, 0, st_>>>(Real(alpha), x, Real(beta), y, n_);
    return cudaGetLastError();
}

template <typename Real>
cudaError_t NkVec<Real>::orthogonalise(const Real* basis, int k, Real* w, double* dev) const {
    double* const h = dev + 2 * grid_;
    for (int i = 0; i <= k; ++i) {
        k_nk_mgs<Real><<<grid_, kNkThreads, 0, st_>>>(i ? basis + size_t(i - 1) * n_ : nullptr,
                                                      i < k ? basis + size_t(i) * n_ : nullptr, w, n_,
                                                      dev + ((i + 1) & 1) * grid_, grid_, h + (i ? i - 1 : 0),
                                                      dev + (i & 1) * grid_);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <typename Real>
cudaError_t NkVec<Real>::read_column(int k, const double* dev, double* host, double* h_out, double* ww_out) const {
    cudaError_t e = cudaMemcpyAsync(host, dev, sizeof(double) * (2 * grid_ + k), cudaMemcpyDeviceToHost, st_);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st_);
    if (e != cudaSuccess) return e;
    for (int i = 0; i < k; ++i) h_out[i] = host[2 * grid_ + i];
    double t = 0.0;
    for (int i = 0; i < grid_; ++i) t += host[(k & 1) * grid_ + i];
    *ww_out = t;
    return cudaSuccess;
}

template <typename Real>
cudaError_t NkVec<Real>::dot(const Real* a, const Real* b, double* partial_dev, double* partial_host, double* out) const {
    k_nk_dot<Real><<<grid_, kNkThreads, 0, st_>>>(a, b, n_, partial_dev);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(partial_host, partial_dev, sizeof(double) * grid_, cudaMemcpyDeviceToHost, st_);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st_);
    if (e != cudaSuccess) return e;
    double t = 0.0;
    for (int i = 0; i < grid_; ++i) t += partial_host[i];
    *out = t;
    return cudaSuccess;
}

template class NkVec<float>;
template class NkVec<double>;
