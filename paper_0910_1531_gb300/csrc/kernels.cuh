// Pass kernels of one residual evaluation G(rho) (Sec. "Discretization and Solution
// in Equilibrium"): every 3D transform is split into an x pass (rows, real <-> half
// spectrum), a y pass and a z pass (column tiles), and the pointwise work rides
// inside those passes:
//
//   first half  (rho -> weighted densities of eq. nDef, bulk-fluid + Poisson spectra)
//     k_xfwd     x R2C of the S densities
//     k_yfft_tma   y forward (k_colfft for lengths without compile-time kernels)
//     k_zconv_fwd_*  z forward, the analytic weights of App. B (n_hat_alpha), the
//                bulk-fluid kernel (eq. CplusPsiHat) and the Poisson symbol
//                (eq. potentialSolution) applied in k space, z inverse of seven
//                weighted-density spectra; or as three passes (k_colfft / k_yfft_tma, k_zmul)
//     k_yfft_tma   y inverse of the nine spectra (the two y derivatives formed on the way in;
//                the x derivatives are formed in k_xphi)
//   second half (weighted densities -> c1 -> G)
//     k_xphi     x C2R to the ten n, dPhi/dn_alpha of eq. Phi (|nV2| <= n2 bound,
//                FP64 log(1-n3) and 1/(1-n3)^m; or another hard-sphere form), x R2C back
//                to nine spectra
//     k_yfft_tma   y forward, the two y-derivative spectra added into two others: seven out
//     k_zconv_bwd_*  z forward, adjoint weights (eq. muHS), + bulk-fluid/Poisson spectra,
//                z inverse of the S one-body correlations; or as three passes (k_zmul_bwd)
//     k_yfft_tma   y inverse
//     k_xupdate  x C2R and the update G_i = rho_bath_i exp(mu_HS_bath_i - V_i + c1_i)
//                (eq. rhoEquation), mixing of rho for the line search, residual sums
//
// Linear stages carry mixing weights (read from the device control block) so that
// n_alpha at a line-search point is the mix of two stored weighted-density sets:
// n3, and every n_alpha, is linear in rho (Sec. "Nonlinear solver").
#pragma once

#include <math_constants.h>

#include <type_traits>

#include "common.cuh"
#include "fft.cuh"
#include "passes.h"
#include "tma.cuh"

namespace dftk {

constexpr int kThreads = 256;
// the one-block line-search bookkeeping kernel: 1024 threads for many partial results, 256 for
// few (small grids, where its latency is all that counts)
constexpr int kFinThreads = 1024, kFinThreadsSmall = 256;


template <typename Real> __device__ __forceinline__ void sc(Real x, Real* s, Real* c);
template <> __device__ __forceinline__ void sc<float>(float x, float* s, float* c) { sincosf(x, s, c); }
template <> __device__ __forceinline__ void sc<double>(double x, double* s, double* c) { sincos(x, s, c); }

// Wave number of index j on an axis of n points (eq. Kvalues); kf = 2 pi / (n h).
template <typename Real> __device__ __forceinline__ Real kval(int j, int n, Real kf) {
    return (2 * j <= n) ? Real(j) * kf : -Real(n - j) * kf;
}

// Power series sum_m (-1)^m y^(2m) / ((2m+1)! (2m+q)) in t = y^2, q = n + 3 of the ball
// integral (4 pi / k) I_n = 4 pi R^(n+3) * series (expansion of sin(k r) under the integral).
__host__ __device__ constexpr double series_coef(int m, int q) {
    double f = 1.0;
    for (int i = 2; i <= 2 * m + 1; ++i) f *= double(i);
    return ((m & 1) ? -1.0 : 1.0) / (f * double(2 * m + q));
}

template <typename Real, int Q> __device__ __forceinline__ Real ball_series(Real t) {
    constexpr int M = sizeof(Real) == 4 ? 9 : 11;
    Real acc = Real(0);
#pragma unroll
    for (int m = M - 1; m >= 0; --m) acc = acc * t + Real(series_coef(m, Q));
    return acc;
}

template <typename Real> __device__ __forceinline__ Real series_cut() { return sizeof(Real) == 4 ? Real(1.5) : Real(1.0); }

// (sin x - x cos x) / x^3 (1/3 at x = 0), s = sin x, c = cos x
template <typename Real> __device__ __forceinline__ Real sinc3(Real x, Real s, Real c) {
    if (x < series_cut<Real>()) return ball_series<Real, 3>(x * x);
    return (s - x * c) / (x * x * x);
}

// FMT scalar weights of App. B for one species at |k| (x = |k| R).  Returns w0 (w1 = R w0,
// w2 = 4 pi R^2 w0) and j3 = (sin x - x cos x)/x^3 (w3 = 4 pi R^3 j3).
template <typename Real> __device__ __forceinline__ void fmt_weights(Real kmag, Real R, Real* w0, Real* j3) {
    const Real x = kmag * R;
    Real s, c;
    sc<Real>(x, &s, &c);
    if (x < series_cut<Real>()) {
        // sin x / x series for accuracy next to the series of j3
        const Real t = x * x;
        *w0 = Real(1) + t * (Real(-1.0 / 6) + t * (Real(1.0 / 120) + t * (Real(-1.0 / 5040) + t * (Real(1.0 / 362880)
              + t * (Real(-1.0 / 39916800) + t * Real(1.0 / 6227020800.0))))));
    } else {
        *w0 = s / x;
    }
    *j3 = sinc3<Real>(x, s, c);
}

// Bulk-fluid kernel DC_ij_hat(|k|) of eq. CplusPsiHat (prefactor 2 pi lambda_B z_i z_j / k, i.e.
// (lambda_B z_i z_j / 2)(4 pi / k) I_n) in kT units.
template <typename Real>
__device__ __forceinline__ Real delta_c_hat(Real kmag, Real R, Real pref, Real a, Real b, Real c,
                                           Real* dGamma = nullptr, Real da = 0, Real db = 0, Real dc = 0) {
    const Real y = kmag * R;
    Real bm1, b0, b1;   // (4 pi / k) I_n / (4 pi R^(n+3))
    if (y < series_cut<Real>()) {
        const Real t = y * y;
        bm1 = ball_series<Real, 2>(t);
        b0 = ball_series<Real, 3>(t);
        b1 = ball_series<Real, 4>(t);
    } else {
        Real s, co;
        sc<Real>(y, &s, &co);
        Real sh, chh;
        sc<Real>(Real(0.5) * y, &sh, &chh);
        const Real omc = Real(2) * sh * sh;           // 1 - cos y, without cancellation
        const Real iy = Real(1) / y;
        const Real iy2 = iy * iy;
        bm1 = omc * iy2;
        b0 = (s - y * co) * iy2 * iy;
        b1 = -co * iy2 + Real(2) * s * iy2 * iy - Real(2) * omc * iy2 * iy2;
    }
    const Real R2 = R * R;
    const Real fourpi = Real(4.0 * CUDART_PI);
    // the Gamma dependence sits in the coefficients only (l_k = R_k + 1/(2 Gamma))
    if (dGamma) *dGamma = pref * fourpi * R2 * (da * R2 * b1 - db * R * b0 + dc * bm1);
    return pref * fourpi * R2 * (a * R2 * b1 - b * R * b0 + c * bm1);
}

// ------------------------------------------------------------------------------------
// Reductions
// ------------------------------------------------------------------------------------
__device__ __forceinline__ double block_sum(double v, double* scratch) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) scratch[w] = v;
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x < 32) {
        r = (l < (int)(blockDim.x >> 5)) ? scratch[l] : 0.0;
        for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    }
    return r;   // valid in thread 0
}

// Block sum of per-thread FP32 pairs (hi, lo) kept as a double-single (hi + lo) through the
// warp shuffles (error-free TwoSum of the high parts, Knuth), then in FP64 across the warps:
// about 48 significant bits at FP32 cost, where FP64 shuffles and adds would queue on the
// narrow FP64 pipe.  Result valid in thread 0.
__device__ __forceinline__ void ds_add(float& hi, float& lo, float bhi, float blo) {
    const float s = hi + bhi;
    const float bb = s - hi;
    const float err = (hi - (s - bb)) + (bhi - bb);
    const float l = err + lo + blo;
    hi = s + l;
    lo = l - (hi - s);
}

__device__ __forceinline__ double block_sum_ds(float hi, float lo, double* scratch) {
    for (int o = 16; o > 0; o >>= 1) {
        const float bh = __shfl_xor_sync(0xffffffffu, hi, o), bl = __shfl_xor_sync(0xffffffffu, lo, o);
        ds_add(hi, lo, bh, bl);
    }
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) scratch[w] = double(hi) + double(lo);
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) r += scratch[i];
    return r;
}

__device__ __forceinline__ float block_max(float v, float* scratch) {
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) scratch[w] = v;
    __syncthreads();
    float r = -CUDART_INF_F;
    if (threadIdx.x < 32) {
        r = (l < (int)(blockDim.x >> 5)) ? scratch[l] : -CUDART_INF_F;
        for (int o = 16; o > 0; o >>= 1) r = fmaxf(r, __shfl_xor_sync(0xffffffffu, r, o));
    }
    return r;
}

// The x passes are compiled for a length NX > 0 or for any length: NX = 0, and NX = -1 for lengths
// with a prime factor of 17..31.  Position of element e within a row (padded in the compile-time
// passes, see ct_xpad) and row pitch (odd in the run-time ones, see RtRows).
template <int NX> __device__ __forceinline__ int xo(int e) { return NX > 0 ? ct_xpad(e) : e; }
template <int NX> __host__ __device__ __forceinline__ int x_pitch(int nx) { return NX > 0 ? ct_row_pitch(NX) : nx | 1; }

// Division of a block's item index by a length that may be known at compile time (D > 0).
template <int D> struct QDiv {
    FastDiv f;
    __device__ __forceinline__ explicit QDiv(int d) : f(D > 0 ? 1 : d) {}
    __device__ __forceinline__ int operator()(int x) const {
        if constexpr (D > 0) return x / D;
        else return f.div(x);
    }
};
template <int NX> using QRow = QDiv<NX>;                              // by nx
template <int NX> using QHalf = QDiv<(NX > 0 ? NX / 2 + 1 : 0)>;      // by nx / 2 + 1

template <typename C> __device__ __forceinline__ C* align_ptr(unsigned char* p) {
    uintptr_t u = reinterpret_cast<uintptr_t>(p);
    u = (u + 15) & ~uintptr_t(15);
    return reinterpret_cast<C*>(u);
}

// ------------------------------------------------------------------------------------
// x pass, forward: S real fields -> half spectra.  Two real rows a, b are packed as a + i b
// into one complex transform of length nx and separated afterwards:
//   X_a[k] = (Z[k] + conj Z[-k]) / 2,  X_b[k] = (Z[k] - conj Z[-k]) / (2 i).
// ------------------------------------------------------------------------------------
template <typename Real, int NX>
__global__ void __launch_bounds__(kThreads) k_xfwd(GridDesc g, AxisPlan px, int ncomp, int lx,
                                                   const Real* __restrict__ in,
                                                   typename Cplx<Real>::type* __restrict__ out,
                                                   const typename Cplx<Real>::type* __restrict__ twx) {
    dep_launch();
    dep_wait();
    using C = typename Cplx<Real>::type;
    extern __shared__ unsigned char smem_raw[];
    const int nx = NX > 0 ? NX : g.nx, nxh = nx / 2 + 1, pitch = x_pitch<NX>(nx);
    const QRow<NX> qx(nx);
    const QHalf<NX> qh(nxh);
    C* tw = align_ptr<C>(smem_raw);
    C* A = tw + nx;
    C* B = A + lx * pitch;
    for (int i = threadIdx.x; i < nx; i += blockDim.x) tw[i] = twx[i];
    const long long rows = (long long)ncomp * g.ny * g.nz;
    const long long pair0 = (long long)blockIdx.x * lx;
    // rows 2(pair0 + l) and 2(pair0 + l) + 1 as the real and imaginary parts of line l; the loads
    // of kU elements per thread are issued before their shared-memory stores
    constexpr int kU = 4;
    const int total = lx * nx;
    for (int base = threadIdx.x; base < total; base += kU * kThreads) {
        Real av[kU], bv[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int idx = base + u * kThreads;
            const int l = qx(idx), x = idx - l * nx;
            const long long ra = 2 * (pair0 + l), rb = ra + 1;
            av[u] = (idx < total && ra < rows) ? in[ra * nx + x] : Real(0);
            bv[u] = (idx < total && rb < rows) ? in[rb * nx + x] : Real(0);
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int idx = base + u * kThreads;
            if (idx >= total) break;
            const int l = qx(idx), x = idx - l * nx;
            A[l * pitch + xo<NX>(x)] = cmake<C>(av[u], bv[u]);
        }
    }
    __syncthreads();
    C* R = any_fft<NX, false>(A, B, px, lx, pitch, tw);
    for (int idx = threadIdx.x; idx < lx * nxh; idx += blockDim.x) {
        const int l = qh(idx), k = idx - l * nxh;
        const long long ra = 2 * (pair0 + l), rb = ra + 1;
        const C zk = R[l * pitch + xo<NX>(k)];
        const C znk = R[l * pitch + xo<NX>(k == 0 ? 0 : nx - k)];
        const C s = cadd(zk, cconj(znk));
        const C d = csub(zk, cconj(znk));
        if (ra < rows) out[ra * g.pxh + k] = cmake<C>(Real(0.5) * s.x, Real(0.5) * s.y);
        if (rb < rows) out[rb * g.pxh + k] = cmake<C>(Real(0.5) * d.y, Real(-0.5) * d.x);
    }
}

// ------------------------------------------------------------------------------------
// Column transforms (y and z passes): what a pass does with the components.
//   COL_PLAIN  every component in place
//   COL_WD     the seven components of each set of nine that the z passes carry (dft_zcomp)
//   COL_DERIV  inverse: those seven in place, and from the inputs of m and n3 also i k times them,
//              transformed into the y-derivative components 5 and 7
//   COL_FOLD   forward: those seven in place, with -i k times the transforms of the y-derivative
//              components 5 and 7 added to components 4 and 3
// A column holds the whole k axis, so both products cost one multiplication per element, and the z
// passes read and write seven components instead of nine (256^3, S = 4, FP32: second-half z pass
// 604 -> 526 us, first half's z inverse 236 -> 184, products 295 -> 265; the y passes as before).
// k is zero on the Nyquist index.
// ------------------------------------------------------------------------------------
__host__ __device__ constexpr bool col_dual(int q) { return q == 3 || q == 4; }
__host__ __device__ constexpr int col_partner(int q) { return q == 3 ? 7 : 5; }

template <typename Real> struct PreDeriv {     // v -> i k v
    const Real* k;
    template <typename C> __device__ __forceinline__ void operator()(C& v, int e) const {
        const Real kk = k[e];
        v = cmake<C>(-kk * v.y, kk * v.x);
    }
};
template <typename Real> struct PostFold {     // *p holds u: v - i k u
    const Real* k;
    template <typename C> __device__ __forceinline__ void operator()(C* p, C v, int e) const {
        const Real kk = k[e];
        const C u = *p;
        *p = cmake<C>(v.x + kk * u.y, v.y - kk * u.x);
    }
};

// Wave numbers of an axis for the two modes above, zero on the Nyquist index.
template <typename Real> __device__ __forceinline__ void fill_axis_k(Real* k, int n, Real kf) {
    for (int i = threadIdx.x; i < n; i += kThreads) k[i] = (2 * i == n) ? Real(0) : kval<Real>(i, n, kf);
}

// A pass's tiles, kx tile fastest, then the index on the other axis, then the item (component or, in
// the modes with sets of nine, q-th component of set m; at most two sets).  per = kx tiles times
// other indices; every thread needs the item, only the one that moves tiles the rest.
struct ColItem {
    int m, q;
    __device__ __forceinline__ ColItem(int tile, const FastDiv& per, bool sets) {
        int c = per.div(tile);
        if (c * per.d > tile) --c;      // tile * per.d may exceed FastDiv's exact range
        m = sets && c >= DFT_NZSPEC ? 1 : 0;
        q = c - m * DFT_NZSPEC;
    }
    __device__ __forceinline__ int comp(bool sets) const { return sets ? m * DFT_NSPEC + dft_zcomp(q) : q; }
    __device__ __forceinline__ int partner() const { return m * DFT_NSPEC + col_partner(q); }
};

// A persistent block's loads in order: tiles b, b + gridDim.x, ...; in COL_FOLD a tile with a
// derivative component takes two, that component's first.
template <int MODE> struct ColCursor {
    int tile, sub;
    __device__ __forceinline__ bool dual(const FastDiv& per) const {
        return MODE == COL_FOLD && col_dual(ColItem(tile, per, true).q);
    }
    __device__ __forceinline__ void next(const FastDiv& per) {
        if (MODE == COL_FOLD && sub == 0 && dual(per)) { sub = 1; return; }
        tile += gridDim.x;
        sub = 0;
    }
};

// ------------------------------------------------------------------------------------
// y pass with TMA tiles (compile-time length NY <= 256 and tile width TY).  Persistent: CTA b
// handles tiles b, b + gridDim.x, ...  Two shared-memory stages are filled by TMA loads (one
// cp.async.bulk.tensor per tile, completing on an mbarrier).  The first of the two FFT stages moves
// a tile out of its TMA stage into scratch X (padded), so the stage is refilled with the tile after
// next at once; the second writes the dense box Y that leaves through a TMA store, whose
// shared-memory reads are awaited only before Y is written again.  The tensor map views the half
// spectra as (x: nxh * E, y: ny, plane: nz * ncomp) 8-byte elements, E = sizeof(complex) / 8; a
// tile is the box (TY * E, NY, 1).  A wait that runs out sets DEV_TIMEOUT and the CTA stops after
// draining the loads it has in flight.
// ZAX: the same pass along z (modes COL_PLAIN, COL_WD): a tile is TY of the ny pxh columns (pitch
// padding included; nothing reads it) of all NY z points of one component; the box lands in shared
// memory with the same layout (element (z, t) at z TY + t).  Tiles of one ky each left most of the last
// one empty, as nx / 2 + 1 is one past a multiple: seven spectra, 128^3 FP64 258 -> 237 us, 256^3 FP32
// 184 -> 158.
// Along y that last tile stays (wd bit 1: it holds one column).  Bound by the FP64 pipe, FP64 from 96 on
// runs the butterflies of that one column only (128^3, Phi' forward of nine spectra 634 -> 603 us); FP32,
// the short lengths and COL_DERIV lose more by the branch (FP32 128^3 COL_DERIV 26 -> 79 us).
// Shared memory: stage 0 | stage 1 (dense tiles) | X (padded) | Y | twiddles | k | 2 mbarriers.
// ------------------------------------------------------------------------------------
template <typename Real, int NY, int TY> __host__ __device__ constexpr size_t yfft_tma_smem() {
    using C = typename Cplx<Real>::type;
    return (3 * size_t(TY) * NY + size_t(ct_gstride(NY, TY, int(sizeof(C)))) + NY) * sizeof(C) + NY * sizeof(Real) +
           2 * sizeof(uint64_t) + 128;
}

template <typename Real, bool INV, int NY, int TY, bool ZAX = false, int MODE = COL_PLAIN>
__global__ void __launch_bounds__(kThreads, dft_yfft_minb<Real>(NY)) k_yfft_tma(const __grid_constant__ CUtensorMap map, int ntiles_x, int other,
                                                       int ntiles, int wd, int* __restrict__ status,
                                                       const typename Cplx<Real>::type* __restrict__ twy, Real kfy,
                                                       long long polls) {
    dep_launch();
    dep_wait();
    static_assert(NY > 0 && NY <= 256 && TY > 0 && ct_nstages(NY) == 2, "compile-time TMA y pass");
    static_assert(MODE == COL_PLAIN || (MODE == (INV ? COL_DERIV : COL_FOLD) && !ZAX), "column mode");
    using C = typename Cplx<Real>::type;
    constexpr int E = int(sizeof(C) / 8);
    constexpr int TILE = TY * NY;
    constexpr int GS = ct_gstride(NY, TY, int(sizeof(C)));
    constexpr uint32_t BYTES = uint32_t(TILE * sizeof(C));
    constexpr bool kSingle = sizeof(Real) == 8 && NY >= 96 && MODE != COL_DERIV && !ZAX;
    static_assert(BYTES % 128 == 0, "TMA stage alignment");
    extern __shared__ unsigned char smem_raw[];
    const uintptr_t base = (reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127);
    C* const stage0 = reinterpret_cast<C*>(base);
    C* const Y = stage0 + 2 * TILE;
    C* const X = Y + TILE;
    C* const tw = X + GS;
    Real* const kt = reinterpret_cast<Real*>(tw + NY);
    uint64_t* const bar = reinterpret_cast<uint64_t*>(kt + NY);
    const bool sets = MODE != COL_PLAIN || (wd & 1);
    if (threadIdx.x == 0) {
        tma::mbar_init(&bar[0], 1);
        tma::mbar_init(&bar[1], 1);
        tma::fence_mbar_init();
    }
    for (int i = threadIdx.x; i < NY; i += kThreads) tw[i] = twy[i];
    if constexpr (MODE != COL_PLAIN) fill_axis_k<Real>(kt, NY, kfy);
    __syncthreads();
    int issued = 0, consumed = 0;   // per stage, packed (stage 1 << 16) | stage 0; thread 0
    const FastDiv per(ntiles_x * other);
    ColCursor<MODE> load{(int)blockIdx.x, 0};
    auto issue = [&](int s) {       // thread 0: the next load in order into stage s
        if (load.tile >= ntiles) return;
        const ColItem t(load.tile, per, sets);
        const int c = (load.sub == 0 && load.dual(per)) ? t.partner() : t.comp(sets);
        const int x = load.tile % ntiles_x, o = load.tile / ntiles_x % other;
        tma::mbar_expect_tx(&bar[s], BYTES);
        tma::load_3d(stage0 + s * TILE, &map, x * TY * E, ZAX ? o : 0, ZAX ? c * NY : c * other + o, &bar[s]);
        issued += 1 << (16 * s);
        load.next(per);
    };
    if (threadIdx.x == 0) { issue(0); issue(1); }
    ColCursor<MODE> at{(int)blockIdx.x, 0};
    for (int it = 0; at.tile < ntiles; ++it, at.next(per)) {
        const int cur = it & 1;
        C* const st = stage0 + cur * TILE;
        const bool ok = tma::mbar_wait(&bar[cur], (it >> 1) & 1, polls);
        if (__syncthreads_or(!ok)) {
            if (threadIdx.x == 0) {
                atomicOr(status, DEV_TIMEOUT);
                for (int s = 0; s < 2; ++s) {
                    const int n_is = (issued >> (16 * s)) & 0xffff, n_co = (consumed >> (16 * s)) & 0xffff;
                    if (n_is > n_co) tma::mbar_wait(&bar[s], (n_is - 1) & 1);
                }
            }
            break;
        }
        consumed += 1 << (16 * cur);
        const ColItem t(at.tile, per, sets);
        const bool dual = MODE != COL_PLAIN && col_dual(t.q);
        const bool add = MODE == COL_FOLD && dual && at.sub == 1;       // Y holds the partner's transform
        const bool hold = MODE == COL_FOLD && dual && at.sub == 0;      // keep it there
        const bool single = kSingle && (wd & 2) && at.tile % ntiles_x == ntiles_x - 1;
        // COL_DERIV: the derivative first (from the same stage), then the component itself
        for (int pass = (MODE == COL_DERIV && dual) ? 0 : 1; pass < 2; ++pass) {
            if (MODE == COL_DERIV && pass == 0)
                ct_stage_grouped<NY, ct_radix_at(NY, 0), 1, INV, TY, GS, true, false, kThreads>(
                    st, X, 1, tw, PreDeriv<Real>{kt}, PostStore{}, single);
            else
                ct_stage_grouped<NY, ct_radix_at(NY, 0), 1, INV, TY, GS, true, false, kThreads>(
                    st, X, 1, tw, PreNone{}, PostStore{}, single);
            // the previous store has finished reading Y
            if (threadIdx.x == 0 && !add) tma::wait_read_all();
            __syncthreads();
            if (threadIdx.x == 0 && pass == 1) issue(cur);
            if (MODE == COL_FOLD && add)
                ct_stage_grouped<NY, ct_radix_at(NY, 1), ct_ns_at(NY, 1), INV, TY, GS, false, true, kThreads>(
                    X, Y, 1, tw, PreNone{}, PostFold<Real>{kt}, single);
            else
                ct_stage_grouped<NY, ct_radix_at(NY, 1), ct_ns_at(NY, 1), INV, TY, GS, false, true, kThreads>(
                    X, Y, 1, tw, PreNone{}, PostStore{}, single);
            tma::fence_proxy_async();
            __syncthreads();
            if (threadIdx.x == 0 && !hold) {
                const int c = (MODE == COL_DERIV && pass == 0) ? t.partner() : t.comp(sets);
                const int x = at.tile % ntiles_x, o = at.tile / ntiles_x % other;
                tma::store_3d(&map, x * TY * E, ZAX ? o : 0, ZAX ? c * NY : c * other + o, Y);
                tma::commit();
            }
        }
    }
    if (threadIdx.x == 0) tma::wait_all();
}

// ------------------------------------------------------------------------------------
// Column transform of a run-time length along y or z, in place, of every component: the
// persistent TMA pipeline of k_yfft_tma with the stages of an AxisPlan.  The tensor map views the
// half spectra as (x: nxh E, y, z, component) 8-byte elements; a tile is T kx columns of the whole
// axis at `planes` indices of the other axis (`other` such groups; indices past the axis read as
// zero and are not written) of one component, moved as one box, or, past 256 rows, two.
// Memory-bound in FP32: at 160^3 8.9 us a component (3.8 TB/s; a column pass of plain tile loads,
// divisions by run-time integers and odd primes by their R^2 terms took 44).  FP64 is bound by the
// FP64 pipe: 21 x 21 x 161 (161 = 7 x 23), z forward 6.9 us a component.
// Shared memory: stage 0 | stage 1 | X | Y (only with two or more stages) | twiddles | 2 mbarriers.
// ------------------------------------------------------------------------------------
struct ColBox {
    int n, nbox, rows;      // axis length; boxes of a tile and rows of a box
    int planes;             // planes of the other axis in a tile (1 with two boxes)
    int elems;              // shared-memory elements of one tile buffer (128-byte multiple)
};

template <typename Real, bool INV, int T, bool BIG, int MODE>
__global__ void __launch_bounds__(kThreads, BIG ? 1 : (sizeof(Real) == 4 && T < 16 ? 3 : 2)) k_colfft(const __grid_constant__ CUtensorMap map, AxisPlan pa,
                                                                  ColBox cb, int zax, int ntiles_x, int other,
                                                                  int ntiles, int wd, int* __restrict__ status,
                                                                  const typename Cplx<Real>::type* __restrict__ twd,
                                                                  Real kf, long long polls) {
    dep_launch();
    dep_wait();
    static_assert(MODE == COL_PLAIN || MODE == (INV ? COL_DERIV : COL_FOLD), "column mode");
    using C = typename Cplx<Real>::type;
    constexpr int E = int(sizeof(C) / 8);
    extern __shared__ unsigned char smem_raw[];
    const uintptr_t base = (reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127);
    C* const stage0 = reinterpret_cast<C*>(base);
    C* const X = stage0 + 2 * cb.elems;
    C* const Y = X + cb.elems;
    C* const tw = pa.nstages > 1 ? Y + cb.elems : Y;
    Real* const kt = reinterpret_cast<Real*>(tw + cb.n);
    uint64_t* const bar = reinterpret_cast<uint64_t*>(kt + ((cb.n + 1) & ~1));
    const uint32_t bytes = uint32_t(cb.nbox) * uint32_t(cb.rows * cb.planes) * uint32_t(T * sizeof(C));
    const RtCols<T> cols(cb.planes, cb.n, zax != 0);
    const bool sets = MODE != COL_PLAIN || wd;
    const int nst = pa.nstages;     // 1 to DFT_RT_STAGES
    static_assert(DFT_RT_STAGES == 3, "the buffers below rotate over three stages");
    if (threadIdx.x == 0) {
        tma::mbar_init(&bar[0], 1);
        tma::mbar_init(&bar[1], 1);
        tma::fence_mbar_init();
    }
    for (int i = threadIdx.x; i < cb.n; i += kThreads) tw[i] = twd[i];
    if constexpr (MODE != COL_PLAIN) fill_axis_k<Real>(kt, cb.n, kf);
    __syncthreads();
    int issued = 0, consumed = 0;   // per stage, packed (stage 1 << 16) | stage 0; thread 0
    const FastDiv per(ntiles_x * other);
    ColCursor<MODE> load{(int)blockIdx.x, 0};
    auto issue = [&](int s) {       // thread 0: the next load in order into stage s
        if (load.tile >= ntiles) return;
        const ColItem t(load.tile, per, sets);
        const int c = (load.sub == 0 && load.dual(per)) ? t.partner() : t.comp(sets);
        const int x = load.tile % ntiles_x, o = load.tile / ntiles_x % other * cb.planes;
        tma::mbar_expect_tx(&bar[s], bytes);
        for (int b = 0; b < cb.nbox; ++b)
            tma::load_4d(stage0 + s * cb.elems + b * cb.rows * T, &map, x * T * E, zax ? o : b * cb.rows,
                         zax ? b * cb.rows : o, c, &bar[s]);
        issued += 1 << (16 * s);
        load.next(per);
    };
    if (threadIdx.x == 0) { issue(0); issue(1); }
    ColCursor<MODE> at{(int)blockIdx.x, 0};
    for (int it = 0; at.tile < ntiles; ++it, at.next(per)) {
        const int cur = it & 1;
        C* const st = stage0 + cur * cb.elems;
        const bool ok = tma::mbar_wait(&bar[cur], (it >> 1) & 1, polls);
        // the previous store has finished reading X or Y
        if (threadIdx.x == 0) tma::wait_read_all();
        if (__syncthreads_or(!ok)) {
            if (threadIdx.x == 0) {
                atomicOr(status, DEV_TIMEOUT);
                for (int s = 0; s < 2; ++s) {
                    const int n_is = (issued >> (16 * s)) & 0xffff, n_co = (consumed >> (16 * s)) & 0xffff;
                    if (n_is > n_co) tma::mbar_wait(&bar[s], (n_is - 1) & 1);
                }
            }
            break;
        }
        consumed += 1 << (16 * cur);
        const ColItem t(at.tile, per, sets);
        const bool dual = MODE != COL_PLAIN && col_dual(t.q);
        const bool add = MODE == COL_FOLD && dual && at.sub == 1;       // X or Y holds the partner's transform
        const bool hold = MODE == COL_FOLD && dual && at.sub == 0;      // keep it there
        // The buffers: the stage, X, Y, X ...; the last one (of one to three stages X, Y, X) ends up
        // with the result.  A tile to be added to its partner's transform must not pass through that
        // buffer before its last stage: with three stages it goes through Y and its TMA stage.
        C* const res = nst == 2 ? Y : X;
        const bool spare = add && nst == 3;
        for (int pass = (MODE == COL_DERIV && dual) ? 0 : 1; pass < 2; ++pass) {
            if (MODE == COL_DERIV && pass == 1 && dual) {               // after the derivative's store
                if (threadIdx.x == 0) tma::wait_read_all();
                __syncthreads();
            }
            const C* src = st;
            for (int s = 0; s < nst; ++s) {
                C* const dst = s == nst - 1 ? res : (spare ? (s == 0 ? Y : st) : (s == 0 ? X : Y));
                if (MODE == COL_DERIV && s == 0 && pass == 0)
                    rt_stage_any<INV, kThreads, BIG>(src, dst, pa, s, cols, tw, PreDeriv<Real>{kt});
                else if (MODE == COL_FOLD && add && s == nst - 1)
                    rt_stage_any<INV, kThreads, BIG>(src, dst, pa, s, cols, tw, PreNone{}, PostFold<Real>{kt});
                else
                    rt_stage_any<INV, kThreads, BIG>(src, dst, pa, s, cols, tw);
                if (s == nst - 1) tma::fence_proxy_async();
                __syncthreads();
                // the stage is free: refill it
                if (threadIdx.x == 0 && pass == 1 && s == (spare ? nst - 1 : 0)) issue(cur);
                src = dst;
            }
            if (threadIdx.x == 0 && !hold) {
                const int c = (MODE == COL_DERIV && pass == 0) ? t.partner() : t.comp(sets);
                const int x = at.tile % ntiles_x, o = at.tile / ntiles_x % other * cb.planes;
                for (int q = 0; q < cb.nbox; ++q)
                    tma::store_4d(&map, x * T * E, zax ? o : q * cb.rows, zax ? q * cb.rows : o, c,
                                  res + q * cb.rows * T);
                tma::commit();
            }
        }
    }
    if (threadIdx.x == 0) tma::wait_all();
}

// Wave vector components of tile point (kz index, t) in a z-pass tile at (kx0, ky index)
template <typename Real> struct KPoint {
    Real kx, ky, kz;
    bool zero;
    __device__ __forceinline__ Real kmag() const { return sqrt(kx * kx + ky * ky + kz * kz); }
};

template <typename Real>
__device__ __forceinline__ KPoint<Real> kpoint(const GridDesc& g, int kxi, int kyi, int kzi, Real kfx, Real kfy,
                                               Real kfz) {
    KPoint<Real> p;
    p.kx = kval<Real>(kxi, g.nx, kfx);
    p.ky = kval<Real>(kyi, g.ny, kfy);
    p.kz = kval<Real>(kzi, g.nz, kfz);
    p.zero = (kxi == 0) && (kyi == 0) && (kzi == 0);
    return p;
}

// Bulk-fluid + mean-field kernel K_ij(k) = DC_ij_hat(k) - 4 pi lambda_B z_i z_j / lap(k) (k != 0),
// lap(k) = sum_d 4 sin^2(k_d h_d / 2) / h_d^2 (eq. potentialSolution), psi_hat(0) = 0.
template <typename Real>
__device__ __forceinline__ Real es_kernel(const SpeciesDesc<Real>& sp, int i, int j, const KPoint<Real>& p, Real inv_lap,
                                         Real* dGamma = nullptr) {
    Real K = delta_c_hat<Real>(p.kmag(), sp.es_R[i][j], sp.es_pref[i][j], sp.es_a[i][j], sp.es_b[i][j], sp.es_c[i][j],
                               dGamma, sp.es_da[i][j], sp.es_db[i][j], sp.es_dc[i][j]);
    if (!p.zero) K -= sp.pois[i][j] * inv_lap;
    return K;
}

// One axis's term of lap(k): sin^2(k_d h_d / 2) / h_d^2.
template <typename Real> __device__ __forceinline__ Real lap_term(Real k, Real h) {
    const Real s = sin(Real(0.5) * k * h);
    return s * s / (h * h);
}

template <typename Real>
__device__ __forceinline__ Real inverse_laplacian(const KPoint<Real>& p, Real hx, Real hy, Real hz) {
    if (p.zero) return Real(0);
    const Real lap = Real(4) * (lap_term(p.kx, hx) + lap_term(p.ky, hy) + lap_term(p.kz, hz));
    return Real(1) / lap;
}

// The same from the plan's per-axis table (sp.lap1d, the lap_term values by FFT index, evaluated
// by k_laptab with the same expression: equal bit for bit) where it has one.
// ALWAYS: it has one.
template <typename Real, bool ALWAYS = false>
__device__ __forceinline__ Real inverse_laplacian(const SpeciesDesc<Real>& sp, const GridDesc& g, const KPoint<Real>& p,
                                                  int kxi, int kyi, int kzi, Real hx, Real hy, Real hz) {
    if constexpr (!ALWAYS)
        if (!sp.lap1d) return inverse_laplacian<Real>(p, hx, hy, hz);
    if (p.zero) return Real(0);
    const Real lap = Real(4) * (__ldg(sp.lap1d + kxi) + __ldg(sp.lap1d + g.nx + kyi) + __ldg(sp.lap1d + g.nx + g.ny + kzi));
    return Real(1) / lap;
}

// The per-axis Laplacian terms of a grid: out[i] for x indices i < nx, out[nx + j] for y, out[nx +
// ny + l] for z (wave numbers kval of the FFT index, as the z passes form them); then, in the same
// order, the wave numbers themselves, zero on the Nyquist index.
template <typename Real>
__global__ void k_laptab(GridDesc g, Real kfx, Real kfy, Real kfz, Real* __restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.nx + g.ny + g.nz) return;
    Real v;
    if (i < g.nx) v = lap_term(kval<Real>(i, g.nx, kfx), Real(g.hx));
    else if (i < g.nx + g.ny) v = lap_term(kval<Real>(i - g.nx, g.ny, kfy), Real(g.hy));
    else v = lap_term(kval<Real>(i - g.nx - g.ny, g.nz, kfz), Real(g.hz));
    out[i] = v;
    const int j = i < g.nx ? i : (i < g.nx + g.ny ? i - g.nx : i - g.nx - g.ny);
    const int n = i < g.nx ? g.nx : (i < g.nx + g.ny ? g.ny : g.nz);
    const Real kf = i < g.nx ? kfx : (i < g.nx + g.ny ? kfy : kfz);
    out[g.nx + g.ny + g.nz + i] = 2 * j == n ? Real(0) : kval<Real>(j, n, kf);
}

// Wave number of z index kzi, zero on the Nyquist index, from the plan's table where it has one (an
// int-to-FP64 conversion and a product otherwise, on the FP64 pipe).
template <typename Real>
__device__ __forceinline__ Real kz_of(const SpeciesDesc<Real>& sp, const GridDesc& g, int kzi, Real kfz) {
    if (sp.kax) return __ldg(sp.kax + g.nx + g.ny + kzi);
    return 2 * kzi == g.nz ? Real(0) : kval<Real>(kzi, g.nz, kfz);
}

// ------------------------------------------------------------------------------------
// The z passes.  First half: the S half spectra of the densities after x, y forward (kx, ky, z) ->
//   slot_n:  seven of the nine weighted-density spectra (dft_zcomp), 1/N applied, after z inverse (kx, ky, z)
//   slot_es: S (+1 with psi) unnormalised bulk-fluid/Poisson spectra sum_j K_ij drho_hat_j (kx, ky, kz)
// Second half: seven Phi' spectra after x, y forward (kx, ky, z), the y derivatives added ->
//   the S one-body correlation spectra after z inverse, 1/N applied (kx, ky, z), in their place.
//   mu_hat_i = sum_alpha Phi_hat_alpha w_hat_i^alpha(+k) (eq. muHS): with the vector weights
//   w_hat^V2 = -i k w_hat^3 and w_hat^V1 = w_hat^V2/(4 pi R) the k-space sum needs only the five
//   species-independent spectra Phi0, Phi1, Phi2, Phi3 + div(PhiV2), div(PhiV1).
//   c_hat_i = (-mu_hat_i + wA es_A_i + wB es_B_i) / N.
//   flags: 1 = hard-sphere part, 2 = electrostatic part; ncomp_out = S (or S + 1 for psi).
// FP32 plans do a half of a compile-time length in one pass (below); FP64 plans, run-time lengths, plans
// without |k| tables and a first half where it is faster run a z transform (k_colfft / k_yfft_tma), a
// k-space products pass (k_zmul, k_zmul_bwd) and another z transform.
// ------------------------------------------------------------------------------------
// ------------------------------------------------------------------------------------
// Grouped z passes (compile-time length NZ, tile width TZ), grid (ceil(nxh/TZ), ny).  All
// components of a column tile are loaded in one batch of in-flight loads and transformed by
// one grouped FFT (ct_fft_grouped), so every stage keeps the CTA's threads busy and a tile
// costs a handful of barriers instead of a dozen transforms of one component each.
// Shared memory: twiddles | 7 tiles | 7 tiles (ct_gstride(NZ, TZ, csize) elements each).
// ------------------------------------------------------------------------------------
// One species' contribution, 1/N applied, to the spectra acc = (n0, n1, n2, n3, m) at a k point:
// the weights are w0 (1, R, 4 pi R^2) and j3 (4 pi R^3, R^2), so v is scaled by each of w0 and j3
// once.  These sums and the back convolution's are written for the fewest FP64 instructions: at
// 128^3, S = 3, FP64 the second half's products pass issues 58 per k point and takes 128 us (206 and
// 428 us with a run-time choice between tables and evaluation, wave numbers converted per point and
// each weight formed by itself).
template <typename Real>
__device__ __forceinline__ void wd_add_species(typename Cplx<Real>::type* acc, const SpeciesDesc<Real>& sp, int s,
                                               typename Cplx<Real>::type v, Real w0, Real j3) {
    const typename Cplx<Real>::type u = cscale(v, w0 * sp.inv_n), t = cscale(v, j3 * sp.inv_n);
    acc[0] = cadd(acc[0], u);
    acc[1] = cadd(acc[1], cscale(u, sp.R[s]));
    acc[2] = cadd(acc[2], cscale(u, sp.a2[s]));
    acc[3] = cadd(acc[3], cscale(t, sp.v3[s]));
    acc[4] = cadd(acc[4], cscale(t, sp.r2[s]));       // w3 / (4 pi R)
}

// The seven weighted-density spectra of one k point that the z passes carry into groups (group
// stride GS, position pos; q-th of them = component dft_zcomp(q)): acc, then i k_z m and i k_z n3
// (kz zero on the Nyquist index).  The y pass forms the y derivatives, the x pass the x derivatives.
template <typename Real>
__device__ __forceinline__ void store_wd_spectra(typename Cplx<Real>::type* O, int GS, int pos,
                                                 const typename Cplx<Real>::type* acc, Real kz) {
    using C = typename Cplx<Real>::type;
#pragma unroll
    for (int a = 0; a < 5; ++a) O[a * GS + pos] = acc[a];
    O[5 * GS + pos] = cmake<C>(-kz * acc[4].y, kz * acc[4].x);
    O[6 * GS + pos] = cmake<C>(-kz * acc[3].y, kz * acc[3].x);
}

// Species-independent sums of the back convolution at one k point from the seven Phi' spectra of
// the y pass (groups as above): a0..a2 = Phi_0..Phi_2, a3 = B3 - i k_z Phi_V2z,
// a4 = B4 - i k_z Phi_V1z, where the x pass formed B3 = Phi_3 - i k_x Phi_V2x, B4 = -i k_x Phi_V1x
// and the y pass added their y terms (Nyquist terms dropped: kz zero there).
template <typename Real>
__device__ __forceinline__ void bwd_sums(const typename Cplx<Real>::type* X, int GS, int pos, Real kz,
                                         typename Cplx<Real>::type* a) {
    using C = typename Cplx<Real>::type;
#pragma unroll
    for (int q = 0; q < 5; ++q) a[q] = X[q * GS + pos];
    const C u1 = X[5 * GS + pos], u2 = X[6 * GS + pos];
    a[4] = cmake<C>(a[4].x + kz * u1.y, a[4].y - kz * u1.x);
    a[3] = cmake<C>(a[3].x + kz * u2.y, a[3].y - kz * u2.x);
}

// es - mu_hat of species s: mu_hat = w0 (a0 + R a1 + 4 pi R^2 a2) + j3 (4 pi R^3 a3 + R^2 a4).
template <typename Real>
__device__ __forceinline__ typename Cplx<Real>::type bwd_species(const typename Cplx<Real>::type* a,
                                                                 const SpeciesDesc<Real>& sp, int s, Real w0, Real j3,
                                                                 typename Cplx<Real>::type es) {
    using C = typename Cplx<Real>::type;
    const Real R = sp.R[s], A = sp.a2[s], V = sp.v3[s], R2 = sp.r2[s];
    const C P = cmake<C>(a[0].x + R * a[1].x + A * a[2].x, a[0].y + R * a[1].y + A * a[2].y);
    const C Q = cmake<C>(V * a[3].x + R2 * a[4].x, V * a[3].y + R2 * a[4].y);
    return cmake<C>(es.x - w0 * P.x - j3 * Q.x, es.y - w0 * P.y - j3 * Q.y);
}

template <int TT, int NN> __host__ __device__ constexpr size_t zg_smem_bytes(size_t csize) {
    return (size_t(NN) + 2 * size_t(DFT_NZSPEC) * ct_gstride(NN, TT, int(csize))) * csize + 16;
}

// Load `groups` column tiles (component c at src + c * cstride; WD: the q-th is component
// dft_zcomp(q); global row stride rs, columns t < valid, zero elsewhere) into the grouped layout;
// every load of a thread is issued before its first shared-memory store.
template <int TT, int NN, int GMAX, bool WD, typename C>
__device__ __forceinline__ void tiles_load_grouped(C* __restrict__ dst, const C* __restrict__ src, long long cstride,
                                                   int groups, long long rs, int valid) {
    constexpr int TILE = TT * NN;
    constexpr int PER = (TILE + kThreads - 1) / kThreads;
    constexpr int GS = ct_gstride(NN, TT, int(sizeof(C)));
    C reg[GMAX][PER];
#pragma unroll
    for (int gi = 0; gi < GMAX; ++gi) {
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int idx = threadIdx.x + i * kThreads;
            const int e = idx / TT, t = idx % TT;
            reg[gi][i] = cmake<C>(0, 0);
            if (gi < groups && (TILE % kThreads == 0 || idx < TILE) && t < valid)
                reg[gi][i] = src[(WD ? dft_zcomp(gi) : gi) * cstride + e * rs + t];
        }
    }
#pragma unroll
    for (int gi = 0; gi < GMAX; ++gi) {
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int idx = threadIdx.x + i * kThreads;
            const int e = idx / TT, t = idx % TT;
            if (gi < groups && (TILE % kThreads == 0 || idx < TILE)) dst[gi * GS + ct_gpos(e, TT) + t] = reg[gi][i];
        }
    }
}

template <int TT, int NN, bool WD, typename C>
__device__ __forceinline__ void tiles_store_grouped(C* __restrict__ dst, const C* __restrict__ src, long long cstride,
                                                    int groups, long long rs, int valid) {
    constexpr int TILE = TT * NN;
    constexpr int GS = ct_gstride(NN, TT, int(sizeof(C)));
    for (int gi = 0; gi < groups; ++gi) {
#pragma unroll
        for (int idx = threadIdx.x; idx < TILE; idx += kThreads) {
            const int e = idx / TT, t = idx % TT;
            if (t < valid) dst[(WD ? dft_zcomp(gi) : gi) * cstride + e * rs + t] = src[gi * GS + ct_gpos(e, TT) + t];
        }
    }
}

// Load the first n entries of a table record (16-byte aligned) with 16-byte loads.
template <typename Real, int MAXN>
__device__ __forceinline__ void load_record(Real (&dst)[MAXN], const Real* __restrict__ rec, int n) {
    constexpr int V = int(16 / sizeof(Real));
    static_assert(MAXN % V == 0, "record capacity");
#pragma unroll
    for (int v = 0; v < MAXN / V; ++v) {
        if (v * V < n) {
            if constexpr (sizeof(Real) == 4) {
                const float4 t = __ldg(reinterpret_cast<const float4*>(rec) + v);
                dst[4 * v] = t.x; dst[4 * v + 1] = t.y; dst[4 * v + 2] = t.z; dst[4 * v + 3] = t.w;
            } else {
                const double2 t = __ldg(reinterpret_cast<const double2*>(rec) + v);
                dst[2 * v] = t.x; dst[2 * v + 1] = t.y;
            }
        }
    }
}

__device__ __forceinline__ int signed_index(int j, int n) { return (2 * j <= n) ? j : j - n; }

// Register capacity of a table record of n entries: whole 16-byte loads.
template <typename Real> __host__ __device__ constexpr int tab_capacity(int n) {
    const int v = int(16 / sizeof(Real));
    return (n + v - 1) / v * v;
}

// Tables of the |k|-only factors: the FMT weights w0, j3 of each species and the bulk-fluid kernel
// DC_ij_hat with its Gamma derivative.  On a cubic box (kf equal on the three axes) one record per
// integer m2 = mx^2 + my^2 + mz^2, |k| = kf sqrt(m2); on other boxes (sp.tab_oct) one per (kx, |ky|,
// |kz|), |k| as kpoint forms it.  Evaluated once per plan with the functions the z passes call
// where there is no table; a null table is left out.
template <typename Real>
__global__ void k_ktab(GridDesc g, SpeciesDesc<Real> sp, double kf, Real kfx, Real kfy, Real kfz, long long rows,
                       Real* tab_w, Real* tab_k, Real* tab_dk) {
    const long long row = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (row >= rows) return;
    const int S = sp.S;
    Real kmag;
    if (sp.tab_oct) {
        const int ix = int(row % g.nxh), rest = int(row / g.nxh), nyh = g.ny / 2 + 1;
        const int iy = rest % nyh, iz = rest / nyh;
        kmag = kpoint<Real>(g, ix, iy, iz, kfx, kfy, kfz).kmag();
    } else {
        kmag = Real(kf * sqrt(double(row)));
    }
    if (tab_w)
        for (int s = 0; s < S; ++s) {
            Real w0, j3;
            fmt_weights<Real>(kmag, sp.R[s], &w0, &j3);
            tab_w[row * sp.tab_ws + 2 * s] = w0;
            tab_w[row * sp.tab_ws + 2 * s + 1] = j3;
        }
    for (int j = 0; j < S; ++j)
        for (int i = 0; i <= j; ++i) {
            Real dG = Real(0);
            const Real K = delta_c_hat<Real>(kmag, sp.es_R[i][j], sp.es_pref[i][j], sp.es_a[i][j], sp.es_b[i][j],
                                             sp.es_c[i][j], &dG, sp.es_da[i][j], sp.es_db[i][j], sp.es_dc[i][j]);
            if (tab_k) tab_k[row * sp.tab_ks + dft_pair(i, j)] = K;
            if (tab_dk) tab_dk[row * sp.tab_ks + dft_pair(i, j)] = dG;
        }
}

// Table row of the mode (kx index kxi >= 0, signed y index my, z index kzi).
template <typename Real>
__device__ __forceinline__ long long tab_row(const SpeciesDesc<Real>& sp, const GridDesc& g, int kxi, int my, int kzi) {
    const int mz = signed_index(kzi, g.nz);
    if (sp.tab_oct) return ((long long)abs(mz) * (g.ny / 2 + 1) + abs(my)) * g.nxh + kxi;
    return kxi * kxi + my * my + mz * mz;
}

// First-half z pass: S species spectra in, seven weighted-density
// spectra (z inverse, 1/N applied) and the bulk-fluid/Poisson spectra out.  Per-species loops
// run to DFT_MAXS with guards so that every per-point array stays in registers.
template <typename Real, int NZ, int TZ>
__global__ void __launch_bounds__(kThreads, 2) k_zconv_fwd_g(GridDesc g, SpeciesDesc<Real> sp, Real kfx, Real kfy,
                                                             Real kfz, int want_psi,
                                                             const typename Cplx<Real>::type* __restrict__ in,
                                                             typename Cplx<Real>::type* __restrict__ slot_n,
                                                             typename Cplx<Real>::type* __restrict__ slot_es,
                                                             const typename Cplx<Real>::type* __restrict__ twz) {
    dep_launch();
    dep_wait();
    using C = typename Cplx<Real>::type;
    constexpr int TILE = TZ * NZ;
    constexpr int GS = ct_gstride(NZ, TZ, int(sizeof(C)));
    extern __shared__ unsigned char smem_raw[];
    const int ny = g.ny, nxh = g.nxh, S = sp.S;
    const int Pn = S * (S + 1) / 2;
    C* tw = align_ptr<C>(smem_raw);
    C* A = tw + NZ;
    C* B = A + DFT_NZSPEC * GS;
    for (int i = threadIdx.x; i < NZ; i += kThreads) tw[i] = twz[i];
    const int kx0 = blockIdx.x * TZ;
    const int kyi = blockIdx.y;
    const long long zstride = (long long)ny * g.pxh;
    const long long col0 = (long long)kyi * g.pxh + kx0;
    tiles_load_grouped<TZ, NZ, DFT_MAXS, false>(A, in + col0, g.nc, S, zstride, nxh - kx0);
    __syncthreads();
    C* R = ct_fft_grouped<NZ, false, TZ, GS>(A, B, S, tw);
    C* O = (R == A) ? B : A;

    const Real hx = Real(g.hx), hy = Real(g.hy), hz = Real(g.hz);
    const int my = signed_index(kyi, ny);
    Real flb = Real(0);      // 4 pi lambda_B = pois[s][s] / z_s^2 of a charged species
    for (int s = 0; s < S; ++s)
        if (sp.z[s] != Real(0)) { flb = sp.pois[s][s] / (sp.z[s] * sp.z[s]); break; }
    for (int idx = threadIdx.x; idx < TILE; idx += kThreads) {
        const int kzi = idx / TZ, t = idx % TZ;
        const int pos = ct_gpos(kzi, TZ) + t;
        const int kxi = kx0 + t;
        const bool live = kxi < nxh;
        const KPoint<Real> p = kpoint<Real>(g, kxi, kyi, kzi, kfx, kfy, kfz);
        const long long row = live ? tab_row(sp, g, kxi, my, kzi) : 0;
        Real wr[DFT_TAB_W];
        Real kr[DFT_TAB_K];
        load_record(wr, sp.tab_w + row * sp.tab_ws, 2 * S);
        if (live) load_record(kr, sp.tab_k + row * sp.tab_ks, Pn);
        C v[DFT_MAXS];
#pragma unroll
        for (int s = 0; s < DFT_MAXS; ++s)
            if (s < S) v[s] = R[s * GS + pos];
        C acc[5];
#pragma unroll
        for (int a = 0; a < 5; ++a) acc[a] = cmake<C>(Real(0), Real(0));
#pragma unroll
        for (int s = 0; s < DFT_MAXS; ++s) {
            if (s >= S) break;
            wd_add_species<Real>(acc, sp, s, v[s], wr[2 * s], wr[2 * s + 1]);
        }
        if (live) {
            const Real inv_lap = inverse_laplacian<Real, true>(sp, g, p, kxi, kyi, kzi, hx, hy, hz);
            C dv[DFT_MAXS], es[DFT_MAXS];
#pragma unroll
            for (int s = 0; s < DFT_MAXS; ++s) {
                if (s < S) {
                    dv[s] = v[s];
                    if (p.zero) dv[s].x -= sp.n_rho_b[s];       // DFT(rho - rho_bath) at k = 0
                }
                es[s] = cmake<C>(Real(0), Real(0));
            }
#pragma unroll
            for (int j = 0; j < DFT_MAXS; ++j) {
#pragma unroll
                for (int i = 0; i <= j; ++i) {
                    if (j >= S) continue;
                    const Real K = kr[dft_pair(i, j)] - sp.pois[i][j] * inv_lap;    // inv_lap is zero at k = 0
                    es[i] = cadd(es[i], cscale(dv[j], K));
                    if (j != i) es[j] = cadd(es[j], cscale(dv[i], K));
                }
            }
            const long long o = (long long)kzi * zstride + col0 + t;
#pragma unroll
            for (int s = 0; s < DFT_MAXS; ++s) {
                if (s >= S) break;
                slot_es[(long long)s * g.nc + o] = es[s];
            }
            if (want_psi) {
                C q = cmake<C>(Real(0), Real(0));
#pragma unroll
                for (int s = 0; s < DFT_MAXS; ++s)
                    if (s < S) q = cadd(q, cscale(v[s], sp.z[s]));
                // psi_hat = 4 pi lambda_B q_hat / lap
                slot_es[(long long)S * g.nc + o] = cscale(q, flb * inv_lap);
            }
        }
        store_wd_spectra<Real>(O, GS, pos, acc, kz_of(sp, g, kzi, kfz));
    }
    __syncthreads();
    C* Q = ct_fft_grouped<NZ, true, TZ, GS>(O, R, DFT_NZSPEC, tw);
    tiles_store_grouped<TZ, NZ, true>(slot_n + col0, Q, g.nc, DFT_NZSPEC, zstride, nxh - kx0);
}

// Second-half z pass: seven Phi' spectra in (flags & 1), the
// bulk-fluid/Poisson spectra mixed in (flags & 2), ncomp_out one-body correlation spectra out.
// The points of a thread are handled together so that all of their global and table loads are
// in flight at once.
template <typename Real, int NZ, int TZ>
__global__ void __launch_bounds__(kThreads, 2) k_zconv_bwd_g(GridDesc g, SpeciesDesc<Real> sp, Real kfx, Real kfy,
                                                             Real kfz, int flags, int ncomp_out,
                                                             const Ctl* __restrict__ ctl,
                                                             typename Cplx<Real>::type* phi,
                                                             const typename Cplx<Real>::type* esA,
                                                             const typename Cplx<Real>::type* esB,
                                                             typename Cplx<Real>::type* es_mat,
                                                             const typename Cplx<Real>::type* __restrict__ twz) {
    dep_launch();
    dep_wait();
    using C = typename Cplx<Real>::type;
    constexpr int TILE = TZ * NZ;
    constexpr int GS = ct_gstride(NZ, TZ, int(sizeof(C)));
    constexpr int PER = (TILE + kThreads - 1) / kThreads;
    constexpr int EMAX = DFT_MAXS + 1;
    extern __shared__ unsigned char smem_raw[];
    const int ny = g.ny, nxh = g.nxh, S = sp.S;
    C* tw = align_ptr<C>(smem_raw);
    C* A = tw + NZ;
    C* B = A + DFT_NZSPEC * GS;
    for (int i = threadIdx.x; i < NZ; i += kThreads) tw[i] = twz[i];
    const int kx0 = blockIdx.x * TZ;
    const int kyi = blockIdx.y;
    const long long zstride = (long long)ny * g.pxh;
    const long long col0 = (long long)kyi * g.pxh + kx0;
    const bool hs = (flags & 1) != 0, es_on = (flags & 2) != 0;
    const Real wA = CtlW<Real>::wA(ctl), wB = CtlW<Real>::wB(ctl);
    C* R = A;
    if (hs) {
        tiles_load_grouped<TZ, NZ, DFT_NZSPEC, true>(A, phi + col0, g.nc, DFT_NZSPEC, zstride, nxh - kx0);
        __syncthreads();
        R = ct_fft_grouped<NZ, false, TZ, GS>(A, B, DFT_NZSPEC, tw);
    }
    C* O = (R == A) ? B : A;
    const int my = signed_index(kyi, ny);

    // loads first: bulk-fluid/Poisson spectra and table records of all of this thread's points
    C ea[PER][EMAX];
    Real wr[PER][DFT_TAB_W];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int idx = threadIdx.x + i * kThreads;
        const int kzi = idx / TZ, t = idx % TZ;
        const int kxi = kx0 + t;
        const bool in_tile = (TILE % kThreads == 0) || idx < TILE;
        const bool live = in_tile && kxi < nxh;
        const long long o = (long long)kzi * zstride + col0 + t;
#pragma unroll
        for (int s = 0; s < EMAX; ++s) {
            ea[i][s] = cmake<C>(Real(0), Real(0));
            if (es_on && live && s < ncomp_out) {
                C e = cscale(esA[(long long)s * g.nc + o], wA);
                if (esB) e = cadd(e, cscale(esB[(long long)s * g.nc + o], wB));
                ea[i][s] = e;
            }
        }
        if (hs) {
            load_record(wr[i], sp.tab_w + (live ? tab_row(sp, g, kxi, my, kzi) : 0) * sp.tab_ws, 2 * S);
        }
    }
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int idx = threadIdx.x + i * kThreads;
        if ((TILE % kThreads != 0) && idx >= TILE) break;
        const int kzi = idx / TZ, t = idx % TZ;
        const int pos = ct_gpos(kzi, TZ) + t;
        const int kxi = kx0 + t;
        C out[EMAX];
#pragma unroll
        for (int s = 0; s < EMAX; ++s) out[s] = ea[i][s];
        if (es_on && es_mat && kxi < nxh) {
            const long long o = (long long)kzi * zstride + col0 + t;
#pragma unroll
            for (int s = 0; s < EMAX; ++s)
                if (s < ncomp_out) es_mat[(long long)s * g.nc + o] = ea[i][s];
        }
        if (hs) {
            C asum[5];
            bwd_sums<Real>(R, GS, pos, kz_of(sp, g, kzi, kfz), asum);
#pragma unroll
            for (int s = 0; s < DFT_MAXS; ++s) {
                if (s >= S) break;
                out[s] = bwd_species<Real>(asum, sp, s, wr[i][2 * s], wr[i][2 * s + 1], out[s]);
            }
        }
#pragma unroll
        for (int s = 0; s < EMAX; ++s)
            if (s < ncomp_out) O[s * GS + pos] = cscale(out[s], sp.inv_n);
    }
    __syncthreads();
    C* Q = ct_fft_grouped<NZ, true, TZ, GS>(O, R, ncomp_out, tw);
    tiles_store_grouped<TZ, NZ, false>(phi + col0, Q, g.nc, ncomp_out, zstride, nxh - kx0);
}

// ------------------------------------------------------------------------------------
// First-half z pass with TMA tiles (without the grand-potential sums), persistent like k_zconv_bwd_tma: two stages of S species tiles are filled by TMA loads
// while the previous tile is transformed; the seven weighted-density spectra are transformed back
// and leave through TMA stores, the bulk-fluid/Poisson spectra through plain stores.  A tensor map views a half-spectrum
// array as (x: nxh * E, y: ny, plane: nz * ncomp) 8-byte elements; a tile is the box
// (TZ * E, 1, NZ) at plane c * nz.  A wait that runs out sets DEV_TIMEOUT and the CTA stops
// after draining the loads it has in flight.
// Shared memory: stage 0 | stage 1 (S padded groups each) | W | V (seven padded groups each) |
// twiddles | two mbarriers.
// ------------------------------------------------------------------------------------
template <typename Real, int NZ, int TZ> __host__ __device__ constexpr size_t zfwd_tma_smem(int S) {
    using C = typename Cplx<Real>::type;
    constexpr size_t GS = size_t(ct_gstride(NZ, TZ, int(sizeof(C))));
    return ((2 * size_t(S) + 2 * DFT_NZSPEC) * GS + NZ) * sizeof(C) + 2 * sizeof(uint64_t) + 128;
}

template <typename Real, int NZ, int TZ, int NT, int MINB, int SM = DFT_MAXS>
__global__ void __launch_bounds__(NT, MINB) k_zconv_fwd_tma(const __grid_constant__ CUtensorMap map_in,
                                                                         const __grid_constant__ CUtensorMap map_n,
                                                                         GridDesc g, SpeciesDesc<Real> sp, Real kfx,
                                                                         Real kfy, Real kfz, int want_psi,
                                                                         typename Cplx<Real>::type* __restrict__ slot_es,
                                                                         int ntiles_x, int ntiles,
                                                                         int* __restrict__ status,
                                                                         const typename Cplx<Real>::type* __restrict__ twz) {
    dep_launch();
    dep_wait();
    using C = typename Cplx<Real>::type;
    constexpr int E = int(sizeof(C) / 8);
    constexpr int TILE = TZ * NZ;
    constexpr int GS = ct_gstride(NZ, TZ, int(sizeof(C)));
    constexpr int PER = (TILE + NT - 1) / NT;
    constexpr uint32_t BOX = uint32_t(TILE * sizeof(C));
    static_assert(NZ > 0 && NZ <= 256 && (TZ * sizeof(C)) % 16 == 0 && BOX % 128 == 0, "z TMA tile");
    extern __shared__ unsigned char smem_raw[];
    const int S = sp.S, ny = g.ny, nxh = g.nxh;
    const int Pn = S * (S + 1) / 2;
    const int stage_elems = S * GS;
    const uintptr_t base = (reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127);
    C* const stage0 = reinterpret_cast<C*>(base);
    C* W = stage0 + 2 * stage_elems;
    C* Vb = W + DFT_NZSPEC * GS;
    C* tw = Vb + DFT_NZSPEC * GS;
    uint64_t* bar = reinterpret_cast<uint64_t*>(tw + NZ);
    const uint32_t tile_bytes = uint32_t(S) * BOX;
    const long long zstride = (long long)ny * g.pxh;

    auto issue = [&](int tile, int s) {
        C* st = stage0 + s * stage_elems;
        const int x = (tile % ntiles_x) * TZ * E, y = tile / ntiles_x;
        tma::mbar_expect_tx(&bar[s], tile_bytes);
        for (int c = 0; c < S; ++c) tma::load_3d(st + c * GS, &map_in, x, y, c * NZ, &bar[s]);
    };
    if (threadIdx.x == 0) {
        tma::mbar_init(&bar[0], 1);
        tma::mbar_init(&bar[1], 1);
        tma::fence_mbar_init();
    }
    for (int i = threadIdx.x; i < NZ; i += NT) tw[i] = twz[i];
    __syncthreads();
    int issued = 0, consumed = 0;   // per stage, packed (stage 1 << 16) | stage 0; thread 0
    if (threadIdx.x == 0) {
        for (int s = 0; s < 2; ++s) {
            const int tile = blockIdx.x + s * gridDim.x;
            if (tile < ntiles) { issue(tile, s); issued += 1 << (16 * s); }
        }
    }
    const Real hx = Real(g.hx), hy = Real(g.hy), hz = Real(g.hz);
    Real flb = Real(0);      // 4 pi lambda_B = pois[s][s] / z_s^2 of a charged species
    for (int s = 0; s < S; ++s)
        if (sp.z[s] != Real(0)) { flb = sp.pois[s][s] / (sp.z[s] * sp.z[s]); break; }
    int it = 0;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++it) {
        const int cur = it & 1;
        const int kx0 = (tile % ntiles_x) * TZ, kyi = tile / ntiles_x;
        const int my = signed_index(kyi, ny);
        // table records of this thread's points, in flight while the tile arrives
        // (the first point's; a thread's later points load theirs at the top of their iteration)
        Real wr[tab_capacity<Real>(2 * SM)];
        Real kr[tab_capacity<Real>(SM * (SM + 1) / 2)];
        auto load_tab = [&](int idx) {
            const int kxi = kx0 + idx % TZ;
            const long long row =
                (((TILE % NT == 0) || idx < TILE) && kxi < nxh) ? tab_row(sp, g, kxi, my, idx / TZ) : 0;
            load_record(wr, sp.tab_w + row * sp.tab_ws, 2 * S);
            load_record(kr, sp.tab_k + row * sp.tab_ks, Pn);
        };
        load_tab(threadIdx.x);
        const bool ok = tma::mbar_wait(&bar[cur], (it >> 1) & 1);
        // the previous tile's TMA stores have finished reading shared memory
        if (threadIdx.x == 0) tma::wait_read_all();
        if (__syncthreads_or(!ok)) {
            if (threadIdx.x == 0) {
                atomicOr(status, DEV_TIMEOUT);
                for (int s = 0; s < 2; ++s) {
                    const int n_is = (issued >> (16 * s)) & 0xffff, n_co = (consumed >> (16 * s)) & 0xffff;
                    if (n_is > n_co) tma::mbar_wait(&bar[s], (n_is - 1) & 1);
                }
            }
            break;
        }
        consumed += 1 << (16 * cur);
        C* st = stage0 + cur * stage_elems;
        C* X = ct_fft_grouped<NZ, false, TZ, GS, true, false, NT>(st, Vb, S, tw);
#pragma unroll 1
        for (int i = 0; i < PER; ++i) {
            const int idx = threadIdx.x + i * NT;
            if ((TILE % NT != 0) && idx >= TILE) break;
            if (i > 0) load_tab(idx);
            const int kzi = idx / TZ, t = idx % TZ;
            const int pos = ct_gpos(kzi, TZ) + t;
            const int kxi = kx0 + t;
            const bool live = kxi < nxh;
            const KPoint<Real> p = kpoint<Real>(g, kxi, kyi, kzi, kfx, kfy, kfz);
            C v[SM];
#pragma unroll
            for (int s = 0; s < SM; ++s)
                if (s < S) v[s] = X[s * GS + pos];
            C acc[5];
#pragma unroll
            for (int a = 0; a < 5; ++a) acc[a] = cmake<C>(Real(0), Real(0));
#pragma unroll
            for (int s = 0; s < SM; ++s) {
                if (s >= S) break;
                wd_add_species<Real>(acc, sp, s, v[s], wr[2 * s], wr[2 * s + 1]);
            }
            if (live) {
                const Real inv_lap = inverse_laplacian<Real, true>(sp, g, p, kxi, kyi, kzi, hx, hy, hz);
                C dv[SM], es[SM];
#pragma unroll
                for (int s = 0; s < SM; ++s) {
                    if (s < S) {
                        dv[s] = v[s];
                        if (p.zero) dv[s].x -= sp.n_rho_b[s];       // DFT(rho - rho_bath) at k = 0
                    }
                    es[s] = cmake<C>(Real(0), Real(0));
                }
#pragma unroll
                for (int j = 0; j < SM; ++j) {
#pragma unroll
                    for (int i2 = 0; i2 <= j; ++i2) {
                        if (j >= S) continue;
                        const Real K = kr[dft_pair(i2, j)] - sp.pois[i2][j] * inv_lap;  // inv_lap is zero at k = 0
                        es[i2] = cadd(es[i2], cscale(dv[j], K));
                        if (j != i2) es[j] = cadd(es[j], cscale(dv[i2], K));
                    }
                }
                const long long o = (long long)kzi * zstride + (long long)kyi * g.pxh + kxi;
#pragma unroll
                for (int s = 0; s < SM; ++s)
                    if (s < S) slot_es[(long long)s * g.nc + o] = es[s];
                if (want_psi) {
                    C q = cmake<C>(Real(0), Real(0));
#pragma unroll
                    for (int s = 0; s < SM; ++s)
                        if (s < S) q = cadd(q, cscale(v[s], sp.z[s]));
                    slot_es[(long long)S * g.nc + o] = cscale(q, flb * inv_lap);
                }
            }
            store_wd_spectra<Real>(W, GS, pos, acc, kz_of(sp, g, kzi, kfz));
        }
        __syncthreads();
        // the stage is free now: refill it with the tile after next while the inverse runs
        if (threadIdx.x == 0) {
            const int next = tile + 2 * gridDim.x;
            if (next < ntiles) { issue(next, cur); issued += 1 << (16 * cur); }
        }
        C* Q = ct_fft_grouped<NZ, true, TZ, GS, false, true, NT>(W, Vb, DFT_NZSPEC, tw);
        tma::fence_proxy_async();
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int q = 0; q < DFT_NZSPEC; ++q)
                tma::store_3d(&map_n, kx0 * E, kyi, dft_zcomp(q) * NZ, Q + q * GS);
            tma::commit();
        }
    }
    if (threadIdx.x == 0) tma::wait_all();
}

// ------------------------------------------------------------------------------------
// The k-space products of the first half as a pass of their own (the first-half z stage in three:
// z forward transform of the S species, this pass, z inverse transform of seven weighted-density
// spectra).  At each k point of the S species spectra (after the x, y and z forward
// transforms) the seven weighted-density spectra, 1/N applied, into slot_n and the S
// bulk-fluid/Poisson spectra into slot_es, both in (kx, ky, kz); the same arithmetic per point as
// k_zconv_fwd_tma.  One thread per k point, kx fastest.
// ------------------------------------------------------------------------------------
// GRAD: also the two grand-potential sums per block, red_energy[2 b] = sum_k w Re(conj(drho_hat_i)
// es_hat_i) and red_energy[2 b + 1] = sum_k w Re(conj(drho_hat_i) dK_ij/dGamma drho_hat_j), w = 1 on
// the kx = 0 and Nyquist planes and 2 elsewhere (the half spectrum standing for the full one).
// TAB: the |k| factors come from the plan's tables (kernels that could also evaluate them, and that
// carried arrays for five species, spilled 316 bytes in FP64).  SM: most species.
template <typename Real, bool GRAD, bool TAB, int SM>
__global__ void __launch_bounds__(kThreads, sizeof(Real) == 4 && !GRAD ? 3 : 2) k_zmul(GridDesc g, SpeciesDesc<Real> sp, Real kfx, Real kfy, Real kfz,
                                                   int want_psi,
                                                   const typename Cplx<Real>::type* __restrict__ in,
                                                   typename Cplx<Real>::type* __restrict__ slot_n,
                                                   typename Cplx<Real>::type* __restrict__ slot_es,
                                                   double* __restrict__ red_energy) {
    dep_launch();
    dep_wait();
    using C = typename Cplx<Real>::type;
    constexpr int TW = tab_capacity<Real>(2 * SM), TK = tab_capacity<Real>(SM * (SM + 1) / 2);
    const int S = sp.S;
    const unsigned nxh = g.nxh, npt = (unsigned)g.nz * g.ny * nxh;
    const int Pn = S * (S + 1) / 2;
    double e_acc = 0.0, q_acc = 0.0;
    for (unsigned q = blockIdx.x * kThreads + threadIdx.x; q < npt; q += gridDim.x * kThreads) {
        const unsigned rz = q / nxh;
        const int kxi = int(q - rz * nxh), kzi = int(rz / (unsigned)g.ny), kyi = int(rz - kzi * g.ny);
        const long long o = (long long)rz * g.pxh + kxi;
        const KPoint<Real> p = kpoint<Real>(g, kxi, kyi, kzi, kfx, kfy, kfz);
        const long long row = TAB ? tab_row(sp, g, kxi, signed_index(kyi, g.ny), kzi) : 0;
        C v[SM];
#pragma unroll
        for (int s = 0; s < SM; ++s)
            if (s < S) v[s] = in[(long long)s * g.nc + o];
        {   // the seven weighted-density spectra the z inverse transforms, 1/N applied
            Real wr[TW];
            if constexpr (TAB) load_record(wr, sp.tab_w + row * sp.tab_ws, 2 * S);
            C acc[5];
#pragma unroll
            for (int a = 0; a < 5; ++a) acc[a] = cmake<C>(Real(0), Real(0));
#pragma unroll
            for (int s = 0; s < SM; ++s) {
                if (s >= S) break;
                Real w0, j3;
                if constexpr (TAB) { w0 = wr[2 * s]; j3 = wr[2 * s + 1]; }
                else fmt_weights<Real>(p.kmag(), sp.R[s], &w0, &j3);
                wd_add_species<Real>(acc, sp, s, v[s], w0, j3);
            }
            C wd[DFT_NZSPEC];
            store_wd_spectra<Real>(wd, 1, 0, acc, kz_of(sp, g, kzi, kfz));
#pragma unroll
            for (int c = 0; c < DFT_NZSPEC; ++c) slot_n[(long long)dft_zcomp(c) * g.nc + o] = wd[c];
        }
        // the bulk-fluid/Poisson spectra
        Real kr[TK];
        Real dkr[GRAD ? TK : 4];
        if constexpr (TAB) {
            load_record(kr, sp.tab_k + row * sp.tab_ks, Pn);
            if constexpr (GRAD) load_record(dkr, sp.tab_dk + row * sp.tab_ks, Pn);
        }
        const Real inv_lap =
            inverse_laplacian<Real, TAB>(sp, g, p, kxi, kyi, kzi, Real(g.hx), Real(g.hy), Real(g.hz));
        if (want_psi) {
            C ps = cmake<C>(Real(0), Real(0));
            Real flb = Real(0);      // 4 pi lambda_B = pois[s][s] / z_s^2 of a charged species
#pragma unroll
            for (int s = 0; s < SM; ++s) {
                if (s >= S) break;
                ps = cadd(ps, cscale(v[s], sp.z[s]));
                if (flb == Real(0) && sp.z[s] != Real(0)) flb = sp.pois[s][s] / (sp.z[s] * sp.z[s]);
            }
            slot_es[(long long)S * g.nc + o] = cscale(ps, flb * inv_lap);   // psi_hat = 4 pi lambda_B q_hat / lap
        }
        const double wk = GRAD ? ((kxi == 0 || (g.nx % 2 == 0 && 2 * kxi == g.nx)) ? 1.0 : 2.0) : 0.0;
        C es[SM];
#pragma unroll
        for (int s = 0; s < SM; ++s) {
            if (s < S && p.zero) v[s].x -= sp.n_rho_b[s];       // DFT(rho - rho_bath) at k = 0
            es[s] = cmake<C>(Real(0), Real(0));
        }
#pragma unroll
        for (int j = 0; j < SM; ++j) {
            if (j >= S) break;
#pragma unroll
            for (int i2 = 0; i2 <= j; ++i2) {
                Real K, dK = Real(0);
                if constexpr (TAB) {
                    K = kr[dft_pair(i2, j)] - sp.pois[i2][j] * inv_lap;     // inv_lap is zero at k = 0
                    if constexpr (GRAD) dK = dkr[dft_pair(i2, j)];
                } else {
                    K = es_kernel<Real>(sp, i2, j, p, inv_lap, GRAD ? &dK : nullptr);
                }
                es[i2] = cadd(es[i2], cscale(v[j], K));
                if (j != i2) es[j] = cadd(es[j], cscale(v[i2], K));
                if constexpr (GRAD) {
                    const double re = double(v[i2].x) * v[j].x + double(v[i2].y) * v[j].y;
                    q_acc += wk * double(dK) * re * (j != i2 ? 2.0 : 1.0);
                }
            }
        }
#pragma unroll
        for (int s = 0; s < SM; ++s) {
            if (s >= S) break;
            if constexpr (GRAD) e_acc += wk * (double(v[s].x) * es[s].x + double(v[s].y) * es[s].y);
            slot_es[(long long)s * g.nc + o] = es[s];
        }
    }
    if constexpr (GRAD) {
        __shared__ double scratch_d[32];
        const double be = block_sum(e_acc, scratch_d);
        const double bq = block_sum(q_acc, scratch_d);
        if (threadIdx.x == 0) {
            red_energy[2 * (long long)blockIdx.x] = be;
            red_energy[2 * (long long)blockIdx.x + 1] = bq;
        }
    }
}

// ------------------------------------------------------------------------------------
// The k-space products of the second half as a pass of their own (between its z transforms): at
// each k point the seven Phi' spectra and the mixed bulk-fluid/Poisson spectra into the ncomp_out
// correlation spectra, 1/N applied.  `samples` 2: the line search's two samples, sample m's Phi'
// spectra at components 9 m .., its weights in ctl[m], its results at components m ncomp_out ..; the
// ES spectra are read once for both.  One thread per k point, kx fastest; a thread reads a sample's
// components before it writes, and a second sample's results end before that sample's own Phi' or
// inside what the same thread has read (2 ncomp_out <= 12 < 18).  TAB, SM as in k_zmul.
// ------------------------------------------------------------------------------------
template <typename Real, bool TAB, int SM>
__global__ void __launch_bounds__(kThreads, sizeof(Real) == 4 ? 3 : 2) k_zmul_bwd(GridDesc g, SpeciesDesc<Real> sp, Real kfx, Real kfy, Real kfz,
                                                       int flags, int ncomp_out, int samples,
                                                       const Ctl* __restrict__ ctl, typename Cplx<Real>::type* phi,
                                                       const typename Cplx<Real>::type* esA,
                                                       const typename Cplx<Real>::type* esB,
                                                       typename Cplx<Real>::type* es_mat) {
    dep_launch();
    dep_wait();
    using C = typename Cplx<Real>::type;
    constexpr int EMAX = SM + 1, TW = tab_capacity<Real>(2 * SM);
    const int S = sp.S;
    const unsigned nxh = g.nxh, npt = (unsigned)g.nz * g.ny * nxh;
    const bool hs = (flags & 1) != 0, es_on = (flags & 2) != 0;
    for (unsigned q = blockIdx.x * kThreads + threadIdx.x; q < npt; q += gridDim.x * kThreads) {
        const unsigned rz = q / nxh;
        const int kxi = int(q - rz * nxh), kzi = int(rz / (unsigned)g.ny), kyi = int(rz - kzi * g.ny);
        const long long o = (long long)rz * g.pxh + kxi;
        Real wr[TW];
        if constexpr (TAB)
            if (hs) load_record(wr, sp.tab_w + tab_row(sp, g, kxi, signed_index(kyi, g.ny), kzi) * sp.tab_ws, 2 * S);
        const Real kz = kz_of(sp, g, kzi, kfz);
        C ea[EMAX], eb[EMAX];
#pragma unroll
        for (int s = 0; s < EMAX; ++s) {
            ea[s] = eb[s] = cmake<C>(Real(0), Real(0));
            if (es_on && s < ncomp_out) {
                ea[s] = esA[(long long)s * g.nc + o];
                if (esB) eb[s] = esB[(long long)s * g.nc + o];
            }
        }
#pragma unroll 1
        for (int m = 0; m < samples; ++m) {
            C* const ph = phi + (long long)m * DFT_NSPEC * g.nc;
            const Real wA = CtlW<Real>::wA(ctl + m), wB = CtlW<Real>::wB(ctl + m);
            C a[5];
            if (hs) {
                C x[DFT_NZSPEC];
#pragma unroll
                for (int c = 0; c < DFT_NZSPEC; ++c) x[c] = ph[(long long)dft_zcomp(c) * g.nc + o];
                bwd_sums<Real>(x, 1, 0, kz, a);
            }
#pragma unroll
            for (int s = 0; s < EMAX; ++s) {
                if (s >= ncomp_out) break;
                C out = cscale(ea[s], wA);
                if (esB) out = cadd(out, cscale(eb[s], wB));
                if (es_mat) es_mat[(long long)s * g.nc + o] = out;
                if (hs && s < S && s < SM) {        // a psi component (s = S) has no hard-sphere part
                    Real w0, j3;
                    if constexpr (TAB) { w0 = wr[2 * (s < SM ? s : 0)]; j3 = wr[2 * (s < SM ? s : 0) + 1]; }
                    else fmt_weights<Real>(kpoint<Real>(g, kxi, kyi, kzi, kfx, kfy, kfz).kmag(), sp.R[s], &w0, &j3);
                    out = bwd_species<Real>(a, sp, s, w0, j3, out);
                }
                phi[(long long)(m * ncomp_out + s) * g.nc + o] = cscale(out, sp.inv_n);
            }
        }
    }
}

// ------------------------------------------------------------------------------------
// Second-half z pass with TMA tiles, persistent: CTA b handles
// tiles b, b + gridDim.x, ...  Two shared-memory stages, each holding one tile's seven Phi'
// spectra, are filled by TMA loads (one cp.async.bulk.tensor per component, completing on the
// stage's mbarrier) while the previous tile is transformed; the tile's bulk-fluid/Poisson spectra arrive in one single-buffered area (third mbarrier), loaded while the previous tile's
// inverse and this tile's forward transform run.  The ncomp_out results are written over the
// first groups of the transformed tile and leave through TMA stores.  At length 256 both
// transforms run in place (ct_fft_grouped_ip), which keeps the CTA within half an SM's shared
// memory (two CTAs per SM instead of one); shorter lengths, where two CTAs fit anyway,
// alternate with a scratch area W (one barrier per stage instead of two).  A tensor map views a
// half-spectrum array as (x: nxh * E, y: ny, plane: nz * ncomp) 8-byte elements, E =
// sizeof(complex) / 8; a component tile is the box (TZ * E, 1, NZ) at plane c * nz.  Columns
// past nxh read as zero and are not written.  The results go to map_out (map_phi's array for a
// single evaluation).  pair: the two line-search samples in one pass, each tile taken for both in
// turn: sample m's Phi' spectra are components 9 m .. 9 m + 8 of map_phi, its mixing weights
// ctl[m], its results components m ncomp_out .. of map_out, and the tile's ES spectra serve both.
// A tile's components are read and written only by the CTA that takes it, loads before stores,
// so map_out may overlap map_phi.  A wait that runs out sets DEV_TIMEOUT and the CTA stops after
// draining the loads it has in flight.
// Shared memory: stage 0 | stage 1 (seven padded groups each) | W (seven padded groups, below
// length 256) | ES (nes dense tiles) | twiddles | three mbarriers.
// ------------------------------------------------------------------------------------
__host__ __device__ constexpr bool zbwd_in_place(int nz) { return nz >= 256; }

template <typename Real, int NZ, int TZ> __host__ __device__ constexpr size_t zbwd_tma_smem(int nes) {
    using C = typename Cplx<Real>::type;
    constexpr size_t GS = size_t(ct_gstride(NZ, TZ, int(sizeof(C))));
    constexpr size_t groups = (zbwd_in_place(NZ) ? 2 : 3) * size_t(DFT_NZSPEC);
    return (groups * GS + size_t(nes) * TZ * NZ + NZ) * sizeof(C) + 3 * sizeof(uint64_t) + 128;
}

template <typename Real, int NZ, int TZ, int NT, int MINB, int SM>
__global__ void __launch_bounds__(NT, MINB) k_zconv_bwd_tma(const __grid_constant__ CUtensorMap map_phi,
                                                            const __grid_constant__ CUtensorMap map_esA,
                                                            const __grid_constant__ CUtensorMap map_esB,
                                                            const __grid_constant__ CUtensorMap map_out, GridDesc g,
                                                            SpeciesDesc<Real> sp, Real kfx, Real kfy, Real kfz,
                                                            int flags, int ncomp_out, int has_esB, int pair,
                                                            const Ctl* __restrict__ ctl,
                                                            typename Cplx<Real>::type* es_mat, int ntiles_x,
                                                            int ntiles, int* __restrict__ status,
                                                            const typename Cplx<Real>::type* __restrict__ twz) {
    dep_launch();
    dep_wait();
    using C = typename Cplx<Real>::type;
    constexpr int E = int(sizeof(C) / 8);
    constexpr int TILE = TZ * NZ;
    constexpr int GS = ct_gstride(NZ, TZ, int(sizeof(C)));
    constexpr int PER = (TILE + NT - 1) / NT;
    constexpr int EMAX = SM + 1;
    constexpr uint32_t BOX = uint32_t(TILE * sizeof(C));
    static_assert(NZ > 0 && NZ <= 256 && (TZ * sizeof(C)) % 16 == 0 && BOX % 128 == 0, "z TMA tile");
    extern __shared__ unsigned char smem_raw[];
    const bool hs = (flags & 1) != 0, es_on = (flags & 2) != 0;
    const int nes = es_on ? ncomp_out * (has_esB ? 2 : 1) : 0;
    constexpr int stage_elems = DFT_NZSPEC * GS;
    constexpr bool IP = zbwd_in_place(NZ);
    const uintptr_t base = (reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127);
    C* const stage0 = reinterpret_cast<C*>(base);
    C* const W = stage0 + 2 * stage_elems;
    C* const es_t = W + (IP ? 0 : stage_elems);
    C* tw = es_t + nes * TILE;
    uint64_t* bar = reinterpret_cast<uint64_t*>(tw + NZ);
    const int S = sp.S, ny = g.ny, nxh = g.nxh;
    const long long zstride = (long long)ny * g.pxh;
    // Work items: tiles, or (pair) each tile twice, for the two line-search samples in turn
    // (sample m's Phi' spectra at components 9 m + dft_zcomp(q) of map_phi, its weights in
    // ctl[m], its results to components m ncomp_out .. of map_out); the ES tiles of a tile are
    // loaded once for both.
    const int shift = pair ? 1 : 0;
    auto item_tile = [&](int item) { return blockIdx.x + (item >> shift) * gridDim.x; };

    auto issue_phi = [&](int item, int s) {
        C* st = stage0 + s * stage_elems;
        const int tile = item_tile(item), m = pair ? (item & 1) : 0;
        const int x = (tile % ntiles_x) * TZ * E, y = tile / ntiles_x;
        tma::mbar_expect_tx(&bar[s], uint32_t(DFT_NZSPEC) * BOX);
        for (int q = 0; q < DFT_NZSPEC; ++q)
            tma::load_3d(st + q * GS, &map_phi, x, y, (m * DFT_NSPEC + dft_zcomp(q)) * NZ, &bar[s]);
    };
    auto issue_es = [&](int tile) {
        const int x = (tile % ntiles_x) * TZ * E, y = tile / ntiles_x;
        tma::mbar_expect_tx(&bar[2], uint32_t(nes) * BOX);
        for (int c = 0; c < ncomp_out; ++c) tma::load_3d(es_t + c * TILE, &map_esA, x, y, c * NZ, &bar[2]);
        if (has_esB)
            for (int c = 0; c < ncomp_out; ++c)
                tma::load_3d(es_t + (ncomp_out + c) * TILE, &map_esB, x, y, c * NZ, &bar[2]);
    };
    if (threadIdx.x == 0) {
        for (int b = 0; b < 3; ++b) tma::mbar_init(&bar[b], 1);
        tma::fence_mbar_init();
    }
    for (int i = threadIdx.x; i < NZ; i += NT) tw[i] = twz[i];
    __syncthreads();
    // Phi' loads issued / consumed per stage, packed as (stage 1 << 16) | stage 0, and ES loads
    // issued / consumed; meaningful in thread 0
    int issued = 0, consumed = 0, es_issued = 0, es_consumed = 0;
    if (threadIdx.x == 0) {
        if (hs)
            for (int s = 0; s < 2; ++s)
                if (item_tile(s) < ntiles) { issue_phi(s, s); issued += 1 << (16 * s); }
        if (es_on && blockIdx.x < ntiles) { issue_es(blockIdx.x); ++es_issued; }
    }
    // on a wait that ran out: record it, let the copies in flight land, stop
    auto drain = [&]() {
        if (threadIdx.x == 0) {
            atomicOr(status, DEV_TIMEOUT);
            for (int s = 0; s < 2; ++s) {
                const int n_is = (issued >> (16 * s)) & 0xffff, n_co = (consumed >> (16 * s)) & 0xffff;
                if (n_is > n_co) tma::mbar_wait(&bar[s], (n_is - 1) & 1);
            }
            if (es_issued > es_consumed) tma::mbar_wait(&bar[2], (es_issued - 1) & 1);
        }
    };
    for (int it = 0;; ++it) {
        const int tile = item_tile(it);
        if (tile >= ntiles) break;
        const int m = pair ? (it & 1) : 0;
        const int ti = it >> shift;                 // this CTA's tile count so far
        const bool last_of_tile = !pair || m == 1;
        const Real wA = CtlW<Real>::wA(ctl + m), wB = CtlW<Real>::wB(ctl + m);
        const int cur = it & 1;
        const int kx0 = (tile % ntiles_x) * TZ, kyi = tile / ntiles_x;
        const int my = signed_index(kyi, ny);
        // the first point's table record is in flight while the tile arrives; a thread's later
        // points load theirs where they are used
        Real wr[tab_capacity<Real>(2 * SM)];
        if (hs) {
            const int idx = threadIdx.x;
            const int kxi = kx0 + idx % TZ;
            const long long row =
                (((TILE % NT == 0) || idx < TILE) && kxi < nxh) ? tab_row(sp, g, kxi, my, idx / TZ) : 0;
            load_record(wr, sp.tab_w + row * sp.tab_ws, 2 * S);
        }
        C* const st = stage0 + cur * stage_elems;
        C* X = st;
        if (hs) {
            const bool ok = tma::mbar_wait(&bar[cur], (it >> 1) & 1);
            if (__syncthreads_or(!ok)) { drain(); break; }
            if (threadIdx.x == 0) consumed += 1 << (16 * cur);
            if constexpr (IP) ct_fft_grouped_ip<NZ, false, TZ, GS, true, false, NT>(X, DFT_NZSPEC, tw);
            else X = ct_fft_grouped<NZ, false, TZ, GS, true, false, NT>(st, W, DFT_NZSPEC, tw);
        }
        // the ES tiles of this tile (loaded since the previous tile's pointwise phase; a pair's
        // second item reuses them); the barrier also ends the forward transform
        const bool ok_es = (es_on && m == 0) ? tma::mbar_wait(&bar[2], ti & 1) : true;
        if (__syncthreads_or(!ok_es)) { drain(); break; }
        if (threadIdx.x == 0 && es_on && m == 0) ++es_consumed;
#pragma unroll 1
        for (int i = 0; i < PER; ++i) {
            const int idx = threadIdx.x + i * NT;
            if ((TILE % NT != 0) && idx >= TILE) break;
            const int kzi = idx / TZ, t = idx % TZ;
            const int pos = ct_gpos(kzi, TZ) + t;
            const int kxi = kx0 + t;
            C out[EMAX];
#pragma unroll
            for (int s = 0; s < EMAX; ++s) {
                out[s] = cmake<C>(Real(0), Real(0));
                if (es_on && s < ncomp_out) {
                    C e = cscale(es_t[s * TILE + idx], wA);
                    if (has_esB) e = cadd(e, cscale(es_t[(ncomp_out + s) * TILE + idx], wB));
                    out[s] = e;
                }
            }
            if (es_on && es_mat && kxi < nxh) {
                const long long o = (long long)kzi * zstride + (long long)kyi * g.pxh + kxi;
#pragma unroll
                for (int s = 0; s < EMAX; ++s)
                    if (s < ncomp_out) es_mat[(long long)s * g.nc + o] = out[s];
            }
            if (hs) {
                if (i > 0)
                    load_record(wr, sp.tab_w + (kxi < nxh ? tab_row(sp, g, kxi, my, kzi) : 0) * sp.tab_ws, 2 * S);
                C asum[5];
                bwd_sums<Real>(X, GS, pos, kz_of(sp, g, kzi, kfz), asum);
#pragma unroll
                for (int s = 0; s < SM; ++s) {
                    if (s >= S) break;
                    out[s] = bwd_species<Real>(asum, sp, s, wr[2 * s], wr[2 * s + 1], out[s]);
                }
            }
            // over the first groups at this thread's own position (read above, by this thread only)
#pragma unroll
            for (int s = 0; s < EMAX; ++s)
                if (s < ncomp_out) X[s * GS + pos] = cscale(out[s], sp.inv_n);
        }
        __syncthreads();
        // the ES area is free after a tile's last item: load the next tile's while this one is
        // finished
        if (threadIdx.x == 0 && es_on && last_of_tile) {
            const int next = tile + gridDim.x;
            if (next < ntiles) { issue_es(next); ++es_issued; }
        }
        C* Q = X;
        if constexpr (IP) ct_fft_grouped_ip<NZ, true, TZ, GS, false, true, NT>(X, ncomp_out, tw);
        else Q = ct_fft_grouped<NZ, true, TZ, GS, false, true, NT>(X, X == st ? W : st, ncomp_out, tw);
        tma::fence_proxy_async();
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int s = 0; s < ncomp_out; ++s)
                tma::store_3d(&map_out, kx0 * E, kyi, (m * ncomp_out + s) * NZ, Q + s * GS);
            tma::commit();
            // the stores read the stage or W: let them finish reading before either is written
            tma::wait_read_all();
            if (hs && item_tile(it + 2) < ntiles) { issue_phi(it + 2, cur); issued += 1 << (16 * cur); }
        }
    }
    if (threadIdx.x == 0) tma::wait_all();
}

// ------------------------------------------------------------------------------------
// Pointwise derivatives of eq. Phi; xi = |nV2|^2/n2^2 is clamped to [0, 1] (Sec. "Numerical
// Stability") and the xi terms vanish where n2 <= 1e-30.  log(1 - n3) and 1/(1 - n3)^m are
// formed in FP64 where n3 >= 0.5, i.e. where n3 approaches 1; below, 1 - n3 is exact in the
// working precision and log1p / the reciprocal are within 2 ulp.  Returns false if n3 >= 1.
// ------------------------------------------------------------------------------------
// White Bear g(n3) = (n3 + D^2 ln D) / n3^2 and g'(n3), D = 1 - n3 (the other forms' last term
// is (n2^3 - 3 n2 nV2.nV2) f(n3), f = g / (36 pi D^2) for White Bear).  Below n3 = 1/2 the closed
// form cancels, so the power series of ln D is summed: g = 3/2 - sum_{k>=3} 2 n3^(k-2) /
// (k (k-1) (k-2)), g' = -sum_{k>=3} 2 n3^(k-3) / (k (k-1)), to k = 24 (FP32) / 52 (FP64), where
// the truncation is below the working precision; from 1/2 up the closed form in FP64 with
// lnD_hi = ln D.
template <typename Real>
__device__ __forceinline__ void wb_g(Real n3, double lnD_hi, Real* g, Real* dg) {
    if (n3 < Real(0.5)) {
        constexpr int K = sizeof(Real) == 4 ? 24 : 52;
        Real sg = Real(0), sd = Real(0);
#pragma unroll
        for (int k = K; k >= 3; --k) {
            sg = sg * n3 + Real(2.0 / (double(k) * double(k - 1) * double(k - 2)));
            sd = sd * n3 + Real(2.0 / (double(k) * double(k - 1)));
        }
        *g = Real(1.5) - n3 * sg;
        *dg = -sd;
    } else {
        const double u = double(n3), d = 1.0 - u, num = u + d * d * lnD_hi;
        *g = Real(num / (u * u));
        *dg = Real((u - 2.0 * d * lnD_hi) / (u * u) - 2.0 * num / (u * u * u));
    }
}

// Phi itself (eq. Phi, or the form `kind`), in FP64, for the grand potential; same clamp as the
// derivatives.  Bounds the Phi' pass of an FP32 plan where it is asked for (64^3: 52 us with it).
template <typename Real> __device__ __forceinline__ double phi_value(const Real* n, int kind) {
    const double n0 = n[0], n1 = n[1], n2 = n[2], n3 = n[3];
    const double D = 1.0 - n3;
    const double q = double(n[7]) * n[7] + double(n[8]) * n[8] + double(n[9]) * n[9];
    const double dot = double(n[4]) * n[7] + double(n[5]) * n[8] + double(n[6]) * n[9];
    const double base = -n0 * log(D) + (n1 * n2 - dot) / D;
    if (kind == DFT_PHI_ROSENFELD) return base + (n2 * n2 * n2 - 3.0 * n2 * q) / (24.0 * CUDART_PI * D * D);
    if (kind == DFT_PHI_WHITE_BEAR) {
        double g, dg;
        wb_g<double>(n3, log(D), &g, &dg);
        return base + (n2 * n2 * n2 - 3.0 * n2 * q) * g / (36.0 * CUDART_PI * D * D);
    }
    double xi = (n2 > 1e-30) ? q / (n2 * n2) : 1.0;
    xi = xi < 0.0 ? 0.0 : (xi > 1.0 ? 1.0 : xi);
    const double om = 1.0 - xi;
    return base + n2 * n2 * n2 * om * om * om / (24.0 * CUDART_PI * D * D);
}

// The derivatives of eq. Phi (kind DFT_PHI_RSLT) or of the other forms, whose last term
// T f(n3), T = n2^3 - 3 n2 nV2.nV2, gives dPhi/dn2 += 3 (n2^2 - nV2.nV2) f, dPhi/dn3 += T f',
// dPhi/dnV2 += -6 n2 f nV2 (no clamp); f = 1/(24 pi D^2) (Rosenfeld) or g/(36 pi D^2) (White
// Bear, f' = (g' D + 2 g)/(36 pi D^3)).
template <typename Real> __device__ __forceinline__ bool phi_derivatives(Real* n, int kind) {
    const Real n0 = n[0], n1 = n[1], n2 = n[2], n3 = n[3];
    const Real v1x = n[4], v1y = n[5], v1z = n[6], v2x = n[7], v2y = n[8], v2z = n[9];
    Real lnD, fiD;
    double lnD_hi = 0.0;
    bool ok = true;
    if (n3 < Real(0.5)) {
        lnD = log1p(-n3);
        fiD = Real(1) / (Real(1) - n3);
    } else {
        const double D = 1.0 - double(n3);
        ok = D > 0.0;
        lnD_hi = log(D);
        lnD = Real(lnD_hi);
        fiD = Real(1.0 / D);
    }
    const Real fiD2 = fiD * fiD, fiD3 = fiD2 * fiD;
    const Real q = v2x * v2x + v2y * v2y + v2z * v2z;
    const Real dot = v1x * v2x + v1y * v2y + v1z * v2z;
    // the constant denominators as products with their reciprocals (rounded once, from double)
    const Real i4pi = Real(1.0 / (4.0 * CUDART_PI)), i8pi = Real(1.0 / (8.0 * CUDART_PI));
    const Real i12pi = Real(1.0 / (12.0 * CUDART_PI)), i24pi = Real(1.0 / (24.0 * CUDART_PI));
    const Real i36pi = Real(1.0 / (36.0 * CUDART_PI));
    n[0] = -lnD;
    n[1] = n2 * fiD;
    n[4] = -v2x * fiD;
    n[5] = -v2y * fiD;
    n[6] = -v2z * fiD;
    if (kind != DFT_PHI_RSLT) {
        Real f, df;
        if (kind == DFT_PHI_ROSENFELD) {
            f = fiD2 * i24pi;
            df = fiD3 * i12pi;
        } else {
            Real g, dg;
            wb_g<Real>(n3, lnD_hi, &g, &dg);
            f = g * fiD2 * i36pi;
            df = (dg * fiD2 + Real(2) * g * fiD3) * i36pi;
        }
        const Real T = n2 * n2 * n2 - Real(3) * n2 * q;
        const Real c6 = Real(6) * n2 * f;
        n[2] = n1 * fiD + Real(3) * (n2 * n2 - q) * f;
        n[3] = n0 * fiD + (n1 * n2 - dot) * fiD2 + T * df;
        n[7] = -v1x * fiD - c6 * v2x;
        n[8] = -v1y * fiD - c6 * v2y;
        n[9] = -v1z * fiD - c6 * v2z;
        return ok;
    }
    Real xi = (n2 > Real(1e-30)) ? q / (n2 * n2) : Real(1);
    xi = xi < Real(0) ? Real(0) : (xi > Real(1) ? Real(1) : xi);
    const Real om = Real(1) - xi;
    n[2] = n1 * fiD + n2 * n2 * om * om * (Real(1) + xi) * fiD2 * i8pi;
    n[3] = n0 * fiD + (n1 * n2 - dot) * fiD2 + n2 * n2 * n2 * om * om * om * fiD3 * i12pi;
    const Real cv = n2 * om * om * fiD2 * i4pi;
    n[7] = -v1x * fiD - cv * v2x;
    n[8] = -v1y * fiD - cv * v2y;
    n[9] = -v1z * fiD - cv * v2z;
    return ok;
}

// The ten weighted densities in the x passes: five complex lines of two real rows each,
// (n0, n1), (n2, nV1y), (n3, nV2x), (nV1x, nV1z), (nV2y, nV2z) (line 2 carries n3 and
// nV2x = i k_x n3, line 3 nV1x = i k_x m; on the way back, line 2 gives B3 and line 3 B4).
// wd_comp(l, j): component of slot j of line l; wd_line / wd_slot: the inverse.
__host__ __device__ constexpr int wd_comp(int l, int j) {
    return l == 0 ? j : (l == 1 ? (j ? 5 : 2) : (l == 2 ? (j ? 7 : 3) : (l == 3 ? (j ? 6 : 4) : 8 + j)));
}
__host__ __device__ constexpr int wd_line(int c) {
    return c < 2 ? 0 : (c == 2 || c == 5 ? 1 : (c == 3 || c == 7 ? 2 : (c == 4 || c == 6 ? 3 : 4)));
}
__host__ __device__ constexpr int wd_slot(int c) { return (c == 1 || c == 5 || c == 7 || c == 6 || c == 9) ? 1 : 0; }

// Items in flight per thread in the update pass's pointwise phase (build flag).
#ifndef DFT_XUPD_BATCH
#define DFT_XUPD_BATCH 1
#endif

// One real value, or 16 bytes of consecutive ones (four floats or two doubles), as a thread's unit
// of global loads and stores.
template <typename Real> struct Vec1 {
    using type = Real;
    static constexpr int n = 1;
    static __device__ __forceinline__ type load(const Real* p) { return *p; }
    static __device__ __forceinline__ void store(Real* p, type v) { *p = v; }
};
template <typename Real> struct Vec16;
template <> struct Vec16<float> {
    using type = float4;
    static constexpr int n = 4;
    static __device__ __forceinline__ type load(const float* p) { return *reinterpret_cast<const float4*>(p); }
    static __device__ __forceinline__ void store(float* p, type v) { *reinterpret_cast<float4*>(p) = v; }
};
template <> struct Vec16<double> {
    using type = double2;
    static constexpr int n = 2;
    static __device__ __forceinline__ type load(const double* p) { return *reinterpret_cast<const double2*>(p); }
    static __device__ __forceinline__ void store(double* p, type v) { *reinterpret_cast<double2*>(p) = v; }
};
__device__ __forceinline__ float& vel(float& v, int) { return v; }
__device__ __forceinline__ double& vel(double& v, int) { return v; }
__device__ __forceinline__ float& vel(float4& v, int e) { return e == 0 ? v.x : (e == 1 ? v.y : (e == 2 ? v.z : v.w)); }
__device__ __forceinline__ double& vel(double2& v, int e) { return e == 0 ? v.x : v.y; }
template <typename V> __device__ __forceinline__ V vzero() { V v; memset(&v, 0, sizeof(V)); return v; }

// Load the Hermitian half rows of two components (mixed wA * A + wB * B) as Z = a + i b over the
// full length nx (Z[nx-k] = conj(a_k) + i conj(b_k)).  Optionally stores the mixed half rows.
// Loads are issued in batches of kBatch elements per thread before any store, so that several
// are in flight at once.
template <typename Real, int NX>
__device__ __forceinline__ void load_pair_rows(const GridDesc& g, int lines, int lines_per_row, long long row0,
                                               long long nrows, int ncomp,
                                               const typename Cplx<Real>::type* A,
                                               const typename Cplx<Real>::type* Bm, Real wA, Real wB,
                                               typename Cplx<Real>::type* mat_out,
                                               typename Cplx<Real>::type* dst) {
    using C = typename Cplx<Real>::type;
    constexpr int kBatch = 4;
    const int nx = NX > 0 ? NX : g.nx, nxh = nx / 2 + 1, pitch = x_pitch<NX>(nx);
    const QHalf<NX> qh(nxh);
    const FastDiv ql(lines_per_row);
    const bool even = (nx % 2) == 0;
    const int total = lines * nxh;
    for (int base = threadIdx.x; base < total; base += kBatch * kThreads) {
        C av[kBatch], bv[kBatch], aB[kBatch], bB[kBatch];
        long long oa[kBatch], ob[kBatch];
        bool live[kBatch], hasb[kBatch];
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
            const int idx = base + j * kThreads;
            const int l = qh(idx), k = idx - l * nxh;
            const int lr = ql.div(l);
            const long long row = row0 + lr;
            const int ca = 2 * (l - lr * lines_per_row), cb = ca + 1;
            live[j] = idx < total && row < nrows;
            hasb[j] = cb < ncomp;
            oa[j] = (long long)ca * g.nc + row * g.pxh + k;
            ob[j] = (long long)cb * g.nc + row * g.pxh + k;
            av[j] = bv[j] = aB[j] = bB[j] = cmake<C>(Real(0), Real(0));
            if (live[j]) {
                av[j] = A[oa[j]];
                if (hasb[j]) bv[j] = A[ob[j]];
                if (Bm) {
                    aB[j] = Bm[oa[j]];
                    if (hasb[j]) bB[j] = Bm[ob[j]];
                }
            }
        }
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
            const int idx = base + j * kThreads;
            if (idx >= total) continue;
            const int l = qh(idx), k = idx - l * nxh;
            C a = cadd(cscale(av[j], wA), cscale(aB[j], wB));
            C b = cadd(cscale(bv[j], wA), cscale(bB[j], wB));
            if (k == 0 || (even && 2 * k == nx)) { a.y = Real(0); b.y = Real(0); }
            if (mat_out && live[j]) {
                mat_out[oa[j]] = a;
                if (hasb[j]) mat_out[ob[j]] = b;
            }
            dst[l * pitch + xo<NX>(k)] = cmake<C>(a.x - b.y, a.y + b.x);
            if (k != 0 && !(even && 2 * k == nx)) dst[l * pitch + xo<NX>(nx - k)] = cmake<C>(a.x + b.y, b.x - a.y);
        }
    }
}

// The S species' half rows of `rows` grid rows as ceil(S/2) complex lines each (species 2l and
// 2l + 1 in line l of a row's lines), for NM sets of spectra (spec, then spec2 into the lines
// after the first set's).  Items are (set, line, k), k fastest; each thread issues the loads of
// kBatch items before any store, so that they are in flight together.
template <typename Real, int NX, int NM = 1>
__device__ __forceinline__ void load_species_rows(const GridDesc& g, int rows, long long row0, long long nrows, int S,
                                                  const typename Cplx<Real>::type* __restrict__ spec,
                                                  const typename Cplx<Real>::type* __restrict__ spec2,
                                                  typename Cplx<Real>::type* dst) {
    using C = typename Cplx<Real>::type;
    constexpr int kBatch = 4;
    const int nx = NX > 0 ? NX : g.nx, nxh = nx / 2 + 1, pitch = x_pitch<NX>(nx);
    const QHalf<NX> qh(nxh);
    const bool even = (nx % 2) == 0;
    const int lpr = (S + 1) / 2;
    const FastDiv ql(lpr);
    const int lines = rows * lpr;                 // lines of one set
    const int total = NM * lines * nxh;
    for (int base = threadIdx.x; base < total; base += kBatch * kThreads) {
        C av[kBatch], bv[kBatch];
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
            const int idx = base + j * kThreads;
            const int ml = qh(idx), k = idx - ml * nxh;
            const int m = NM == 1 ? 0 : (ml >= lines ? 1 : 0), l = ml - m * lines;
            const int lr = ql.div(l);
            const long long row = row0 + lr;
            const int ca = 2 * (l - lr * lpr), cb = ca + 1;
            const C* src = (NM == 2 && m == 1) ? spec2 : spec;
            const long long o = row * g.pxh + k;
            av[j] = bv[j] = cmake<C>(Real(0), Real(0));
            if (idx < total && row < nrows) {
                av[j] = src[(long long)ca * g.nc + o];
                if (cb < S) bv[j] = src[(long long)cb * g.nc + o];
            }
        }
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
            const int idx = base + j * kThreads;
            if (idx >= total) continue;
            const int ml = qh(idx), k = idx - ml * nxh;
            C a = av[j], b = bv[j];
            const bool edge = k == 0 || (even && 2 * k == nx);
            if (edge) { a.y = Real(0); b.y = Real(0); }
            dst[ml * pitch + xo<NX>(k)] = cmake<C>(a.x - b.y, a.y + b.x);
            if (!edge) dst[ml * pitch + xo<NX>(nx - k)] = cmake<C>(a.x + b.y, b.x - a.y);
        }
    }
}

// One component's half rows of `rows` grid rows, two grid rows per complex line (rows 2l and
// 2l + 1 of the block in line l; a missing partner row reads as zero).
template <typename Real, int NX>
__device__ __forceinline__ void load_row_pairs(const GridDesc& g, int rows, long long row0, long long nrows,
                                               const typename Cplx<Real>::type* __restrict__ spec,
                                               typename Cplx<Real>::type* dst) {
    using C = typename Cplx<Real>::type;
    const int nx = NX > 0 ? NX : g.nx, nxh = nx / 2 + 1, pitch = x_pitch<NX>(nx);
    const QHalf<NX> qh(nxh);
    const bool even = (nx % 2) == 0;
    const int lines = (rows + 1) / 2;
    const int total = lines * nxh;
    // the loads of kBatch items per thread in flight together
    constexpr int kBatch = 4;
    for (int base = threadIdx.x; base < total; base += kBatch * kThreads) {
        C av[kBatch], bv[kBatch];
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
            const int idx = base + j * kThreads;
            const int l = qh(idx), k = idx - l * nxh;
            const int ra = 2 * l, rb = 2 * l + 1;
            av[j] = bv[j] = cmake<C>(Real(0), Real(0));
            if (idx < total) {
                if (row0 + ra < nrows) av[j] = spec[(row0 + ra) * g.pxh + k];
                if (rb < rows && row0 + rb < nrows) bv[j] = spec[(row0 + rb) * g.pxh + k];
            }
        }
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
            const int idx = base + j * kThreads;
            if (idx >= total) continue;
            const int l = qh(idx), k = idx - l * nxh;
            C a = av[j], b = bv[j];
            const bool edge = k == 0 || (even && 2 * k == nx);
            if (edge) { a.y = Real(0); b.y = Real(0); }
            dst[l * pitch + xo<NX>(k)] = cmake<C>(a.x - b.y, a.y + b.x);
            if (!edge) dst[l * pitch + xo<NX>(nx - k)] = cmake<C>(a.x + b.y, b.x - a.y);
        }
    }
}

// The ten weighted-density rows of `rows` grid rows as five complex lines each (wd_comp
// arrangement), built from the nine kept spectra mixed as wA * A + wB * B (B optional), with
// n_V1x = i k_x m and n_V2x = i k_x n3 (zero on the Nyquist index); mat_out (optional) receives
// the nine mixed spectra.  One thread handles all lines of one (row, k): the index arithmetic is
// shared and its eighteen loads are in flight together.  NM mixtures (weights wA[a], wB[a]) of
// the same loads: mixture a of row r goes to lines (r NM + a) 5 .. + 4.
// STAGED: the spectra come from shared memory instead, component c of the block's rows at
// stage[c cstride + r pxh + k] (slot B's at components 9..17; Bm only tells that they are there).
template <typename Real, int NX, int NM = 1, bool STAGED = false>
__device__ __forceinline__ void load_wd_rows(const GridDesc& g, int rows, long long row0, long long nrows,
                                             const typename Cplx<Real>::type* A,
                                             const typename Cplx<Real>::type* Bm, const Real* wA,
                                             const Real* wB, typename Cplx<Real>::type* mat_out, Real kfx,
                                             typename Cplx<Real>::type* dst,
                                             const typename Cplx<Real>::type* stage = nullptr, int cstride = 0) {
    using C = typename Cplx<Real>::type;
    const int nx = NX > 0 ? NX : g.nx, nxh = nx / 2 + 1, pitch = x_pitch<NX>(nx);
    const QHalf<NX> qh(nxh);
    const bool even = (nx % 2) == 0;
    for (int idx = threadIdx.x; idx < rows * nxh; idx += blockDim.x) {
        const int r = qh(idx), k = idx - r * nxh;
        const unsigned row = (unsigned)row0 + r;
        const bool live = row < (unsigned)nrows;
        const unsigned o = row * (unsigned)g.pxh + k;      // 32-bit: a component has < 2^27 elements
        C v[DFT_NSPEC], vb[DFT_NSPEC];
#pragma unroll
        for (int c = 0; c < DFT_NSPEC; ++c) {
            v[c] = vb[c] = cmake<C>(Real(0), Real(0));
            if (live) {
                if constexpr (STAGED) {
                    v[c] = stage[c * cstride + r * g.pxh + k];
                    if (Bm) vb[c] = stage[(DFT_NSPEC + c) * cstride + r * g.pxh + k];
                } else {
                    v[c] = (A + (long long)c * g.nc)[o];
                    if (Bm) vb[c] = (Bm + (long long)c * g.nc)[o];
                }
            }
        }
        const bool edge = k == 0 || (even && 2 * k == nx);
        const bool nyq = even && 2 * k == nx;
        const Real kx = Real(k) * kfx;
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            C u[DFT_NSPEC];
#pragma unroll
            for (int c = 0; c < DFT_NSPEC; ++c) {
                u[c] = cadd(cscale(v[c], wA[m]), cscale(vb[c], wB[m]));
                if (edge) u[c].y = Real(0);
                if (NM == 1 && mat_out && live) (mat_out + (long long)c * g.nc)[o] = u[c];
            }
            const C zero = cmake<C>(Real(0), Real(0));
            const C dm = nyq ? zero : cmake<C>(-kx * u[4].y, kx * u[4].x);     // i k_x m
            const C dn3 = nyq ? zero : cmake<C>(-kx * u[3].y, kx * u[3].x);    // i k_x n3
            // line l holds (a, b) = (wd_comp(l, 0), wd_comp(l, 1))
            const C la[5] = {u[0], u[2], u[3], dm, u[7]};
            const C lb[5] = {u[1], u[5], dn3, u[6], u[8]};
            const int l0 = (r * NM + m) * 5;
#pragma unroll
            for (int l = 0; l < 5; ++l) {
                const C a = la[l], b = lb[l];
                dst[(l0 + l) * pitch + xo<NX>(k)] = cmake<C>(a.x - b.y, a.y + b.x);
                if (!edge) dst[(l0 + l) * pitch + xo<NX>(nx - k)] = cmake<C>(a.x + b.y, b.x - a.y);
            }
        }
    }
}

// Separate Z = FFT(a + i b) of two real rows into their half spectra and store them.
template <typename Real, int NX>
__device__ __forceinline__ void store_pair_rows(const GridDesc& g, int lines, int lines_per_row, long long row0,
                                                long long nrows, int ncomp, const typename Cplx<Real>::type* R,
                                                typename Cplx<Real>::type* out) {
    using C = typename Cplx<Real>::type;
    const int nx = NX > 0 ? NX : g.nx, nxh = nx / 2 + 1, pitch = x_pitch<NX>(nx);
    const QHalf<NX> qh(nxh);
    const FastDiv ql(lines_per_row);
    for (int idx = threadIdx.x; idx < lines * nxh; idx += blockDim.x) {
        const int l = qh(idx), k = idx - l * nxh;
        const int lr = ql.div(l);
        const long long row = row0 + lr;
        if (row >= nrows) continue;
        const int ca = 2 * (l - lr * lines_per_row), cb = ca + 1;
        const C zk = R[l * pitch + xo<NX>(k)];
        const C znk = R[l * pitch + xo<NX>(k == 0 ? 0 : nx - k)];
        const C s = cadd(zk, cconj(znk));
        const C d = csub(zk, cconj(znk));
        out[(long long)ca * g.nc + row * g.pxh + k] = cmake<C>(Real(0.5) * s.x, Real(0.5) * s.y);
        if (cb < ncomp) out[(long long)cb * g.nc + row * g.pxh + k] = cmake<C>(Real(0.5) * d.y, Real(-0.5) * d.x);
    }
}

// Half spectra of the ten dPhi/dn_alpha rows of `rows` grid rows (five complex lines each, in the
// wd_comp arrangement of load_pair_rows) into the nine spectra the y pass takes:
// Phi_0..Phi_2, B3 = Phi_3 - i k_x Phi_V2x, B4 = -i k_x Phi_V1x, Phi_V1y, Phi_V1z, Phi_V2y,
// Phi_V2z (the -i k_x terms dropped on the Nyquist index).  Each line maps to its own outputs:
// line 2 holds Phi_3 and Phi_V2x, line 3 Phi_V1x and Phi_V1z.
// NM mixtures: those of sub-row r NM + m (lines (r NM + m) 5 ..) go to out + m DFT_NSPEC nc.
template <typename Real, int NX, int NM = 1>
__device__ __forceinline__ void store_phi_spectra(const GridDesc& g, int rows, long long row0, long long nrows,
                                                  Real kfx, const typename Cplx<Real>::type* R,
                                                  typename Cplx<Real>::type* out0) {
    using C = typename Cplx<Real>::type;
    const int nx = NX > 0 ? NX : g.nx, nxh = nx / 2 + 1, pitch = x_pitch<NX>(nx);
    const QHalf<NX> qh(nxh);
    const bool even = (nx % 2) == 0;
    for (int idx = threadIdx.x; idx < rows * NM * nxh; idx += blockDim.x) {
        const int rr = qh(idx), k = idx - rr * nxh;
        const int r = rr / NM;
        const unsigned row = (unsigned)row0 + r;
        if (row >= (unsigned)nrows) continue;
        C* out = out0 + (long long)(rr - r * NM) * DFT_NSPEC * g.nc;
        C a[5], b[5];
#pragma unroll
        for (int l = 0; l < 5; ++l) {
            const C zk = R[(rr * 5 + l) * pitch + xo<NX>(k)];
            const C znk = R[(rr * 5 + l) * pitch + xo<NX>(k == 0 ? 0 : nx - k)];
            const C s = cadd(zk, cconj(znk));
            const C d = csub(zk, cconj(znk));
            a[l] = cmake<C>(Real(0.5) * s.x, Real(0.5) * s.y);
            b[l] = cmake<C>(Real(0.5) * d.y, Real(-0.5) * d.x);
        }
        const Real kx = (even && 2 * k == nx) ? Real(0) : Real(k) * kfx;
        const unsigned o = row * (unsigned)g.pxh + k;
        (out + 0 * g.nc)[o] = a[0];
        (out + 1 * g.nc)[o] = b[0];
        (out + 2 * g.nc)[o] = a[1];
        (out + 5 * g.nc)[o] = b[1];
        (out + 3 * g.nc)[o] = cadd(a[2], cmake<C>(kx * b[2].y, -kx * b[2].x));   // Phi_3 - i k_x Phi_V2x
        (out + 4 * g.nc)[o] = cmake<C>(kx * a[3].y, -kx * a[3].x);               // -i k_x Phi_V1x
        (out + 6 * g.nc)[o] = b[3];
        (out + 7 * g.nc)[o] = a[4];
        (out + 8 * g.nc)[o] = b[4];
    }
}

// ------------------------------------------------------------------------------------
// x pass of the second half's start: n_alpha (mixed from slots A and B) -> real space ->
// dPhi/dn_alpha -> half spectra.  grid: ceil(ny nz / LR); 5 lines (component pairs) per row.
// ------------------------------------------------------------------------------------
// NM = 2: the two line-search samples at once (weights from ctl[1] and ctl[2]; the same loads
// of both slots serve both; sample m's nine Phi' spectra go to phi_out + m DFT_NSPEC nc).
template <typename Real, int NX, int NM = 1>
__global__ void __launch_bounds__(kThreads) k_xphi(GridDesc g, AxisPlan px, int LR, const Ctl* __restrict__ ctl,
                                                   const typename Cplx<Real>::type* slotA,
                                                   const typename Cplx<Real>::type* slotB,
                                                   typename Cplx<Real>::type* mat_out,
                                                   typename Cplx<Real>::type* __restrict__ phi_out,
                                                   float* __restrict__ red_max, int* __restrict__ status,
                                                   double* __restrict__ red_phi, Real kfx,
                                                   const typename Cplx<Real>::type* __restrict__ twx) {
    dep_launch();
    dep_wait();
    using C = typename Cplx<Real>::type;
    extern __shared__ unsigned char smem_raw[];
    __shared__ float scratch_f[32];
    __shared__ double scratch_d[32];
    double phi_acc = 0.0;   // sum of Phi(n) over the block's points (grand potential only)
    const int nx = NX > 0 ? NX : g.nx, pitch = x_pitch<NX>(nx);
    const QRow<NX> qx(nx);
    const int lines = 5 * NM * LR;
    C* tw = align_ptr<C>(smem_raw);
    C* A = tw + nx;
    C* B = A + lines * pitch;
    for (int i = threadIdx.x; i < nx; i += blockDim.x) tw[i] = twx[i];
    const long long nrows = (long long)g.ny * g.nz;
    const long long row0 = (long long)blockIdx.x * LR;
    Real wA[NM], wB[NM];
#pragma unroll
    for (int m = 0; m < NM; ++m) {
        const Ctl* cw = NM == 1 ? ctl : ctl + 1 + m;
        wA[m] = CtlW<Real>::wA(cw);
        wB[m] = CtlW<Real>::wB(cw);
    }
    load_wd_rows<Real, NX, NM>(g, LR, row0, nrows, slotA, slotB, wA, wB, mat_out, kfx, A);
    __syncthreads();
    C* R = any_fft<NX, true>(A, B, px, lines, pitch, tw);
    float mx = -CUDART_INF_F;
    bool bad = false;
    for (int idx = threadIdx.x; idx < LR * NM * nx; idx += blockDim.x) {
        const int rr = qx(idx), x = idx - rr * nx;
        const int r = rr / NM;
        C* base = R + (rr * 5) * pitch + xo<NX>(x);
        Real n[DFT_NCOMP];
        {   // lines (n0, n1), (n2, nV1y), (n3, nV2x), (nV1x, nV1z), (nV2y, nV2z): see wd_comp
            const C v0 = base[0], v1 = base[pitch], v2 = base[2 * pitch], v3 = base[3 * pitch], v4 = base[4 * pitch];
            n[0] = v0.x; n[1] = v0.y; n[2] = v1.x; n[5] = v1.y; n[3] = v2.x;
            n[7] = v2.y; n[4] = v3.x; n[6] = v3.y; n[8] = v4.x; n[9] = v4.y;
        }
        if (row0 + r < nrows) mx = fmaxf(mx, float(n[3]));
        if (red_phi && row0 + r < nrows) phi_acc += phi_value<Real>(n, g.phi);
        const bool ok = phi_derivatives<Real>(n, g.phi);
        if (!ok && row0 + r < nrows) bad = true;
        base[0] = cmake<C>(n[0], n[1]);
        base[pitch] = cmake<C>(n[2], n[5]);
        base[2 * pitch] = cmake<C>(n[3], n[7]);
        base[3 * pitch] = cmake<C>(n[4], n[6]);
        base[4 * pitch] = cmake<C>(n[8], n[9]);
    }
    if (bad) atomicOr(status, DEV_N3BOUND);
    __syncthreads();
    C* other = (R == A) ? B : A;
    C* F = any_fft<NX, false>(R, other, px, lines, pitch, tw);
    store_phi_spectra<Real, NX, NM>(g, LR, row0, nrows, kfx, F, phi_out);
    const float bm = block_max(mx, scratch_f);
    if (threadIdx.x == 0 && red_max) red_max[blockIdx.x] = bm;
    if (red_phi) {
        const double bp = block_sum(phi_acc, scratch_d);
        if (threadIdx.x == 0) red_phi[blockIdx.x] = bp;
    }
}

// ------------------------------------------------------------------------------------
// The part of the persistent Phi' x passes after the weighted-density lines of a block's LR rows
// (NM mixtures, the load_wd_rows arrangement) are in A (synced): x C2R, dPhi/dn_alpha at each
// point (the maximum of n3 over the live rows into *mx, n3 >= 1 met into *bad), x R2C, and the
// nine Phi' spectra of each mixture out.  The line buffers stay in use until the caller's next
// barrier.
// ------------------------------------------------------------------------------------
template <typename Real, int NX, int NM>
__device__ __forceinline__ void xphi_rows_ct(const GridDesc& g, int LR, long long row0, long long nrows,
                                             typename Cplx<Real>::type* A, typename Cplx<Real>::type* B,
                                             const typename Cplx<Real>::type* tw, Real kfx,
                                             typename Cplx<Real>::type* __restrict__ phi_out, float* mx,
                                             bool* bad) {
    using C = typename Cplx<Real>::type;
    constexpr int pitch = ct_row_pitch(NX);
    const int lines = 5 * NM * LR;
    C* R = ct_fft<NX, true, false, 0>(A, B, lines, pitch, tw);
    for (int idx = threadIdx.x; idx < LR * NM * NX; idx += kThreads) {
        const int rr = idx / NX, x = idx - (idx / NX) * NX;
        const int r = rr / NM;
        C* bp = R + (rr * 5) * pitch + xo<NX>(x);
        Real n[DFT_NCOMP];
        {   // lines (n0, n1), (n2, nV1y), (n3, nV2x), (nV1x, nV1z), (nV2y, nV2z): see wd_comp
            const C v0 = bp[0], v1 = bp[pitch], v2 = bp[2 * pitch], v3 = bp[3 * pitch], v4 = bp[4 * pitch];
            n[0] = v0.x; n[1] = v0.y; n[2] = v1.x; n[5] = v1.y; n[3] = v2.x;
            n[7] = v2.y; n[4] = v3.x; n[6] = v3.y; n[8] = v4.x; n[9] = v4.y;
        }
        if (row0 + r < nrows) *mx = fmaxf(*mx, float(n[3]));
        const bool okp = phi_derivatives<Real>(n, g.phi);
        if (!okp && row0 + r < nrows) *bad = true;
        bp[0] = cmake<C>(n[0], n[1]);
        bp[pitch] = cmake<C>(n[2], n[5]);
        bp[2 * pitch] = cmake<C>(n[3], n[7]);
        bp[3 * pitch] = cmake<C>(n[4], n[6]);
        bp[4 * pitch] = cmake<C>(n[8], n[9]);
    }
    __syncthreads();
    C* other = (R == A) ? B : A;
    C* F = ct_fft<NX, false, false, 0>(R, other, lines, pitch, tw);
    store_phi_spectra<Real, NX, NM>(g, LR, row0, nrows, kfx, F, phi_out);
}

// ------------------------------------------------------------------------------------
// Persistent form of k_xphi for compile-time lengths (same contract, same arithmetic per block):
// CTA b takes the row blocks b, b + gridDim.x, ...  The nine (one slot) or eighteen (two slots)
// half-spectrum components of a block's LR rows are contiguous in each component, so they
// arrive by one bulk copy each (cp.async.bulk, completing on the stage's mbarrier) into one of
// two staging areas, requested two blocks ahead: the transforms and Phi' of one block run
// while the next blocks' spectra are in flight.  A wait that runs out sets DEV_TIMEOUT and the
// CTA stops after draining the copies it has in flight.
// Shared memory: twiddles | stage 0 | stage 1 (nsrc components of LR rows each) | line
// buffers A, B | two mbarriers.
// ------------------------------------------------------------------------------------
template <typename Real, int NX> __host__ __device__ constexpr size_t xphi_tma_smem(int nm, int LR, int nsrc, int pxh) {
    using C = typename Cplx<Real>::type;
    return (size_t(NX) + 2 * size_t(nsrc) * LR * pxh + 2 * size_t(5 * nm * LR) * ct_row_pitch(NX)) * sizeof(C) +
           2 * sizeof(uint64_t) + 256;
}

template <typename Real, int NX, int NM>
__global__ void __launch_bounds__(kThreads, sizeof(Real) == 4 ? 3 : 1) k_xphi_tma(GridDesc g, int LR, const Ctl* __restrict__ ctl,
                                                       const typename Cplx<Real>::type* slotA,
                                                       const typename Cplx<Real>::type* slotB,
                                                       typename Cplx<Real>::type* mat_out,
                                                       typename Cplx<Real>::type* __restrict__ phi_out,
                                                       float* __restrict__ red_max, int* __restrict__ status,
                                                       Real kfx, const typename Cplx<Real>::type* __restrict__ twx) {
    dep_launch();
    dep_wait();
    static_assert(NX > 0, "compile-time lengths only");
    using C = typename Cplx<Real>::type;
    extern __shared__ unsigned char smem_raw[];
    __shared__ float scratch_f[32];
    constexpr int pitch = ct_row_pitch(NX);
    const int nsrc = slotB ? 2 * DFT_NSPEC : DFT_NSPEC;
    const int cstride = LR * g.pxh;                       // elements per staged component
    const int lines = 5 * NM * LR;
    const uintptr_t base = (reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127);
    C* tw = reinterpret_cast<C*>(base);
    C* stage0 = tw + ((NX + 15) & ~15);                   // 128-byte aligned (NX a multiple of 16)
    C* A = stage0 + 2 * nsrc * cstride;
    C* B = A + lines * pitch;
    uint64_t* bar = reinterpret_cast<uint64_t*>(B + lines * pitch);
    const long long nrows = (long long)g.ny * g.nz;
    const int nblk = (int)((nrows + LR - 1) / LR);
    Real wA[NM], wB[NM];
#pragma unroll
    for (int m = 0; m < NM; ++m) {
        const Ctl* cw = NM == 1 ? ctl : ctl + 1 + m;
        wA[m] = CtlW<Real>::wA(cw);
        wB[m] = CtlW<Real>::wB(cw);
    }
    auto issue = [&](int blk, int s) {
        const long long r0 = (long long)blk * LR;
        const int rows = (int)(nrows - r0 < LR ? nrows - r0 : LR);
        const uint32_t bytes = uint32_t(rows) * uint32_t(g.pxh) * uint32_t(sizeof(C));
        C* st = stage0 + s * nsrc * cstride;
        tma::mbar_expect_tx(&bar[s], bytes * uint32_t(nsrc));
        for (int c = 0; c < nsrc; ++c) {
            const C* src = (c < DFT_NSPEC ? slotA + (long long)c * g.nc : slotB + (long long)(c - DFT_NSPEC) * g.nc) +
                           r0 * g.pxh;
            tma::bulk_load(st + c * cstride, src, bytes, &bar[s]);
        }
    };
    if (threadIdx.x == 0) {
        tma::mbar_init(&bar[0], 1);
        tma::mbar_init(&bar[1], 1);
        tma::fence_mbar_init();
    }
    for (int i = threadIdx.x; i < NX; i += kThreads) tw[i] = twx[i];
    __syncthreads();
    int issued = 0, consumed = 0;   // per stage, packed (stage 1 << 16) | stage 0; thread 0
    if (threadIdx.x == 0) {
        for (int s = 0; s < 2; ++s) {
            const int blk = blockIdx.x + s * gridDim.x;
            if (blk < nblk) { issue(blk, s); issued += 1 << (16 * s); }
        }
    }
    bool bad = false;
    int it = 0;
    for (int blk = blockIdx.x; blk < nblk; blk += gridDim.x, ++it) {
        const int cur = it & 1;
        const long long row0 = (long long)blk * LR;
        const bool ok = tma::mbar_wait(&bar[cur], (it >> 1) & 1);
        if (__syncthreads_or(!ok)) {
            if (threadIdx.x == 0) {
                atomicOr(status, DEV_TIMEOUT);
                for (int s = 0; s < 2; ++s) {
                    const int n_is = (issued >> (16 * s)) & 0xffff, n_co = (consumed >> (16 * s)) & 0xffff;
                    if (n_is > n_co) tma::mbar_wait(&bar[s], (n_is - 1) & 1);
                }
            }
            break;
        }
        consumed += 1 << (16 * cur);
        const C* st = stage0 + cur * nsrc * cstride;
        load_wd_rows<Real, NX, NM, true>(g, LR, row0, nrows, nullptr, slotB, wA, wB, mat_out, kfx, A, st, cstride);
        __syncthreads();
        // the stage is free: request the block after next into it while this one is transformed
        if (threadIdx.x == 0) {
            const int next = blk + 2 * gridDim.x;
            if (next < nblk) { issue(next, cur); issued += 1 << (16 * cur); }
        }
        float mx = -CUDART_INF_F;
        xphi_rows_ct<Real, NX, NM>(g, LR, row0, nrows, A, B, tw, kfx, phi_out, &mx, &bad);
        const float bm = block_max(mx, scratch_f);
        if (threadIdx.x == 0 && red_max) red_max[blk] = bm;
        __syncthreads();   // the line buffers are rewritten by the next block
    }
    if (bad) atomicOr(status, DEV_N3BOUND);
}

// ------------------------------------------------------------------------------------
// Persistent form of k_xphi with one staging area filled by per-thread 16-byte asynchronous
// copies (cp.async; same contract, same arithmetic per block): the spectra of a CTA's next row
// block are requested as soon as the current block's have been turned into lines, and arrive
// while it is transformed.  Each thread waits for its own copies, then a barrier: no mbarrier,
// no bound needed.  Shared memory: twiddles | stage (nsrc components of LR rows) | line buffers
// A, B.  Row blocks of a component are contiguous and start on 16-byte boundaries (pxh even).
// ------------------------------------------------------------------------------------
template <typename Real, int NX> __host__ __device__ constexpr size_t xphi_cpa_smem(int nm, int LR, int nsrc, int pxh) {
    using C = typename Cplx<Real>::type;
    return (size_t(NX) + size_t(nsrc) * LR * pxh + 2 * size_t(5 * nm * LR) * ct_row_pitch(NX)) * sizeof(C) + 128;
}

template <typename Real, int NX, int NM>
__global__ void __launch_bounds__(kThreads, sizeof(Real) == 4 ? 3 : 1) k_xphi_cpa(GridDesc g, int LR, const Ctl* __restrict__ ctl,
                                                       const typename Cplx<Real>::type* slotA,
                                                       const typename Cplx<Real>::type* slotB,
                                                       typename Cplx<Real>::type* mat_out,
                                                       typename Cplx<Real>::type* __restrict__ phi_out,
                                                       float* __restrict__ red_max, int* __restrict__ status,
                                                       Real kfx, const typename Cplx<Real>::type* __restrict__ twx) {
    static_assert(NX > 0, "compile-time lengths only");
    using C = typename Cplx<Real>::type;
    extern __shared__ unsigned char smem_raw[];
    __shared__ float scratch_f[32];
    const int nsrc = slotB ? 2 * DFT_NSPEC : DFT_NSPEC;
    const int cstride = LR * g.pxh;                       // elements per staged component
    const int lines = 5 * NM * LR;
    constexpr int pitch = ct_row_pitch(NX);
    const uintptr_t base = (reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127);
    C* tw = reinterpret_cast<C*>(base);
    C* stage = tw + ((NX + 15) & ~15);                    // 128-byte aligned (NX a multiple of 16)
    C* A = stage + nsrc * cstride;
    C* B = A + lines * pitch;
    const long long nrows = (long long)g.ny * g.nz;
    const int nblk = (int)((nrows + LR - 1) / LR);
    for (int i = threadIdx.x; i < NX; i += kThreads) tw[i] = twx[i];
    dep_launch();
    dep_wait();
    Real wA[NM], wB[NM];
#pragma unroll
    for (int m = 0; m < NM; ++m) {
        const Ctl* cw = NM == 1 ? ctl : ctl + 1 + m;
        wA[m] = CtlW<Real>::wA(cw);
        wB[m] = CtlW<Real>::wB(cw);
    }
    // the nsrc components of row block blk, in 16-byte chunks spread over the threads
    auto issue = [&](int blk) {
        const long long r0 = (long long)blk * LR;
        const int rows = (int)(nrows - r0 < LR ? nrows - r0 : LR);
        const int per = int((long long)rows * g.pxh * sizeof(C) / 16);
        for (int i = threadIdx.x; i < nsrc * per; i += kThreads) {
            const int c = i / per, q = i - c * per;
            const C* src = (c < DFT_NSPEC ? slotA + (long long)c * g.nc : slotB + (long long)(c - DFT_NSPEC) * g.nc) +
                           r0 * g.pxh;
            tma::cp16(reinterpret_cast<char*>(stage + c * cstride) + 16 * q, reinterpret_cast<const char*>(src) + 16 * q);
        }
        tma::cp_commit();
    };
    if (blockIdx.x < nblk) issue(blockIdx.x);
    bool bad = false;
    for (int blk = blockIdx.x; blk < nblk; blk += gridDim.x) {
        const long long row0 = (long long)blk * LR;
        tma::cp_wait_all();
        __syncthreads();
        load_wd_rows<Real, NX, NM, true>(g, LR, row0, nrows, nullptr, slotB, wA, wB, mat_out, kfx, A, stage, cstride);
        __syncthreads();
        // the stage is free: request the next block into it while this one is transformed
        if (blk + gridDim.x < nblk) issue(blk + gridDim.x);
        float mx = -CUDART_INF_F;
        xphi_rows_ct<Real, NX, NM>(g, LR, row0, nrows, A, B, tw, kfx, phi_out, &mx, &bad);
        const float bm = block_max(mx, scratch_f);
        if (threadIdx.x == 0 && red_max) red_max[blk] = bm;
        __syncthreads();   // the line buffers are rewritten by the next block
    }
    if (bad) atomicOr(status, DEV_N3BOUND);
}

// ------------------------------------------------------------------------------------
// Normalisation of fixed-number species: per block, sum over accessible points of
// e_i = exp(-V_i + c_i) for the species with canon[i] (c_i from the half spectra cspec),
// red[block * DFT_MAXS + i].  Only the complex lines holding such species are transformed.
// grid: ceil(ny nz / LR); nl lines per row (line l = species pair (2 line_of[l], +1)).
// ------------------------------------------------------------------------------------
template <typename Real, int NX>
__global__ void __launch_bounds__(kThreads) k_xcanon(GridDesc g, AxisPlan px, SpeciesDesc<Real> sp, int LR, int nl,
                                                     int line0, int line1, int line2,
                                                     const typename Cplx<Real>::type* __restrict__ cspec,
                                                     const Real* __restrict__ V, double* __restrict__ red,
                                                     const typename Cplx<Real>::type* __restrict__ twx) {
    dep_launch();
    dep_wait();
    using C = typename Cplx<Real>::type;
    extern __shared__ unsigned char smem_raw[];
    __shared__ double scratch_d[32];
    const int nx = NX > 0 ? NX : g.nx, nxh = nx / 2 + 1, pitch = x_pitch<NX>(nx), S = sp.S;
    const QRow<NX> qx(nx);
    const QHalf<NX> qh(nxh);
    const bool even = (nx % 2) == 0;
    const int lines = nl * LR;
    C* tw = align_ptr<C>(smem_raw);
    C* A = tw + nx;
    C* B = A + lines * pitch;
    const long long nrows = (long long)g.ny * g.nz;
    const long long row0 = (long long)blockIdx.x * LR;
    // A confined species is excluded from most rows, whose sums are zero: only blocks with a point
    // accessible to one transform theirs (pore at 256^3, eight ions in a hundredth of a per cent of
    // the box: 215 us without this, 33 with, most of it reading V).
    {
        const int pts = (int)(nrows - row0 < LR ? nrows - row0 : LR) * nx;
        bool open = false;
        for (int s = 0; s < S; ++s) {
            if (!sp.canon[s]) continue;
            const Real* v = V + (long long)s * g.n + row0 * nx;
            using VT = typename std::conditional<(NX > 0), Vec16<Real>, Vec1<Real>>::type;
            constexpr int VW = VT::n, KB = 4;       // KB loads in flight per thread
            for (int i0 = threadIdx.x * VW; i0 < pts; i0 += KB * kThreads * VW) {
                typename VT::type x[KB];
#pragma unroll
                for (int u = 0; u < KB; ++u) {
                    const int i = i0 + u * kThreads * VW;
                    x[u] = VT::load(v + (i < pts ? i : i0));
                }
#pragma unroll
                for (int u = 0; u < KB; ++u)
#pragma unroll
                    for (int e = 0; e < VW; ++e) open = open || !(vel(x[u], e) == Real(CUDART_INF));
            }
        }
        if (!__syncthreads_or(open)) {
            if (threadIdx.x < S && sp.canon[threadIdx.x]) red[(long long)blockIdx.x * DFT_MAXS + threadIdx.x] = 0.0;
            return;
        }
    }
    for (int i = threadIdx.x; i < nx; i += blockDim.x) tw[i] = twx[i];
    const int line_of[3] = {line0, line1, line2};
    const FastDiv ql(nl);
    for (int idx = threadIdx.x; idx < lines * nxh; idx += blockDim.x) {
        const int l = qh(idx), k = idx - l * nxh;
        const int r = ql.div(l), j = l - r * nl;
        const long long row = row0 + r;
        const int ca = 2 * line_of[j], cb = ca + 1;
        C a = cmake<C>(Real(0), Real(0)), b = a;
        if (row < nrows) {
            a = cspec[(long long)ca * g.nc + row * g.pxh + k];
            if (cb < S) b = cspec[(long long)cb * g.nc + row * g.pxh + k];
        }
        const bool edge = k == 0 || (even && 2 * k == nx);
        if (edge) { a.y = Real(0); b.y = Real(0); }
        A[l * pitch + xo<NX>(k)] = cmake<C>(a.x - b.y, a.y + b.x);
        if (!edge) A[l * pitch + xo<NX>(nx - k)] = cmake<C>(a.x + b.y, b.x - a.y);
    }
    __syncthreads();
    C* R = any_fft<NX, true>(A, B, px, lines, pitch, tw);
    Real acc[DFT_MAXS], comp[DFT_MAXS];
#pragma unroll
    for (int s = 0; s < DFT_MAXS; ++s) acc[s] = comp[s] = Real(0);
    for (int idx = threadIdx.x; idx < LR * nx; idx += blockDim.x) {
        const int r = qx(idx), x = idx - r * nx;
        const long long row = row0 + r;
        if (row >= nrows) continue;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            if (j >= nl) continue;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int s = 2 * line_of[j] + h;
                if (s >= S || !sp.canon[s]) continue;
                const C pr = R[(r * nl + j) * pitch + xo<NX>(x)];
                const Real c = h ? pr.y : pr.x;
                const Real v = V[(long long)s * g.n + row * nx + x];
                const Real e = (isinf(v) && v > Real(0)) ? Real(0) : exp(-v + c);
#pragma unroll
                for (int q = 0; q < DFT_MAXS; ++q) {
                    if (q != s) continue;
                    const Real y = e - comp[q];
                    const Real t = acc[q] + y;
                    comp[q] = (t - acc[q]) - y;
                    acc[q] = t;
                }
            }
        }
    }
#pragma unroll
    for (int s = 0; s < DFT_MAXS; ++s) {
        if (s >= S || !sp.canon[s]) continue;      // uniform across the block
        double bs;
        if constexpr (sizeof(Real) == 4) bs = block_sum_ds(acc[s], -comp[s], scratch_d);
        else bs = block_sum(double(acc[s]) - double(comp[s]), scratch_d);
        if (threadIdx.x == 0) red[(long long)blockIdx.x * DFT_MAXS + s] = bs;
    }
}

// canon_scale_i = (N_i / h^3) / sum over blocks of the k_xcanon partial sums (one block, four loads
// in flight per thread: 256^3 21 -> 9 us).
template <typename Real>
__global__ void __launch_bounds__(kFinThreads) k_canon_scale(Ctl* ctl, SpeciesDesc<Real> sp, const double* __restrict__ red,
                                                             int nblocks) {
    dep_launch();
    dep_wait();
    __shared__ double scratch_d[32];
    for (int s = 0; s < sp.S; ++s) {
        if (!sp.canon[s]) continue;
        double t[4] = {0.0, 0.0, 0.0, 0.0};
        for (int b = threadIdx.x; b < nblocks; b += 4 * kFinThreads) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int q = b + u * kFinThreads;
                if (q < nblocks) t[u] += red[(long long)q * DFT_MAXS + s];
            }
        }
        const double tot = block_sum((t[0] + t[1]) + (t[2] + t[3]), scratch_d);
        if (threadIdx.x == 0) {
            ctl->canon_scale[s] = sp.nfix_dv[s] / tot;
            if (!(tot > 0.0) || !isfinite(tot)) ctl->status |= DEV_NONFINITE;
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------------------------------
// Final x pass: one-body correlations c_i (half spectra) -> real space -> Picard map
//   G_i = rho_bath_i exp(beta mu_HS_bath_i - V_i + c_i)   (0 where V_i = +inf)
// at rho = w0 rho0 + w1 rho1, with the residual sum_i sum_x ((rho_i - G_i)/rho_bath_i)^2
// accumulated in FP64.  grid: ceil(ny nz / LR); ceil(S/2) lines per row.
// rho_out may alias rho0 and g_out may alias rho1 (each point is read before it is written).
// ------------------------------------------------------------------------------------
// NM = 2: the two line-search samples at once -- the c spectra of sample m at cspec (m = 0) and
// cspec2 (m = 1), weights from ctl[1 + m], rho0, rho1, V (and the low part) read once for both;
// the residual sums of sample m go to red_sum / red_sum2; nothing is written to rho or G.
template <typename Real, int NX, int NM = 1>
__global__ void __launch_bounds__(kThreads, NX < 0 ? 1 : (sizeof(Real) == 4 ? 3 : 2)) k_xupdate(GridDesc g, AxisPlan px, SpeciesDesc<Real> sp, int LR,
                                                      const Ctl* __restrict__ ctl,
                                                      const typename Cplx<Real>::type* __restrict__ cspec,
                                                      const typename Cplx<Real>::type* __restrict__ cspec2,
                                                      const Real* rho0, const Real* rho1,
                                                      const Real* __restrict__ V, Real* rho_out, Real* g_out,
                                                      typename Cplx<Real>::type* __restrict__ gspec_out,
                                                      Real* rho_lo, double* __restrict__ red_sum,
                                                      double* __restrict__ red_sum2, int* __restrict__ status,
                                                      const typename Cplx<Real>::type* __restrict__ twx) {
    dep_launch();
    dep_wait();
    using C = typename Cplx<Real>::type;
    extern __shared__ unsigned char smem_raw[];
    __shared__ double scratch_d[32];
    const int nx = NX > 0 ? NX : g.nx, pitch = x_pitch<NX>(nx), S = sp.S;
    const QRow<NX> qx(nx);
    const int lpr = (S + 1) / 2;
    const int lines = NM * lpr * LR;
    C* tw = align_ptr<C>(smem_raw);
    C* A = tw + nx;
    C* B = A + lines * pitch;
    for (int i = threadIdx.x; i < nx; i += blockDim.x) tw[i] = twx[i];
    const long long nrows = (long long)g.ny * g.nz;
    const long long row0 = (long long)blockIdx.x * LR;
    load_species_rows<Real, NX, NM>(g, LR, row0, nrows, S, cspec, cspec2, A);
    const int total = LR * nx;
    // G_i = pref_i exp(mu0_i - V_i + c_i): the bath (rho_b, beta mu_HS,b), or for a
    // fixed-number species the normalisation of this evaluation and no bath constant
    __shared__ Real s_pref[DFT_MAXS], s_mu0[DFT_MAXS], s_irb[DFT_MAXS];
    if (threadIdx.x < DFT_MAXS) {
        const int s = threadIdx.x;
        const bool cn = s < S && sp.canon[s];
        s_pref[s] = cn ? Real(ctl->canon_scale[s]) : sp.rho_b[s];
        s_mu0[s] = cn ? Real(0) : sp.mu_hs_b[s];
        s_irb[s] = sp.inv_rho_b[s];
    }
    __syncthreads();
    C* R = any_fft<NX, true>(A, B, px, lines, pitch, tw);
    Real w0[NM], w1[NM];
#pragma unroll
    for (int m = 0; m < NM; ++m) {
        const Ctl* cw = NM == 1 ? ctl : ctl + 1 + m;
        w0[m] = CtlW<Real>::w0(cw);
        w1[m] = CtlW<Real>::w1(cw);
    }
    // per-thread partial sums in the working precision with Kahan compensation, then
    // double-single (FP32) or FP64 across threads, FP64 across blocks
    Real acc[NM], comp[NM];
#pragma unroll
    for (int m = 0; m < NM; ++m) acc[m] = comp[m] = Real(0);
    bool bad = false;
    // one point of species s under mixture m: new iterate (and its low part), G, squared
    // weighted residual
    auto point = [&](int m, int s, Real c, Real r0, Real r1, Real v, Real l0, Real& rho, Real& lo, Real& gval) {
        lo = Real(0);
        if (rho_lo) {
            // extended iterate rho0 = r0 + l0 (a value and its rounding error):
            // rho = rho0 + w1 (rho1 - rho0) formed so that steps below half an ulp of rho0
            // accumulate in the low part instead of rounding away (w0 = 1 - w1), then split
            // again into rho + lo by an error-free sum (Knuth's TwoSum)
            const Real t = l0 + w1[m] * ((r1 - r0) - l0);
            rho = r0 + t;
            const Real bv = rho - r0;
            lo = (r0 - (rho - bv)) + (t - bv);
        } else {
            rho = w0[m] * r0 + w1[m] * r1;
        }
        if (isinf(v) && v > Real(0)) gval = Real(0);
        else gval = s_pref[s] * exp(s_mu0[s] - v + c);
        if (!isfinite(gval) || !isfinite(rho)) bad = true;
        const Real d = ((rho - gval) + lo) * s_irb[s];
        const Real y = d * d - comp[m];
        const Real t = acc[m] + y;
        comp[m] = (t - acc[m]) - y;
        acc[m] = t;
    };
    // rho_out / g_out / rho_lo may alias rho0 / rho1 / the low part read: every value is read
    // before the same thread writes that element, and the threads' elements are distinct
    // items (species, group of VW consecutive points of the block's rows), KB items per thread with
    // their loads of rho0, rho1, V (and the low part) issued before any is used: 16-byte accesses
    // for compile-time lengths (KB 2 measured 144 us per 128^3 iteration against 133), single values
    // for run-time ones, whose rows need not start on a 16-byte boundary
    {
        using VT = typename std::conditional<(NX > 0), Vec16<Real>, Vec1<Real>>::type;
        using V16 = typename VT::type;
        constexpr int VW = VT::n;
        constexpr int KB = NX > 0 ? DFT_XUPD_BATCH : 4;
        static_assert(NX <= 0 || NX % VW == 0, "row length a multiple of the vector width");
        const int groups = total / VW;
        const int items = S * groups;
        // item it = s groups + gi, kept as (s, gi) and advanced without dividing
        int s_b = threadIdx.x / groups, gi_b = threadIdx.x - s_b * groups;
        for (int base = threadIdx.x; base < items; base += KB * kThreads) {
            V16 a0[KB], a1[KB], av[KB], al[KB];
            int sj[KB], gj[KB];
#pragma unroll
            for (int j = 0; j < KB; ++j) {
                if (j == 0) { sj[0] = s_b; gj[0] = gi_b; }
                else {
                    sj[j] = sj[j - 1];
                    gj[j] = gj[j - 1] + kThreads;
                    while (gj[j] >= groups) { gj[j] -= groups; ++sj[j]; }
                }
                const int it = base + j * kThreads;
                const int s = sj[j], gi = gj[j];
                const bool live = it < items && row0 + qx(gi * VW) < nrows;
                const long long o = (long long)s * g.n + row0 * nx + (long long)gi * VW;
                a0[j] = a1[j] = av[j] = al[j] = vzero<V16>();
                if (live) {
                    a0[j] = VT::load(rho0 + o);
                    if (rho1) a1[j] = VT::load(rho1 + o);
                    av[j] = VT::load(V + o);
                    if (rho_lo) al[j] = VT::load(rho_lo + o);
                }
            }
            gi_b += KB * kThreads;
            while (gi_b >= groups) { gi_b -= groups; ++s_b; }
#pragma unroll
            for (int j = 0; j < KB; ++j) {
                const int it = base + j * kThreads;
                const int s = sj[j], gi = gj[j];
                const int idx = gi * VW, r = qx(idx), x = idx - r * nx;
                if (!(it < items && row0 + r < nrows)) continue;
                const long long o = (long long)s * g.n + row0 * nx + idx;
#pragma unroll
                for (int m = 0; m < NM; ++m) {
                    C* Rl = R + (m * lpr * LR + r * lpr + s / 2) * pitch;
                    V16 orho, og, olo;
#pragma unroll
                    for (int e = 0; e < VW; ++e) {
                        // this species' half of the line (the other species of the line is another
                        // item's); with gspec_out, G goes back into the same half
                        Real* hp = reinterpret_cast<Real*>(Rl + xo<NX>(x + e)) + (s & 1);
                        point(m, s, *hp, vel(a0[j], e), vel(a1[j], e), vel(av[j], e), vel(al[j], e), vel(orho, e),
                              vel(olo, e), vel(og, e));
                        if (NM == 1 && gspec_out) *hp = vel(og, e);
                    }
                    if (NM == 1 && rho_out) {
                        VT::store(rho_out + o, orho);
                        if (rho_lo) VT::store(rho_lo + o, olo);
                    }
                    if (NM == 1 && g_out) VT::store(g_out + o, og);
                }
            }
        }
    }
    if (bad) atomicOr(status, DEV_NONFINITE);
    if (NM == 1 && gspec_out) {
        // the x half spectra of the G rows just formed (the next first half's input): the lines
        // now hold G in place of c1, two species per complex line
        __syncthreads();
        C* other = (R == A) ? B : A;
        C* F = any_fft<NX, false>(R, other, px, lines, pitch, tw);
        store_pair_rows<Real, NX>(g, lines, lpr, row0, nrows, S, F, gspec_out);
    }
#pragma unroll
    for (int m = 0; m < NM; ++m) {
        double bs;
        if constexpr (sizeof(Real) == 4) bs = block_sum_ds(acc[m], -comp[m], scratch_d);
        else bs = block_sum(double(acc[m]) - double(comp[m]), scratch_d);
        if (threadIdx.x == 0) (m == 0 ? red_sum : red_sum2)[blockIdx.x] = bs;
    }
}

// ------------------------------------------------------------------------------------
// Gradient pass: x inverse of the one-body correlations c_i, then at each point
//   dOmega/drho_i = h^3 [ln(rho_i / rho_bath_i) + V_i - beta mu_HS_bath_i - c_i]   (accessible, rho > 0)
//   dOmega/dV_i   = h^3 rho_i
// and per-block sums red[b (S + 1) + 0] = sum_i sum_x [rho_i (ln(rho_i/rho_bath_i) - 1) + rho_i (V_i -
// beta mu_ex_bath_i)] (accessible points), red[b (S + 1) + 1 + i] = sum_x rho_i, all in FP64.  In FP32
// plans too, where the logarithm and products per point and species bound the pass on the FP64 pipe (64^3, two
// species: 52 us).
// ------------------------------------------------------------------------------------
template <typename Real, int NX>
__global__ void __launch_bounds__(kThreads) k_xgrad(GridDesc g, AxisPlan px, SpeciesDesc<Real> sp, int LR, Real dv,
                                                    const typename Cplx<Real>::type* __restrict__ cspec,
                                                    const Real* __restrict__ rho, const Real* __restrict__ V,
                                                    Real* __restrict__ grad_rho, Real* __restrict__ grad_V,
                                                    double* __restrict__ red,
                                                    const typename Cplx<Real>::type* __restrict__ twx) {
    dep_launch();
    dep_wait();
    using C = typename Cplx<Real>::type;
    extern __shared__ unsigned char smem_raw[];
    __shared__ double scratch_d[32];
    const int nx = NX > 0 ? NX : g.nx, pitch = x_pitch<NX>(nx), S = sp.S;
    const QRow<NX> qx(nx);
    const int lpr = (S + 1) / 2;
    const int lines = lpr * LR;
    C* tw = align_ptr<C>(smem_raw);
    C* A = tw + nx;
    C* B = A + lines * pitch;
    for (int i = threadIdx.x; i < nx; i += blockDim.x) tw[i] = twx[i];
    const long long nrows = (long long)g.ny * g.nz;
    const long long row0 = (long long)blockIdx.x * LR;
    load_pair_rows<Real, NX>(g, lines, lpr, row0, nrows, S, cspec, nullptr, Real(1), Real(0), nullptr, A);
    __syncthreads();
    C* R = any_fft<NX, true>(A, B, px, lines, pitch, tw);
    double ideal = 0.0, num[DFT_MAXS];
#pragma unroll
    for (int s = 0; s < DFT_MAXS; ++s) num[s] = 0.0;
    for (int idx = threadIdx.x; idx < LR * nx; idx += blockDim.x) {
        const int r = qx(idx), x = idx - r * nx;
        const long long row = row0 + r;
        if (row >= nrows) continue;
#pragma unroll
        for (int s = 0; s < DFT_MAXS; ++s) {
            if (s >= S) break;
            const C pr = R[(r * lpr + s / 2) * pitch + xo<NX>(x)];
            const Real c = (s & 1) ? pr.y : pr.x;
            const long long o = (long long)s * g.n + row * nx + x;
            const Real rv = rho[o];
            const Real v = V[o];
            const bool acc_ok = !(isinf(v) && v > Real(0)) && rv > Real(0);
            Real gr = Real(0);
            if (acc_ok) {
                const double lr = log(double(rv) * double(sp.inv_rho_b[s]));
                gr = Real(dv * (lr + double(v) - double(sp.mu_hs_b[s]) - double(c)));
                ideal += double(rv) * (lr - 1.0) + double(rv) * (double(v) - double(sp.mu_ex_b[s]));
            }
            num[s] += double(rv);
            if (grad_rho) grad_rho[o] = gr;
            if (grad_V) grad_V[o] = dv * rv;
        }
    }
#pragma unroll
    for (int s = -1; s < DFT_MAXS; ++s) {
        if (s >= S) break;
        const double b = block_sum(s < 0 ? ideal : num[s < 0 ? 0 : s], scratch_d);
        if (threadIdx.x == 0) red[(long long)blockIdx.x * (S + 1) + 1 + s] = b;
    }
}

// ------------------------------------------------------------------------------------
// Plain x inverse of ncomp half spectra to real fields, out[c] = value + offset[c].
// Optional max of component cmax into red_max.  grid: ceil(ny nz / LR).
// ------------------------------------------------------------------------------------
template <typename Real, int NX>
__global__ void __launch_bounds__(kThreads) k_xinv(GridDesc g, AxisPlan px, int LR, int ncomp,
                                                   const typename Cplx<Real>::type* __restrict__ spec,
                                                   Real* __restrict__ out, Real* __restrict__ out_last,
                                                   Offsets<Real> off, int cmax,
                                                   float* __restrict__ red_max, int wd, Real kfx,
                                                   const typename Cplx<Real>::type* __restrict__ twx) {
    dep_launch();
    dep_wait();
    using C = typename Cplx<Real>::type;
    extern __shared__ unsigned char smem_raw[];
    __shared__ float scratch_f[32];
    const int nx = NX > 0 ? NX : g.nx, pitch = x_pitch<NX>(nx);
    const QRow<NX> qx(nx);
    // one component without outputs (the maximum only): two grid rows per complex line
    const bool rows2 = ncomp == 1 && !wd && !out && !out_last;
    const int lpr = (ncomp + 1) / 2;
    const int lines = rows2 ? (LR + 1) / 2 : lpr * LR;
    C* tw = align_ptr<C>(smem_raw);
    C* A = tw + nx;
    C* B = A + lines * pitch;
    for (int i = threadIdx.x; i < nx; i += blockDim.x) tw[i] = twx[i];
    const long long nrows = (long long)g.ny * g.nz;
    const long long row0 = (long long)blockIdx.x * LR;
    const Real one = Real(1), zero = Real(0);
    if (wd) load_wd_rows<Real, NX>(g, LR, row0, nrows, spec, nullptr, &one, &zero, nullptr, kfx, A);
    else if (rows2) load_row_pairs<Real, NX>(g, LR, row0, nrows, spec, A);
    else load_pair_rows<Real, NX>(g, lines, lpr, row0, nrows, ncomp, spec, nullptr, Real(1), Real(0), nullptr, A);
    __syncthreads();
    C* R = any_fft<NX, true>(A, B, px, lines, pitch, tw);
    float mx = -CUDART_INF_F;
    for (int idx = threadIdx.x; idx < LR * nx; idx += blockDim.x) {
        const int r = qx(idx), x = idx - r * nx;
        const long long row = row0 + r;
        if (row >= nrows) continue;
        if (rows2) {
            const C pr = R[(r / 2) * pitch + xo<NX>(x)];
            mx = fmaxf(mx, float(((r & 1) ? pr.y : pr.x) + off.v[0]));
            continue;
        }
        for (int c = 0; c < ncomp; ++c) {
            const int l = wd ? wd_line(c) : c / 2, j = wd ? wd_slot(c) : (c & 1);
            const C pr = R[(r * lpr + l) * pitch + xo<NX>(x)];
            const Real v = (j ? pr.y : pr.x) + off.v[c];
            if (out_last && c == ncomp - 1) out_last[row * nx + x] = v;
            else if (out) out[(long long)c * g.n + row * nx + x] = v;
            if (c == cmax) mx = fmaxf(mx, float(v));
        }
    }
    if (red_max) {
        const float bm = block_max(mx, scratch_f);
        if (threadIdx.x == 0) red_max[blockIdx.x] = bm;
    }
}

#ifdef DFT_DEFINE_FINALIZE
// ------------------------------------------------------------------------------------
// Line-search bookkeeping on the device (Sec. "Nonlinear solver"), one block.
// ------------------------------------------------------------------------------------
__device__ __forceinline__ void set_weights(Ctl* c, double a) {
    c->wA = 1.0 - a; c->wB = a; c->w0 = 1.0 - a; c->w1 = a;
    c->wAf = float(c->wA); c->wBf = float(c->wB); c->w0f = float(c->w0); c->w1f = float(c->w1);
}

// Start of an evaluation: the status words of the three control blocks cleared and the weights of a
// plain G evaluation (1, 0) set.  One launch of 1.5 us where three memsets and a bookkeeping kernel
// took eight between the passes of a small grid.
__global__ void k_ctl_reset(Ctl* ctl) {
    dep_launch();
    dep_wait();
    if (threadIdx.x < 3) ctl[threadIdx.x].status = 0;
    if (threadIdx.x == 0) {
        set_weights(ctl, 0.0);
        ctl->alpha = 0.5;   // no previous step: the first sampled interval is alpha_max (<= 1 = 2 * 0.5)
    }
}

// ctl points at three control blocks: the iteration's, then the weights of the two line-search
// samples (ctl[1], ctl[2]: wA, wB, w0, w1 only), which FIN_AMAX sets for the paired evaluation.
template <int B>
__device__ __forceinline__ double partial_sum(const double* __restrict__ red_sum, int nsum) {
    // four independent partial results per thread, so that a thread's loads are all in flight
    // at once (the partial sums are L2-resident: the kernel is a few load latencies long)
    double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
    int i = threadIdx.x;
    for (; i + 3 * B < nsum; i += 4 * B) {
        s0 += red_sum[i];
        s1 += red_sum[i + B];
        s2 += red_sum[i + 2 * B];
        s3 += red_sum[i + 3 * B];
    }
    for (; i < nsum; i += B) s0 += red_sum[i];
    return (s0 + s1) + (s2 + s3);
}

template <int B>
__global__ void __launch_bounds__(B) k_finalize(Ctl* ctl, const double* __restrict__ red_sum,
                                                          const double* __restrict__ red_sum2, int nsum,
                                                          const float* __restrict__ red_max, int nmax, int op,
                                                          double inv_count, double alpha_fixed, double n3_bound,
                                                          double alpha_floor) {
    dep_launch();
    dep_wait();
    __shared__ double scratch_d[64];
    __shared__ float scratch_f[32];
    double s = partial_sum<B>(red_sum, nsum);
    double s_2 = red_sum2 ? partial_sum<B>(red_sum2, nsum) : 0.0;
    float m0 = -CUDART_INF_F, m1 = -CUDART_INF_F, m2 = -CUDART_INF_F, m3 = -CUDART_INF_F;
    int i = threadIdx.x;
    for (; i + 3 * B < nmax; i += 4 * B) {
        m0 = fmaxf(m0, red_max[i]);
        m1 = fmaxf(m1, red_max[i + B]);
        m2 = fmaxf(m2, red_max[i + 2 * B]);
        m3 = fmaxf(m3, red_max[i + 3 * B]);
    }
    for (; i < nmax; i += B) m0 = fmaxf(m0, red_max[i]);
    float m = fmaxf(fmaxf(m0, m1), fmaxf(m2, m3));
    // the two sums and the maximum through one pair of barriers (the same order of operations
    // per quantity as block_sum / block_max)
    for (int o = 16; o > 0; o >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, o);
        s_2 += __shfl_xor_sync(0xffffffffu, s_2, o);
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    }
    {
        const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
        if (l == 0) { scratch_d[w] = s; scratch_d[32 + w] = s_2; scratch_f[w] = m; }
        __syncthreads();
        if (threadIdx.x >= 32) return;
        const bool in = l < B / 32;
        s = in ? scratch_d[l] : 0.0;
        s_2 = in ? scratch_d[32 + l] : 0.0;
        m = in ? scratch_f[l] : -CUDART_INF_F;
        for (int o = 16; o > 0; o >>= 1) {
            s += __shfl_xor_sync(0xffffffffu, s, o);
            s_2 += __shfl_xor_sync(0xffffffffu, s_2, o);
            m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        }
    }
    const double tot = s, tot2 = s_2;
    const float mx = m;
    if (threadIdx.x != 0) return;
    Ctl* c = ctl;
    const double f = tot * inv_count;
    if (op & FIN_F0) {
        c->f[0] = f;
        c->resid = sqrt(f);
        if (!isfinite(f)) c->status |= DEV_NONFINITE;
    }
    if (op & FIN_N3CUR) c->n3max_cur = mx;
    if (op & FIN_AMAX) {
        c->n3max_next = mx;
        c->resid_prev = c->resid;
        const double m0 = c->n3max_cur, m1 = mx;
        double am = 1.0;
        if (m1 > m0) am = fmin(1.0, (n3_bound - m0) / (m1 - m0));
        c->alpha_max = am;
        c->alpha_fixed = alpha_fixed;
        if (alpha_fixed >= 0.0) {
            const double a = fmin(alpha_fixed, am);
            c->alpha = a;
            set_weights(c, a);
        } else {
            const double as = fmin(am, 2.0 * c->alpha);
            c->alpha_s = as;
            c->sample_alpha[0] = 0.5 * as;
            c->sample_alpha[1] = as;
            set_weights(c, 0.5 * as);
            set_weights(c + 1, 0.5 * as);
            set_weights(c + 2, as);
        }
    }
    if (op & FIN_F1) {
        c->f[1] = f;
        c->sample_alpha[1] = c->alpha_s;
        set_weights(c, c->alpha_s);
    }
    if (op & (FIN_F2_CHOOSE | FIN_F12_CHOOSE)) {
        // FIN_F12_CHOOSE: both samples' sums at once (f1 in red_sum, f2 in red_sum2); the z
        // passes of the samples recorded their status in the samples' blocks
        if (op & FIN_F12_CHOOSE) {
            c->f[1] = f;
            c->status |= c[1].status | c[2].status;
            c[1].status = 0;
            c[2].status = 0;
        }
        c->f[2] = (op & FIN_F12_CHOOSE) ? tot2 * inv_count : f;
        const double am = c->alpha_s, a = 0.5 * am;
        const double f0 = c->f[0], f1 = c->f[1], f2 = c->f[2];
        const double c2 = (f0 - 2.0 * f1 + f2) / (2.0 * a * a);
        const double c1 = (-3.0 * f0 + 4.0 * f1 - f2) / (2.0 * a);
        double al;
        if (c2 > 0.0) al = fmin(fmax(-c1 / (2.0 * c2), alpha_floor * am), am);
        else al = (f1 <= f2) ? a : am;
        c->alpha = al;
        set_weights(c, al);
    }
    if (op & FIN_ACCEPT) {
        c->f[3] = f;
        c->f[0] = f;
        c->resid = sqrt(f);
        c->n3max_cur = mx;
        c->iter += 1;
        if (!isfinite(f)) c->status |= DEV_NONFINITE;
    }
}

#endif  // DFT_DEFINE_FINALIZE

}  // namespace dftk
