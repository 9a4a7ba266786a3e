// Shared definitions of the GB300 classical-DFT kernels: complex arithmetic,
// per-axis FFT plans, grid / species descriptors and the device control block.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

#include "gb300dft.h"

#define DFT_MAXS 5          // species (the back-convolution keeps 5 k-space accumulators)
#define DFT_MAXSTAGES 8     // radix stages per axis
#define DFT_NCOMP 10        // n0 n1 n2 n3 nV1(xyz) nV2(xyz)
// Weighted-density spectra kept between the passes: n0 n1 n2 n3, m (n_V1 = grad m), then
// i k_y m, i k_z m, i k_y n3, i k_z n3.  The x components i k_x m and i k_x n3 are formed in
// the x pass that takes the spectra to real space (and the divergence terms of the back
// convolution in the x pass that leaves it), so the y passes carry nine components.
#define DFT_NSPEC 9
// Of these the z passes carry seven: i k_y m and i k_y n3 (and on the way back the -i k_y terms) are
// formed in the y pass, whose tiles hold all k_y.  Component of the q-th of them:
#define DFT_NZSPEC 7
__host__ __device__ constexpr int dft_zcomp(int q) { return q < 5 ? q : 2 * q - 4; }
// Modes of the column passes (k_yfft_tma, k_colfft)
enum { COL_PLAIN = 0, COL_WD = 1, COL_DERIV = 2, COL_FOLD = 3 };
// Polls of a TMA tile wait before it gives up (the plans' default; dft_set_wait_polls)
#define DFT_WAIT_POLLS (1LL << 24)

template <typename Real> struct Cplx;
template <> struct Cplx<float> { using type = float2; };
template <> struct Cplx<double> { using type = double2; };

template <typename C> __host__ __device__ __forceinline__ C cmake(decltype(C().x) re, decltype(C().x) im) {
    C c; c.x = re; c.y = im; return c;
}
template <typename C> __device__ __forceinline__ C cadd(C a, C b) { return cmake<C>(a.x + b.x, a.y + b.y); }
template <typename C> __device__ __forceinline__ C csub(C a, C b) { return cmake<C>(a.x - b.x, a.y - b.y); }
template <typename C> __device__ __forceinline__ C cmul(C a, C b) {
    return cmake<C>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
template <typename C> __device__ __forceinline__ C cscale(C a, decltype(C().x) s) { return cmake<C>(a.x * s, a.y * s); }
template <typename C> __device__ __forceinline__ C cconj(C a) { return cmake<C>(a.x, -a.y); }
// multiply by +i or -i
template <typename C> __device__ __forceinline__ C cmul_i(C a) { return cmake<C>(-a.y, a.x); }
template <typename C> __device__ __forceinline__ C cmul_mi(C a) { return cmake<C>(a.y, -a.x); }

// Division by a positive run-time constant d: floor(x / d) = hi32(x ceil(2^32 / d)) for
// 0 <= x with x d < 2^32 (the tasks and items of one block: both factors below 2^16).
struct FastDiv {
    unsigned mul;   // 0 for d = 1
    int d;
    FastDiv() = default;
    __host__ __device__ explicit FastDiv(int dd) : mul(dd > 1 ? 0xffffffffu / (unsigned)dd + 1u : 0u), d(dd) {}
    __device__ __forceinline__ int div(int x) const { return mul ? (int)__umulhi((unsigned)x, mul) : x; }
};

// Radix decomposition of one axis length: n = prod radix[s]; the radices of dft_small and the
// primes up to DFT_MAX_PRIME (run-time transforms only; see dft_radix_plan, dft_mixed_plan).
// Stage s: ns = product of the earlier radices, m = n / radix butterflies per line, twiddle step
// n / (ns radix).
struct AxisPlan {
    int n;
    int nstages;
    int radix[DFT_MAXSTAGES];
    int m[DFT_MAXSTAGES];
    int tws[DFT_MAXSTAGES];
    FastDiv ns[DFT_MAXSTAGES];
    FastDiv dm[DFT_MAXSTAGES];      // division by m
};

// Fill the per-stage constants from n and the radices.
inline void dft_finish_plan(AxisPlan* p) {
    int ns = 1;
    for (int s = 0; s < p->nstages; ++s) {
        p->m[s] = p->n / p->radix[s];
        p->tws[s] = p->n / (ns * p->radix[s]);
        p->ns[s] = FastDiv(ns);
        p->dm[s] = FastDiv(p->m[s]);
        ns *= p->radix[s];
    }
}

// Largest prime factor an axis length may have.  Factors 11..31 take a stage of their own
// (rt_stage_prime); lengths with one of 17..31 ("big" primes) run kernels compiled for them.
#define DFT_MAX_PRIME 31
inline bool dft_has_big_prime(int n) {
    for (int p : {17, 19, 23, 29, 31})
        if (n % p == 0) return true;
    return false;
}

// Radix plan of an axis length: the 3s, then the other odd primes up to DFT_MAX_PRIME, then
// 16s and one of 2 / 4 / 8.  False if n has a larger prime factor or needs more than
// DFT_MAXSTAGES stages.
inline bool dft_radix_plan(int n, AxisPlan* out) {
    out->n = n;
    out->nstages = 0;
    int m = n;
    auto push = [&](int r) {
        if (out->nstages >= DFT_MAXSTAGES) return false;
        out->radix[out->nstages++] = r;
        return true;
    };
    while (m % 3 == 0) { if (!push(3)) return false; m /= 3; }
    for (int p = 5; p <= DFT_MAX_PRIME; p += 2)
        while (m % p == 0) { if (!push(p)) return false; m /= p; }
    while (m >= 16 && m % 16 == 0) { if (!push(16)) return false; m /= 16; }
    if (m == 2 || m == 4 || m == 8) { if (!push(m)) return false; m = 1; }
    dft_finish_plan(out);
    return m == 1 && out->nstages > 0;
}

// Radix plan of the run-time transforms: the factorisation into the radices 2..10, 12, 14, 15, 16
// and the primes 11..31 with the least estimated work, larger radices first (a first stage takes
// no twiddles).  A stage of radix R costs its threads R (memory and index work + flops of an
// R-point DFT, per element) for every wave of a block's 256 threads over the m T butterflies of a
// 16-column tile, averaged with the same without the rounding to whole waves (other tiles of the
// SM fill it), and a barrier.  Two stages of near-equal radices win for most lengths (160 =
// 16 x 10, 120 = 12 x 10, 84 = 12 x 7), three above 256.
// At most DFT_RT_STAGES of them: k_colfft's buffers rotate over three stages, and every length up to 512 with
// prime factors up to 31 has such a plan.
#define DFT_RT_STAGES 3
inline bool dft_mixed_plan(int n, AxisPlan* out) {
    static const struct { int r; double flops; } kR[] = {
        {31, 55}, {29, 52}, {23, 44}, {19, 39}, {17, 36}, {13, 27}, {11, 24}, {16, 10.5}, {15, 10}, {14, 11},
        {12, 7.5}, {10, 7.5}, {9, 8.5}, {8, 6.5}, {7, 9}, {6, 5}, {5, 6.5}, {4, 4}, {3, 4}, {2, 2}};
    AxisPlan cur{}, best{};
    double best_cost = 1e30;
    cur.n = n;
    auto search = [&](auto&& self, int rem, int from, double cost) -> void {
        if (cost >= best_cost) return;
        if (rem == 1) {
            best = cur;
            best_cost = cost;
            return;
        }
        if (cur.nstages == DFT_RT_STAGES) return;
        for (int i = from; i < int(sizeof(kR) / sizeof(kR[0])); ++i) {
            const int r = kR[i].r;
            if (rem % r) continue;
            const double waves = double(n / r) * 16.0 / 256.0;
            const double whole = double((n / r * 16 + 255) / 256);
            cur.radix[cur.nstages++] = r;
            self(self, rem / r, i, cost + 0.5 * (waves + whole) * r * (7.0 + kR[i].flops) + 40.0);
            --cur.nstages;
        }
    };
    search(search, n, 0, 0.0);
    if (best.nstages == 0) return false;
    *out = best;
    dft_finish_plan(out);
    return true;
}

// Axis lengths a plan accepts: 4 <= n <= 512 with a radix plan.
inline bool dft_valid_length(int n) {
    AxisPlan p;
    return n >= 4 && n <= 512 && dft_radix_plan(n, &p);
}

// Grid of one state point.  Real fields: [c][nz][ny][nx]; half spectra after the
// x transform: [c][nz][ny][pxh], of which kx < nxh = nx/2 + 1 are used; the row pitch
// pxh is nxh rounded up to even so that every row starts on a 16-byte boundary (a TMA
// requirement).
struct GridDesc {
    int nx, ny, nz, nxh, pxh;
    long long n;     // nx * ny * nz
    long long nc;    // nz * ny * pxh (elements per half-spectrum component)
    double hx, hy, hz;
    int phi;         // hard-sphere free-energy density of the state point (DFT_PHI_*; 0 = eq. Phi)
    // transform variants chosen by the autotuner (0 for all: the compile-time passes where a
    // length has them): x passes by the run-time kernels with the plan's AxisPlan; y passes by
    // the run-time column kernel; z passes by the one-tile-per-CTA grouped kernels instead of
    // the persistent TMA ones
    int xrt, yrt, zgrp;
    int xpers;       // the Phi' x passes as a persistent kernel: 1 bulk-copy prefetch, 2 cp.async prefetch
    int zsplit;      // the first-half z stage as three passes: z transform, k-space products, z transform
    int pdl;         // launch the passes with programmatic dependent launch (launch_k)
};

// Programmatic dependent launch.  With GridDesc::pdl set the passes are launched with the
// programmatic-stream-serialization attribute, so that the launch of one pass overlaps the
// completion of the previous one.  dep_wait() (griddepcontrol.wait) returns once every grid
// the kernel depends on has completed and its memory writes are visible; each pass calls it
// before its first access to memory an earlier kernel may write (for a kernel launched without
// the attribute it returns at once).  dep_launch() (griddepcontrol.launch_dependents) lets the
// next kernel be scheduled once every CTA of this one has issued it or exited.
__device__ __forceinline__ void dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Where a pass lets the next one be scheduled (build flag): 0 (default) = never, the next pass
// is scheduled as this one's CTAs exit (its launch still overlaps this one's completion); 1 = at
// its start.  Measured on the 128^3 iteration: 0 runs 0.5 % faster than plain stream order, 1
// 13 % slower (the next pass's waiting CTAs become resident beside the persistent passes).
#ifndef DFT_DEP_TRIGGER
#define DFT_DEP_TRIGGER 0
#endif
__device__ __forceinline__ void dep_launch() {
#if DFT_DEP_TRIGGER
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
#endif
}

// Launch `kernel` on `st`, with the programmatic-serialization attribute when pdl != 0.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_k(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, int pdl,
                            Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// Species constants in the kernels' precision (host fills them in double, then converts).
template <typename Real>
struct SpeciesDesc {
    int S;
    Real R[DFT_MAXS];
    Real z[DFT_MAXS];
    Real rho_b[DFT_MAXS];
    Real inv_rho_b[DFT_MAXS];   // residual weights 1 / rho_bath
    Real mu_hs_b[DFT_MAXS];     // beta mu^{HS,bath}
    Real mu_ex_b[DFT_MAXS];     // beta mu^{ex,bath} = beta (mu^{HS,bath} + mu^{ES,bath})
    Real n_rho_b[DFT_MAXS];     // N * rho_bath: DFT of the bath density at k = 0
    // bulk-fluid kernel per pair (i, j), in kT units
    Real es_pref[DFT_MAXS][DFT_MAXS];   // lambda_B z_i z_j / 2
    Real es_a[DFT_MAXS][DFT_MAXS];      // 1 / (2 l_i l_j)
    Real es_b[DFT_MAXS][DFT_MAXS];      // (l_i + l_j) / (l_i l_j)
    Real es_c[DFT_MAXS][DFT_MAXS];      // (l_i - l_j)^2 / (2 l_i l_j) + 2
    Real es_R[DFT_MAXS][DFT_MAXS];      // R_ij = R_i + R_j
    Real pois[DFT_MAXS][DFT_MAXS];      // 4 pi lambda_B z_i z_j
    Real es_da[DFT_MAXS][DFT_MAXS];     // d es_a / d Gamma  (gradient with respect to the bath)
    Real es_db[DFT_MAXS][DFT_MAXS];     // d es_b / d Gamma
    Real es_dc[DFT_MAXS][DFT_MAXS];     // d es_c / d Gamma
    Real inv_n;                         // 1 / N
    int coulomb_limit;                  // Gamma == 0: kernel is lambda_B z_i z_j / r inside R_ij
    // Optional tables of the |k|-only factors: on a cubic box by the integer m2 = mx^2 + my^2 + mz^2
    // (|k| = kf sqrt(m2)), else (tab_oct) by (kx, |ky|, |kz|); null: the kernels evaluate them per
    // point.
    const Real* tab_w;                  // [row][tab_ws]: w0_s at 2 s, j3_s at 2 s + 1
    const Real* tab_k;                  // [row][tab_ks]: DC_ij_hat at j (j + 1) / 2 + i, i <= j
    const Real* tab_dk;                 // [row][tab_ks]: d DC_ij_hat / d Gamma, same order (or null)
    int tab_oct;
    int tab_ws, tab_ks;                 // record lengths: 2 S and S (S + 1) / 2 rounded up to 16 bytes
    // Optional per-axis terms of the discrete Laplacian, sin^2(k_d h_d / 2) / h_d^2 by FFT index:
    // x indices at 0, y at nx, z at nx + ny (k_laptab); null: the kernels evaluate them per point.
    const Real* lap1d;
    // Optional wave numbers by FFT index, same layout, zero on the Nyquist index (k_laptab); null:
    // evaluated per point.
    const Real* kax;
    Real r2[DFT_MAXS], a2[DFT_MAXS], v3[DFT_MAXS];   // R^2, 4 pi R^2, 4 pi R^3
    // fixed-number species (canonical form of eq. rhoEquation): canon[i] != 0, target sum of G_i
    // over the grid N_i / h^3; ncanon of them
    int canon[DFT_MAXS];
    double nfix_dv[DFT_MAXS];
    int ncanon;
};

// Index of the pair (i, j), i <= j, in a table record (independent of S).
__host__ __device__ constexpr int dft_pair(int i, int j) { return j * (j + 1) / 2 + i; }

// Register capacity of a table record (a multiple of 16 bytes of either precision).
#define DFT_TAB_W 12        // >= 2 DFT_MAXS
#define DFT_TAB_K 16        // >= DFT_MAXS (DFT_MAXS + 1) / 2

// Per-component additive constants of the plain x inverse.
template <typename Real> struct Offsets { Real v[DFT_NCOMP + 2]; };

// Device-resident control block of the Picard iteration.  Kernels read the mixing
// weights from here, so a whole iteration can be queued (or captured) without a
// host round trip.
struct Ctl {
    double wA, wB;          // weights of slot A / slot B weighted densities (XPHI, ZK2)
    double w0, w1;          // weights of rho^(0) / rho^(1) (XU)
    double f[4];            // squared residuals: f0 = r^2(rho0), f1, f2 samples, f3 = accepted point
    double alpha_max;       // n3 bound of the step
    double alpha_s;         // sampled interval min(alpha_max, 2 alpha_prev)
    double alpha;           // accepted alpha of the last step (alpha_prev of the next)
    double alpha_fixed;     // < 0: line search
    double n3max_cur;       // max n3 of the current iterate
    double n3max_next;      // max n3 of G(current)
    double resid;           // sqrt(f0)
    double resid_prev;      // r of the iterate a step started from
    double sample_alpha[2];
    int status;             // dft_status bits raised on the device (see DEV_* below)
    int iter;
    int loop_left;          // iterations left in an on-device loop of dft_iter_run / dft_batch_iterate
    // fixed-number species: G_i = canon_scale[i] exp(-V_i + c_i), canon_scale = N_i / (h^3 sum e)
    double canon_scale[DFT_MAXS];
    // the four weights rounded to float when they are set: the FP32 passes read these, since a
    // double-to-float conversion in every thread queues on the narrow FP64 pipe
    float wAf, wBf, w0f, w1f;
};

// The weights of a control block in the working precision.
template <typename Real> struct CtlW;
template <> struct CtlW<float> {
    static __device__ __forceinline__ float wA(const Ctl* c) { return c->wAf; }
    static __device__ __forceinline__ float wB(const Ctl* c) { return c->wBf; }
    static __device__ __forceinline__ float w0(const Ctl* c) { return c->w0f; }
    static __device__ __forceinline__ float w1(const Ctl* c) { return c->w1f; }
};
template <> struct CtlW<double> {
    static __device__ __forceinline__ double wA(const Ctl* c) { return c->wA; }
    static __device__ __forceinline__ double wB(const Ctl* c) { return c->wB; }
    static __device__ __forceinline__ double w0(const Ctl* c) { return c->w0; }
    static __device__ __forceinline__ double w1(const Ctl* c) { return c->w1; }
};

enum {
    DEV_N3BOUND = 1,        // n3 >= 1 met
    DEV_NONFINITE = 2,      // non-finite density or residual met
    DEV_TIMEOUT = 4         // a bounded wait on an asynchronous copy gave up
};

// finalize() operations
enum {
    FIN_F0 = 1,             // f0 = sum, resid = sqrt(f0)
    FIN_N3CUR = 2,          // n3max_cur = max
    FIN_AMAX = 4,           // n3max_next = max; alpha_max; weights for the first sample (or the fixed alpha)
    FIN_F1 = 8,             // f1 = sum; weights for the second sample
    FIN_F2_CHOOSE = 16,     // f2 = sum; alpha from the parabola; weights for the accepted point
    FIN_ACCEPT = 32,        // f0 = f3 = sum; n3max_cur = max; resid; iter++
    FIN_F12_CHOOSE = 128    // f1 = sum, f2 = second sum (paired samples); alpha; weights for the accepted point
};
