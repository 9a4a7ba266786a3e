// Host-side launchers of the pass kernels.
//
// Passes<Real> is the interface the plan code calls; it dispatches on the axis length to
// LaunchX / LaunchY / LaunchZ<Real, N>, whose kernels have the transform length N (and the
// column tile width) fixed at compile time.  N = 0 is the run-time path for any length.
// Each (Real, N) pair is compiled in its own translation unit (kinst.cu).
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>

#include "common.cuh"

// Axis lengths with compile-time kernels.
#define DFT_CT_SIZES(X) X(32) X(48) X(64) X(96) X(128) X(256)

__host__ __device__ constexpr bool dft_is_ct_size(int n) {
    return n == 32 || n == 48 || n == 64 || n == 96 || n == 128 || n == 256;
}

// Column-tile widths of the compile-time y and z passes (kx columns per tile).
#ifndef DFT_TILE_Y_SHIFT
#define DFT_TILE_Y_SHIFT 0
#endif
template <typename Real> __host__ __device__ constexpr int dft_tile_y(int n) {
    return (sizeof(Real) == 4 ? 16 : 8) >> DFT_TILE_Y_SHIFT;
}
// The one-pass z kernels (FP32) transform all components of a tile together (two pools of seven
// tiles in shared memory): the width keeps a CTA near 61 KB (their register budget is for two on an SM).
// DFT_TILE_ZG_SHIFT (build flag, default 0) narrows the tiles by that power of two.
#ifndef DFT_TILE_ZG_SHIFT
#define DFT_TILE_ZG_SHIFT 0
#endif
__host__ __device__ constexpr int dft_tile_z(int n) {
    const int t = n <= 32 ? 16 : (n <= 64 ? 8 : (n <= 128 ? 4 : 2));
    return (t >> DFT_TILE_ZG_SHIFT) > 0 ? (t >> DFT_TILE_ZG_SHIFT) : 1;
}

// The z stages that run as three passes (z transform, k-space products, z transform): run-time
// lengths, and FP64, where the one-pass kernels' narrow tiles (one or two columns at 128) leave lanes
// of the FP64 pipe's warps idle: three species, FP64, one line-search iteration at 128^3 12.2 ms with
// the one-pass kernels, 11.4 with three passes (two species at 64^3 1407 -> 1323 us, 32^3 263 -> 253).
template <typename Real> __host__ __device__ constexpr bool dft_zsplit(int n) { return n == 0 || sizeof(Real) == 8; }

// Persistent TMA z passes: half the grouped width (at least 16 bytes of a row, the TMA
// minimum).
__host__ __device__ constexpr int dft_tile_zb(int n) {
    const int t = dft_tile_z(n) / 2;
    return t > 2 ? t : 2;
}
// Tile width of the persistent TMA first-half z pass: the second half's (DFT_ZFWD_WIDE: the
// grouped width).
__host__ __device__ constexpr int dft_tile_zf(int n) {
#ifdef DFT_ZFWD_WIDE
    return dft_tile_z(n);
#else
    return dft_tile_zb(n);
#endif
}

// Tile buffer of the run-time column transform (k_colfft) in elements: the axis in boxes of at most
// 256 rows (a second one starts at a multiple of four rows, so that every box lands on a 128-byte
// boundary), rounded up to 128 bytes.
inline int dft_col_box_rows(int n) { return n <= 256 ? n : ((n + 1) / 2 + 3) & ~3; }
template <typename Real> inline int dft_col_elems(int n, int T, int planes = 1) {
    const int e = (n <= 256 ? 1 : 2) * dft_col_box_rows(n) * T * planes, q = 128 / int(2 * sizeof(Real));
    return (e + q - 1) / q * q;
}
// Shared memory of k_colfft: two TMA stages, X and (from two radix stages) Y, twiddles, wave
// numbers, mbarriers.
template <typename Real> inline size_t dft_col_smem(int n, int T, int nstages, int planes = 1) {
    return (size_t(nstages > 1 ? 4 : 3) * dft_col_elems<Real>(n, T, planes) + n) * 2 * sizeof(Real) +
           ((n + 1) & ~1) * sizeof(Real) + 2 * sizeof(uint64_t) + 128;
}
// Elements of a run-time column tile up to which it takes several planes (dft_col_planes).
template <typename Real> constexpr int dft_col_fill() { return sizeof(Real) == 4 ? 2048 : 1024; }
// Whether a z transform's tiles may cut the ny pxh columns of a plane as one row (padding included;
// nothing reads it): where they divide it, as chunks of T in the place of the ky, or where a tile takes one
// plane anyway.  Tiles of one ky each leave most of their last one empty, as nx / 2 + 1 is one past a
// multiple: 160^3 FP32, three species, an iteration 1970 -> 1917 us; 100^3 FP64 5960 -> 5817.
template <typename Real> inline bool dft_col_flat(int n, int ny, int pxh, int T) {
    return ny * pxh % T == 0 || n > 256 || dft_col_fill<Real>() / (n * T) < 2;
}
// Tile width of a run-time column transform (128-, 64- or 32-byte rows): of the widths that leave two blocks on an
// SM, the one with the least work per column in use, where a narrower tile's shorter rows and fewer butterflies per block count as 2 / T columns
// (FP64, bound by its arithmetic: 1 / T) and columns past nxh as work.
// Along z (ny > 0: the rows of a plane) the columns of a plane count together where dft_col_flat allows.
template <typename Real> inline int dft_tile_rt(int n, int nxh, int ny = 0, int pxh = 0) {
    constexpr bool f32 = sizeof(Real) == 4;
    int best = 4;
    double best_cost = 1e30;
    for (int T = f32 ? 16 : 8; T >= 4; T /= 2) {
        if (T > 4 && dft_col_smem<Real>(n, T, 2) > 113 * 1024) continue;
        const int cols = ny > 0 && dft_col_flat<Real>(n, ny, pxh, T) ? pxh : (nxh + T - 1) / T * T;
        const double cost = double(cols) * (1.0 + (f32 ? 2.0 : 1.0) / T);
        if (cost < best_cost) { best_cost = cost; best = T; }
    }
    return best;
}

// Resident CTAs per SM that the compile-time column pass's register budget is sized for: what its
// shared memory allows (at 256 one), and no more than its radices' registers (FP64 radix 16: two).  FP64 32
// and 64 (8 x 4, 8 x 8) at four against three: 32^3, two species, y passes of nine spectra 13.0 -> 10.7 us, z
// transforms 7.1 -> 6.0, an iteration 250.6 -> 241.6; 64^3 1256 -> 1248; 48 (8 x 6) 598 -> 604, so three there.
template <typename Real> __host__ __device__ constexpr int dft_yfft_minb(int n) {
    if (n >= 256) return 1;
    if (sizeof(Real) == 4) return n >= 128 ? 3 : 4;
    return n >= 96 ? 2 : (n == 48 ? 3 : 4);
}

// Planes of the other axis (`other` of them) in a tile of a run-time column transform of `items`
// components: as many as a buffer of 2048 elements (FP64 1024) takes, while four tiles per SM remain, so
// that short axes do not pay a tile's latency (a few us) for some hundred elements.  One plane against this:
// 21 x 21 x 161, FP64, S = 2, a y forward pass 69 -> 37 us, an iteration 979 -> 752; 4 x 4 x 512, FP64, a y
// pass 19 -> 13; 100^3 FP32 an iteration 644 -> 537.
template <typename Real> inline int dft_col_planes(int n, int nxh, int T, int other, int items, int sms) {
    if (n > 256) return 1;
    const int most = dft_col_fill<Real>() / (n * T);
    const long long tiles = (long long)((nxh + T - 1) / T) * other * items;
    const long long spread = tiles / (4LL * sms);
    const long long p = spread < most ? spread : most;
    return p < 1 ? 1 : (p > 256 ? 256 : (int)p);
}

// Threads of the persistent TMA z passes and the resident CTAs per SM their register budget
// is sized for.  First half: 256 threads, two CTAs per SM, up to length 128; 512 threads, one
// CTA, at 256.  Second half: 256 threads, three CTAs per SM, up to 128; at 256 (one pass of the
// threads covers the radix-16 butterflies of the seven Phi' groups of a two-column tile) two (its
// shared memory allows no more).  DFT_ZFWD_THREADS / DFT_ZFWD_MINB / DFT_ZBWD_THREADS / DFT_ZBWD_MINB (build
// flags) override.
__host__ __device__ constexpr int dft_zfwd_threads(int n) {
#ifdef DFT_ZFWD_THREADS
    return DFT_ZFWD_THREADS;
#else
    return n >= 256 ? 512 : 256;
#endif
}
__host__ __device__ constexpr int dft_zfwd_minb(int n) {
#ifdef DFT_ZFWD_MINB
    return DFT_ZFWD_MINB;
#else
    return dft_zfwd_threads(n) <= 256 ? 2 : 1;
#endif
}
// The first-half pass for at most three species (its table records and species loops sized for
// three): resident CTAs per SM its register budget is sized for (DFT_ZFWD_MINB_S3 overrides).
__host__ __device__ constexpr int dft_zfwd_minb_s3(int n) {
#ifdef DFT_ZFWD_MINB_S3
    return DFT_ZFWD_MINB_S3;
#else
    return n <= 64 ? 3 : dft_zfwd_minb(n);   // radix 16 at 128 spills under a budget for three
#endif
}
__host__ __device__ constexpr int dft_zbwd_threads(int n) {
#ifdef DFT_ZBWD_THREADS
    return DFT_ZBWD_THREADS;
#else
    return 256;
#endif
}
__host__ __device__ constexpr int dft_zbwd_minb(int n) {
#ifdef DFT_ZBWD_MINB
    return DFT_ZBWD_MINB;
#else
    return n < 256 ? 3 : 2;
#endif
}

template <typename Real, int N>
struct LaunchX {
    using C = typename Cplx<Real>::type;
    static cudaError_t init();
    static cudaError_t xfwd(cudaStream_t st, const GridDesc& g, const AxisPlan& px, int ncomp, int lx, const Real* in,
                     C* out, const C* tw);
    static cudaError_t xphi(cudaStream_t st, const GridDesc& g, const AxisPlan& px, int LR, const Ctl* ctl, const C* A,
                     const C* B, C* mat, C* phi, float* red_max, int* status, double* red_phi, Real kfx,
                     const C* tw);
    static cudaError_t xupdate(cudaStream_t st, const GridDesc& g, const AxisPlan& px, const SpeciesDesc<Real>& sp, int LR,
                        const Ctl* ctl, const C* cspec, const Real* rho0, const Real* rho1, const Real* V,
                        Real* rho_out, Real* g_out, C* gspec_out, Real* rho_lo, double* red_sum, int* status,
                        const C* tw);
    // the two line-search samples in one pass each (weights from ctl[1] and ctl[2]): Phi' of
    // both mixtures of the slots (sample m's nine spectra at phi + m DFT_NSPEC nc), and the
    // update pass's residual sums of both (c spectra at cspec / cspec2, sums into red_sum /
    // red_sum2; nothing written to rho or G)
    static cudaError_t xphi2(cudaStream_t st, const GridDesc& g, const AxisPlan& px, int LR, const Ctl* ctl,
                             const C* A, const C* B, C* phi, int* status, Real kfx, const C* tw);
    static int xphi_rows(const GridDesc& g, int nm, int LR);
    static cudaError_t xupdate2(cudaStream_t st, const GridDesc& g, const AxisPlan& px, const SpeciesDesc<Real>& sp,
                                int LR, const Ctl* ctl, const C* cspec, const C* cspec2, const Real* rho0,
                                const Real* rho1, const Real* V, Real* rho_lo, double* red_sum, double* red_sum2,
                                int* status, const C* tw);
    static cudaError_t xinv(cudaStream_t st, const GridDesc& g, const AxisPlan& px, int LR, int ncomp, const C* spec,
                     Real* out, Real* out_last, const Offsets<Real>& off, int cmax, float* red_max, int wd,
                     Real kfx, const C* tw);
    static cudaError_t xgrad(cudaStream_t st, const GridDesc& g, const AxisPlan& px, const SpeciesDesc<Real>& sp,
                             int LR, Real dv, const C* cspec, const Real* rho, const Real* V, Real* grad_rho,
                             Real* grad_V, double* red, const C* tw);
    static cudaError_t xcanon(cudaStream_t st, const GridDesc& g, const AxisPlan& px, const SpeciesDesc<Real>& sp,
                              int LR, const C* cspec, const Real* V, double* red, const C* tw);
};

template <typename Real, int N>
struct LaunchY {
    using C = typename Cplx<Real>::type;
    static cudaError_t init();
    static cudaError_t yfft(cudaStream_t st, bool inv, const GridDesc& g, const AxisPlan& py, int T, int ncomp, C* data,
                            int* status, const C* tw, long long polls, int mode, Real kfy);
};

template <typename Real, int N>
struct LaunchZ {
    using C = typename Cplx<Real>::type;
    static cudaError_t init();
    static cudaError_t zconv_fwd(cudaStream_t st, const GridDesc& g, const SpeciesDesc<Real>& sp, Real kfx, Real kfy,
                                 Real kfz, int want_psi, const C* in, C* slot_n, C* slot_es, const C* tw, int* status);
    static cudaError_t zconv_bwd(cudaStream_t st, const GridDesc& g, const SpeciesDesc<Real>& sp, Real kfx, Real kfy,
                                 Real kfz, int flags, int ncomp_out, const Ctl* ctl, C* phi, const C* esA,
                                 const C* esB, C* es_mat, const C* tw);
    static cudaError_t zconv_bwd_pair(cudaStream_t st, const GridDesc& g, const SpeciesDesc<Real>& sp, Real kfx,
                                      Real kfy, Real kfz, int ncomp_out, const Ctl* ctl, C* phi, const C* esA,
                                      const C* esB, const C* tw);
    static bool has_zbwd_pair(const GridDesc& g, int ncomp_out);
    static cudaError_t zfft(cudaStream_t st, bool inv, const GridDesc& g, const AxisPlan& pz, int T, int ncomp, C* data,
                            int* status, const C* tw, long long polls, int mode);
};

// Column transform of a run-time length in place (k_colfft; colfft.cu): along z (zax) or y, tiles of
// T columns (16, 8, 4; FP64 8, 4).  mode: COL_*; ncomp counts components, or with the modes of sets
// the sets of nine; kf: the axis's wave number unit (COL_DERIV, COL_FOLD).
template <typename Real>
struct ColFft {
    using C = typename Cplx<Real>::type;
    static cudaError_t init();
    static cudaError_t run(cudaStream_t st, bool inv, const GridDesc& g, const AxisPlan& pa, bool zax, int T, int ncomp,
                           C* data, int* status, const C* tw, long long polls, int mode, Real kf);
};

template <typename Real>
struct Passes {
    using C = typename Cplx<Real>::type;
    // allow the kernels of a grid's lengths (nullptr: of every length) their shared memory
    static cudaError_t init_attributes(const GridDesc* g = nullptr);
    // dynamic shared memory of an x pass with `lines` lines
    static size_t smem_x(int nx, int lines) { return (size_t(nx) + 2 * size_t(lines) * (nx + 1)) * sizeof(C) + 16; }
    // column tile widths of the y passes and of a run-time length's z transforms
    static int tile_y(const GridDesc& g);
    static int tile_z(const GridDesc& g);

    static cudaError_t xfwd(cudaStream_t st, const GridDesc& g, const AxisPlan& px, int ncomp, int lx, const Real* in,
                     C* out, const C* tw);
    // polls: bound of each TMA tile wait (DFT_WAIT_POLLS; the drains after a give-up keep it);
    // mode COL_PLAIN: ncomp components in place; COL_DERIV (inverse) / COL_FOLD (forward): ncomp sets
    // of the nine weighted-density / Phi' spectra, with the y derivatives formed / added
    static cudaError_t yfft(cudaStream_t st, bool inv, const GridDesc& g, const AxisPlan& py, int T, int ncomp, C* data,
                     int* status, const C* tw, long long polls = DFT_WAIT_POLLS, int mode = COL_PLAIN, Real kfy = 0);
    // Whether a half's z stage can only run as three passes (zfft, zmul or zmul_bwd, zfft); the zconv
    // passes, a half in one, need FP32, a compile-time length and the |k| tables, and return
    // cudaErrorNotSupported otherwise.
    static bool z_three(const GridDesc& g, const SpeciesDesc<Real>& sp) {
        return dft_zsplit<Real>(dft_is_ct_size(g.nz) ? g.nz : 0) || !sp.tab_w;
    }
    static cudaError_t zconv_fwd(cudaStream_t st, const GridDesc& g, const SpeciesDesc<Real>& sp, Real kfx, Real kfy,
                                 Real kfz, int want_psi, const C* in, C* slot_n, C* slot_es, const C* tw, int* status);
    static cudaError_t xphi(cudaStream_t st, const GridDesc& g, const AxisPlan& px, int LR, const Ctl* ctl, const C* A,
                     const C* B, C* mat, C* phi, float* red_max, int* status, double* red_phi, Real kfx,
                     const C* tw);
    static cudaError_t zconv_bwd(cudaStream_t st, const GridDesc& g, const SpeciesDesc<Real>& sp, Real kfx, Real kfy,
                                 Real kfz, int flags, int ncomp_out, const Ctl* ctl, C* phi, const C* esA,
                                 const C* esB, C* es_mat, const C* tw);
    // The two line-search samples' second-half z passes in one launch (both hard-sphere and ES
    // parts): phi holds sample 1's nine Phi' spectra then sample 2's, ctl[0] / ctl[1] their
    // weights; sample m's ncomp_out results go to phi components m ncomp_out ...  Only where
    // has_zbwd_pair (the persistent TMA pass); cudaErrorNotSupported otherwise.
    static cudaError_t zconv_bwd_pair(cudaStream_t st, const GridDesc& g, const SpeciesDesc<Real>& sp, Real kfx,
                                      Real kfy, Real kfz, int ncomp_out, const Ctl* ctl, C* phi, const C* esA,
                                      const C* esB, const C* tw);
    static bool has_zbwd_pair(const GridDesc& g, int ncomp_out);
    // The z stages in three passes: zfft = the z transform of ncomp components (COL_WD: of the seven of
    // ncomp sets of nine) in place (k_yfft_tma or k_colfft along z), zmul = the first half's k-space
    // products from the S species spectra into seven weighted-density spectra (slot_n, 1/N applied) and
    // the S (want_psi: S + 1) ES spectra (slot_es); red_energy (or nullptr): energy_blocks pairs of partial
    // sums of the grand potential.
    static cudaError_t zfft(cudaStream_t st, bool inv, const GridDesc& g, const AxisPlan& pz, int T, int ncomp, C* data,
                            int* status, const C* tw, long long polls, int mode = COL_PLAIN);
    static cudaError_t zmul(cudaStream_t st, const GridDesc& g, const SpeciesDesc<Real>& sp, Real kfx, Real kfy,
                            Real kfz, int want_psi, const C* in, C* slot_n, C* slot_es, double* red_energy);
    // the second half's products between its z transforms: one sample or the line search's two
    static cudaError_t zmul_bwd(cudaStream_t st, const GridDesc& g, const SpeciesDesc<Real>& sp, Real kfx, Real kfy,
                                Real kfz, int flags, int ncomp_out, int samples, const Ctl* ctl, C* phi, const C* esA,
                                const C* esB, C* es_mat);
    // pairs of partial sums zmul writes to red_energy
    static long long energy_blocks(const GridDesc& g);
    // rho_lo (or nullptr): low part of an extended iterate rho0 + rho_lo, read
    // with rho0 and, when rho_out is written, replaced by the low part of the new iterate;
    // gspec_out (or nullptr): also the x half spectra of G (S components, the layout of xfwd's
    // output), the next first half's input
    static cudaError_t xupdate(cudaStream_t st, const GridDesc& g, const AxisPlan& px, const SpeciesDesc<Real>& sp, int LR,
                        const Ctl* ctl, const C* cspec, const Real* rho0, const Real* rho1, const Real* V,
                        Real* rho_out, Real* g_out, C* gspec_out, Real* rho_lo, double* red_sum, int* status,
                        const C* tw);
    // the two line-search samples in one pass each (weights from ctl[1] and ctl[2]): Phi' of
    // both mixtures of the slots (sample m's nine spectra at phi + m DFT_NSPEC nc), and the
    // update pass's residual sums of both (c spectra at cspec / cspec2, sums into red_sum /
    // red_sum2; nothing written to rho or G)
    static cudaError_t xphi2(cudaStream_t st, const GridDesc& g, const AxisPlan& px, int LR, const Ctl* ctl,
                             const C* A, const C* B, C* phi, int* status, Real kfx, const C* tw);
    // Rows per block, at most LR, with which the persistent form of g.xpers of the Phi' pass of nm mixtures
    // fits the shared memory (LR itself where none is asked for or not even one row fits).
    static int xphi_rows(const GridDesc& g, int nm, int LR);
    static cudaError_t xupdate2(cudaStream_t st, const GridDesc& g, const AxisPlan& px, const SpeciesDesc<Real>& sp,
                                int LR, const Ctl* ctl, const C* cspec, const C* cspec2, const Real* rho0,
                                const Real* rho1, const Real* V, Real* rho_lo, double* red_sum, double* red_sum2,
                                int* status, const C* tw);
    static cudaError_t xinv(cudaStream_t st, const GridDesc& g, const AxisPlan& px, int LR, int ncomp, const C* spec,
                     Real* out, Real* out_last, const Offsets<Real>& off, int cmax, float* red_max, int wd,
                     Real kfx, const C* tw);
    static cudaError_t xgrad(cudaStream_t st, const GridDesc& g, const AxisPlan& px, const SpeciesDesc<Real>& sp,
                             int LR, Real dv, const C* cspec, const Real* rho, const Real* V, Real* grad_rho,
                             Real* grad_V, double* red, const C* tw);
    // sums for the normalisation of fixed-number species (red: [blocks][DFT_MAXS]) and the
    // scale factors they give (into ctl->canon_scale)
    static cudaError_t xcanon(cudaStream_t st, const GridDesc& g, const AxisPlan& px, const SpeciesDesc<Real>& sp,
                              int LR, const C* cspec, const Real* V, double* red, const C* tw);
    static cudaError_t canon_scale(cudaStream_t st, Ctl* ctl, const SpeciesDesc<Real>& sp, const double* red,
                                   int nblocks, int pdl);
    // fill the `rows` rows of the |k| tables of sp (tab_w and tab_k unless !all, tab_dk where it is not
    // null; they and tab_oct set by the caller); kf: the wave number of a cubic box
    static cudaError_t build_ktab(cudaStream_t st, const GridDesc& g, const SpeciesDesc<Real>& sp, double kf, Real kfx,
                                  Real kfy, Real kfz, long long rows, bool all);
    // fill out[nx + ny + nz] with the per-axis Laplacian terms of grid g (SpeciesDesc::lap1d)
    static cudaError_t build_laptab(cudaStream_t st, const GridDesc& g, Real kfx, Real kfy, Real kfz, Real* out);
};

// The plan's three control blocks at the start of an evaluation: status cleared, weights (1, 0).
cudaError_t launch_ctl_reset(cudaStream_t st, Ctl* ctl, int pdl);

// ctl: the plan's three control blocks (iteration, sample 1 weights, sample 2 weights);
// red_sum2 (or nullptr): the second sample's partial sums for FIN_F12_CHOOSE; pdl: launch with
// programmatic dependent launch (GridDesc::pdl)
cudaError_t launch_finalize(cudaStream_t st, Ctl* ctl, const double* red_sum, const double* red_sum2, int nsum,
                            const float* red_max, int nmax, int op, double inv_count, double alpha_fixed,
                            double n3_bound, double alpha_floor, int pdl);

inline long long ceil_div(long long a, long long b) { return (a + b - 1) / b; }
