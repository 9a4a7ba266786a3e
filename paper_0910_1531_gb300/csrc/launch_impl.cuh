// Definitions of LaunchX / LaunchY / LaunchZ<Real, N> (included by kinst.cu once per pair).
#pragma once

#include "kernels.cuh"
#include "launch.cuh"
#include "passes.h"

namespace {
// x pass: twiddles (nx) + two buffers of `lines` rows at the kernel's row pitch
template <typename C, int N> size_t smem_x_of(int nx, int lines) {
    const int pitch = dftk::x_pitch<N>(nx);
    return (size_t(nx) + 2 * size_t(lines) * pitch) * sizeof(C) + 16;
}
}  // namespace

// ---------------------------------------------------------------------------------- x
template <typename Real, int N>
cudaError_t LaunchX<Real, N>::init() {
    cudaError_t e = cudaSuccess, r;
    if ((r = set_max_smem(dftk::k_xfwd<Real, N>)) != cudaSuccess) e = r;
    if ((r = set_max_smem(dftk::k_xphi<Real, N, 1>)) != cudaSuccess) e = r;
    if ((r = set_max_smem(dftk::k_xphi<Real, N, 2>)) != cudaSuccess) e = r;
    if constexpr (N > 0) {
        if ((r = set_max_smem(dftk::k_xphi_tma<Real, N, 1>)) != cudaSuccess) e = r;
        if ((r = set_max_smem(dftk::k_xphi_tma<Real, N, 2>)) != cudaSuccess) e = r;
        if ((r = set_max_smem(dftk::k_xphi_cpa<Real, N, 1>)) != cudaSuccess) e = r;
        if ((r = set_max_smem(dftk::k_xphi_cpa<Real, N, 2>)) != cudaSuccess) e = r;
    }
    if ((r = set_max_smem(dftk::k_xupdate<Real, N, 1>)) != cudaSuccess) e = r;
    if ((r = set_max_smem(dftk::k_xupdate<Real, N, 2>)) != cudaSuccess) e = r;
    if ((r = set_max_smem(dftk::k_xcanon<Real, N>)) != cudaSuccess) e = r;
    if ((r = set_max_smem(dftk::k_xinv<Real, N>)) != cudaSuccess) e = r;
    if ((r = set_max_smem(dftk::k_xgrad<Real, N>)) != cudaSuccess) e = r;
    return e;
}

template <typename Real, int N>
cudaError_t LaunchX<Real, N>::xfwd(cudaStream_t st, const GridDesc& g, const AxisPlan& px, int ncomp, int lx,
                            const Real* in, C* out, const C* tw) {
    const long long rows = (long long)ncomp * g.ny * g.nz;
    const unsigned blocks = (unsigned)ceil_div((rows + 1) / 2, lx);
    launch_k(dftk::k_xfwd<Real, N>, blocks, dftk::kThreads, smem_x_of<C, N>(g.nx, lx), st, g.pdl, g, px, ncomp, lx, in, out, tw);
    return cudaSuccess;
}

namespace {
// The persistent Phi' x passes (compile-time lengths, no grand-potential sums): g.xpers 1 =
// bulk copies two blocks ahead, 2 = per-thread cp.async one block ahead; grid = the row blocks,
// at most the CTAs that fit on the GPU at once.  False if neither applies.
template <typename Real, int N, int NM, typename C>
bool launch_xphi_tma(cudaStream_t st, const GridDesc& g, int LR, const Ctl* ctl, const C* A, const C* B, C* mat,
                     C* phi, float* red_max, int* status, Real kfx, const C* tw) {
    if constexpr (N <= 0) {
        return false;
    } else {
        if (!g.xpers || !status) return false;
        const int nsrc = B ? 2 * DFT_NSPEC : DFT_NSPEC;
        const bool cpa = g.xpers == 2;
        const size_t sm = cpa ? dftk::xphi_cpa_smem<Real, N>(NM, LR, nsrc, g.pxh)
                              : dftk::xphi_tma_smem<Real, N>(NM, LR, nsrc, g.pxh);
        static int optin = 0, sms = 0;
        if (optin == 0) {
            int dev = 0;
            cudaGetDevice(&dev);
            cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        }
        if (sm > size_t(optin)) return false;
        int occ = 0;
        if (cpa) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, dftk::k_xphi_cpa<Real, N, NM>, dftk::kThreads, sm);
        else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, dftk::k_xphi_tma<Real, N, NM>, dftk::kThreads, sm);
        if (occ < 1) occ = 1;
        const long long nblk = ceil_div((long long)g.ny * g.nz, LR);
        const int grid = (int)(nblk < (long long)sms * occ ? nblk : (long long)sms * occ);
        if (cpa)
            launch_k(dftk::k_xphi_cpa<Real, N, NM>, grid, dftk::kThreads, sm, st, g.pdl, g, LR, ctl, A, B, mat, phi,
                     red_max, status, kfx, tw);
        else
            launch_k(dftk::k_xphi_tma<Real, N, NM>, grid, dftk::kThreads, sm, st, g.pdl, g, LR, ctl, A, B, mat, phi,
                     red_max, status, kfx, tw);
        return true;
    }
}
}  // namespace

template <typename Real, int N>
cudaError_t LaunchX<Real, N>::xphi(cudaStream_t st, const GridDesc& g, const AxisPlan& px, int LR, const Ctl* ctl,
                            const C* A, const C* B, C* mat, C* phi, float* red_max, int* status, double* red_phi,
                            Real kfx, const C* tw) {
    if (!red_phi && launch_xphi_tma<Real, N, 1>(st, g, LR, ctl, A, B, mat, phi, red_max, status, kfx, tw))
        return cudaSuccess;
    const unsigned blocks = (unsigned)ceil_div((long long)g.ny * g.nz, LR);
    launch_k(dftk::k_xphi<Real, N, 1>, blocks, dftk::kThreads, smem_x_of<C, N>(g.nx, 5 * LR), st, g.pdl, g, px, LR, ctl,
             A, B, mat, phi, red_max, status, red_phi, kfx, tw);
    return cudaSuccess;
}

template <typename Real, int N>
int LaunchX<Real, N>::xphi_rows(const GridDesc& g, int nm, int LR) {
    if constexpr (N > 0) {
        int dev = 0, optin = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        auto smem = [&](int L) {        // both slots read
            return g.xpers == 2 ? dftk::xphi_cpa_smem<Real, N>(nm, L, 2 * DFT_NSPEC, g.pxh)
                                : dftk::xphi_tma_smem<Real, N>(nm, L, 2 * DFT_NSPEC, g.pxh);
        };
        for (int L = LR; g.xpers && L >= 1; --L)
            if (smem(L) <= size_t(optin)) return L;
    }
    return LR;
}

template <typename Real, int N>
cudaError_t LaunchX<Real, N>::xphi2(cudaStream_t st, const GridDesc& g, const AxisPlan& px, int LR, const Ctl* ctl,
                                    const C* A, const C* B, C* phi, int* status, Real kfx, const C* tw) {
    if (launch_xphi_tma<Real, N, 2>(st, g, LR, ctl, A, B, static_cast<C*>(nullptr), phi, static_cast<float*>(nullptr),
                                    status, kfx, tw))
        return cudaSuccess;
    const unsigned blocks = (unsigned)ceil_div((long long)g.ny * g.nz, LR);
    launch_k(dftk::k_xphi<Real, N, 2>, blocks, dftk::kThreads, smem_x_of<C, N>(g.nx, 10 * LR), st, g.pdl,
        g, px, LR, ctl, A, B, nullptr, phi, nullptr, status, nullptr, kfx, tw);
    return cudaSuccess;
}

template <typename Real, int N>
cudaError_t LaunchX<Real, N>::xupdate(cudaStream_t st, const GridDesc& g, const AxisPlan& px, const SpeciesDesc<Real>& sp,
                               int LR, const Ctl* ctl, const C* cspec, const Real* rho0, const Real* rho1,
                               const Real* V, Real* rho_out, Real* g_out, C* gspec_out, Real* rho_lo,
                               double* red_sum, int* status, const C* tw) {
    const unsigned blocks = (unsigned)ceil_div((long long)g.ny * g.nz, LR);
    const int lpr = (sp.S + 1) / 2;
    launch_k(dftk::k_xupdate<Real, N, 1>, blocks, dftk::kThreads, smem_x_of<C, N>(g.nx, lpr * LR), st, g.pdl,
        g, px, sp, LR, ctl, cspec, nullptr, rho0, rho1, V, rho_out, g_out, gspec_out, rho_lo, red_sum, nullptr,
        status, tw);
    return cudaSuccess;
}

template <typename Real, int N>
cudaError_t LaunchX<Real, N>::xupdate2(cudaStream_t st, const GridDesc& g, const AxisPlan& px,
                                       const SpeciesDesc<Real>& sp, int LR, const Ctl* ctl, const C* cspec,
                                       const C* cspec2, const Real* rho0, const Real* rho1, const Real* V,
                                       Real* rho_lo, double* red_sum, double* red_sum2, int* status, const C* tw) {
    const unsigned blocks = (unsigned)ceil_div((long long)g.ny * g.nz, LR);
    const int lpr = (sp.S + 1) / 2;
    launch_k(dftk::k_xupdate<Real, N, 2>, blocks, dftk::kThreads, smem_x_of<C, N>(g.nx, 2 * lpr * LR), st, g.pdl,
        g, px, sp, LR, ctl, cspec, cspec2, rho0, rho1, V, nullptr, nullptr, static_cast<C*>(nullptr), rho_lo,
        red_sum, red_sum2, status, tw);
    return cudaSuccess;
}

template <typename Real, int N>
cudaError_t LaunchX<Real, N>::xinv(cudaStream_t st, const GridDesc& g, const AxisPlan& px, int LR, int ncomp,
                            const C* spec, Real* out, Real* out_last, const Offsets<Real>& off, int cmax,
                            float* red_max, int wd, Real kfx, const C* tw) {
    const unsigned blocks = (unsigned)ceil_div((long long)g.ny * g.nz, LR);
    // one component and no outputs: the kernel pairs grid rows in its lines
    const bool rows2 = ncomp == 1 && !wd && !out && !out_last;
    const int lines = rows2 ? (LR + 1) / 2 : (ncomp + 1) / 2 * LR;
    launch_k(dftk::k_xinv<Real, N>, blocks, dftk::kThreads, smem_x_of<C, N>(g.nx, lines), st, g.pdl,
        g, px, LR, ncomp, spec, out, out_last, off, cmax, red_max, wd, kfx, tw);
    return cudaSuccess;
}

template <typename Real, int N>
cudaError_t LaunchX<Real, N>::xgrad(cudaStream_t st, const GridDesc& g, const AxisPlan& px,
                                    const SpeciesDesc<Real>& sp, int LR, Real dv, const C* cspec, const Real* rho,
                                    const Real* V, Real* grad_rho, Real* grad_V, double* red, const C* tw) {
    const unsigned blocks = (unsigned)ceil_div((long long)g.ny * g.nz, LR);
    const int lpr = (sp.S + 1) / 2;
    launch_k(dftk::k_xgrad<Real, N>, blocks, dftk::kThreads, smem_x_of<C, N>(g.nx, lpr * LR), st, g.pdl,
        g, px, sp, LR, dv, cspec, rho, V, grad_rho, grad_V, red, tw);
    return cudaSuccess;
}

// Lines (species pairs) of the x transform that hold a fixed-number species.
template <typename Real> inline int canon_lines(const SpeciesDesc<Real>& sp, int* lines) {
    int nl = 0;
    for (int l = 0; 2 * l < sp.S; ++l)
        if (sp.canon[2 * l] || (2 * l + 1 < sp.S && sp.canon[2 * l + 1])) lines[nl++] = l;
    return nl;
}

template <typename Real, int N>
cudaError_t LaunchX<Real, N>::xcanon(cudaStream_t st, const GridDesc& g, const AxisPlan& px,
                                     const SpeciesDesc<Real>& sp, int LR, const C* cspec, const Real* V,
                                     double* red, const C* tw) {
    int lines[3] = {0, 0, 0};
    const int nl = canon_lines(sp, lines);
    if (nl == 0) return cudaSuccess;
    const unsigned blocks = (unsigned)ceil_div((long long)g.ny * g.nz, LR);
    launch_k(dftk::k_xcanon<Real, N>, blocks, dftk::kThreads, smem_x_of<C, N>(g.nx, nl * LR), st, g.pdl,
        g, px, sp, LR, nl, lines[0], lines[1], lines[2], cspec, V, red, tw);
    return cudaSuccess;
}

// ---------------------------------------------------------------------------------- y
template <typename Real, int N>
cudaError_t LaunchY<Real, N>::init() {
    cudaError_t e = cudaSuccess, r;
    if constexpr (N > 0) {
        constexpr int TY = dft_tile_y<Real>(N);
        if ((r = set_max_smem(dftk::k_yfft_tma<Real, false, N, TY>)) != cudaSuccess) e = r;
        if ((r = set_max_smem(dftk::k_yfft_tma<Real, true, N, TY>)) != cudaSuccess) e = r;
        if ((r = set_max_smem(dftk::k_yfft_tma<Real, false, N, TY, false, COL_FOLD>)) != cudaSuccess) e = r;
        if ((r = set_max_smem(dftk::k_yfft_tma<Real, true, N, TY, false, COL_DERIV>)) != cudaSuccess) e = r;
    }
    (void)r;
    return e;
}

namespace {
// One launch of the compile-time column pass along y or (ZAX) z.
template <typename Real, bool INV, int N, bool ZAX, int MODE, typename C>
cudaError_t launch_col_ct(cudaStream_t st, const GridDesc& g, int ncomp, C* data, int* status, const C* tw,
                          long long polls, int mode, Real kf) {
    constexpr int TY = dft_tile_y<Real>(N);
    constexpr int E = int(sizeof(C) / 8);
    const int planes = mode == COL_PLAIN ? ncomp : ncomp * DFT_NSPEC, items = mode == COL_PLAIN ? ncomp : ncomp * DFT_NZSPEC;
    CUtensorMap map;
    // along z the ny rows of a plane are one row of ny pxh columns
    const int cols = ZAX ? g.ny * g.pxh : g.nxh, rows = ZAX ? 1 : g.ny;
    cudaError_t e = tma_encode_3d(&map, data, (unsigned long long)cols * E, (unsigned long long)rows,
                                  (unsigned long long)g.nz * planes, (unsigned long long)g.pxh * sizeof(C),
                                  (unsigned long long)g.ny * g.pxh * sizeof(C), TY * E, ZAX ? 1 : N, ZAX ? N : 1);
    if (e != cudaSuccess) return e;
    const int ntx = (int)ceil_div(cols, TY), other = ZAX ? 1 : g.nz;
    const int ntiles = ntx * other * items;
    const size_t sm = dftk::yfft_tma_smem<Real, N, TY>();
    auto kern = dftk::k_yfft_tma<Real, INV, N, TY, ZAX, MODE>;
    const int fit = resident_blocks(kern, dftk::kThreads, sm);
    return launch_k(kern, ntiles < fit ? ntiles : fit, dftk::kThreads, sm, st, g.pdl, map, ntx, other, ntiles,
                    (mode != COL_PLAIN ? 1 : 0) | (cols % TY == 1 ? 2 : 0), status, tw, kf, polls);
}
}  // namespace

template <typename Real, int N>
cudaError_t LaunchY<Real, N>::yfft(cudaStream_t st, bool inv, const GridDesc& g, const AxisPlan& py, int T, int ncomp,
                                   C* data, int* status, const C* tw, long long polls, int mode, Real kfy) {
    if constexpr (N > 0) {
        if (mode == COL_DERIV)
            return launch_col_ct<Real, true, N, false, COL_DERIV>(st, g, ncomp, data, status, tw, polls, mode, kfy);
        if (mode == COL_FOLD)
            return launch_col_ct<Real, false, N, false, COL_FOLD>(st, g, ncomp, data, status, tw, polls, mode, kfy);
        return inv ? launch_col_ct<Real, true, N, false, COL_PLAIN>(st, g, ncomp, data, status, tw, polls, mode, kfy)
                   : launch_col_ct<Real, false, N, false, COL_PLAIN>(st, g, ncomp, data, status, tw, polls, mode, kfy);
    } else {
        return ColFft<Real>::run(st, inv, g, py, false, T, ncomp, data, status, tw, polls, mode, kfy);
    }
}

// ---------------------------------------------------------------------------------- z
// The z transforms of any length, and the halves in one pass (FP32, compile-time lengths).
template <typename Real, int N>
cudaError_t LaunchZ<Real, N>::init() {
    cudaError_t e = cudaSuccess, r;
    if constexpr (!dft_zsplit<Real>(N)) {
        constexpr int TZ = dft_tile_z(N);
        if ((r = set_max_smem(dftk::k_zconv_fwd_g<Real, N, TZ>)) != cudaSuccess) e = r;
        if ((r = set_max_smem(dftk::k_zconv_bwd_g<Real, N, TZ>)) != cudaSuccess) e = r;
        constexpr int TB = dft_tile_zb(N), TF = dft_tile_zf(N);
        constexpr int NB = dft_zbwd_threads(N), MBB = dft_zbwd_minb(N);
        constexpr int NF = dft_zfwd_threads(N), MBF = dft_zfwd_minb(N), MBF3 = dft_zfwd_minb_s3(N);
        if ((r = set_max_smem(dftk::k_zconv_bwd_tma<Real, N, TB, NB, MBB, 3>)) != cudaSuccess) e = r;
        if ((r = set_max_smem(dftk::k_zconv_bwd_tma<Real, N, TB, NB, MBB, DFT_MAXS>)) != cudaSuccess) e = r;
        if ((r = set_max_smem(dftk::k_zconv_fwd_tma<Real, N, TF, NF, MBF, DFT_MAXS>)) != cudaSuccess) e = r;
        if ((r = set_max_smem(dftk::k_zconv_fwd_tma<Real, N, TF, NF, MBF3, 3>)) != cudaSuccess) e = r;
    }
    if constexpr (N > 0) {
        constexpr int TY = dft_tile_y<Real>(N);
        if ((r = set_max_smem(dftk::k_yfft_tma<Real, false, N, TY, true>)) != cudaSuccess) e = r;
        if ((r = set_max_smem(dftk::k_yfft_tma<Real, true, N, TY, true>)) != cudaSuccess) e = r;
    }
    (void)r;
    return e;
}

template <typename Real, int N>
cudaError_t LaunchZ<Real, N>::zfft(cudaStream_t st, bool inv, const GridDesc& g, const AxisPlan& pz, int T, int ncomp,
                                   C* data, int* status, const C* tw, long long polls, int mode) {
    if constexpr (N > 0) {
        return inv ? launch_col_ct<Real, true, N, true, COL_PLAIN>(st, g, ncomp, data, status, tw, polls, mode, Real(0))
                   : launch_col_ct<Real, false, N, true, COL_PLAIN>(st, g, ncomp, data, status, tw, polls, mode, Real(0));
    } else {
        return ColFft<Real>::run(st, inv, g, pz, true, T, ncomp, data, status, tw, polls, mode, Real(0));
    }
}

template <typename Real, int N>
cudaError_t LaunchZ<Real, N>::zconv_fwd(cudaStream_t st, const GridDesc& g, const SpeciesDesc<Real>& sp, Real kfx,
                                        Real kfy, Real kfz, int want_psi, const C* in, C* slot_n, C* slot_es,
                                        const C* tw, int* status) {
    if constexpr (!dft_zsplit<Real>(N)) {
        constexpr int TZ = dft_tile_z(N);
        constexpr int TB = dft_tile_zf(N);
        static int optin = 0, sms = 0;
        if (optin == 0) {
            int dev = 0;
            cudaGetDevice(&dev);
            cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        }
        const size_t sm = dftk::zfwd_tma_smem<Real, N, TB>(sp.S);
        if (status && !g.zgrp && sm <= size_t(optin)) {
            constexpr int NT = dft_zfwd_threads(N), MB = dft_zfwd_minb(N);
            constexpr int E = int(sizeof(C) / 8);
            CUtensorMap map_in, map_n;
            auto encode = [&](CUtensorMap* m, const C* data, int ncomp) {
                return tma_encode_3d(m, const_cast<C*>(data), (unsigned long long)g.nxh * E, (unsigned long long)g.ny,
                                     (unsigned long long)g.nz * ncomp, (unsigned long long)g.pxh * sizeof(C),
                                     (unsigned long long)g.ny * g.pxh * sizeof(C), TB * E, 1, N);
            };
            cudaError_t e = encode(&map_in, in, sp.S);
            if (e == cudaSuccess) e = encode(&map_n, slot_n, DFT_NSPEC);
            if (e != cudaSuccess) return e;
            const int ntx = (int)ceil_div(g.nxh, TB);
            const int ntiles = ntx * g.ny;
            // at most three species: the instance whose records and species loops are sized for three
            constexpr int MB3 = dft_zfwd_minb_s3(N);
            auto kern = sp.S <= 3 ? dftk::k_zconv_fwd_tma<Real, N, TB, NT, MB3, 3>
                                  : dftk::k_zconv_fwd_tma<Real, N, TB, NT, MB, DFT_MAXS>;
            const int fit = resident_blocks(kern, NT, sm), grid = ntiles < fit ? ntiles : fit;
            launch_k(kern, grid, NT, sm, st, g.pdl, map_in, map_n, g, sp, kfx, kfy, kfz, want_psi, slot_es, ntx, ntiles,
                     status, tw);
            return cudaSuccess;
        }
        dim3 grid((unsigned)ceil_div(g.nxh, TZ), (unsigned)g.ny);
        return launch_k(dftk::k_zconv_fwd_g<Real, N, TZ>, grid, dftk::kThreads, dftk::zg_smem_bytes<TZ, N>(sizeof(C)), st,
                        g.pdl, g, sp, kfx, kfy, kfz, want_psi, in, slot_n, slot_es, tw);
    }
    return cudaErrorNotSupported;
}

namespace {
// The persistent TMA second-half z pass: single (pair = 0: a set of nine Phi' spectra at phi, seven of them
// read, results over its first ncomp_out) or the two line-search samples (pair = 1: two sets, weights in
// ctl[0], ctl[1], results at phi components 0 .. 2 ncomp_out - 1).  False if it does not apply (no
// one-pass kernel, the grouped variant chosen, or too little shared memory).
template <typename Real, int N, typename C>
bool launch_zbwd_tma(cudaStream_t st, const GridDesc& g, const SpeciesDesc<Real>& sp, Real kfx, Real kfy, Real kfz,
                     int flags, int ncomp_out, int pair, const Ctl* ctl, C* phi, const C* esA, const C* esB, C* es_mat,
                     const C* tw) {
    if constexpr (dft_zsplit<Real>(N)) {
        return false;
    } else {
        constexpr int TB = dft_tile_zb(N);
        const bool es_on = (flags & 2) != 0;
        const int nes = es_on ? ncomp_out * (esB ? 2 : 1) : 0;
        static int optin = 0, sms = 0;
        if (optin == 0) {
            int dev = 0;
            cudaGetDevice(&dev);
            cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        }
        const size_t sm = dftk::zbwd_tma_smem<Real, N, TB>(nes);
        if (g.zgrp || sm > size_t(optin)) return false;
        // persistent CTAs, two TMA-filled stages of seven Phi' tiles, one area of ES tiles
        constexpr int NT = dft_zbwd_threads(N), MB = dft_zbwd_minb(N);
        constexpr int E = int(sizeof(C) / 8);
        CUtensorMap map_phi, map_esA, map_esB, map_out;
        auto encode = [&](CUtensorMap* m, const C* data, int ncomp) {
            return tma_encode_3d(m, const_cast<C*>(data), (unsigned long long)g.nxh * E, (unsigned long long)g.ny,
                                 (unsigned long long)g.nz * ncomp, (unsigned long long)g.pxh * sizeof(C),
                                 (unsigned long long)g.ny * g.pxh * sizeof(C), TB * E, 1, N);
        };
        const int nphi = (pair ? 2 : 1) * DFT_NSPEC;
        cudaError_t e = encode(&map_phi, phi, nphi);
        if (e == cudaSuccess) e = encode(&map_esA, es_on ? esA : phi, es_on ? ncomp_out : DFT_NSPEC);
        if (e == cudaSuccess) e = encode(&map_esB, (es_on && esB) ? esB : phi, (es_on && esB) ? ncomp_out : DFT_NSPEC);
        if (e == cudaSuccess) e = encode(&map_out, phi, nphi);
        if (e != cudaSuccess) return false;
        const int ntx = (int)ceil_div(g.nxh, TB);
        const int ntiles = ntx * g.ny;
        // at most three species: the instance whose records and species loops are sized for three
        auto kern = sp.S <= 3 ? dftk::k_zconv_bwd_tma<Real, N, TB, NT, MB, 3>
                              : dftk::k_zconv_bwd_tma<Real, N, TB, NT, MB, DFT_MAXS>;
        const int fit = resident_blocks(kern, NT, sm), grid = ntiles < fit ? ntiles : fit;
        // the status word of the device control block records a TMA wait that ran out
        int* status = const_cast<int*>(&ctl->status);
        launch_k(kern, grid, NT, sm, st, g.pdl, map_phi, map_esA, map_esB,
                 map_out, g, sp, kfx, kfy, kfz, flags, ncomp_out, esB ? 1 : 0, pair, ctl, es_mat, ntx, ntiles, status,
                 tw);
        return true;
    }
}
}  // namespace

template <typename Real, int N>
cudaError_t LaunchZ<Real, N>::zconv_bwd(cudaStream_t st, const GridDesc& g, const SpeciesDesc<Real>& sp, Real kfx,
                                        Real kfy, Real kfz, int flags, int ncomp_out, const Ctl* ctl, C* phi,
                                        const C* esA, const C* esB, C* es_mat, const C* tw) {
    if (launch_zbwd_tma<Real, N>(st, g, sp, kfx, kfy, kfz, flags, ncomp_out, 0, ctl, phi, esA, esB, es_mat, tw))
        return cudaSuccess;
    if constexpr (!dft_zsplit<Real>(N)) {
        constexpr int TZ = dft_tile_z(N);
        dim3 grid((unsigned)ceil_div(g.nxh, TZ), (unsigned)g.ny);
        return launch_k(dftk::k_zconv_bwd_g<Real, N, TZ>, grid, dftk::kThreads, dftk::zg_smem_bytes<TZ, N>(sizeof(C)), st,
                        g.pdl, g, sp, kfx, kfy, kfz, flags, ncomp_out, ctl, phi, esA, esB, es_mat, tw);
    }
    return cudaErrorNotSupported;
}

template <typename Real, int N>
cudaError_t LaunchZ<Real, N>::zconv_bwd_pair(cudaStream_t st, const GridDesc& g, const SpeciesDesc<Real>& sp, Real kfx,
                                             Real kfy, Real kfz, int ncomp_out, const Ctl* ctl, C* phi, const C* esA,
                                             const C* esB, const C* tw) {
    if (launch_zbwd_tma<Real, N>(st, g, sp, kfx, kfy, kfz, 3, ncomp_out, 1, ctl, phi, esA, esB,
                                 static_cast<C*>(nullptr), tw))
        return cudaSuccess;
    return cudaErrorNotSupported;
}

template <typename Real, int N>
bool LaunchZ<Real, N>::has_zbwd_pair(const GridDesc& g, int ncomp_out) {
    if constexpr (dft_zsplit<Real>(N)) {
        return false;
    } else {
        constexpr int TB = dft_tile_zb(N);
        int dev = 0, optin = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        return !g.zgrp && dftk::zbwd_tma_smem<Real, N, TB>(2 * ncomp_out) <= size_t(optin);
    }
}
