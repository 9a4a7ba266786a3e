// Launchers of the run-time column transform, compiled once per precision (DFT_INST_REAL).
#include "kernels.cuh"
#include "launch.cuh"
#include "passes.h"

namespace {
template <typename Real, bool INV, int T, bool BIG, int MODE>
cudaError_t launch(cudaStream_t st, const GridDesc& g, const AxisPlan& pa, bool zax, int ncomp,
                   typename Cplx<Real>::type* data, int* status, const typename Cplx<Real>::type* tw, long long polls,
                   int mode, Real kf) {
    using C = typename Cplx<Real>::type;
    constexpr int E = int(sizeof(C) / 8);
    dftk::ColBox cb;
    cb.n = pa.n;
    cb.nbox = pa.n <= 256 ? 1 : 2;
    cb.rows = dft_col_box_rows(pa.n);
    // the planes as nxh columns x ny rows; along z as chunks of T columns, or all columns as one row
    const bool flat = zax && dft_col_flat<Real>(pa.n, g.ny, g.pxh, T), chunks = flat && g.ny * g.pxh % T == 0;
    const int nxh = !flat ? g.nxh : (chunks ? T : g.ny * g.pxh), ny = !flat ? g.ny : (chunks ? g.ny * g.pxh / T : 1);
    const int ntx = (int)ceil_div(nxh, T), across = zax ? ny : g.nz;
    const int items = mode == COL_PLAIN ? ncomp : ncomp * DFT_NZSPEC;
    cb.planes = dft_col_planes<Real>(pa.n, nxh, T, across, items, sm_count());
    cb.elems = dft_col_elems<Real>(pa.n, T, cb.planes);
    CUtensorMap map;
    const unsigned long long dims[4] = {(unsigned long long)nxh * E, (unsigned long long)ny, (unsigned long long)g.nz,
                                        (unsigned long long)(mode == COL_PLAIN ? ncomp : ncomp * DFT_NSPEC)};
    const unsigned long long strides[3] = {(unsigned long long)(flat ? T : g.pxh) * sizeof(C),
                                           (unsigned long long)g.ny * g.pxh * sizeof(C),
                                           (unsigned long long)g.nc * sizeof(C)};
    const unsigned pl = unsigned(cb.planes), rows = unsigned(cb.rows);
    const unsigned box[4] = {unsigned(T * E), zax ? pl : rows, zax ? rows : pl, 1u};
    cudaError_t e = tma_encode_4d(&map, data, dims, strides, box);
    if (e != cudaSuccess) return e;
    const int other = (int)ceil_div(across, cb.planes);
    const int ntiles = ntx * other * items;
    const size_t sm = dft_col_smem<Real>(pa.n, T, pa.nstages, cb.planes);
    auto kern = dftk::k_colfft<Real, INV, T, BIG, MODE>;
    const int fit = resident_blocks(kern, dftk::kThreads, sm);
    return launch_k(kern, ntiles < fit ? ntiles : fit, dftk::kThreads, sm, st, g.pdl, map, pa, cb, zax ? 1 : 0, ntx,
                    other, ntiles, mode != COL_PLAIN ? 1 : 0, status, tw, kf, polls);
}

template <typename Real, bool INV, int T>
cudaError_t launch_m(cudaStream_t st, const GridDesc& g, const AxisPlan& pa, bool zax, int ncomp,
                     typename Cplx<Real>::type* data, int* status, const typename Cplx<Real>::type* tw,
                     long long polls, int mode, Real kf) {
    constexpr int kDual = INV ? COL_DERIV : COL_FOLD;
    const bool big = dft_has_big_prime(pa.n);
    if (mode == kDual)
        return big ? launch<Real, INV, T, true, kDual>(st, g, pa, zax, ncomp, data, status, tw, polls, mode, kf)
                   : launch<Real, INV, T, false, kDual>(st, g, pa, zax, ncomp, data, status, tw, polls, mode, kf);
    return big ? launch<Real, INV, T, true, COL_PLAIN>(st, g, pa, zax, ncomp, data, status, tw, polls, mode, kf)
               : launch<Real, INV, T, false, COL_PLAIN>(st, g, pa, zax, ncomp, data, status, tw, polls, mode, kf);
}

template <typename Real, bool INV, int T> cudaError_t init_m() {
    constexpr int kDual = INV ? COL_DERIV : COL_FOLD;
    cudaError_t e = cudaSuccess, r;
    if ((r = set_max_smem(dftk::k_colfft<Real, INV, T, false, COL_PLAIN>)) != cudaSuccess) e = r;
    if ((r = set_max_smem(dftk::k_colfft<Real, INV, T, true, COL_PLAIN>)) != cudaSuccess) e = r;
    if ((r = set_max_smem(dftk::k_colfft<Real, INV, T, false, kDual>)) != cudaSuccess) e = r;
    if ((r = set_max_smem(dftk::k_colfft<Real, INV, T, true, kDual>)) != cudaSuccess) e = r;
    return e;
}

template <typename Real, int T>
cudaError_t launch_t(cudaStream_t st, bool inv, const GridDesc& g, const AxisPlan& pa, bool zax, int ncomp,
                     typename Cplx<Real>::type* data, int* status, const typename Cplx<Real>::type* tw,
                     long long polls, int mode, Real kf) {
    return inv ? launch_m<Real, true, T>(st, g, pa, zax, ncomp, data, status, tw, polls, mode, kf)
               : launch_m<Real, false, T>(st, g, pa, zax, ncomp, data, status, tw, polls, mode, kf);
}

template <typename Real, int T> cudaError_t init_t() {
    const cudaError_t e = init_m<Real, false, T>(), r = init_m<Real, true, T>();
    return e != cudaSuccess ? e : r;
}
}  // namespace

template <typename Real>
cudaError_t ColFft<Real>::init() {
    cudaError_t e = init_t<Real, 8>(), r = init_t<Real, 4>();
    if (r == cudaSuccess) r = init_t<Real, sizeof(Real) == 4 ? 16 : 2>();
    return e != cudaSuccess ? e : r;
}

template <typename Real>
cudaError_t ColFft<Real>::run(cudaStream_t st, bool inv, const GridDesc& g, const AxisPlan& pa, bool zax, int T,
                              int ncomp, C* data, int* status, const C* tw, long long polls, int mode, Real kf) {
    if constexpr (sizeof(Real) == 4)
        if (T >= 16) return launch_t<Real, 16>(st, inv, g, pa, zax, ncomp, data, status, tw, polls, mode, kf);
    // FP64: half-width tiles where four columns would leave SMs without a tile (4 x 4 x 512, three columns)
    if constexpr (sizeof(Real) == 8)
        if (T == 4 && ceil_div(g.nxh, 4) * (zax ? g.ny : g.nz) * ncomp * (mode == COL_PLAIN ? 1 : DFT_NZSPEC) < sm_count())
            return launch_t<Real, 2>(st, inv, g, pa, zax, ncomp, data, status, tw, polls, mode, kf);
    return T >= 8 ? launch_t<Real, 8>(st, inv, g, pa, zax, ncomp, data, status, tw, polls, mode, kf)
                  : launch_t<Real, 4>(st, inv, g, pa, zax, ncomp, data, status, tw, polls, mode, kf);
}

template struct ColFft<DFT_INST_REAL>;
