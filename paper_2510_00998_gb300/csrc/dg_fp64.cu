// FP64 on the DG levels: the dispatch to the block fixed-point kernels (dg_fx.cuh)
// and the FP64 transfers of gradual p-hierarchies.
#include <array>
#include <mutex>

#include "internal.h"

#include "dg_transfer.cuh"

namespace dgmg {

namespace {

// f(FxRun<dim, q>) for the run-time (dim, q)
template <typename F>
auto fx_dispatch(int dim, int q, F f) {
    switch (dim * 16 + q) {
        case 2 * 16 + 2: return f(FxRun<2, 2>{});
        case 2 * 16 + 3: return f(FxRun<2, 3>{});
        case 2 * 16 + 4: return f(FxRun<2, 4>{});
        case 2 * 16 + 5: return f(FxRun<2, 5>{});
        case 2 * 16 + 6: return f(FxRun<2, 6>{});
        case 2 * 16 + 7: return f(FxRun<2, 7>{});
        case 3 * 16 + 2: return f(FxRun<3, 2>{});
        case 3 * 16 + 3: return f(FxRun<3, 3>{});
        case 3 * 16 + 4: return f(FxRun<3, 4>{});
        case 3 * 16 + 5: return f(FxRun<3, 5>{});
        case 3 * 16 + 6: return f(FxRun<3, 6>{});
        default: return f(FxRun<3, 7>{});
    }
}
bool fx_valid(int dim, int q) { return (dim == 2 || dim == 3) && q >= 2 && q <= QMAX; }

// Tables of the batched launches (GLL nodes, the degree's own penalty), formed
// once per degree.
const FxTab &batch_tables(int q) {
    static std::array<FxTab, QMAX + 1> tabs;
    static std::array<std::once_flag, QMAX + 1> once;
    std::call_once(once[q], [q] { fx_tables(make_refelem(q - 1), q - 1, tabs[q]); });
    return tabs[q];
}

}  // namespace

int fx_cells_per_cta(int dim, int q, int64_t ncell) {
    return fx_dispatch(dim, q, [&](auto run) { return decltype(run)::cells_per_cta(ncell); });
}

template <>
cudaError_t launch_project<double>(int dim, int q, const DGConst<double> &c, int, double *u, const double *e0,
                                   double *tr, cudaStream_t s) {
    if (!fx_valid(dim, q)) return cudaErrorInvalidValue;
    return fx_dispatch(dim, q, [&](auto run) { return decltype(run)::project(c, false, u, e0, tr, s); });
}
cudaError_t launch_project_user(int dim, int q, const DGConst<double> &c, double *u, const double *e0, double *tr,
                                cudaStream_t s) {
    if (!fx_valid(dim, q)) return cudaErrorInvalidValue;
    return fx_dispatch(dim, q, [&](auto run) { return decltype(run)::project(c, true, u, e0, tr, s); });
}

template <>
cudaError_t launch_smooth<double>(int dim, int q, const DGConst<double> &c, int, int exact, int flags, double *u,
                                  const double *b, const double *kappa, const double *fd, const double *linv,
                                  const double *tr_in, double *tr_out, cudaStream_t s) {
    if (!fx_valid(dim, q)) return cudaErrorInvalidValue;
    return fx_dispatch(dim, q, [&](auto run) {
        return decltype(run)::smooth(c, exact != 0, flags, u, b, kappa, fd, linv, tr_in, tr_out, s);
    });
}

template <>
cudaError_t launch_residual<double>(int dim, int q, const DGConst<double> &c, int, int mode, const double *u,
                                    const double *b, const double *kappa, const double *tr, double *r, double *corners,
                                    const double *, cudaStream_t s) {
    if (!fx_valid(dim, q)) return cudaErrorInvalidValue;
    return fx_dispatch(
        dim, q, [&](auto run) { return decltype(run)::residual(c, false, mode, u, b, kappa, tr, r, corners, s); });
}
cudaError_t launch_residual_user(int dim, int q, const DGConst<double> &c, int mode, const double *u, const double *b,
                                 const double *kappa, const double *tr, double *r, double *corners, cudaStream_t s) {
    if (!fx_valid(dim, q)) return cudaErrorInvalidValue;
    return fx_dispatch(
        dim, q, [&](auto run) { return decltype(run)::residual(c, true, mode, u, b, kappa, tr, r, corners, s); });
}

template <>
cudaError_t launch_project_batch<double>(int dim, int q, const BatchDG<double> *D, const BlockMap *map, int nblocks,
                                         int cpb, double *u, int with_e0, cudaStream_t s) {
    if (!fx_valid(dim, q)) return cudaErrorInvalidValue;
    return fx_dispatch(dim, q, [&](auto run) {
        return decltype(run)::project_batch(batch_tables(q), cpb, D, map, nblocks, u, with_e0, s);
    });
}
template <>
cudaError_t launch_smooth_batch<double>(int dim, int q, const BatchDG<double> *D, const BlockMap *map, int nblocks, int cpb,
                                        int exact, int flags, double *u, const double *b, int cur, cudaStream_t s) {
    if (!fx_valid(dim, q)) return cudaErrorInvalidValue;
    return fx_dispatch(dim, q, [&](auto run) {
        return decltype(run)::smooth_batch(batch_tables(q), cpb, exact != 0, D, map, nblocks, flags, u, b, cur, s);
    });
}
template <>
cudaError_t launch_residual_batch<double>(int dim, int q, const BatchDG<double> *D, const BlockMap *map, int nblocks,
                                          int cpb, int mode, const double *u, const double *b, double *r, int cur,
                                          cudaStream_t s) {
    if (!fx_valid(dim, q)) return cudaErrorInvalidValue;
    return fx_dispatch(dim, q, [&](auto run) {
        return decltype(run)::residual_batch(batch_tables(q), cpb, D, map, nblocks, mode, u, b, r, cur, s);
    });
}

template <>
cudaError_t launch_dg_transfer<double>(int dim, int qf, bool prolong, int64_t ncell, const DGInterp<double> &P,
                                       const double *in, double *out, cudaStream_t s) {
    return launch_dg_transfer_impl<double>(dim, qf, prolong, ncell, P, in, out, s);
}

}  // namespace dgmg
