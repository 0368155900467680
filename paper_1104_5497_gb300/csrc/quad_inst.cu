// quad_inst.cu -- the generic quadratic-system kernels for one system size per
// compilation.  Compiled with -DNPHC_QUAD_NV=<n> (unknowns, 1 .. NPHC_QUAD_MAX_N).
#include "quad.cuh"
#include "smem_optin.h"
#include "xy_dispatch.cuh"

namespace {

template <auto Kernel>
cudaError_t persistent_grid(int block, size_t smem, int &grid) {
    int dev = 0, sms = 0, per = 0;
    cudaError_t e = allow_dynamic_smem<Kernel>(smem);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, Kernel, block, smem);
    if (e != cudaSuccess) return e;
    grid = sms * (per > 0 ? per : 1);
    return cudaSuccess;
}

}  // namespace

constexpr int QUAD_WARPS = 4;   // warps per block of the one-path-per-warp kernels

cudaError_t NPHC_CAT(launch_quad_track_n, NPHC_QUAD_NV)(const QSys &sys, const XYCtl &ctl,
                                                        const EPView &ep, const WorkList &wl,
                                                        cudaStream_t st) {
    if (ep.count <= 0) return cudaSuccess;
    const size_t smem = sizeof(cx<double>) * QuadLayout<NPHC_QUAD_NV>::TOTAL * QUAD_WARPS;
    constexpr auto k = quad_track_warp_kernel<NPHC_QUAD_NV, QUAD_WARPS>;
    int full = 0;
    cudaError_t e = persistent_grid<k>(32 * QUAD_WARPS, smem, full);
    if (e != cudaSuccess) return e;
    const int64_t need = (ep.count + QUAD_WARPS - 1) / QUAD_WARPS;   // a list is at most ep.count long
    k<<<(int)(need < full ? need : full), 32 * QUAD_WARPS, smem, st>>>(sys, ctl, ep, wl);
    nphc_launch_counter(1);
    return cudaGetLastError();
}

cudaError_t NPHC_CAT(launch_quad_refine_certify_n, NPHC_QUAD_NV)(const QSys &sys, double tol_sol,
                                                                 double refine_eps,
                                                                 int refine_iters,
                                                                 const EPView &ep, int64_t cap,
                                                                 const WorkList &wl,
                                                                 cudaStream_t st) {
    if (cap <= 0) return cudaSuccess;
    const size_t smem = sizeof(cx<double>) * QuadRefineLayout<NPHC_QUAD_NV>::TOTAL * QUAD_WARPS;
    constexpr auto k = quad_refine_warp_kernel<NPHC_QUAD_NV, QUAD_WARPS>;
    int full = 0;
    cudaError_t e = persistent_grid<k>(32 * QUAD_WARPS, smem, full);
    if (e != cudaSuccess) return e;
    const int64_t need = (cap + QUAD_WARPS - 1) / QUAD_WARPS;
    k<<<(int)(need < full ? need : full), 32 * QUAD_WARPS, smem, st>>>(sys, tol_sol, refine_eps, refine_iters,
                                                                       ep, wl);
    nphc_launch_counter(1);
    return cudaGetLastError();
}

cudaError_t NPHC_CAT(launch_quad_cauchy_n, NPHC_QUAD_NV)(const QSys &sys, const EGCtl &ctl,
                                                         const EPView &ep, const WorkList &wl,
                                                         int32_t *cyc, int32_t *egst,
                                                         cudaStream_t st) {
    using P = QuadProblem<NPHC_QUAD_NV>;
    if (ep.count <= 0) return cudaSuccess;
    const size_t smem = track_smem_per_thread<P>() * P::BLOCK;
    constexpr auto k = quad_cauchy_kernel<NPHC_QUAD_NV>;
    int full = 0;
    cudaError_t e = persistent_grid<k>(P::BLOCK, smem, full);
    if (e != cudaSuccess) return e;
    const int64_t need = (ep.count + P::BLOCK - 1) / P::BLOCK;   // the list is at most ep.count long
    const int64_t cap = wl.state_threads / P::BLOCK;
    int64_t grid = need < full ? need : full;
    if (grid > cap) grid = cap;
    if (grid <= 0) return cudaErrorInvalidValue;
    k<<<(int)grid, P::BLOCK, smem, st>>>(sys, ctl, ep, wl, cyc, egst);
    nphc_launch_counter(1);
    return cudaGetLastError();
}
