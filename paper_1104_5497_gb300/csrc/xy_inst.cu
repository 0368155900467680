// xy_inst.cu -- one ring size of one kernel family per compilation, so that the build
// compiles the heavily unrolled kernels in parallel.  Compiled with
//   -DNPHC_INST_M=<M>  (free sites, N = M + 1)
//   -DNPHC_INST_KIND=0 (FP32 tracker), 1 (FP64 tracker), 2 (FP64 refinement,
//   certification, classification, adjoint) or 3 (Cauchy endgame)
#include <algorithm>

#include "smem_optin.h"
#include "xy_dispatch.cuh"

#if NPHC_INST_KIND == 3
#include "cauchy_warp.cuh"

// one path per warp, 4 warps per block
cudaError_t NPHC_CAT(launch_xy_cauchy_m, NPHC_INST_M)(const XYSys &sys, const EGCtl &ctl,
                                                      const EPView &ep, const WorkList &wl,
                                                      int32_t *cyc, int32_t *egst,
                                                      cudaStream_t st) {
    constexpr int M = NPHC_INST_M, WARPS = 4;
    if (ep.count <= 0) return cudaSuccess;
    const size_t smem = cauchy_warp_smem_per_warp<M>() * WARPS;
    constexpr auto k = xy_cauchy_warp_kernel<M, WARPS>;
    int dev = 0, sms = 0, per = 0;
    cudaError_t e = allow_dynamic_smem<k>(smem);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, 32 * WARPS, smem);
    if (e != cudaSuccess) return e;
    const int64_t full = (int64_t)sms * (per > 0 ? per : 1);
    const int64_t need = (ep.count + WARPS - 1) / WARPS;   // the list is at most ep.count long
    const int grid = (int)(need < full ? need : full);
    k<<<grid, 32 * WARPS, smem, st>>>(sys, ctl, ep, wl, cyc, egst);
    nphc_launch_counter(1);
    return cudaGetLastError();
}
#endif

#if NPHC_INST_KIND == 0 || NPHC_INST_KIND == 1
#include "xy_track.cuh"

// The per-thread tracker (xy_track.cuh) over the list or every entry of the launch.
template <int M, class R>
static cudaError_t launch_per_thread(const XYSys &sys, const XYCtl &ctl, const EPView &ep,
                                     const WorkList &wl, int grid, int64_t min_paths, cudaStream_t st) {
    constexpr int BLK = NPHC_TRACK_BLOCK;
    const size_t smem = xy_smem_per_thread<M, R>() * BLK;
    constexpr auto k = xy_track_kernel<M, R, BLK>;
    int dev = 0, sms = 0, per = 0;
    cudaError_t e = allow_dynamic_smem<k>(smem);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, BLK, smem);
    if (e != cudaSuccess) return e;
    const int full = sms * (per > 0 ? per : 1);   // persistent grid: every SM filled
    if (grid <= 0 || grid > full) grid = full;
    const int cap = (int)(wl.state_threads / BLK);  // the scratch holds state for this many
    if (grid > cap) grid = cap;
    if (grid <= 0) return cudaErrorInvalidValue;
    k<<<grid, BLK, smem, st>>>(sys, ctl, ep, wl, min_paths);
    nphc_launch_counter(1);
    return cudaGetLastError();
}
#endif

#if NPHC_INST_KIND == 0
#include "xy_track_group.cuh"
#include "xy_track_lane.cuh"
#include "xy_track_warp32.cuh"

static cudaError_t device_sms(int &sms) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return e;
}

cudaError_t NPHC_CAT(launch_xy_track_f32t_m, NPHC_INST_M)(const XYSys &sys, const XYCtl &ctl,
                                                          const EPView &ep, const WorkList &wl,
                                                          int grid, int64_t min_paths,
                                                          cudaStream_t st) {
    if (ep.count < min_paths) return cudaSuccess;   // a list is at most ep.count long
    return launch_per_thread<NPHC_INST_M, float>(sys, ctl, ep, wl, grid, min_paths, st);
}

// one path per warp, 4 warps per block
cudaError_t NPHC_CAT(launch_xy_track_f32w_m, NPHC_INST_M)(const XYSys &sys, const XYCtl &ctl,
                                                          const EPView &ep, const WorkList &wl,
                                                          int64_t max_paths, cudaStream_t st) {
    constexpr int M = NPHC_INST_M, WARPS = 4;
    if (ep.count <= 0) return cudaSuccess;
    constexpr auto k = xy_track_warp32_kernel<M, WARPS>;
    int sms = 0, per = 0;
    cudaError_t e = device_sms(sms);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, 32 * WARPS, 0);
    if (e != cudaSuccess) return e;
    const int64_t full = (int64_t)sms * std::max(per, 1);
    const int64_t need = (std::min(ep.count, max_paths) + WARPS - 1) / WARPS;
    k<<<(int)std::min(full, need), 32 * WARPS, 0, st>>>(sys, ctl, ep, wl, max_paths);
    nphc_launch_counter(1);
    return cudaGetLastError();
}

cudaError_t NPHC_CAT(launch_xy_track_far_batch_m, NPHC_INST_M)(const BatchGroup &bg, const XYCtl &ctl,
                                                               cudaStream_t st) {
    constexpr int M = NPHC_INST_M, WARPS = 4;
    if (bg.total <= 0) return cudaSuccess;
    far_list_batch_kernel<M><<<(int)((bg.total + 127) / 128), 128, 0, st>>>(bg.sys, bg.ep, bg.off, bg.n, bg.far + 1,
                                                                            bg.far);
    nphc_launch_counter(1);
    cudaError_t e = cudaGetLastError();
    constexpr auto k = xy_track_warp32_batch_kernel<M, WARPS>;
    int sms = 0, per = 0;
    if (e == cudaSuccess) e = device_sms(sms);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, 32 * WARPS, 0);
    if (e != cudaSuccess) return e;
    const int64_t full = (int64_t)sms * std::max(per, 1), need = (bg.total + WARPS - 1) / WARPS;
    k<<<(int)std::min(full, need), 32 * WARPS, 0, st>>>(bg.sys, bg.ep, bg.off, bg.n, ctl, bg.far + 1, bg.far,
                                                        bg.far_queue);
    nphc_launch_counter(1);
    return cudaGetLastError();
}

// The FP32 pass has two kernels: one path per thread (xy_track_lane.cuh) and four lanes per path
// (xy_track_group.cuh).  The first takes fewer instructions per path but one wave of it (38,912 paths
// up to M = 8, where registers hold it to eight warps per SM, 34,048 at M = 9, 29,184 at M = 10)
// takes its paths' latency however few they are; four lanes shorten every solve, and eight (M = 12)
// to fourteen warps per SM hide each other's latency better than six to eight, at the price of
// the rows that pad M to a multiple of four.  Measured (GB300, FP32 pass alone or the whole batch,
// group / lane, ms; in brackets the waves of lanes; M >= 11 before it lost its lane kernel):
//   no padding    N = 9 65,536 (1.7) 12.5 / 16.9, batches of 262,144 (6.7) 62 / 67, 524,288 (13.5) 184 / 168;
//                 N = 13 262,144 (13.5) 126 / 186
//   one row       N = 8 batches of 65,536 (1.7) 17.4 / 18.8, 196,608 (5.1) 61.4 / 59.6, 393,216 (10.1)
//                 123 / 119; N = 12 262,144 (10.8) 114 / 133
//   two rows      N = 7 batch of 163,840 (4.2) 46.1 / 47.5; N = 11 65,536 (2.2) 26.7 / 29.9, 131,072 (4.5)
//                 49.6 / 50.6, 262,144 (9.0) 95.3 / 93.3
//   three rows    N = 10 20,000 (0.6) 10.5 / 13.7, 32,768 (1.0) 14.2 / 14.0, 65,536 (1.9) 25.1 / 22.8,
//                 262,144 (7.7) 96 / 73; N = 6 batch of 131,072 (3.4) 76.5 / 74.4
// So lanes from that many waves on, by the number of padding rows, and never at M >= 11 (five
// and four warps per SM): LANE_MAX_M.  One ring has at most 4^M paths, less than the line's waves up
// to M = 8: only batches run the per-thread kernel there.
constexpr int LANE_MAX_M = 10, LANE_MIN_M_SINGLE = 9;
template <int M, bool BATCH>
constexpr bool has_lanes = M <= LANE_MAX_M && (BATCH || M >= LANE_MIN_M_SINGLE);
template <int M, bool BATCH>
static bool use_group(int64_t items, int64_t wave) {
    constexpr int waves[4] = {8, 4, 6, 1};
    return !has_lanes<M, BATCH> || items < waves[GrpLayout<M>::ROWS - M] * wave;
}

// Shared memory opt-in and resident blocks per SM of a kernel.
template <auto Kernel>
static cudaError_t kernel_blocks(int threads, size_t smem, int &per) {
    cudaError_t e = allow_dynamic_smem<Kernel>(smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, Kernel, threads, smem);
    per = std::max(per, 1);
    return e;
}

// The per-thread kernel where it exists: resident blocks per SM, and the launches.
template <int M, bool BATCH>
static cudaError_t lane_blocks(int &per) {
    per = 0;
    if constexpr (has_lanes<M, BATCH>) {
        const size_t smem = lane_smem_per_block<M>(BATCH);
        if constexpr (BATCH) return kernel_blocks<xy_track_lane_batch_kernel<M>>(NPHC_TRACK_BLOCK, smem, per);
        else return kernel_blocks<xy_track_lane_kernel<M>>(NPHC_TRACK_BLOCK, smem, per);
    }
    return cudaSuccess;
}
template <int M>
static void launch_lanes(int grid, const XYSys &sys, const XYCtl &ctl, const EPView &ep, const WorkList &wl,
                         cudaStream_t st) {
    if constexpr (has_lanes<M, false>)
        xy_track_lane_kernel<M><<<grid, NPHC_TRACK_BLOCK, lane_smem_per_block<M>(false), st>>>(sys, ctl, ep, wl);
}
template <int M>
static void launch_lanes_batch(int grid, const BatchGroup &bg, const XYCtl &ctl, const WorkList &wl, cudaStream_t st) {
    if constexpr (has_lanes<M, true>)
        xy_track_lane_batch_kernel<M><<<grid, NPHC_TRACK_BLOCK, lane_smem_per_block<M>(true), st>>>(
            bg.sys, bg.ep, bg.off, bg.n, ctl, wl);
}

// Grid of a group launch over `items` paths: every SM filled (or with `warps` warps in all, if
// given), but no more blocks than the paths need at one warp per scheduler first and eight
// paths per warp then.
static int group_grid(int sms, int per, int warps, int64_t items, int64_t state_threads) {
    int64_t full = (int64_t)sms * per;
    if (warps > 0) full = std::min<int64_t>(full, (warps + GRP_WARPS - 1) / GRP_WARPS);
    const int64_t one = (int64_t)sms * GRP_WARPS;
    const int64_t paths = std::min<int64_t>(std::max<int64_t>((items + one - 1) / one, 1), GRP_PATHS);
    const int64_t need = std::max<int64_t>((items + paths * GRP_WARPS - 1) / (paths * GRP_WARPS), 1);
    const int64_t cap = state_threads / (32 * GRP_WARPS);   // its checkpoints live in the scratch
    return (int)std::min(std::min(full, need), cap);
}

cudaError_t NPHC_CAT(launch_xy_track_f32_m, NPHC_INST_M)(const XYSys &sys, const XYCtl &ctl,
                                                         const EPView &ep, const WorkList &wl,
                                                         int grid, cudaStream_t st) {
    constexpr int M = NPHC_INST_M, BLK = NPHC_TRACK_BLOCK;
    const size_t smem_g = grp_smem_per_block<M>(false);
    constexpr auto kg = xy_track_group_kernel<M>;
    int sms = 0, per_t = 0, per_g = 0;
    cudaError_t e = device_sms(sms);
    if (e == cudaSuccess) e = lane_blocks<M, false>(per_t);
    if (e == cudaSuccess) e = kernel_blocks<kg>(32 * GRP_WARPS, smem_g, per_g);
    if (e != cudaSuccess) return e;
    if (use_group<M, false>(ep.count, (int64_t)sms * per_t * BLK)) {
        const int gg = group_grid(sms, per_g, grid, ep.count, wl.state_threads);
        if (gg <= 0) return cudaErrorInvalidValue;
        kg<<<gg, 32 * GRP_WARPS, smem_g, st>>>(sys, ctl, ep, wl);
    } else {
        const int full = sms * per_t;   // persistent grid: every SM filled
        if (grid <= 0 || grid > full) grid = full;
        grid = std::min(grid, (int)(wl.state_threads / BLK));   // the scratch holds state for this many
        if (grid <= 0) return cudaErrorInvalidValue;
        launch_lanes<M>(grid, sys, ctl, ep, wl, st);
    }
    nphc_launch_counter(1);
    return cudaGetLastError();
}

// The FP32 pass of a batch group: one persistent grid over every path of the group's
// instances (one queue), at most every SM filled.
cudaError_t NPHC_CAT(launch_xy_track_f32_batch_m, NPHC_INST_M)(const BatchGroup &bg,
                                                               const XYCtl &ctl,
                                                               const WorkList &wl, int grid,
                                                               cudaStream_t st) {
    constexpr int M = NPHC_INST_M, BLK = NPHC_TRACK_BLOCK;
    if (bg.total <= 0) return cudaSuccess;
    const size_t smem_g = grp_smem_per_block<M>(true);
    constexpr auto kg = xy_track_group_batch_kernel<M>;
    int sms = 0, per_t = 0, per_g = 0;
    cudaError_t e = device_sms(sms);
    if (e == cudaSuccess) e = lane_blocks<M, true>(per_t);
    if (e == cudaSuccess) e = kernel_blocks<kg>(32 * GRP_WARPS, smem_g, per_g);
    if (e != cudaSuccess) return e;
    if (use_group<M, true>(bg.total, (int64_t)sms * per_t * BLK)) {
        const int gg = group_grid(sms, per_g, grid, bg.total, wl.state_threads);
        if (gg <= 0) return cudaErrorInvalidValue;
        kg<<<gg, 32 * GRP_WARPS, smem_g, st>>>(bg.sys, bg.ep, bg.off, bg.n, ctl, wl);
    } else {
        const int full = sms * per_t;
        if (grid <= 0 || grid > full) grid = full;
        const int64_t need = (bg.total + BLK - 1) / BLK;   // no more threads than paths
        if (grid > need) grid = (int)need;
        grid = std::min(grid, (int)(wl.state_threads / BLK));
        if (grid <= 0) return cudaErrorInvalidValue;
        launch_lanes_batch<M>(grid, bg, ctl, wl, st);
    }
    nphc_launch_counter(1);
    return cudaGetLastError();
}
#endif

#if NPHC_INST_KIND == 1
#include "xy_track_group64.cuh"

// one path per warp (short FP64 lists), 4 warps per block, blocks_per_sm blocks per SM
// (0: two)
cudaError_t NPHC_CAT(launch_xy_track_f64w_m, NPHC_INST_M)(const XYSys &sys, const XYCtl &ctl,
                                                          const EPView &ep, const WorkList &wl,
                                                          int blocks_per_sm, int64_t max_paths,
                                                          cudaStream_t st) {
    constexpr int M = NPHC_INST_M, WARPS = 4;
    if (ep.count <= 0) return cudaSuccess;
    const size_t smem = warp_track_smem_per_warp<M>() * WARPS;
    constexpr auto k = xy_track_warp64_kernel<M, WARPS>;
    int dev = 0, sms = 0, per = 0;
    cudaError_t e = allow_dynamic_smem<k>(smem);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, 32 * WARPS, smem);
    if (e != cudaSuccess) return e;
    // by default two blocks (8 warps) per SM, each warp pulling paths until the list is
    // drained: the FP64 pipe is already busy at 8 warps, and with more warps than paths
    // each warp would take at most one path, whose SM is then chance (some SMs got twice
    // the mean and the others idled half the launch)
    const int want = blocks_per_sm > 0 ? blocks_per_sm : 2;
    const int64_t full = (int64_t)sms * (per < want ? (per > 0 ? per : 1) : want);
    // at most max_paths run here, and the list is at most ep.count long
    const int64_t most = ep.count < max_paths ? ep.count : max_paths;
    const int64_t need = (most + WARPS - 1) / WARPS;
    const int grid = (int)(need < full ? need : full);
    k<<<grid, 32 * WARPS, smem, st>>>(sys, ctl, ep, wl, max_paths);
    nphc_launch_counter(1);
    return cudaGetLastError();
}

// four lanes per path, for min_paths paths or more
#if NPHC_INST_M < NPHC_GROUP64_MIN_M
cudaError_t NPHC_CAT(launch_xy_track_f64g_m, NPHC_INST_M)(const XYSys &, const XYCtl &, const EPView &ep,
                                                          const WorkList &, int64_t min_paths, cudaStream_t) {
    return ep.count < min_paths ? cudaSuccess : cudaErrorInvalidValue;
}
#else
cudaError_t NPHC_CAT(launch_xy_track_f64g_m, NPHC_INST_M)(const XYSys &sys, const XYCtl &ctl,
                                                          const EPView &ep, const WorkList &wl,
                                                          int64_t min_paths, cudaStream_t st) {
    constexpr int M = NPHC_INST_M;
    if (ep.count <= 0 || ep.count < min_paths) return cudaSuccess;
    const size_t smem = g64_smem_per_block<M>();
    constexpr auto k = xy_track_group64_kernel<M>;
    int dev = 0, sms = 0, per = 0;
    cudaError_t e = allow_dynamic_smem<k>(smem);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, 32, smem);
    if (e != cudaSuccess) return e;
    // one or two warps on each scheduler (paths are pulled from a queue)
    const int64_t grid = (int64_t)sms * (per >= 8 ? 8 : per >= 4 ? 4 : per > 0 ? per : 1);
    k<<<(int)std::min(grid, ep.count), 32, smem, st>>>(sys, ctl, ep, wl, min_paths);
    nphc_launch_counter(1);
    return cudaGetLastError();
}
#endif

cudaError_t NPHC_CAT(launch_xy_track_f64_m, NPHC_INST_M)(const XYSys &sys, const XYCtl &ctl,
                                                         const EPView &ep, const WorkList &wl,
                                                         int grid, cudaStream_t st) {
    return launch_per_thread<NPHC_INST_M, double>(sys, ctl, ep, wl, grid, 0, st);
}
#endif

#if NPHC_INST_KIND == 2
#include "xy_refine_group.cuh"

cudaError_t NPHC_CAT(launch_xy_refine_certify_m, NPHC_INST_M)(const XYSys &sys, double tol_sol,
                                                             double refine_eps, int refine_iters,
                                                             const EPView &ep, int64_t cap,
                                                             const WorkList &wl, int shortcut,
                                                             cudaStream_t st) {
    if (cap <= 0) return cudaSuccess;
    constexpr int M = NPHC_INST_M;
    const size_t smem = rg_smem_per_block<M>();
    constexpr auto k = xy_refine_group_kernel<M>;
    int dev = 0, sms = 0, per = 0;
    cudaError_t e = allow_dynamic_smem<k>(smem);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, 32, smem);
    if (e != cudaSuccess) return e;
    // one or two warps on each of an SM's four schedulers (the FP64 pipes are per scheduler,
    // and the entries are dealt out evenly), at most one entry per warp
    const int64_t full = (int64_t)sms * (per >= 8 ? 8 : per >= 4 ? 4 : per > 0 ? per : 1);
    const int grid = (int)(cap < full ? cap : full);
    k<<<grid, 32, smem, st>>>(sys, tol_sol, refine_eps, refine_iters, ep, wl, shortcut,
                              far_exponent(refine_eps));
    nphc_launch_counter(1);
    return cudaGetLastError();
}

cudaError_t NPHC_CAT(launch_xy_adjoint_m, NPHC_INST_M)(const XYSys &sys, int64_t count,
                                                      const double *theta, const double *g_energy,
                                                      const double *g_theta, double *dJ,
                                                      cudaStream_t st) {
    if (count <= 0) return cudaSuccess;
    constexpr int M = NPHC_INST_M;
    const size_t smem = adj_smem_per_block<M>();
    constexpr auto k = xy_adjoint_kernel<M>;
    int dev = 0, sms = 0;
    cudaError_t e = allow_dynamic_smem<k>(smem);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    // a warp per scheduler (the FP64 pipe is busy with one), fewer when a warp per point is fewer
    const int64_t need = (count + ADJ_WARPS - 1) / ADJ_WARPS;
    const int grid = (int)(need < sms ? need : sms);
    k<<<grid, 32 * ADJ_WARPS, smem, st>>>(sys, count, theta, g_energy, g_theta, dJ);
    nphc_launch_counter(1);
    return cudaGetLastError();
}

cudaError_t NPHC_CAT(launch_xy_classify_m, NPHC_INST_M)(const XYSys &sys, const EPView &ep,
                                                       double *theta, int32_t *index,
                                                       double *energy, double *min_eig,
                                                       double *log_abs_det, const int32_t *list,
                                                       const int32_t *list_count,
                                                       cudaStream_t st) {
    if (ep.count <= 0) return cudaSuccess;
    constexpr int M = NPHC_INST_M;
    const size_t smem = cls_smem_per_block<M>();
    constexpr auto k = xy_classify_kernel<M>;
    int dev = 0, sms = 0;
    cudaError_t e = allow_dynamic_smem<k>(smem);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    // a warp per scheduler, at most one point per warp (a list is at most ep.count long)
    const int64_t full = (int64_t)sms * 4;
    const int grid = (int)(ep.count < full ? ep.count : full);
    k<<<grid, 32, smem, st>>>(sys, ep, theta, index, energy, min_eig, log_abs_det, list, list_count);
    nphc_launch_counter(1);
    return cudaGetLastError();
}
#endif
