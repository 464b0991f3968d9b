// lb_tile_impl.cuh -- instantiates the tile kernels (lb_step_tile.cuh) of one
// storage precision.  Included by lb_tile_<name>.cu after defining LBGB_PREC
// (an LB_PREC_* value) and LBGB_NAME (the suffix of the launch functions); with
// LBGB_BATCH also the batched tile step.  A unit
// of its own: a thread of these kernels has one site, so the parameters are read
// as float copies (LB_KP_FLOAT) where the strip kernels convert the doubles once
// per chunk of rows.
#pragma once

#include <atomic>

#include "lb_fd_tile.cuh"
#include "lb_launch.h"
#include "lb_step_cluster.cuh"
#include "lb_step_tile.cuh"

namespace lbgb {

#define LBGB_CAT2(a, b) a##b
#define LBGB_CAT(a, b) LBGB_CAT2(a, b)

namespace {  // (see lb_prec_impl.cuh: depends on LBGB_PREC, internal linkage)

template <int BX, int WALLS>
auto tile_kernel(const StepLaunch& L) -> void (*)(const typename Store<LBGB_PREC>::elem*,
                                                   typename Store<LBGB_PREC>::elem*, const KParams, int) {
    if (L.eq24) {
        if (L.bmode == BETA_ZERO) return k_step_tile<LBGB_PREC, BX, WALLS, true, BETA_ZERO>;
        if (L.bmode == BETA_ONE) return k_step_tile<LBGB_PREC, BX, WALLS, true, BETA_ONE>;
        return k_step_tile<LBGB_PREC, BX, WALLS, true, BETA_MIXED>;
    }
    if (L.bmode == BETA_ZERO) return k_step_tile<LBGB_PREC, BX, WALLS, false, BETA_ZERO>;
    if (L.bmode == BETA_ONE) return k_step_tile<LBGB_PREC, BX, WALLS, false, BETA_ONE>;
    return k_step_tile<LBGB_PREC, BX, WALLS, false, BETA_MIXED>;
}

// Dynamic shared memory of a launch of `tiles` blocks: what the psi window needs,
// or more where at most eight blocks run per SM, so that no SM takes more than
// ceil(tiles / SMs) of them.  The blocks of a step are dispatched while the step
// before it still runs, and an SM that happens to be free then would take several,
// which keeps the next steps unbalanced as well (FP64 150 x 150 cavity, 150 tiles of
// five rows: 32.4 us per step without, 19.0 us with).
size_t tile_smem(int sms, long long tiles, size_t need) {
    const long long k = (tiles + sms - 1) / sms;
    if (k > 8) return need;
    const size_t pad = TILE_SM_SMEM / (size_t)(k + 1);  // k + 1 blocks (and 1 KB each) do not fit
    return pad > need ? pad : need;
}

// Lets a kernel have the padded size; once per kernel (`done`) and device.
template <class K>
cudaError_t opt_in_smem(std::atomic<unsigned long long>& done, K kern) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 64 && (done.load() >> dev & 1ULL)) return cudaSuccess;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(TILE_SM_SMEM / 2));
    if (e == cudaSuccess && dev < 64) done.fetch_or(1ULL << dev);
    return e;
}

template <int BX, int WALLS>
cudaError_t step_tile(const StepLaunch& L, int by) {
    using E = typename Store<LBGB_PREC>::elem;
    auto kern = tile_kernel<BX, WALLS>(L);
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((L.kp.nx + BX - 1) / BX, (L.kp.ny - 2 * L.kp.halo_rows + by - 1) / by);
    cfg.blockDim = dim3(tile_threads(BX, by));
    cfg.dynamicSmemBytes = tile_smem(L.sms, (long long)cfg.gridDim.x * cfg.gridDim.y,
                                     L.bmode == BETA_MIXED ? tile_smem_bytes<LBGB_PREC, BETA_MIXED>(BX, by)
                                                           : tile_smem_bytes<LBGB_PREC, BETA_ONE>(BX, by));
    cfg.stream = L.stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    if (cfg.dynamicSmemBytes > 48 * 1024) {
        static std::atomic<unsigned long long> configured[6];
        cudaError_t e = opt_in_smem(configured[(L.eq24 ? 3 : 0) + L.bmode], kern);
        if (e != cudaSuccess) return e;
    }
    return launch_kernel(cfg, kern, static_cast<const E*>(L.src), static_cast<E*>(L.dst), L.kp, by);
}

}  // namespace

cudaError_t LBGB_CAT(launch_tile_, LBGB_NAME)(const StepLaunch& L) {
    if (L.kp.walls) {
        if constexpr (LBGB_PREC == LB_PREC_FP64 || LBGB_PREC == LB_PREC_FP32) {
            if (L.kp.walls == LB_WALLS_CAVITY) return step_tile<32, LB_WALLS_CAVITY>(L, L.tile_by);
            return step_tile<32, LB_WALLS_CHANNEL>(L, L.tile_by);
        }
        return cudaErrorNotSupported;
    }
    if (L.by == 0) return step_tile<32, 0>(L, L.tile_by);
    if (L.bx == 32 && (L.by == 8 || L.by == 16)) return step_tile<32, 0>(L, L.by);
    if (L.bx == 64 && L.by == 4) return step_tile<64, 0>(L, L.by);
    return cudaErrorInvalidValue;
}

// `steps` steps of a tiny lattice in one cluster (see lb_step_cluster.cuh); steps = 0
// only asks whether the device can hold such a cluster.
cudaError_t LBGB_CAT(launch_cluster_, LBGB_NAME)(const StepLaunch& L, int steps) {
    if constexpr (LBGB_PREC == LB_PREC_FP64) {
        return cudaErrorNotSupported;
    } else {
        using E = typename Store<LBGB_PREC>::elem;
        const int nc = cluster_blocks(L.kp.nx, L.kp.ny);
        if (!nc || L.kp.walls || L.kp.halo_rows) return cudaErrorInvalidValue;
        void (*kern)(const E*, E*, const KParams, int);
        if (L.eq24)
            kern = L.bmode == BETA_ZERO  ? k_steps_cluster<LBGB_PREC, true, BETA_ZERO>
                   : L.bmode == BETA_ONE ? k_steps_cluster<LBGB_PREC, true, BETA_ONE>
                                         : k_steps_cluster<LBGB_PREC, true, BETA_MIXED>;
        else
            kern = L.bmode == BETA_ZERO  ? k_steps_cluster<LBGB_PREC, false, BETA_ZERO>
                   : L.bmode == BETA_ONE ? k_steps_cluster<LBGB_PREC, false, BETA_ONE>
                                         : k_steps_cluster<LBGB_PREC, false, BETA_MIXED>;
        // opt in once per kernel and device: 16 blocks and the largest bands
        static std::atomic<unsigned long long> configured[6];
        auto& done = configured[(L.eq24 ? 3 : 0) + L.bmode];
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev >= 64 || !(done.load() >> dev & 1ULL)) {
            e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
            if (e != cudaSuccess) return e;
            if (dev < 64) done.fetch_or(1ULL << dev);
        }
        const int rows = (L.kp.ny + nc - 1) / nc;
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = (unsigned)nc;
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)nc);
        cfg.blockDim = dim3((unsigned)((L.kp.nx * (rows + 2) + 31) / 32 * 32));
        cfg.dynamicSmemBytes = L.bmode == BETA_MIXED ? cluster_smem_bytes<LBGB_PREC, BETA_MIXED>(L.kp.nx, rows)
                                                     : cluster_smem_bytes<LBGB_PREC, BETA_ONE>(L.kp.nx, rows);
        cfg.stream = L.stream;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        if (steps == 0) {
            int clusters = 0;
            e = cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg);
            return e == cudaSuccess && clusters == 0 ? cudaErrorNotSupported : e;
        }
        return launch_kernel(cfg, kern, static_cast<const E*>(L.src), static_cast<E*>(L.dst), L.kp, steps);
    }
}

#ifdef LBGB_BATCH
namespace {
auto batch_tile_kernel(int eq24, int bmode)
    -> void (*)(const typename Store<LBGB_PREC>::elem*, typename Store<LBGB_PREC>::elem*, const BatchDomain*,
                const BatchStepTile*, const int*, int) {
    if (eq24) {
        if (bmode == BETA_ZERO) return k_batch_tile<LBGB_PREC, true, BETA_ZERO>;
        if (bmode == BETA_ONE) return k_batch_tile<LBGB_PREC, true, BETA_ONE>;
        return k_batch_tile<LBGB_PREC, true, BETA_MIXED>;
    }
    if (bmode == BETA_ZERO) return k_batch_tile<LBGB_PREC, false, BETA_ZERO>;
    if (bmode == BETA_ONE) return k_batch_tile<LBGB_PREC, false, BETA_ONE>;
    return k_batch_tile<LBGB_PREC, false, BETA_MIXED>;
}
}  // namespace

cudaError_t LBGB_CAT(launch_batch_tile_, LBGB_NAME)(const BatchTileLaunch& L) {
    using E = typename Store<LBGB_PREC>::elem;
    auto kern = batch_tile_kernel(L.eq24, L.bmode);
    if (!L.src) {
        static std::atomic<unsigned long long> configured[6];
        return opt_in_smem(configured[(L.eq24 ? 3 : 0) + L.bmode], kern);
    }
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(L.grid);
    cfg.blockDim = dim3(tile_threads(32, L.by));
    cfg.dynamicSmemBytes = tile_smem(L.sms, L.grid, L.bmode == BETA_MIXED
                                                        ? tile_smem_bytes<LBGB_PREC, BETA_MIXED>(32, L.by)
                                                        : tile_smem_bytes<LBGB_PREC, BETA_ONE>(32, L.by));
    cfg.stream = L.stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return launch_kernel(cfg, kern, static_cast<const E*>(L.src), static_cast<E*>(L.dst), L.doms, L.tiles,
                         L.n_tiles, L.by);
}
#endif

// ------------------------------------------------ finite-difference T (Eqs. 26-27)
namespace {
constexpr bool kFdTile = LBGB_PREC == LB_PREC_FP64 || LBGB_PREC == LB_PREC_FP32;

// Launch over the lattice's 32-column tiles, programmatic and evenly shared (tile_smem).
template <class K, class... A>
cudaError_t fd_launch(std::atomic<unsigned long long>& done, const FdLaunch& L, size_t need, K kern, A... args) {
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((L.kp.nx + 31) / 32, (L.kp.ny + L.tile_by - 1) / L.tile_by);
    cfg.blockDim = dim3(tile_threads(32, L.tile_by));
    cfg.dynamicSmemBytes = tile_smem(L.sms, (long long)cfg.gridDim.x * cfg.gridDim.y, need);
    cfg.stream = L.stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    if (cfg.dynamicSmemBytes > 48 * 1024) {
        cudaError_t e = opt_in_smem(done, kern);
        if (e != cudaSuccess) return e;
    }
    return launch_kernel(cfg, kern, args...);
}

template <int BM, bool STEP>
cudaError_t fd_front(const FdLaunch& L) {
    using E = typename Store<LBGB_PREC>::elem;
    using R = typename Store<LBGB_PREC>::real;
    static std::atomic<unsigned long long> done;
    return fd_launch(done, L, tile_smem_bytes<LBGB_PREC, BM>(32, L.tile_by), k_fd_front<LBGB_PREC, BM, STEP>,
                     static_cast<const E*>(L.src), static_cast<E*>(L.dst), static_cast<const R*>(L.T),
                     static_cast<R*>(L.rho), static_cast<R*>(L.ux), static_cast<R*>(L.uy), L.m_rho, L.m_ux, L.m_uy,
                     L.m_T, L.kp, L.tile_by);
}
template <bool STEP>
cudaError_t fd_front(const FdLaunch& L) {
    if (L.bmode == BETA_ZERO) return fd_front<BETA_ZERO, STEP>(L);
    if (L.bmode == BETA_ONE) return fd_front<BETA_ONE, STEP>(L);
    return fd_front<BETA_MIXED, STEP>(L);
}
}  // namespace

cudaError_t LBGB_CAT(launch_fd_tile_, LBGB_NAME)(const FdLaunch& L) {
    if constexpr (!kFdTile) {
        return cudaErrorNotSupported;
    } else {
        using R = typename Store<LBGB_PREC>::real;
        const cudaError_t e = fd_front<true>(L);
        if (e != cudaSuccess) return e;
        static std::atomic<unsigned long long> done;
        return fd_launch(done, L, fd_rk2_smem_bytes<R>(L.tile_by), k_fd_rk2<R>, static_cast<const R*>(L.T),
                         static_cast<const R*>(L.rho), static_cast<const R*>(L.ux), static_cast<const R*>(L.uy),
                         static_cast<R*>(L.T_next), L.kp, (R)L.chi, (R)L.a, L.tile_by);
    }
}

cudaError_t LBGB_CAT(launch_fd_moments_, LBGB_NAME)(const FdLaunch& L) {
    if constexpr (!kFdTile)
        return cudaErrorNotSupported;
    else
        return fd_front<false>(L);
}

namespace {
template <int BM, bool PART>
void moments(const MomentsLaunch& L, dim3 grid) {
    using E = typename Store<LBGB_PREC>::elem;
    k_moments<LBGB_PREC, BM, PART><<<grid, tile_threads(MOM_BX, MOM_BY), 0, L.stream>>>(
        static_cast<const E*>(L.src), L.kp, L.rho, L.ux, L.uy, L.T, L.ref_rho, L.ref_T, L.part);
}
}  // namespace

cudaError_t LBGB_CAT(launch_moments_, LBGB_NAME)(const MomentsLaunch& L) {
    static_assert(MOM_BX == 32 && MOM_BY == 8, "the tile of k_moments");
    const dim3 grid((L.kp.nx + MOM_BX - 1) / MOM_BX, (L.kp.ny + MOM_BY - 1) / MOM_BY);
    if (L.bmode == BETA_ZERO)
        L.part ? moments<BETA_ZERO, true>(L, grid) : moments<BETA_ZERO, false>(L, grid);
    else if (L.bmode == BETA_ONE)
        L.part ? moments<BETA_ONE, true>(L, grid) : moments<BETA_ONE, false>(L, grid);
    else
        L.part ? moments<BETA_MIXED, true>(L, grid) : moments<BETA_MIXED, false>(L, grid);
    return cudaGetLastError();
}

}  // namespace lbgb
