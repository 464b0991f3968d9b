// lb_prec_impl.cuh -- instantiates the kernels of one storage precision.
// Included by lb_prec_<name>.cu after defining LBGB_PREC (an LB_PREC_*
// value) and LBGB_NAME (the suffix of the launch functions).
#pragma once

#include "lb_fd.cuh"
#include "lb_fd_strip.cuh"
#include "lb_launch.h"
#include "lb_step_strip.cuh"
#include "lb_step_strip_dev.cuh"

namespace lbgb {

#define LBGB_CAT2(a, b) a##b
#define LBGB_CAT(a, b) LBGB_CAT2(a, b)

namespace {

// Everything in this anonymous namespace depends on LBGB_PREC without carrying
// it as a template argument, so it must have internal linkage: each precision
// translation unit gets its own copy (shared weak symbols would let the linker
// pick one precision's launcher for all).

// Stage count per strip width: the deepest ring that still lets two CTAs
// share an SM (228 KB of shared memory).  The 16-bit kernel also holds
// DEV_OUT_BUFS row buffers of the collided rows and a six-row psi ring.
template <int BX>
constexpr int strip_stages() {
    using C = StripCfg<LBGB_PREC>;
    constexpr int NPL = Store<LBGB_PREC>::NPLANES;
    constexpr bool DEV = Store<LBGB_PREC>::SPLIT;
    constexpr size_t stage = [] {
        if constexpr (DEV)
            return (size_t)dev_stage<BX + 2 * C::HALO>() * C::ES;
        else
            return (size_t)NPL * (BX + 2 * C::HALO) * C::ES;
    }();
    constexpr size_t ring = (size_t)(DEV ? 2 * DEV_PSI_ROWS : 8) * (BX + 2) * sizeof(typename C::real);
    constexpr size_t out = DEV ? (size_t)DEV_OUT_BUFS * NPL * BX * C::ES : 0;
    constexpr size_t budget = 110 * 1024 - 32 - (DEV ? (2 * 12 + 2) * 8 : 0);
    constexpr size_t s = (budget - ring - out) / stage;
    return s > 12 ? 12 : (int)s;
}

// 16-bit deviation storage: k_step_strip_dev; FP32 / FP64: k_step_strip.
// (TAIL: the width is not in whole 16-byte units)
template <int BX, int ST, bool EQ24, int BM, bool TAIL>
auto strip_kernel() {
    if constexpr (Store<LBGB_PREC>::SPLIT)
        return k_step_strip_dev<LBGB_PREC, BX, ST, EQ24, BM, TAIL>;
    else
        return k_step_strip<LBGB_PREC, BX, ST, EQ24, BM>;
}

template <int BX, bool EQ24, int BM, bool TAIL = false>
cudaError_t strip_launch(const StepLaunch& L) {
    if constexpr (Store<LBGB_PREC>::SPLIT && !TAIL) {
        if (dev_map_columns(L.kp.nx) != L.kp.nx) return strip_launch<BX, EQ24, BM, true>(L);
    }
    using E = typename Store<LBGB_PREC>::elem;
    constexpr int ST = strip_stages<BX>();
    static_assert(ST >= 3, "strip kernel needs at least three stages");
    constexpr bool DEV = Store<LBGB_PREC>::SPLIT;
    constexpr size_t smem = [] {
        if constexpr (DEV)
            return strip_dev_smem_bytes<LBGB_PREC, BX, ST>();
        else
            return strip_smem_bytes<LBGB_PREC, BX, ST>();
    }();
    static_assert(smem <= 110 * 1024, "two CTAs per SM");
    auto kern = strip_kernel<BX, ST, EQ24, BM, TAIL>();
    static unsigned long long configured = 0;  // per instantiation, one bit per device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !(configured >> dev & 1ULL)) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        if (dev < 64) configured |= 1ULL << dev;
    }
    const dim3 grid((L.kp.nx + BX - 1) / BX, L.nchunks);
    if constexpr (DEV) {
        if (!L.dst_map || !L.src_maps) return cudaErrorInvalidValue;  // the kernel loads and stores through them
        kern<<<grid, strip_threads<BX>(), smem, L.stream>>>(static_cast<E*>(L.dst), L.kp, L.nchunks, *L.dst_map,
                                                             *L.src_maps);
    } else {
        kern<<<grid, strip_threads<BX>(), smem, L.stream>>>(static_cast<const E*>(L.src), static_cast<E*>(L.dst),
                                                             L.kp, L.nchunks);
    }
    return cudaGetLastError();
}

template <int BX>
cudaError_t step_strip(const StepLaunch& L) {
    if (L.eq24) {
        switch (L.bmode) {
            case BETA_ZERO: return strip_launch<BX, true, BETA_ZERO>(L);
            case BETA_ONE: return strip_launch<BX, true, BETA_ONE>(L);
            default: return strip_launch<BX, true, BETA_MIXED>(L);
        }
    }
    switch (L.bmode) {
        case BETA_ZERO: return strip_launch<BX, false, BETA_ZERO>(L);
        case BETA_ONE: return strip_launch<BX, false, BETA_ONE>(L);
        default: return strip_launch<BX, false, BETA_MIXED>(L);
    }
}

}  // namespace

cudaError_t LBGB_CAT(launch_step_, LBGB_NAME)(const StepLaunch& L) {
    if (L.by != 0 || L.tile_by) return LBGB_CAT(launch_tile_, LBGB_NAME)(L);
    if (L.bx == 128) return step_strip<128>(L);
    // (LB_PREC_* are enum constants, invisible to the preprocessor)
    if constexpr (LBGB_PREC != LB_PREC_FP64) {
        if (L.bx == 256) return step_strip<256>(L);
    }
    return cudaErrorInvalidValue;
}

namespace {
int elementwise_blocks(const KParams& kp) {
    const long long n = (long long)kp.nx * kp.ny;
    long long b = (n + 255) / 256;
    return (int)(b < 152 * 16 ? (b < 1 ? 1 : b) : 152 * 16);
}
}  // namespace

cudaError_t LBGB_CAT(launch_init_, LBGB_NAME)(void* dst, const KParams& kp, const double* rho0,
                                             const double* T0, cudaStream_t st) {
    using E = typename Store<LBGB_PREC>::elem;
    k_init<LBGB_PREC><<<elementwise_blocks(kp), 256, 0, st>>>(static_cast<E*>(dst), kp, rho0, T0);
    return cudaGetLastError();
}

cudaError_t LBGB_CAT(launch_gather_, LBGB_NAME)(const void* src, const KParams& kp, double* out,
                                               cudaStream_t st) {
    using E = typename Store<LBGB_PREC>::elem;
    k_gather<LBGB_PREC><<<elementwise_blocks(kp), 256, 0, st>>>(static_cast<const E*>(src), kp, out);
    return cudaGetLastError();
}

cudaError_t LBGB_CAT(launch_scatter_, LBGB_NAME)(void* dst, const KParams& kp, const double* in,
                                                cudaStream_t st) {
    using E = typename Store<LBGB_PREC>::elem;
    k_scatter<LBGB_PREC><<<elementwise_blocks(kp), 256, 0, st>>>(static_cast<E*>(dst), kp, in);
    return cudaGetLastError();
}

// ------------------------------------------------ finite-difference T (Eqs. 26-27)
namespace {
constexpr bool kFdSupported = LBGB_PREC == LB_PREC_FP64 || LBGB_PREC == LB_PREC_FP32;

// The whole FD step on a strip context (k_fd_fused).
template <int BM>
cudaError_t fd_fused_launch(const FdLaunch& L) {
    using S = Store<LBGB_PREC>;
    using E = typename S::elem;
    using R = typename S::real;
    constexpr int BX = LBGB_PREC == LB_PREC_FP64 ? 128 : 256;
    constexpr int ST = fd_fused_stages<LBGB_PREC, BX>();
    static_assert(ST >= 3, "FD strip kernel needs at least three stages");
    constexpr size_t smem = fd_fused_smem_bytes<LBGB_PREC, BX, ST>();
    auto kern = k_fd_fused<LBGB_PREC, BX, ST, BM>;
    static unsigned long long configured = 0;  // per instantiation, one bit per device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !(configured >> dev & 1ULL)) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        if (dev < 64) configured |= 1ULL << dev;
    }
    const dim3 grid((L.kp.nx + BX - 1) / BX, L.nchunks);
    kern<<<grid, strip_threads<BX>(), smem, L.stream>>>(static_cast<const E*>(L.src), static_cast<E*>(L.dst),
                                                         static_cast<const R*>(L.T), static_cast<R*>(L.T_next),
                                                         L.kp, L.nchunks, (R)L.chi, (R)L.a);
    return cudaGetLastError();
}

}  // namespace

cudaError_t LBGB_CAT(launch_fd_step_, LBGB_NAME)(const FdLaunch& L) {
    if constexpr (!kFdSupported) {
        return cudaErrorNotSupported;
    } else {
        if (L.strip) {
            switch (L.bmode) {
                case BETA_ZERO: return fd_fused_launch<BETA_ZERO>(L);
                case BETA_ONE: return fd_fused_launch<BETA_ONE>(L);
                default: return fd_fused_launch<BETA_MIXED>(L);
            }
        }
        return LBGB_CAT(launch_fd_tile_, LBGB_NAME)(L);
    }
}

cudaError_t LBGB_CAT(launch_fd_set_T_, LBGB_NAME)(void* T, const double* T0, const KParams& kp, cudaStream_t st) {
    if constexpr (!kFdSupported) {
        return cudaErrorNotSupported;
    } else {
        using R = typename Store<LBGB_PREC>::real;
        const long long n = (long long)kp.nx * kp.ny;
        long long b = (n + 255) / 256;
        k_fd_set_T<R><<<(int)(b < 2432 ? (b < 1 ? 1 : b) : 2432), 256, 0, st>>>(static_cast<R*>(T), T0, kp);
        return cudaGetLastError();
    }
}

}  // namespace lbgb
