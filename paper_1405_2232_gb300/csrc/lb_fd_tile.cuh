// lb_fd_tile.cuh -- the finite-difference temperature treatment (Eqs. 26-27) on tiles:
// two launches per step on small lattices, in FP64, and in the cavity and channel.
//
// Both kernels have the structure of lb_step_tile.cuh: tiles of 32 columns and a height
// that balances them over the SMs, one site per thread, the ring around the tile in
// threads of its own, launched before the kernel ahead of them ends (whose outputs they
// read: grid_wait).
//  k_fd_front: rho (pulled f), T and psi of the tile and a ring of one site; force,
//   u and the f collision of the tile.  STEP stores f and writes rho^n, u^n; else the
//   moments outputs.
//  k_fd_rk2: T^{n+1} = T^n + (h1 + K(T^n + a h1))/2, h1 = K(T^n): T^n and rho^n staged
//   with a ring of two sites, h1 and the intermediate T on the tile and a ring of one,
//   then the second stage on the tile; grad(rho) is formed once for both stages.
// Per step, before (FP32: the strip kernel; FP64: a 32 x 8 front and a two-row RK2
// tile) and now: FP32 64^2 14.4 -> 4.9 us, 256^2 16.5 -> 6.2, 512^2 16.5 -> 13.5; FP64
// 64^2 67.7 -> 20.2 us, 256^2 90 -> 68.
#pragma once

#include "lb_fd.cuh"
#include "lb_step_tile.cuh"

namespace lbgb {

// Ghost value of a temperature-like field X at (rx, ry) outside the lattice
// of a cavity (walls 1) or channel (walls 2) context, from the value Xm at the
// mirror node (the clamped position): reflected about the boundary value,
// 2 T_b - Xm, across an isothermal boundary (cavity side walls; channel
// plates at T_w and inlet at T_in); Xm across an adiabatic one (cavity bottom
// and top, channel lower plate in Case B, channel outlet).  A position outside
// in both directions takes the side-wall rule in the cavity and the plate
// rule in the channel.
template <typename real>
__device__ __forceinline__ real fd_ghost(const KParams& kp, int rx, int ry, real Xm) {
    const int nx = kp.nx, ny = kp.ny;
    if (kp.walls == 1) {
        if (rx < 0) return (real)2.0 * KPR(kp, T_hot) - Xm;
        if (rx >= nx) return (real)2.0 * KPR(kp, T_cold) - Xm;
        return Xm;
    }
    if (ry < 0 || ry >= ny) {
        if (ry < 0 && kp.adiabatic_bottom) return Xm;
        return (real)2.0 * KPR(kp, T_w) - Xm;
    }
    if (rx < 0) return (real)2.0 * KPR(kp, T_in) - Xm;
    return Xm;
}

template <int PREC, int BMODE, bool STEP>
__global__ void __launch_bounds__(tile_threads(32, tile_max_by(32)))
    k_fd_front(const typename Store<PREC>::elem* src, typename Store<PREC>::elem* __restrict__ dst,
               const typename Store<PREC>::real* Tf, typename Store<PREC>::real* __restrict__ rho_n,
               typename Store<PREC>::real* __restrict__ ux_n, typename Store<PREC>::real* __restrict__ uy_n,
               double* __restrict__ m_rho, double* __restrict__ m_ux, double* __restrict__ m_uy,
               double* __restrict__ m_T, const KParams kp, int by) {
    using S = Store<PREC>;
    using real = typename S::real;
    static_assert(!S::SPLIT, "the FD treatment stores FP64 or FP32");
    constexpr int BX = 32, WX = BX + 2;
    extern __shared__ __align__(16) unsigned char tile_smem[];
    real* s_psi = reinterpret_cast<real*>(tile_smem);
    real* s_psi2 = BMODE == BETA_MIXED ? s_psi + WX * (by + 2) : s_psi;
    const int tid = threadIdx.x, nx = kp.nx, ny = kp.ny;
    const int x0 = blockIdx.x * BX, y0 = blockIdx.y * by;
    int lx, ly, flags = 0;
    tile_site<BX>(tid, by, lx, ly);
    const int W = min(BX, nx - x0), Hh = min(by, ny - y0);
    const bool need = tid - BX * by < tile_ring(BX, by) && lx <= W && ly <= Hh;
    int gx = x0 + lx, gy = y0 + ly;
    gx = kp.walls ? clampc(gx, nx) : (gx < 0 ? gx + nx : (gx >= nx ? gx - nx : gx));
    gy = kp.walls ? clampc(gy, ny) : (gy < 0 ? gy + ny : (gy >= ny ? gy - ny : gy));
    const long long off = (long long)gy * kp.pitch + gx;
    real f[9], g[9], rho = 0, T = 0;
    const int at = (ly + 1) * WX + lx + 1;
    grid_begin();
    if (need) {
        const PullAt<false> pull(kp, gx, gy);
#pragma unroll
        for (int i = 0; i < 9; ++i) f[i] = src[(size_t)i * kp.plane + (kp.walls ? (uint32_t)off : pull(i))];
        rho = f[0];
#pragma unroll
        for (int i = 1; i < 9; ++i) rho += f[i];
        T = Tf[off];
        real psi, psi2;
        site_psi_T<real, BMODE>(kp, rho, T, psi, psi2, flags);
        if (BMODE != BETA_ZERO) s_psi[at] = psi;
        if (BMODE != BETA_ONE) s_psi2[at] = psi2;
    }
    if (flags) atomicOr(kp.err, flags);
    __syncthreads();
    if (!(tid < BX * by && lx < W && ly < Hh)) return;
#pragma unroll
    for (int i = 0; i < 9; ++i) g[i] = (real)0;
    real Fx, Fy, ux, uy, Tg = 0;
    force_from_window<real, BMODE>(kp, s_psi, s_psi2, at, WX, Fx, Fy);
    if (kp.walls) Fy += -rho * KPR(kp, g_grav);  // cavity buoyancy
    // the f half of the collision; g (zero here) is not used (FP32: the fused
    // multiply-add form, as in k_fd_fused)
    collide_et<real, false, true, true>(kp, f, g, rho, (real)0, Tg, Fx, Fy, ux, uy);
    const long long c = (long long)gy * nx + gx;
    if constexpr (!STEP) {
        if (m_rho) m_rho[c] = widen(rho);
        if (m_ux) m_ux[c] = widen(ux);
        if (m_uy) m_uy[c] = widen(uy);
        if (m_T) m_T[c] = widen(T);
        return;
    }
    rho_n[c] = rho;
    ux_n[c] = ux;
    uy_n[c] = uy;
    if (!kp.walls) {
#pragma unroll
        for (int i = 0; i < 9; ++i) dst[(size_t)i * kp.plane + (uint32_t)off] = f[i];
        if (gx < kp.ghost || gx >= nx - kp.ghost) {  // periodic ghost columns (strip contexts)
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                typename S::elem* p = dst + (size_t)i * kp.plane + (uint32_t)off;
                if (gx < kp.ghost) p[nx] = f[i];
                if (gx >= nx - kp.ghost) p[-nx] = f[i];
            }
        }
        return;
    }
    // cavity and channel: push to x + e_i; bounce back from the walls and plates;
    // channel inlet: with the wall velocity; channel outlet: anti-bounce-back at
    // density 1 with the node's velocity
    const real cs2 = (real)(1.0 / 3.0);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const int xd = gx + ex(i), yd = gy + ey(i);
        typename S::elem* pfo = dst + (long long)opp(i) * kp.plane + off;
        if (xd >= 0 && xd < nx && yd >= 0 && yd < ny) {
            dst[(long long)i * kp.plane + (long long)yd * kp.pitch + xd] = f[i];
        } else if (kp.walls != 2 || yd < 0 || yd >= ny) {
            *pfo = f[i];
        } else if (xd < 0) {
            const real eu = (real)ex(i) * KPR(kp, U_in);
            *pfo = f[i] - (real)2.0 * (real)wd(i) * rho * eu / cs2;
        } else {
            const real eu = (real)ex(i) * ux + (real)ey(i) * uy;
            *pfo = -f[i] + (real)2.0 * (real)wd(i) * (real)1.0 *
                               ((real)1.0 + (real)0.5 * eu * eu / (cs2 * cs2) -
                                (real)0.5 * (ux * ux + uy * uy) / cs2);
        }
    }
}

template <typename real>
__host__ __device__ constexpr size_t fd_rk2_smem_bytes(int by) {
    return (size_t)(2 * 36 * (by + 4) + 34 * (by + 2)) * sizeof(real);
}

// T (T^n) and T_next in the context's T layout (row pitch kp.pitch; ghost columns
// written when kp.ghost), rho, ux, uy dense.  Cavity and channel: a neighbour outside
// reads the ghost of fd_ghost; rho and u the mirror node's.
template <typename real>
__global__ void __launch_bounds__(tile_threads(32, tile_max_by(32)))
    k_fd_rk2(const real* T, const real* rho, const real* ux, const real* uy,
             real* __restrict__ T_next, const KParams kp, real chi, real a, int by) {
    constexpr int BX = 32, W2 = BX + 4, W1 = BX + 2;
    extern __shared__ __align__(16) unsigned char tile_smem[];
    real* sT = reinterpret_cast<real*>(tile_smem);  // [by + 4][W2]
    real* sR = sT + W2 * (by + 4);                  // [by + 4][W2]
    real* sTs = sR + W2 * (by + 4);                 // [by + 2][W1]
    const int tid = threadIdx.x, nx = kp.nx, ny = kp.ny;
    const int x0 = blockIdx.x * BX, y0 = blockIdx.y * by;
    const bool walls = kp.walls != 0;
    const int W = min(BX, nx - x0), Hh = min(by, ny - y0);
    auto outside = [&](int rx, int ry) { return walls && (rx < 0 || rx >= nx || ry < 0 || ry >= ny); };
    int lx, ly;
    tile_site<BX>(tid, by, lx, ly);
    const bool need = tid - BX * by < tile_ring(BX, by) && lx <= W && ly <= Hh;
    const int rx = x0 + lx, ry = y0 + ly;
    grid_begin();
    for (int s = tid; s < W2 * (Hh + 4); s += (int)blockDim.x) {
        const int j = s / W2, i = s - j * W2;
        if (i >= W + 4) continue;
        const int px = x0 + i - 2, py = y0 + j - 2;
        const int gx = ringc(kp, px, nx), gy = ringc(kp, py, ny);
        const real Tv = T[(long long)gy * kp.pitch + gx];
        sT[s] = outside(px, py) ? fd_ghost<real>(kp, px, py, Tv) : Tv;
        sR[s] = rho[(long long)gy * nx + gx];
    }
    real u_x = 0, u_y = 0;
    if (need) {
        const long long c = (long long)ringc(kp, ry, ny) * nx + ringc(kp, rx, nx);
        u_x = ux[c];
        u_y = uy[c];
    }
    __syncthreads();
    // stage 1 on the tile and its ring (a ghost site's intermediate T is filled below)
    const int c2 = (ly + 2) * W2 + lx + 2, c1 = (ly + 1) * W1 + lx + 1;
    const bool ghost = need && outside(rx, ry);
    real h1 = 0, ga = 0, gb = 0;  // FP64: grad(rho); FP32: chi grad(rho)/rho - u
    if (need && !ghost) {
        if constexpr (sizeof(real) == 8) {
            real X[9], R[9];
            fd_window(sT + c2 - W2, sT + c2, sT + c2 + W2, X);
            fd_window(sR + c2 - W2, sR + c2, sR + c2 + W2, R);
            fd_grad_fp64(R, ga, gb);
            h1 = fd_K_fp64(X, ga, gb, R[0], u_x, u_y, chi);
        } else {
            fd_a_rows(sR + c2 - W2, sR + c2, sR + c2 + W2, u_x, u_y, chi, ga, gb);
            h1 = fd_K_rows_a(sT + c2 - W2, sT + c2, sT + c2 + W2, ga, gb, chi);
        }
        sTs[c1] = sT[c2] + a * h1;
    }
    __syncthreads();
    if (walls) {
        // ghost sites of the ring, by the same rule from their mirror node
        if (ghost) {
            const int mx = clampc(rx, nx) - x0 + 1, my = clampc(ry, ny) - y0 + 1;
            sTs[c1] = fd_ghost<real>(kp, rx, ry, sTs[my * W1 + mx]);
        }
        __syncthreads();
    }
    // stage 2 on the tile: T^{n+1} = T^n + (h1 + K(Ts)) / 2
    if (!(tid < BX * by && lx < W && ly < Hh)) return;
    real K;
    if constexpr (sizeof(real) == 8) {
        real X[9];
        fd_window(sTs + c1 - W1, sTs + c1, sTs + c1 + W1, X);
        K = fd_K_fp64(X, ga, gb, sR[c2], u_x, u_y, chi);
    } else {
        K = fd_K_rows_a(sTs + c1 - W1, sTs + c1, sTs + c1 + W1, ga, gb, chi);
    }
    const real v = sT[c2] + (real)0.5 * (h1 + K);
    real* p = T_next + (long long)ry * kp.pitch + rx;
    *p = v;
    if (rx < kp.ghost) p[nx] = v;
    if (rx >= nx - kp.ghost) p[-nx] = v;
    if (!finite_bits(v)) atomicOr(kp.err, 1 << LB_ERR_NONFINITE);
}

}  // namespace lbgb
