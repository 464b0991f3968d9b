// lb_fd_strip.cuh -- the finite-difference temperature treatment (Eqs. 26-27)
// in one pass over HBM on strip contexts (k_fd_fused).
//
// k_fd_fused is k_step_strip (lb_step_strip.cuh) with the g populations
// replaced by the temperature field and the RK2 update of Eq. (27) folded in:
// for every pre-collision row the producer streams the 9 f plane rows and the
// row of T^n (both stored in the ghost-column layout), and the consumer warps
// run four phases on rows lagging behind the newest one, with shared-memory
// row rings for psi, rho, T^n, u^n, h1 and the intermediate T.  Per site it
// reads f and T^n and writes f and T^{n+1} once (80 B in FP32).
//
// K uses the isotropic central stencils of the D2Q9 lattice; in FP64 every
// formula is evaluated in its printed order (compiled without contraction),
// so the fused kernel and the tile kernels (lb_fd_tile.cuh) give the same bits.
#pragma once

#include "lb_fd.cuh"
#include "lb_step_strip.cuh"

namespace lbgb {

// Shared memory of k_fd_fused (elements of real unless noted):
//   stages  STAGES x 10 rows (f_0..f_8, T) x (BX + 2 FD_HALO) elements
//   psi     2 x 4 rows x (BX + 4)          columns -2..W+1
//   rho, T  2 x 8 rows x (BX + 4)          columns -2..W+1
//   u, h1, Ts  4 x 4 rows x (BX + 2)       columns -1..W
template <int PREC, int BX>
constexpr size_t fd_fused_ring_bytes() {
    using C = StripCfg<PREC>;
    return ((size_t)24 * (BX + 4) + (size_t)16 * (BX + 2)) * sizeof(typename C::real);
}
template <int PREC, int BX, int STAGES>
constexpr size_t fd_fused_smem_bytes() {
    using C = StripCfg<PREC>;
    return (size_t)STAGES * 10 * (BX + 2 * FD_HALO) * C::ES + fd_fused_ring_bytes<PREC, BX>() +
           (size_t)2 * STAGES * 8 + 16;
}
// Four stages, as the ring rows: the loop is unrolled by four, so that every stage and
// ring row is a constant offset.
template <int PREC, int BX>
constexpr int fd_fused_stages() {
    return 4;
}

// K(X) of Eq. (26) in FP64 from three row pointers (south, centre, north, each at the
// site's column) of X and of rho.
__device__ __forceinline__ double fd_K_rows(const double* Xs, const double* Xc, const double* Xn, const double* Rs,
                                            const double* Rc, const double* Rn, double ux, double uy, double chi) {
    double X[9], R[9], grx, gry;
    fd_window(Xs, Xc, Xn, X);
    fd_window(Rs, Rc, Rn, R);
    fd_grad_fp64(R, grx, gry);
    return fd_K_fp64(X, grx, gry, R[0], ux, uy, chi);
}

// One whole FD step (Eqs. 1, 26, 27) on a strip context, one pass over HBM:
// f and T^n in, f and T^{n+1} out (both in the ghost-column layout, row
// pitch kp.pitch, kp.ghost = FD_GHOST).  Job k is pre-collision row
// y_start - 2 + k (k = 0 .. rows + 3); rows k = 2 .. rows + 1 are the
// chunk's own.  Iteration j, with one named barrier between A and the rest:
//   A(j)    rho (pulled f), T^n and psi of row j, columns -2..W+1
//   B(j-1)  force and u^n of row j-1, columns -1..W (psi rows j-2..j);
//           own rows also collide f and store it (columns 0..W-1)
//   C(j-2)  stage 1: h1 = K(T^n), Ts = T^n + a h1, columns -1..W
//   D(j-4)  stage 2: T^{n+1} = T^n + (h1 + K(Ts)) / 2, own rows, columns 0..W-1
// Each phase reads only rows finished before the barrier it follows.  Column
// thread t owns column t; the halo warp takes the columns outside 0..W-1.
template <int PREC, int BX, int STAGES, int BMODE>
__global__ void __launch_bounds__(strip_threads<BX>(), 2)
    k_fd_fused(const typename Store<PREC>::elem* __restrict__ src, typename Store<PREC>::elem* __restrict__ dst,
               const typename Store<PREC>::real* __restrict__ Tn, typename Store<PREC>::real* __restrict__ Tnext,
               const KParams kp, int nchunks, typename Store<PREC>::real chi, typename Store<PREC>::real a) {
    using S = Store<PREC>;
    using C = StripCfg<PREC>;
    using elem = typename C::elem;
    using real = typename C::real;
    static_assert(sizeof(elem) == sizeof(real), "the FD treatment stores FP64 or FP32");
    constexpr int HALO = FD_HALO;
    constexpr int SEGW = BX + 2 * HALO;
    constexpr int RA = BX + 4;  // ring rows, columns -2..W+1 at index col + 2
    constexpr int RB = BX + 2;  // ring rows, columns -1..W at index col + 1
    constexpr int ES = C::ES;
    constexpr int NCW = BX / 32;
    constexpr int NP = 10;  // rows per stage: f_0..f_8, T

    extern __shared__ __align__(128) unsigned char smem_raw[];
    elem* stage = reinterpret_cast<elem*>(smem_raw);  // [STAGES][NP][SEGW]
    real* r_psi = reinterpret_cast<real*>(stage + (size_t)STAGES * NP * SEGW);  // [4][RA]
    real* r_psi2 = r_psi + 4 * RA;                                               // [4][RA]
    real* r_rho = r_psi2 + 4 * RA;                                               // [8][RA]
    real* r_T = r_rho + 8 * RA;                                                  // [8][RA]
    real* r_ux = r_T + 8 * RA;                                                   // [4][RB]
    real* r_uy = r_ux + 4 * RB;                                                  // [4][RB]
    real* r_h1 = r_uy + 4 * RB;                                                  // [4][RB]
    real* r_Ts = r_h1 + 4 * RB;                                                  // [4][RB]
    uint64_t* full = reinterpret_cast<uint64_t*>(
        (reinterpret_cast<uintptr_t>(r_Ts + 4 * RB) + 7) & ~uintptr_t(7));
    uint64_t* empty = full + STAGES;
    __shared__ int s_abort[2];  // one slot per job parity (see the loop)

    const int t = threadIdx.x;
    const int nx = kp.nx, ny = kp.ny;
    const int x0 = blockIdx.x * BX;
    const int W = min(BX, nx - x0);
    const int y_start = (int)((long long)blockIdx.y * ny / nchunks);
    const int y_end = (int)((long long)(blockIdx.y + 1) * ny / nchunks);
    const int njobs = (y_end - y_start) + 4;  // pre-collision rows y_start-2 .. y_end+1
    const uint32_t plane = (uint32_t)kp.plane, pitch = (uint32_t)kp.pitch;
    const int ghost = kp.ghost;

    if (t == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], NCW);
        }
        fence_mbar_init();
        s_abort[0] = 0;
        s_abort[1] = 0;
    }
    __syncthreads();

    if (t >= BX + 32) {
        // ------------------------------------------------ producer warp
        const int lane = t - BX - 32;
        int issued = 0;
        for (int j = 0; j < njobs; ++j) {
            const int s = j % STAGES;
            if (j >= STAGES) {
                // the warp takes one decision (its lanes poll the barrier independently)
                if (!__all_sync(0xffffffffu, mbar_wait_bounded(&empty[s], (uint32_t)(((j / STAGES) - 1) & 1),
                                                               kp.wait_cycles))) {
                    if (lane == 0) atomicOr(kp.err, 1 << LB_ERR_TIMEOUT);
                    break;
                }
            }
            int y = y_start - 2 + j;
            y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
            if (lane == 0) mbar_arrive_expect_tx(&full[s], (uint32_t)NP * strip_copy_bytes<ES, HALO>(W));
            __syncwarp();
            if (lane < NP) {
                const elem* row;
                if (lane < 9) {
                    int sy = y - ey(lane);
                    sy = sy < 0 ? sy + ny : (sy >= ny ? sy - ny : sy);
                    row = src + (size_t)((uint32_t)lane * plane + (uint32_t)sy * pitch);
                } else {
                    row = reinterpret_cast<const elem*>(Tn) + (size_t)((uint32_t)y * pitch);
                }
                bulk_copy_g2s(stage + ((size_t)s * NP + lane) * SEGW, row + (x0 - HALO),
                              strip_copy_bytes<ES, HALO>(W), &full[s]);
            }
            issued = j + 1;
        }
        if (lane == 0)
            for (int j = (issued > STAGES ? issued - STAGES : 0); j < issued; ++j)
                (void)mbar_wait_bounded(&full[j % STAGES], (uint32_t)((j / STAGES) & 1));
        return;
    }

    // ------------------------------------------ column threads and halo warp
    const bool halo = t >= BX;
    const int hl = t & 31;
    // phase A: column (-2..W+1) of this thread, or none
    const int colA = halo ? (hl < 2 ? hl - 2 : (hl < 4 ? W + hl - 2 : -99)) : (t < W ? t : -99);
    // phases B, C: column (-1..W), or none
    const int colB = halo ? (hl == 0 ? -1 : (hl == 1 ? W : -99)) : (t < W ? t : -99);
    const bool own_col = !halo && t < W;
    int flags = 0;
    bool aborted = false;
    // row r (constant relative to the group of four) of an eight-row ring: `cur` is the
    // half of rows 4 g .. 4 g + 3 of group g, `prv` the other
    static_assert(STAGES == 4, "stages and four-row rings share the unrolled index");
    uint32_t ph = 0;  // parity of "full": the group's
    real *rho_cur = r_rho, *rho_prv = r_rho + 4 * RA, *T_cur = r_T, *T_prv = r_T + 4 * RA;
    for (int jb = 0; jb < njobs + 2 && !aborted; jb += 4) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int j = jb + u;
            if (j >= njobs + 2) break;
            auto row8 = [&](real* cur, real* prv, int r) { return ((r >= 0 || r < -4) ? cur : prv) + (r & 3) * RA; };
            // A(j)
            if (j < njobs) {
                const int s = u;
                if (!mbar_wait_bounded(&full[s], ph, kp.wait_cycles)) s_abort[u & 1] = 1;
                if (colA != -99) {
                    const elem* st = stage + (size_t)s * NP * SEGW;
                    const int c = colA + HALO;
                    real f[9], psi, psi2;
#pragma unroll
                    for (int i = 0; i < 9; ++i) f[i] = S::load(st + i * SEGW + c - ex(i), (real)kp.base_f[i]);
                    real rho = f[0];
#pragma unroll
                    for (int i = 1; i < 9; ++i) rho += f[i];
                    const real T = (real)st[9 * SEGW + c];
                    site_psi_T<real, BMODE>(kp, rho, T, psi, psi2, flags);
                    const int ia = colA + 2;
                    if (BMODE != BETA_ZERO) r_psi[u * RA + ia] = psi;
                    if (BMODE != BETA_ONE) r_psi2[u * RA + ia] = psi2;
                    row8(rho_cur, rho_prv, u)[ia] = rho;
                    row8(T_cur, T_prv, u)[ia] = T;
                }
            }
            consumer_sync<BX + 32>();
            // (a thread that times out at job j + 1 writes the other slot than the
            // one read here, so every consumer leaves at the same job)
            if (s_abort[u & 1]) {
                aborted = true;
                break;
            }
            // B(k), k = j - 1: force, u; own rows: f collision and store
            {
                const int k = j - 1;
                if (k >= 1 && k <= njobs - 2 && colB != -99) {
                    const elem* st = stage + (size_t)((u + 3) & 3) * NP * SEGW;
                    const int c = colB + HALO;
                    real f[9], g[9];
#pragma unroll
                    for (int i = 0; i < 9; ++i) {
                        f[i] = S::load(st + i * SEGW + c - ex(i), (real)kp.base_f[i]);
                        g[i] = (real)0;
                    }
                    const int ia = colB + 2;
                    const real rho = row8(rho_cur, rho_prv, u - 1)[ia];
                    real Fx, Fy, ux, uy, Tg;
                    force_from_rows<real, BMODE>(
                        kp, r_psi + ((u + 2) & 3) * RA + ia, r_psi + ((u + 3) & 3) * RA + ia, r_psi + u * RA + ia,
                        r_psi2 + ((u + 2) & 3) * RA + ia, r_psi2 + ((u + 3) & 3) * RA + ia,
                        r_psi2 + u * RA + ia, Fx, Fy);
                    // the f half of the collision; g (zero here) is not used
                    // (FP32: the fused multiply-add form, faster in this kernel)
                    collide<real, false, true>(kp, f, g, rho, Fx, Fy, ux, uy, Tg);
                    if constexpr (sizeof(real) == 4) {
                        // FP32: the rings keep a = chi grad(rho) / rho - u, which
                        // both stages' K share (fd_K_rows_a)
                        real ax, ay;
                        fd_a_rows(row8(rho_cur, rho_prv, u - 2) + ia, row8(rho_cur, rho_prv, u - 1) + ia,
                                  row8(rho_cur, rho_prv, u) + ia, ux, uy, chi, ax, ay);
                        r_ux[((u + 3) & 3) * RB + colB + 1] = ax;
                        r_uy[((u + 3) & 3) * RB + colB + 1] = ay;
                    } else {
                        r_ux[((u + 3) & 3) * RB + colB + 1] = ux;
                        r_uy[((u + 3) & 3) * RB + colB + 1] = uy;
                    }
                    if (own_col && k >= 2 && k <= njobs - 3) {
                        int y = y_start - 2 + k;
                        y = y >= ny ? y - ny : y;
                        const int xg = x0 + t;
                        const uint32_t off = (uint32_t)y * pitch + (uint32_t)xg;
                        const bool ghost_lo = xg < ghost, ghost_hi = xg >= nx - ghost;
#pragma unroll
                        for (int i = 0; i < 9; ++i) S::put(dst + ((uint32_t)i * plane + off), f[i], (real)kp.base_f[i]);
                        // the periodic ghost copies: one branch per site, not per plane
                        if (ghost_lo || ghost_hi) {
#pragma unroll
                            for (int i = 0; i < 9; ++i) {
                                elem* pf = dst + ((uint32_t)i * plane + off);
                                if (ghost_lo) S::put(pf + nx, f[i], (real)kp.base_f[i]);
                                if (ghost_hi) S::put(pf - nx, f[i], (real)kp.base_f[i]);
                            }
                        }
                    }
                }
            }
            // C(k), k = j - 2: stage 1
            {
                const int k = j - 2;
                if (k >= 1 && k <= njobs - 2 && colB != -99) {
                    const int ia = colB + 2, ib = colB + 1;
                    const real* Ts_ = row8(T_cur, T_prv, u - 3) + ia;
                    const real* Tc_ = row8(T_cur, T_prv, u - 2) + ia;
                    const real* Tn_ = row8(T_cur, T_prv, u - 1) + ia;
                    real K;
                    if constexpr (sizeof(real) == 4)
                        K = fd_K_rows_a(Ts_, Tc_, Tn_, r_ux[((u + 2) & 3) * RB + ib], r_uy[((u + 2) & 3) * RB + ib],
                                        chi);
                    else
                        K = fd_K_rows(Ts_, Tc_, Tn_, row8(rho_cur, rho_prv, u - 3) + ia,
                                      row8(rho_cur, rho_prv, u - 2) + ia, row8(rho_cur, rho_prv, u - 1) + ia,
                                      r_ux[((u + 2) & 3) * RB + ib], r_uy[((u + 2) & 3) * RB + ib], chi);
                    r_h1[((u + 2) & 3) * RB + ib] = K;
                    r_Ts[((u + 2) & 3) * RB + ib] = Tc_[0] + a * K;
                }
            }
            // D(k), k = j - 4: stage 2 on own rows and columns
            {
                const int k = j - 4;
                if (k >= 2 && k <= njobs - 3 && own_col) {
                    const int ia = t + 2, ib = t + 1;
                    real K;
                    if constexpr (sizeof(real) == 4)
                        K = fd_K_rows_a(r_Ts + ((u + 3) & 3) * RB + ib, r_Ts + u * RB + ib,
                                        r_Ts + ((u + 1) & 3) * RB + ib, r_ux[u * RB + ib], r_uy[u * RB + ib],
                                        chi);
                    else
                        K = fd_K_rows(r_Ts + ((u + 3) & 3) * RB + ib, r_Ts + u * RB + ib,
                                      r_Ts + ((u + 1) & 3) * RB + ib, row8(rho_cur, rho_prv, u - 5) + ia,
                                      row8(rho_cur, rho_prv, u - 4) + ia, row8(rho_cur, rho_prv, u - 3) + ia,
                                      r_ux[u * RB + ib], r_uy[u * RB + ib], chi);
                    const real v = row8(T_cur, T_prv, u - 4)[ia] + (real)0.5 * (r_h1[u * RB + ib] + K);
                    int y = y_start - 2 + k;
                    y = y >= ny ? y - ny : y;
                    const int xg = x0 + t;
                    real* p = Tnext + (long long)y * pitch + xg;
                    *p = v;
                    if (xg < ghost) p[nx] = v;
                    if (xg >= nx - ghost) p[-nx] = v;
                    if (!isfinite(v)) flags |= 1 << LB_ERR_NONFINITE;
                }
            }
            // the stage of job j-1 has had its last reader (A at j-1, B at j)
            if (j >= 1 && j <= njobs - 1 && !halo) {
                __syncwarp();
                if ((t & 31) == 0) mbar_arrive(&empty[(u + 3) & 3]);
            }
        }
        ph ^= 1u;
        real* x = rho_cur;
        rho_cur = rho_prv;
        rho_prv = x;
        x = T_cur;
        T_cur = T_prv;
        T_prv = x;
    }
    if (aborted) {
        if (t == 0) atomicOr(kp.err, 1 << LB_ERR_TIMEOUT);
        return;
    }
    if (flags) atomicOr(kp.err, flags);
}

}  // namespace lbgb
