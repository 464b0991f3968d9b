// lb_step_tile.cuh -- the fused step on small tiles, one site per thread: the
// periodic lattice, the natural-convection cavity of Sec. III B and the plate
// channel of Sec. III A.
//
// A CTA owns a tile of BX columns and BY rows (BY chosen at launch).  Its first
// BX * BY threads each pull one site of the tile into registers and form its
// rho, sum g, T and psi; the threads after them do the same for the ring of
// one site around the tile, of which only psi is kept.  After one barrier the
// tile's threads take the force from the psi window in shared memory, collide
// the populations they still hold and store them.  A population is read
// once by its own site (and again by the ring of a neighbouring tile), rho, sum g
// and T are formed once, and no thread has two sites in a row, so the step's
// latency is that of one site.
//
// Bound: the FP64 units in FP64 (about 285 operations for the collision and 65
// for psi per site at one warp instruction per 16 cycles of an SM), where the
// launch takes the height that balances the tiles over the SMs; latency (L2, the
// barrier, the launch) in FP32 and the 16-bit modes on the small lattices this
// kernel is chosen for.  The strip kernels, which re-read and recompute less, take
// the larger lattices (default_tile_rows in lb_capi.cu has the rule).  Per step, before
// (strip kernel; cavity and channel: a tile kernel that pulled its sites twice) and now:
// FP32 64^2 14.4 -> 2.2 us, 512^2 16.4 -> 7.2 us, FP16 1016 x 765 22.6 -> 18.6 us, FP64
// 384 x 320 130 -> 91 us, 150 x 150 cavity 31 -> 19 us, 500 x 60 channel 41 -> 29 us.
//
// Walls: nx-by-ny fluid nodes inside walls half a lattice spacing outside the
// outermost nodes.  The populations are stored pre-collision at their own site and
// pushed after the collision.
//  Cavity: a population whose destination lies beyond a wall comes back to its
//   node in the opposite direction (f: bounce-back on every wall, no slip; g:
//   bounce-back on the adiabatic bottom and top walls, anti-bounce-back
//   -g*_i + 2 w_i rho c_v T_w on the isothermal side walls, the side-wall rule
//   for a link through a corner).  The buoyancy (0, -rho g) is added to the
//   pseudopotential force.
//  Channel: plate rules (f bounce-back; g anti-bounce-back at T_w, or
//   bounce-back on an adiabatic lower plate; a link through a corner takes the
//   plate rule), inlet rules (f bounce-back with the wall velocity (U_in, 0); g
//   anti-bounce-back at T_in with the symmetric equilibrium at u_in); f beyond
//   the outlet anti-bounces back at density 1 with the node's velocity, and the g
//   populations that arrive at column nx - 1 from beyond the outlet are those
//   that arrive at column nx - 2 (zero gradient), which the sites of column nx - 1
//   push: each stores them to both columns.
//  psi at a wall node is that of its nearest fluid node.  FP64: the order of
//  operations of the printed formulas.
#pragma once

#include "lb_device.cuh"
#include "lb_launch.h"

namespace lbgb {

__host__ __device__ constexpr int opp(int i) {
    return i == 0 ? 0 : (i <= 4 ? ((i + 1) % 4) + 1 : ((i - 5 + 2) % 4) + 5);
}

template <int PREC, int BMODE>
__host__ __device__ constexpr size_t tile_smem_bytes(int bx, int by) {
    return (size_t)(BMODE == BETA_MIXED ? 2 : 1) * (bx + 2) * (by + 2) * sizeof(typename Store<PREC>::real);
}

constexpr size_t TILE_SM_SMEM = 228 * 1024;  // shared memory of an SM

// Post-collision populations of fluid node (gx, gy) to the nodes they reach
// (cavity and channel).
template <class S, int WALLS, typename real>
__device__ __forceinline__ void push_walls(typename S::elem* __restrict__ dst, const KParams& kp, int gx, int gy,
                                           const real f[9], const real g[9], real rho, real ux, real uy) {
    const int nx = kp.nx, ny = kp.ny;
    const long long off = (long long)gy * kp.pitch + gx;
    const real cs2 = (real)(1.0 / 3.0);
    const bool interior = gx > 0 && gx < nx - 1 && gy > 0 && gy < ny - 1;
    if (interior) {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const long long d = off + (long long)ey(i) * kp.pitch + ex(i);
            S::put(dst + (long long)i * kp.plane + d, f[i], (real)kp.base_f[i]);
            S::put(dst + (long long)(9 + i) * kp.plane + d, g[i], (real)kp.base_g[i]);
        }
        return;
    }
    const real uin = KPR(kp, U_in);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const int xd = gx + ex(i), yd = gy + ey(i), o = opp(i);
        const bool out_x = xd < 0 || xd >= nx, out_y = yd < 0 || yd >= ny;
        typename S::elem* pfo = dst + (long long)o * kp.plane + off;
        typename S::elem* pgo = dst + (long long)(9 + o) * kp.plane + off;
        if (!out_x && !out_y) {
            const long long d = (long long)yd * kp.pitch + xd;
            S::put(dst + (long long)i * kp.plane + d, f[i], (real)kp.base_f[i]);
            S::put(dst + (long long)(9 + i) * kp.plane + d, g[i], (real)kp.base_g[i]);
            if (WALLS == LB_WALLS_CHANNEL && ex(i) == -1 && gx == nx - 1)
                S::put(dst + (long long)(9 + i) * kp.plane + d + 1, g[i], (real)kp.base_g[i]);
        } else if (WALLS == LB_WALLS_CAVITY) {
            S::put(pfo, f[i], (real)kp.base_f[o]);
            real gb;
            if (out_x) {
                const real Tw = xd < 0 ? KPR(kp, T_hot) : KPR(kp, T_cold);
                gb = -g[i] + (real)2.0 * (real)wd(i) * rho * KPR(kp, cv) * Tw;
            } else {
                gb = g[i];
            }
            S::put(pgo, gb, (real)kp.base_g[o]);
        } else if (out_y) {
            // plate
            S::put(pfo, f[i], (real)kp.base_f[o]);
            real gb;
            if (yd < 0 && kp.adiabatic_bottom)
                gb = g[i];
            else
                gb = -g[i] + (real)2.0 * (real)wd(i) * rho * KPR(kp, cv) * KPR(kp, T_w);
            S::put(pgo, gb, (real)kp.base_g[o]);
        } else if (xd < 0) {
            // inlet
            const real eu = (real)ex(i) * uin;
            S::put(pfo, f[i] - (real)2.0 * (real)wd(i) * rho * eu / cs2, (real)kp.base_f[o]);
            const real gb = -g[i] + (real)2.0 * (real)wd(i) * rho * KPR(kp, cv) * KPR(kp, T_in) *
                                        ((real)1.0 + (real)0.5 * eu * eu / (cs2 * cs2) -
                                         (real)0.5 * uin * uin / cs2);
            S::put(pgo, gb, (real)kp.base_g[o]);
        } else {
            // outlet: f at density 1 with the node's velocity
            const real eu = (real)ex(i) * ux + (real)ey(i) * uy;
            const real fb = -f[i] + (real)2.0 * (real)wd(i) * (real)1.0 *
                                        ((real)1.0 + (real)0.5 * eu * eu / (cs2 * cs2) -
                                         (real)0.5 * (ux * ux + uy * uy) / cs2);
            S::put(pfo, fb, (real)kp.base_f[o]);
        }
    }
}

// Element offsets (within a plane) of the nine pull sources of site (gx, gy): the
// site's own for walls (stored pre-collision), x - e_i on a periodic lattice.
// A plane has fewer than 2^32 elements (two buffers of 18 such planes would not fit
// the device), so each load adds a 32-bit offset to its plane's uniform base.
template <bool WALLED>
struct PullAt {
    uint32_t col[3], row[3];  // by e_ix, e_iy in {0, 1, -1}
    __device__ __forceinline__ PullAt(const KParams& kp, int gx, int gy) {
        const uint32_t pitch = (uint32_t)kp.pitch;
        col[0] = gx;
        row[0] = (uint32_t)gy * pitch;
        if (!WALLED) {
            col[1] = gx == 0 ? kp.nx - 1 : gx - 1;
            col[2] = gx == kp.nx - 1 ? 0 : gx + 1;
            row[1] = (uint32_t)(gy == 0 ? kp.ny - 1 : gy - 1) * pitch;
            row[2] = (uint32_t)(gy == kp.ny - 1 ? 0 : gy + 1) * pitch;
        }
    }
    __device__ __forceinline__ uint32_t operator()(int i) const {
        if (WALLED) return row[0] + col[0];
        return row[ey(i) == 0 ? 0 : (ey(i) > 0 ? 1 : 2)] + col[ex(i) == 0 ? 0 : (ex(i) > 0 ? 1 : 2)];
    }
};

// Site (lx, ly) of thread tid relative to the tile's first: the tile row by row, then
// the ring (the rows below and above with their corners, then the sides in turn).
template <int BX>
__device__ __forceinline__ void tile_site(int tid, int by, int& lx, int& ly) {
    constexpr int WX = BX + 2;
    if (tid < BX * by) {
        lx = tid % BX;
        ly = tid / BX;
        return;
    }
    const int r = tid - BX * by;
    if (r < 2 * WX) {
        lx = (r < WX ? r : r - WX) - 1;
        ly = r < WX ? -1 : by;
    } else {
        lx = (r & 1) ? BX : -1;
        ly = (r - 2 * WX) >> 1;  // (past the ring: ly >= by)
    }
}

// One step of the tile at (x0, y0): see the head of the file.  Every thread of
// the block calls it (one barrier inside).
template <int PREC, int BX, int WALLS, bool EQ24, int BMODE>
__device__ __forceinline__ void tile_step(const typename Store<PREC>::elem* src, typename Store<PREC>::elem* dst,
                                          const KParams& kp, int x0, int y0, int by,
                                          typename Store<PREC>::real* s_psi, typename Store<PREC>::real* s_psi2,
                                          int& flags) {
    using S = Store<PREC>;
    using real = typename S::real;
    constexpr int WX = BX + 2;
    const int tid = threadIdx.x, nx = kp.nx, ny = kp.ny;
    const bool own = tid < BX * by;
    int lx, ly;
    tile_site<BX>(tid, by, lx, ly);
    // rows updated: [H, ny - H) (H = kp.halo_rows; 0 on a periodic lattice)
    const int W = min(BX, nx - x0), Hh = min(by, ny - kp.halo_rows - y0);
    const bool need = tid - BX * by < tile_ring(BX, by) && lx <= W && ly <= Hh;  // the tile and one site around it
    real f[9], g[9], rho = 0, e = 0, T = 0;  // (16-bit modes: the stored deviations)
    float Hf = 0.0f, Hg = 0.0f;
    // (the tile starts inside the lattice: one site past it at most is needed)
    int gx = x0 + lx, gy = y0 + ly;
    gx = WALLS ? clampc(gx, nx) : (gx < 0 ? gx + nx : (gx >= nx ? gx - nx : gx));
    gy = WALLS ? clampc(gy, ny) : (gy < 0 ? gy + ny : (gy >= ny ? gy - ny : gy));
    const int at = (ly + 1) * WX + lx + 1;
    if (need) {
        real psi, psi2;
        const PullAt<WALLS != 0> at_i(kp, gx, gy);
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const typename S::elem *pf = src + (size_t)i * kp.plane, *pg = src + (size_t)(9 + i) * kp.plane;
            const uint32_t o = at_i(i);
            f[i] = dev_of<S>(pf + o, i, rest_lo_offset(i) * kp.plane);
            g[i] = dev_of<S>(pg + o, 9 + i, rest_lo_offset(9 + i) * kp.plane);
        }
        if constexpr (S::SPLIT) {
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                Hf += f[i];
                Hg += g[i];
            }
            rho = kp.sum_bf + Hf;
            T = (kp.sum_bg + Hg) / (rho * KPR(kp, cv));
            site_psi_T<real, BMODE>(kp, rho, T, psi, psi2, flags);
        } else {
            site_psi<real, BMODE>(kp, f, g, rho, e, T, psi, psi2, flags);
        }
        if (BMODE != BETA_ZERO) s_psi[at] = psi;
        if (BMODE != BETA_ONE) s_psi2[at] = psi2;
    }
    __syncthreads();
    if (!(own && lx < W && ly < Hh)) return;
    real Fx, Fy, ux, uy;
    force_from_window<real, BMODE>(kp, s_psi, s_psi2, at, WX, Fx, Fy);
    if (WALLS == LB_WALLS_CAVITY) Fy += -rho * KPR(kp, g_grav);
    const bool glo = kp.ghost && gx < STRIP_GHOST, ghi = kp.ghost && gx >= nx - STRIP_GHOST;
    const long long off = (long long)gy * kp.pitch + gx;
    if constexpr (S::SPLIT) {
        collide_dev<EQ24>(kp, f, g, Hf, Hg, Fx, Fy);
        store_site_dev<S>(dst + off, kp.plane, kp, f, g, Hf, Hg, glo, ghi);
    } else {
        collide_et<real, EQ24, false, true>(kp, f, g, rho, e, T, Fx, Fy, ux, uy);
        if constexpr (WALLS)
            push_walls<S, WALLS, real>(dst, kp, gx, gy, f, g, rho, ux, uy);
        else
            store_site<S>(dst + off, kp.plane, kp, f, g, (real)0, (real)0, glo, ghi);
    }
}

// One step per launch; grid (tiles in x, tiles in y), tile_threads(BX, by)
// threads.  Launched so that its blocks may become resident while the step before
// it still runs (programmatic dependent launch); they wait for its end before
// they read anything (grid_wait: src is not __restrict__).
template <int PREC, int BX, int WALLS, bool EQ24, int BMODE>
__global__ void __launch_bounds__(tile_threads(BX, tile_max_by(BX)))
    k_step_tile(const typename Store<PREC>::elem* src, typename Store<PREC>::elem* __restrict__ dst,
                const KParams kp, int by) {
    using real = typename Store<PREC>::real;
    extern __shared__ __align__(16) unsigned char tile_smem[];
    real* s_psi = reinterpret_cast<real*>(tile_smem);
    real* s_psi2 = BMODE == BETA_MIXED ? s_psi + (BX + 2) * (by + 2) : s_psi;
    int flags = 0;
    grid_begin();
    tile_step<PREC, BX, WALLS, EQ24, BMODE>(src, dst, kp, blockIdx.x * BX, kp.halo_rows + blockIdx.y * by, by, s_psi,
                                            s_psi2, flags);
    if (flags) atomicOr(kp.err, flags);
}

// One step of the active domains of a batch: block b takes tile b of the list (domain
// and first site), with its domain's parameters read from the device table.  The
// list and the table are written before the steps, not by them, so a block has
// read its tile when the step before it ends.  (Each block has its tile whatever the
// others do, so small domains need no balancing; the persistent strip kernel of
// lb_batch_device.cuh re-reads less and takes over for large batches.)
template <int PREC, bool EQ24, int BMODE>
__global__ void __launch_bounds__(tile_threads(32, tile_max_by(32)))
    k_batch_tile(const typename Store<PREC>::elem* src, typename Store<PREC>::elem* __restrict__ dst,
                 const BatchDomain* __restrict__ doms, const BatchStepTile* __restrict__ tiles,
                 const int* __restrict__ n_tiles, int by) {
    using real = typename Store<PREC>::real;
    extern __shared__ __align__(16) unsigned char tile_smem[];
    real* s_psi = reinterpret_cast<real*>(tile_smem);
    real* s_psi2 = BMODE == BETA_MIXED ? s_psi + 34 * (by + 2) : s_psi;
    grid_launch();
    if ((int)blockIdx.x >= *n_tiles) {  // the grid covers the longest list
        grid_wait();         // (no block ends before the step ahead of it)
        return;
    }
    const BatchStepTile t = tiles[blockIdx.x];
    const BatchDomain& D = doms[t.domain];
    const long long off = D.off;
    int flags = 0;
    grid_wait();
    tile_step<PREC, 32, 0, EQ24, BMODE>(src + off, dst + off, D.kp, t.x0, t.y0, by, s_psi, s_psi2, flags);
    if (flags) atomicOr(D.kp.err, flags);
}

// ---------------------------------------------------------------- moments
// Sum of v[0..7] over the warp: halving steps exchange half of the values each
// (nine additions instead of eight times five).  Lane 4 k returns the sum of v[k].
__device__ __forceinline__ double warp_sum8(double v[8], int lane) {
#pragma unroll
    for (int h = 4; h > 0; h >>= 1) {
        const bool up = lane & (4 * h);
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (k < h) {
                const double send = up ? v[k] : v[k + h], keep = up ? v[k + h] : v[k];
                v[k] = keep + __shfl_xor_sync(0xffffffffu, send, 4 * h);
            }
    }
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
    return v[0];
}

// Macroscopic fields of the state as the step forms them: rho, u (with F/2), T (any
// pointer may be null), on the tile and psi ring of tile_step, and with PART the
// FP64 totals of each block:
//   part[blk*8 + k], k = mass, energy, rho ux, rho uy, |d rho|^2, rho^2, |dT|^2, T^2
// against the reference fields ref_rho/ref_T (may be null).  Each site pulled once,
// the parameters read as floats and the results widened on the integer units:
// 4096^2 FP32 fields 340 us, 1,543 us with the two pulls, the FP64 conversions and the
// whole collision of the kernel before (bytes: 72 read, 32 written per site).
template <int PREC, int BMODE, bool PART>
__global__ void __launch_bounds__(tile_threads(32, 8))
    k_moments(const typename Store<PREC>::elem* __restrict__ src, const KParams kp,
              double* __restrict__ o_rho, double* __restrict__ o_ux, double* __restrict__ o_uy,
              double* __restrict__ o_T, const double* __restrict__ ref_rho,
              const double* __restrict__ ref_T, double* __restrict__ part) {
    using S = Store<PREC>;
    using real = typename S::real;
    constexpr int BX = 32, BY = 8, WX = BX + 2, WY = BY + 2;
    __shared__ real s_psi[BMODE != BETA_ZERO ? WX * WY : 1];
    __shared__ real s_psi2[BMODE != BETA_ONE ? WX * WY : 1];
    __shared__ double s_red[BY][8];
    const int tid = threadIdx.x, nx = kp.nx, ny = kp.ny;
    const int x0 = blockIdx.x * BX, y0 = blockIdx.y * BY;
    const bool own = tid < BX * BY;
    int lx, ly;
    tile_site<BX>(tid, BY, lx, ly);
    const int W = min(BX, nx - x0), Hh = min(BY, ny - y0);
    const bool active = own && lx < W && ly < Hh;
    int gx = x0 + lx, gy = y0 + ly, flags = 0;
    real rho = 0, e = 0, T = 0, mx = 0, my = 0;
    double m = 0, en = 0;
    if (tid - BX * BY < tile_ring(BX, BY) && lx <= W && ly <= Hh) {
        gx = kp.walls ? clampc(gx, nx) : (gx < 0 ? gx + nx : (gx >= nx ? gx - nx : gx));
        gy = kp.walls ? clampc(gy, ny) : (gy < 0 ? gy + ny : (gy >= ny ? gy - ny : gy));
        real f[9], g[9], psi, psi2;
        pull18<S>(src, kp, gx, gy, f, g);
        site_psi<real, BMODE>(kp, f, g, rho, e, T, psi, psi2, flags);
        if (BMODE != BETA_ZERO) s_psi[(ly + 1) * WX + lx + 1] = psi;
        if (BMODE != BETA_ONE) s_psi2[(ly + 1) * WX + lx + 1] = psi2;
        if constexpr (sizeof(real) == 8) {
            mx = ((((f[1] - f[3]) + f[5]) - f[6]) - f[7]) + f[8];
            my = ((((f[2] - f[4]) + f[5]) + f[6]) - f[7]) - f[8];
        } else {
            mx = (f[1] - f[3]) + ((f[5] - f[7]) + (f[8] - f[6]));
            my = (f[2] - f[4]) + ((f[5] - f[7]) + (f[6] - f[8]));
        }
        if constexpr (PART) {
            real s;
            m = sum9(f, s);
            en = sum9(g, s);
        }
    }
    if (flags) atomicOr(kp.err, flags);
    __syncthreads();
    double v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (active) {
        real Fx, Fy, ux, uy;
        force_from_window<real, BMODE>(kp, s_psi, s_psi2, (ly + 1) * WX + lx + 1, WX, Fx, Fy);
        if (kp.walls) Fy += -rho * KPR(kp, g_grav);  // cavity buoyancy
        if constexpr (sizeof(real) == 8) {
            ux = (mx + 0.5 * Fx) / rho;
            uy = (my + 0.5 * Fy) / rho;
        } else {
            const real inv_rho = (real)1 / rho;
            ux = (mx + (real)0.5 * Fx) * inv_rho;
            uy = (my + (real)0.5 * Fy) * inv_rho;
        }
        const long long idx = (long long)gy * nx + gx;
        const double dr = widen(rho), dux = widen(ux), duy = widen(uy), dT = widen(T);
        if (o_rho) o_rho[idx] = dr;
        if (o_ux) o_ux[idx] = dux;
        if (o_uy) o_uy[idx] = duy;
        if (o_T) o_T[idx] = dT;
        if constexpr (PART) {
            v[0] = m;
            v[1] = en;
            v[2] = dr * dux;
            v[3] = dr * duy;
            if (ref_rho) {
                const double a = dr - ref_rho[idx], b = dT - ref_T[idx];
                v[4] = a * a;
                v[6] = b * b;
            }
            v[5] = dr * dr;
            v[7] = dT * dT;
        }
    }
    if constexpr (PART) {
        // deterministic block reduction: lanes, then warps in order
        if (own) {
            const double x = warp_sum8(v, tid & 31);
            if ((tid & 3) == 0) s_red[tid >> 5][(tid & 31) >> 2] = x;
        }
        __syncthreads();
        if (tid < 8) {
            double x = 0.0;
            for (int w = 0; w < BY; ++w) x += s_red[w][tid];
            part[(long long)(blockIdx.y * gridDim.x + blockIdx.x) * 8 + tid] = x;
        }
    }
}

}  // namespace lbgb
