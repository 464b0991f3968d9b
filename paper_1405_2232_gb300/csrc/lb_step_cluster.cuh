// lb_step_cluster.cuh -- many steps of a tiny lattice in one launch of one
// thread-block cluster (FP32 and the 16-bit modes, periodic).
//
// A lattice of a few thousand sites takes the tile kernel about 2 us per step, nearly
// all of it the way through the L2 cache and from one launch to the next.  Here the
// lattice stays in the shared memory of a cluster of up to 16 blocks for all steps of a
// call: a block owns a band of rows (two buffers, the stored elements as in device
// memory), each thread one site of the band or of the row above and below it,
// populations from a neighbouring band are pulled through distributed shared memory, and
// one cluster barrier ends a step.  The arithmetic and the rounding to storage of
// a site are the tile kernel's.  Per step in a run of 1,000, FP32: 16^2 0.81 us, 64 x 32
// 1.14, 64^2 1.24, 96 x 64 1.60, 128 x 64 1.92; as tiles 2.2 at all of these (a run of
// 100 steps at 64^2: 150 us, 224).  Below 2,000 sites the chain of one step bounds it
// (remote loads, the collision, two barriers), above them the issue rate of the sixteen
// SMs that do all the work; so the tile kernel takes over at 8,192 sites.
#pragma once

#include <cooperative_groups.h>

#include "lb_step_tile.cuh"

namespace lbgb {

constexpr int CLUSTER_MAX = 16, CLUSTER_THREADS = 768, CLUSTER_SITES = 8192;
// elements from one plane of a band to the next (more than nx * rows; as a constant, the
// addresses of all planes are one register and an immediate)
constexpr int CLUSTER_PLANE = 768;
// fewest steps of a run (a cluster's launch takes some 5 us more than a tile kernel's,
// and a step of 8,192 sites saves 0.3 us: ten steps 28 us against 27) and most of one
// launch (a launch of this many takes a few milliseconds)
constexpr int CLUSTER_RUN = 16, CLUSTER_STEPS = 4096;

// Blocks of the cluster for an nx by ny lattice; 0: it does not fit.
inline int cluster_blocks(int nx, int ny) {
    int nc = CLUSTER_MAX;
    while (nc > ny) nc /= 2;
    const int rows = (ny + nc - 1) / nc;
    return (long long)nx * ny <= CLUSTER_SITES && nx * (rows + 2) <= CLUSTER_THREADS ? nc : 0;
}
template <int PREC, int BMODE>
constexpr size_t cluster_smem_bytes(int nx, int rows) {
    using S = Store<PREC>;
    return (size_t)2 * S::NPLANES * CLUSTER_PLANE * sizeof(typename S::elem) +
           (size_t)(BMODE == BETA_MIXED ? 2 : 1) * (rows + 2) * (nx + 2) * sizeof(float);
}

// src and dst: the lattice before and after (the same buffer for an even number of
// steps, so that a context's current one stays the one that the parity says).
template <int PREC, bool EQ24, int BMODE>
__global__ void __launch_bounds__(CLUSTER_THREADS)
    k_steps_cluster(const typename Store<PREC>::elem* src, typename Store<PREC>::elem* dst, const KParams kp,
                    int steps) {
    namespace cg = cooperative_groups;
    using S = Store<PREC>;
    using elem = typename S::elem;
    using real = float;
    constexpr int NPL = S::NPLANES;
    cg::cluster_group cl = cg::this_cluster();
    const int nc = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int nx = kp.nx, ny = kp.ny, tid = threadIdx.x;
    // band of block c: rows [c ny / nc, (c + 1) ny / nc)
    const int y0 = rank * ny / nc, rows = (rank + 1) * ny / nc - y0, room = (ny + nc - 1) / nc;
    constexpr int PS = CLUSTER_PLANE, BUF = NPL * PS;
    const int W = nx + 2;
    extern __shared__ __align__(16) unsigned char cluster_smem[];
    elem* band = reinterpret_cast<elem*>(cluster_smem);  // [2][NPL][PS]: rows of nx
    float* s_psi = reinterpret_cast<float*>(cluster_smem + (size_t)2 * BUF * sizeof(elem));
    float* s_psi2 = BMODE == BETA_MIXED ? s_psi + (room + 2) * W : s_psi;  // [room + 2][nx + 2]

    // this thread's site: the band row by row, then the rows below and above it
    const bool own = tid < rows * nx, need = tid < (rows + 2) * nx;
    const int ring = tid - rows * nx;
    const int ly = own ? tid / nx : (ring < nx ? -1 : rows), x = own ? tid - ly * nx : (ring < nx ? ring : ring - nx);
    const int at = (ly + 1) * W + x + 1;
    // its three source rows in the blocks that own them, and its source columns
    auto row_of = [&](int y) -> const elem* {
        y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
        const int c = ((y + 1) * nc - 1) / ny;
        return cl.map_shared_rank(band, c) + (y - c * ny / nc) * nx;
    };
    const elem *r0 = band, *rb = band, *ra = band;
    if (need) {
        int y = y0 + ly;
        y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
        r0 = row_of(y);
        rb = row_of(y - 1);
        ra = row_of(y + 1);
    }
    const int xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
    int flags = 0;
    const long long off = (long long)(y0 + ly) * kp.pitch + x;  // (own)
    if (own) {
#pragma unroll
        for (int p = 0; p < NPL; ++p) band[p * PS + tid] = src[(size_t)p * kp.plane + off];
    }
    cl.sync();
    for (int s = 0; s < steps; ++s) {
        const int from = (s & 1) * BUF, to = BUF - from;
        real f[9], g[9], rho = 0, e = 0, T = 0;
        float Hf = 0.0f, Hg = 0.0f;
        if (need) {
            real psi, psi2;
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const elem* a = (ey(i) == 0 ? r0 : (ey(i) > 0 ? rb : ra)) + from + (ex(i) == 0 ? x : (ex(i) > 0 ? xm : xp));
                f[i] = dev_of<S>(a + i * PS, i, rest_lo_offset(i) * PS);
                g[i] = dev_of<S>(a + (9 + i) * PS, 9 + i, rest_lo_offset(9 + i) * PS);
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
            // (with the periodic copies beside the row)
            if (BMODE != BETA_ZERO) {
                s_psi[at] = psi;
                if (x == 0) s_psi[at + nx] = psi;
                if (x == nx - 1) s_psi[at - nx] = psi;
            }
            if (BMODE != BETA_ONE) {
                s_psi2[at] = psi2;
                if (x == 0) s_psi2[at + nx] = psi2;
                if (x == nx - 1) s_psi2[at - nx] = psi2;
            }
        }
        __syncthreads();
        if (own) {
            real Fx, Fy, ux, uy;
            force_from_window<real, BMODE>(kp, s_psi, s_psi2, at, W, Fx, Fy);
            elem* d = band + to + tid;
            if constexpr (S::SPLIT) {
                collide_dev<EQ24>(kp, f, g, Hf, Hg, Fx, Fy);
                store_site_dev<S>(d, PS, kp, f, g, Hf, Hg, false, false);
            } else {
                collide_et<real, EQ24, false, true>(kp, f, g, rho, e, T, Fx, Fy, ux, uy);
                store_site<S>(d, PS, kp, f, g, (real)0, (real)0, false, false);
            }
        }
        // the step's rows are complete, and nobody reads the ones that the next overwrites
        cl.sync();
    }
    if (own) {
        const elem* last = band + (steps & 1) * BUF + tid;
        elem* d = dst + off;
        const bool glo = x < kp.ghost, ghi = x >= nx - kp.ghost;
#pragma unroll
        for (int p = 0; p < NPL; ++p, d += kp.plane) {
            const elem v = last[p * PS];
            *d = v;
            if (glo) d[nx] = v;
            if (ghi) d[-nx] = v;
        }
    }
    if (flags) atomicOr(kp.err, flags);
}

}  // namespace lbgb
