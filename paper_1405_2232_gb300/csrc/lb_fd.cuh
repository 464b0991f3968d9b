// lb_fd.cuh -- the finite-difference temperature treatment, Eqs. (26)-(27).
//
// The density LBE (Eq. 1 with the force of Eq. 2/4) is stepped as in the
// thermal LB path, with psi taken from a temperature field instead of the g
// populations; then T is advanced by the second-order Runge-Kutta update of
// Eq. (27) applied to Eq. (26):
//   K(T) = -u . grad T + chi (lap T + grad rho . grad T / rho),
//   lambda = rho c_v chi, chi = (tau_g - 1/2) c_s^2,
// with the isotropic central stencils of the D2Q9 lattice
//   grad phi = (1/c_s^2) sum_i w_i e_i phi(x + e_i),
//   lap phi  = (2/c_s^2) sum_i w_i (phi(x + e_i) - phi(x)),
// and rho, u (the velocity of the density LBE, with F/2) held at time n for
// both stages.  T^{n+1} = T^n + (h1 + h2)/2, h1 = K(T^n), h2 = K(T^n + a h1),
// a = 1 (Heun) or 1/2 (the form printed with Eq. 27).
//
// Kernels: in lb_fd_strip.cuh k_fd_fused (the whole step in one pass on strip
// contexts), in lb_fd_tile.cuh k_fd_front (tile and psi ring; STEP collides and stores
// f and writes rho^n, u^n; else rho, u, T) and k_fd_rk2 (both RK2 stages in one
// launch, after the front); k_fd_partials (FP64 totals of dense fields).  T is stored like one population plane (row pitch kp.pitch, ghost
// columns on strip contexts).  The FP64 mode evaluates every formula in the
// order of its printed form (compiled without contraction).
#pragma once

#include "lb_device.cuh"

namespace lbgb {

constexpr int FD_BX = 32, FD_BY = 8;

// K of Eq. (26) in FP64, from X and rho of a site (index 0) and its eight neighbours:
// the printed sums in their order, without the products by e_i = 0 (which add
// zero), each w X[i] formed once for both gradient components, and the divisions by
// c_s^2 as div_cs2.  (grx, gry) = grad(rho), which both RK2 stages share.
__device__ __forceinline__ void fd_grad_fp64(const double X[9], double& gx, double& gy) {
    gx = gy = 0.0;
#pragma unroll
    for (int i = 1; i < 9; ++i) {
        const double wX = wd(i) * X[i];
        if (ex(i)) gx = ex(i) > 0 ? gx + wX : gx - wX;
        if (ey(i)) gy = ey(i) > 0 ? gy + wX : gy - wX;
    }
    gx = div_cs2(gx);
    gy = div_cs2(gy);
}
__device__ __forceinline__ double fd_K_fp64(const double X[9], double grx, double gry, double rho, double ux,
                                            double uy, double chi) {
    double gTx, gTy, lap = 0.0;
    fd_grad_fp64(X, gTx, gTy);
#pragma unroll
    for (int i = 1; i < 9; ++i) lap += wd(i) * (X[i] - X[0]);
    lap *= 2.0 / (1.0 / 3.0);
    return -(ux * gTx + uy * gTy) + chi * (lap + (grx * gTx + gry * gTy) / rho);
}

// A site and its neighbours from three row pointers (south, centre, north) at its column.
template <typename real>
__device__ __forceinline__ void fd_window(const real* Xs, const real* Xc, const real* Xn, real X[9]) {
#pragma unroll
    for (int i = 0; i < 9; ++i) X[i] = (ey(i) == 1 ? Xn : (ey(i) == -1 ? Xs : Xc))[ex(i)];
}

// FP32: K with the terms that depend only on the site's density and
// velocity folded into a = chi grad(rho) / rho - u, which both RK2 stages
// share:
// K = a . grad(X) + chi lap(X), the stencil of X alone.
__device__ __forceinline__ float fd_K_rows_a(const float* Xs, const float* Xc, const float* Xn, float ax,
                                             float ay, float chi) {
    float gTx = 0.0f, gTy = 0.0f, lap = 0.0f;
    const float X0 = Xc[0];
#pragma unroll
    for (int i = 1; i < 9; ++i) {
        const float w = (float)wd(i);
        const float* xr = ey(i) == 1 ? Xn : (ey(i) == -1 ? Xs : Xc);
        const float Xv = xr[ex(i)];
        gTx += w * (float)ex(i) * Xv;
        gTy += w * (float)ey(i) * Xv;
        lap += w * (Xv - X0);
    }
    return fmaf(ax, 3.0f * gTx, fmaf(ay, 3.0f * gTy, chi * (6.0f * lap)));
}

// a = chi grad(rho) / rho - u at a site (FP32; see fd_K_rows_a), from the
// density rows (south, centre, north, each at the site's column)
__device__ __forceinline__ void fd_a_rows(const float* Rs, const float* Rc, const float* Rn, float ux, float uy,
                                          float chi, float& ax, float& ay) {
    float grx = 0.0f, gry = 0.0f;
#pragma unroll
    for (int i = 1; i < 9; ++i) {
        const float w = (float)wd(i);
        const float* rr = ey(i) == 1 ? Rn : (ey(i) == -1 ? Rs : Rc);
        const float rn = rr[ex(i)];
        grx += w * (float)ex(i) * rn;
        gry += w * (float)ey(i) * rn;
    }
    const float cr = __fdividef(chi, Rc[0]);
    ax = fmaf(cr, 3.0f * grx, -ux);
    ay = fmaf(cr, 3.0f * gry, -uy);
}

// T field (storage real, row pitch kp.pitch, ghost columns when kp.ghost)
// <- T0 (FP64, dense [ny][nx])
template <typename real>
__global__ void k_fd_set_T(real* __restrict__ T, const double* __restrict__ T0, const KParams kp) {
    const long long n = (long long)kp.nx * kp.ny;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(i % kp.nx), y = (int)(i / kp.nx);
        const real v = (real)T0[i];
        real* p = T + (long long)y * kp.pitch + x;
        *p = v;
        if (x < kp.ghost) p[kp.nx] = v;
        if (x >= kp.nx - kp.ghost) p[-kp.nx] = v;
    }
}

}  // namespace lbgb
