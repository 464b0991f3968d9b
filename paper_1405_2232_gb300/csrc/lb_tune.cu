// lb_tune.cu -- the step-shape autotuner (lb_tune_candidate, lb_autotune, lb_time_step).
//
// Every shape that the fused step can be asked for is timed on a uniform state of
// the caller's lattice, parameters and precision; the fastest wins.  lb_time_step
// times parameters as they are, so also the library's own choice (no shape asked for),
// whose balanced tiles and cluster runs are none of these shapes.  The state is
// uniform so that no candidate can leave the psi domain while it is timed, and
// the timing uses CUDA events on the stream the trial contexts run on.  Results
// do not depend on the shape (FP64: bit for bit), so the choice is free.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <vector>

#include "lb.h"

namespace lbgb {
lb_status record_error(lb_status st, const char* msg);
}

namespace {

// (tile_x, tile_y); tile_y == 0 selects the strip-marching kernel
constexpr int kCand[LB_TUNE_N][2] = {{256, 0}, {128, 0}, {32, 8}, {32, 16}, {64, 4}};

lb_status tune_fail(lb_status st, const char* what, cudaError_t e) {
    char msg[300];
    snprintf(msg, sizeof(msg), "lb_autotune: %s: %s", what, cudaGetErrorString(e));
    return lbgb::record_error(st, msg);
}

// Trial contexts of one tuning: a uniform state, a stream and two events.
struct Trials {
    std::vector<double> rho, T;
    cudaStream_t st = nullptr;
    bool own = false;
    cudaEvent_t ev[2] = {nullptr, nullptr};
    cudaError_t e = cudaSuccess;

    Trials(const lb_params* p, void* stream) : st(static_cast<cudaStream_t>(stream)) {
        const size_t n = (size_t)p->nx * (size_t)p->ny;
        rho.assign(n, p->rho0);
        T.assign(n, p->T0);
        if (st) {
            int dev = 0;
            e = cudaStreamGetDevice(st, &dev);
            if (e == cudaSuccess) e = cudaSetDevice(dev);
        } else {
            e = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking);
            own = e == cudaSuccess;
        }
        if (e == cudaSuccess) e = cudaEventCreate(&ev[0]);
        if (e == cudaSuccess) e = cudaEventCreate(&ev[1]);
    }
    ~Trials() {
        if (ev[0]) cudaEventDestroy(ev[0]);
        if (ev[1]) cudaEventDestroy(ev[1]);
        if (own) cudaStreamDestroy(st);
    }
    // ms per step of q over `steps` steps after `warmup`; e holds an error of the timing
    lb_status time(const lb_params& q, int steps, int warmup, double* per) {
        lb_ctx* c = nullptr;
        lb_status s = lb_init(&q, rho.data(), T.data(), st, &c);
        if (s != LB_OK) return s;
        s = lb_step(c, warmup);
        if (s == LB_OK) e = cudaEventRecord(ev[0], st);
        if (s == LB_OK && e == cudaSuccess) s = lb_step(c, steps);
        if (s == LB_OK && e == cudaSuccess) e = cudaEventRecord(ev[1], st);
        if (s == LB_OK && e == cudaSuccess) e = cudaEventSynchronize(ev[1]);
        float ms = 0.0f;
        if (s == LB_OK && e == cudaSuccess) e = cudaEventElapsedTime(&ms, ev[0], ev[1]);
        if (s == LB_OK && e == cudaSuccess) s = lb_synchronize(c);
        lb_free(c);
        *per = (double)ms / steps;
        return s;
    }
};

}  // namespace

extern "C" {

lb_status lb_tune_candidate(int32_t k, int32_t* tile_x, int32_t* tile_y) {
    if (k < 0 || k >= LB_TUNE_N || !tile_x || !tile_y)
        return lbgb::record_error(LB_ERR_ARG, "lb_tune_candidate: index out of range or NULL output");
    *tile_x = kCand[k][0];
    *tile_y = kCand[k][1];
    return LB_OK;
}

lb_status lb_autotune(const lb_params* p, int32_t steps, void* stream, lb_params* best,
                      double ms_per_step[LB_TUNE_N]) {
    if (!p || !best || steps < 1)
        return lbgb::record_error(LB_ERR_ARG, "lb_autotune: NULL params/best or steps < 1");
    if (p->nx < 3 || p->ny < 3)
        return lbgb::record_error(LB_ERR_ARG, "lb_autotune: nx, ny must be >= 3");
    Trials t(p, stream);
    if (t.e != cudaSuccess) return tune_fail(LB_ERR_CUDA, "stream", t.e);
    double best_ms = INFINITY;
    int best_k = -1;
    for (int k = 0; k < LB_TUNE_N; ++k) {
        if (ms_per_step) ms_per_step[k] = NAN;
        lb_params q = *p;
        q.tile_x = kCand[k][0];
        q.tile_y = kCand[k][1];
        double per = 0.0;
        const lb_status s = t.time(q, steps, 2, &per);
        if (s == LB_ERR_ARG) continue;  // shape not valid for this lattice/precision
        if (s != LB_OK) return s;
        if (t.e != cudaSuccess) return tune_fail(LB_ERR_CUDA, "timing", t.e);
        if (ms_per_step) ms_per_step[k] = per;
        if (per < best_ms) {
            best_ms = per;
            best_k = k;
        }
    }
    if (best_k < 0) return lbgb::record_error(LB_ERR_UNSUPPORTED, "lb_autotune: no step shape is valid");
    *best = *p;
    best->tile_x = kCand[best_k][0];
    best->tile_y = kCand[best_k][1];
    return LB_OK;
}

lb_status lb_time_step(const lb_params* p, int32_t steps, void* stream, double* ms_per_step) {
    if (!p || !ms_per_step || steps < 1)
        return lbgb::record_error(LB_ERR_ARG, "lb_time_step: NULL params/output or steps < 1");
    if (p->nx < 3 || p->ny < 3)
        return lbgb::record_error(LB_ERR_ARG, "lb_time_step: nx, ny must be >= 3");
    Trials t(p, stream);
    if (t.e != cudaSuccess) return tune_fail(LB_ERR_CUDA, "stream", t.e);
    // (warm-up with the same call: a run of steps may take another kernel than two)
    const lb_status s = t.time(*p, steps, steps, ms_per_step);
    if (s != LB_OK) return s;
    return t.e == cudaSuccess ? LB_OK : tune_fail(LB_ERR_CUDA, "timing", t.e);
}

}  // extern "C"
