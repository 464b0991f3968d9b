// unet_kernels.cuh -- device kernels of the warm-start network (include/unet.h).
//
// The 3x3 circular convolutions run as implicit GEMMs on the BF16 tensor
// cores (mma.sync m16n8k16, FP32 accumulation) with cp.async staging:
//   forward / input gradient: out[p][co] = sum_{tap, ci} in[shift_tap(p)][ci] W[co][tap][ci]
//     (the input gradient uses the flipped, transposed weights
//      Wt[ci][8 - tap][co], because shift_{8-tap} = -shift_tap);
//   weight gradient: dW[co][tap][ci] = sum_p g[p][co] in[shift_tap(p)][ci],
//     split over pixel ranges, partials reduced in a fixed order.
// Everything else (pool, upsampling gradients, head, loss, Adam, handoff) is
// element-wise or a small reduction and bound by memory traffic.
//
// Activation layout (every BF16 tensor of the net): per image row
// (row = n H + y), the C / 8 channel groups one after the other, each group
// the row's W pixels x 8 channels (16 bytes per pixel); see act_at.  A
// pixel's 8 channels stay one 16-byte vector, a warp's 32 consecutive pixels
// of one group are 512 contiguous bytes, and a group of a row segment is one
// contiguous block for the tensor copies of the tcgen05 convolution.
#pragma once

#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "lb_device.cuh"

namespace unk {

using lbgb::grid_begin;
using lbgb::grid_launch;
using lbgb::grid_wait;

typedef __nv_bfloat16 bf16;

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// 16-byte asynchronous copy global -> shared; valid == false zero-fills
// (no bytes are read; src must still be a mapped address)
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem, bool valid) {
    const int n = valid ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_addr(smem)), "l"(gmem), "r"(n)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], const void* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(smem_addr(p)));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t (&r)[4], const void* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(smem_addr(p)));
}
__device__ __forceinline__ void ldsm_x2_t(uint32_t& r0, uint32_t& r1, const void* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];\n"
                 : "=r"(r0), "=r"(r1)
                 : "r"(smem_addr(p)));
}

// D += A (16x16, row) * B (16x8, col), BF16 inputs, FP32 accumulators
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ int wrap(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

// element (row, x, c) of an activation tensor with C channels and W pixels
// per row (C a multiple of 8): ((row C + 8 floor(c / 8)) W + 8 x + c mod 8
__host__ __device__ __forceinline__ long long act_at(long long row, int x, int c, int C, int W) {
    return (row * C + (c & ~7)) * (long long)W + x * 8 + (c & 7);
}

__device__ __forceinline__ void unpack8(const uint4& u, float (&f)[8]) {
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float2 t = __bfloat1622float2(h[k]);
        f[2 * k] = t.x;
        f[2 * k + 1] = t.y;
    }
}
__device__ __forceinline__ uint4 pack8(const float (&f)[8]) {
    uint4 u;
    __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&u);
#pragma unroll
    for (int k = 0; k < 4; ++k) h[k] = __floats2bfloat162_rn(f[2 * k], f[2 * k + 1]);
    return u;
}


// ------------------------------------------------------------ convolution
struct ConvArgs {
    const bf16* x;  // input view: channels xoff .. xoff + Cin - 1 of a tensor of xC channels
    int xC, xoff, Cin;
    const bf16* w;  // [Cout][9][Cin]
    const float* bias;  // [Cout] or nullptr
    int Cout;
    bf16* y;  // output view
    int yC, yoff;
    const bf16* mask;  // optional: output *= (mask > 0) (same pixel, channel co)
    int mC, moff;
    int N, H, W;
    int relu;  // forward: ReLU after the bias
    int up;    // store each output pixel to the 2x2 block of a 2H x 2W image
    int* err;  // sticky error word of the net (k_conv3_tc: bit 6 on a wait that gave up)
};

constexpr int CV_MT = 128;   // pixels per CTA
constexpr int CV_KC = 32;    // channels per K step
constexpr int CV_LD = 40;    // shared row stride (halves): conflict-free ldmatrix
constexpr int CV_STAGES = 3;

template <int NT>
__global__ void __launch_bounds__(256) k_conv3(ConvArgs a) {
    grid_begin();
    __shared__ __align__(128) bf16 sA[CV_STAGES][CV_MT * CV_LD];
    __shared__ __align__(128) bf16 sB[CV_STAGES][NT * CV_LD];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int HW = a.H * a.W;
    const int M = a.N * HW;
    const int m0 = blockIdx.x * CV_MT;
    const int co0 = blockIdx.y * NT;
    int an[2], ay[2], ax[2];
    bool av[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int m = m0 + (tid >> 2) + i * 64;
        av[i] = m < M;
        const int mm = av[i] ? m : 0;
        an[i] = mm / HW;
        const int r = mm - an[i] * HW;
        ay[i] = r / a.W;
        ax[i] = r - ay[i] * a.W;
    }
    const int part = tid & 3;
    const int kchunks = a.Cin / CV_KC;
    const int KT = 9 * kchunks;

    auto load_stage = [&](int kt, int s) {
        const int tap = kt / kchunks, c0 = (kt - tap * kchunks) * CV_KC;
        const int dy = tap / 3 - 1, dx = tap % 3 - 1;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int yy = wrap(ay[i] + dy, a.H), xx = wrap(ax[i] + dx, a.W);
            const long long row = (long long)an[i] * a.H + yy;
            cp_async16(&sA[s][((tid >> 2) + i * 64) * CV_LD + part * 8],
                       a.x + act_at(row, xx, a.xoff + c0 + part * 8, a.xC, a.W), av[i]);
        }
        for (int q = tid; q < NT * 4; q += 256) {
            const int r = q >> 2, pp = q & 3;
            cp_async16(&sB[s][r * CV_LD + pp * 8], a.w + ((long long)(co0 + r) * 9 + tap) * a.Cin + c0 + pp * 8,
                       true);
        }
    };

    const int wm = warp & 3, wn = warp >> 2;
    constexpr int WN = NT / 2;
    constexpr int NI = WN / 8;
    float acc[2][NI][4];
#pragma unroll
    for (int mi = 0; mi < 2; ++mi)
#pragma unroll
        for (int ni = 0; ni < NI; ++ni)
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[mi][ni][k] = 0.0f;

#pragma unroll
    for (int s = 0; s < CV_STAGES - 1; ++s) {
        if (s < KT) load_stage(s, s);
        cp_async_commit();
    }
    const int q = lane >> 3, rr = lane & 7;
    for (int kt = 0; kt < KT; ++kt) {
        cp_async_wait<CV_STAGES - 2>();
        __syncthreads();
        {
            const int nk = kt + CV_STAGES - 1;
            if (nk < KT) load_stage(nk, nk % CV_STAGES);
            cp_async_commit();
        }
        const bf16* A = sA[kt % CV_STAGES];
        const bf16* B = sB[kt % CV_STAGES];
#pragma unroll
        for (int kk = 0; kk < CV_KC; kk += 16) {
            uint32_t af[2][4];
#pragma unroll
            for (int mi = 0; mi < 2; ++mi)
                ldsm_x4(af[mi], A + (wm * 32 + mi * 16 + rr + (q & 1) * 8) * CV_LD + kk + (q >> 1) * 8);
#pragma unroll
            for (int nj = 0; nj < NI; nj += 2) {
                uint32_t bf[4];
                ldsm_x4(bf, B + (wn * WN + nj * 8 + rr + (q >> 1) * 8) * CV_LD + kk + (q & 1) * 8);
#pragma unroll
                for (int mi = 0; mi < 2; ++mi) {
                    mma_bf16(acc[mi][nj], af[mi], bf[0], bf[1]);
                    mma_bf16(acc[mi][nj + 1], af[mi], bf[2], bf[3]);
                }
            }
        }
    }
    cp_async_wait<0>();

    const int g = lane >> 2, t4 = lane & 3;
#pragma unroll
    for (int mi = 0; mi < 2; ++mi)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int m = m0 + wm * 32 + mi * 16 + g + h * 8;
            if (m >= M) continue;
            const int n = m / HW;
            const int rem = m - n * HW;
            const int yy = rem / a.W, xx = rem - yy * a.W;
#pragma unroll
            for (int ni = 0; ni < NI; ++ni) {
                const int co = co0 + wn * WN + ni * 8 + 2 * t4;
                float v0 = acc[mi][ni][2 * h], v1 = acc[mi][ni][2 * h + 1];
                if (a.bias) {
                    v0 += a.bias[co];
                    v1 += a.bias[co + 1];
                }
                if (a.relu) {
                    v0 = fmaxf(v0, 0.0f);
                    v1 = fmaxf(v1, 0.0f);
                }
                const long long row = (long long)n * a.H + yy;
                if (a.mask) {
                    const bf16* mp = a.mask + act_at(row, xx, a.moff + co, a.mC, a.W);
                    v0 = __bfloat162float(mp[0]) > 0.0f ? v0 : 0.0f;
                    v1 = __bfloat162float(mp[1]) > 0.0f ? v1 : 0.0f;
                }
                const __nv_bfloat162 o = __floats2bfloat162_rn(v0, v1);
                if (!a.up) {
                    *reinterpret_cast<__nv_bfloat162*>(a.y + act_at(row, xx, a.yoff + co, a.yC, a.W)) = o;
                } else {
#pragma unroll
                    for (int dy = 0; dy < 2; ++dy)
#pragma unroll
                        for (int dx = 0; dx < 2; ++dx)
                            *reinterpret_cast<__nv_bfloat162*>(
                                a.y + act_at(2 * row + dy, 2 * xx + dx, a.yoff + co, a.yC, 2 * a.W)) = o;
                }
            }
        }
}

// ------------------------------------------- convolution, halo-tile form
// For images at least 16 wide: a CTA computes an 8 x 16 pixel tile of one
// image for NT = 32 output channels.  Per 32-channel chunk it stages the
// 10 x 18 input halo once and the weights of all nine taps, then runs the
// nine taps from shared memory (ldmatrix row addresses point at the shifted
// halo pixel), so each input pixel is fetched once per chunk instead of once
// per tap.  Chunks are double buffered.  Same epilogue as k_conv3.
constexpr int HT_H = 8, HT_W = 16, HT_HH = HT_H + 2, HT_HW = HT_W + 2;
constexpr int HT_NT = 32;
constexpr int HT_A = HT_HH * HT_HW * CV_LD;   // halves per halo stage
constexpr int HT_B = 9 * HT_NT * CV_LD;       // halves per weight stage

__host__ __device__ constexpr size_t halo_smem_bytes() { return (size_t)2 * (HT_A + HT_B) * 2; }

__global__ void __launch_bounds__(256) k_conv3_halo(ConvArgs a) {
    grid_begin();
    extern __shared__ __align__(128) bf16 ht_smem[];
    bf16* sA = ht_smem;                 // [2][HT_A]
    bf16* sB = ht_smem + 2 * HT_A;      // [2][HT_B]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int tiles_x = a.W / HT_W, tiles_y = a.H / HT_H;
    int b = blockIdx.x;
    const int tx0 = (b % tiles_x) * HT_W;
    b /= tiles_x;
    const int ty0 = (b % tiles_y) * HT_H;
    const int n = b / tiles_y;
    const int co0 = blockIdx.y * HT_NT;
    const int kchunks = a.Cin / CV_KC;

    auto load_chunk = [&](int c, int s) {
        const int c0 = c * CV_KC;
        bf16* A = sA + s * HT_A;
        // consecutive threads take consecutive halo pixels of one channel group
        for (int q = tid; q < HT_HH * HT_HW * 4; q += 256) {
            const int part = q / (HT_HH * HT_HW), hp = q - part * (HT_HH * HT_HW);
            const int hy = hp / HT_HW, hx = hp - (hp / HT_HW) * HT_HW;
            const int yy = wrap(ty0 + hy - 1, a.H), xx = wrap(tx0 + hx - 1, a.W);
            cp_async16(A + hp * CV_LD + part * 8,
                       a.x + act_at((long long)n * a.H + yy, xx, a.xoff + c0 + part * 8, a.xC, a.W), true);
        }
        bf16* B = sB + s * HT_B;
        for (int q = tid; q < 9 * HT_NT * 4; q += 256) {
            const int row = q >> 2, part = q & 3;  // row = tap * NT + co
            const int tap = row / HT_NT, co = row - (row / HT_NT) * HT_NT;
            cp_async16(B + row * CV_LD + part * 8, a.w + ((long long)(co0 + co) * 9 + tap) * a.Cin + c0 + part * 8,
                       true);
        }
    };

    const int wm = warp & 3, wn = warp >> 2;
    constexpr int WN = HT_NT / 2;   // 16 columns per warp
    constexpr int NI = WN / 8;      // 2
    float acc[2][NI][4];
#pragma unroll
    for (int mi = 0; mi < 2; ++mi)
#pragma unroll
        for (int ni = 0; ni < NI; ++ni)
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[mi][ni][k] = 0.0f;
    const int q = lane >> 3, rr = lane & 7;
    // halo index of this lane's A row (tap centre) for the two m16 tiles
    int hbase[2];
#pragma unroll
    for (int mi = 0; mi < 2; ++mi) {
        const int r = wm * 32 + mi * 16 + rr + (q & 1) * 8;  // pixel row of the tile
        hbase[mi] = (r / HT_W + 1) * HT_HW + (r % HT_W) + 1;
    }

    load_chunk(0, 0);
    cp_async_commit();
    for (int c = 0; c < kchunks; ++c) {
        const int s = c & 1;
        if (c + 1 < kchunks) {
            load_chunk(c + 1, s ^ 1);
            cp_async_commit();
            cp_async_wait<1>();
        } else {
            cp_async_wait<0>();
        }
        __syncthreads();
        const bf16* A = sA + s * HT_A;
        const bf16* B = sB + s * HT_B;
#pragma unroll 1
        for (int tap = 0; tap < 9; ++tap) {
            const int off = (tap / 3 - 1) * HT_HW + (tap % 3 - 1);
#pragma unroll
            for (int kk = 0; kk < CV_KC; kk += 16) {
                uint32_t af[2][4];
#pragma unroll
                for (int mi = 0; mi < 2; ++mi) ldsm_x4(af[mi], A + (hbase[mi] + off) * CV_LD + kk + (q >> 1) * 8);
                uint32_t bf[4];
                ldsm_x4(bf, B + (tap * HT_NT + wn * WN + rr + (q >> 1) * 8) * CV_LD + kk + (q & 1) * 8);
#pragma unroll
                for (int mi = 0; mi < 2; ++mi) {
                    mma_bf16(acc[mi][0], af[mi], bf[0], bf[1]);
                    mma_bf16(acc[mi][1], af[mi], bf[2], bf[3]);
                }
            }
        }
        __syncthreads();  // the stage is refilled two chunks later
    }

    const int g = lane >> 2, t4 = lane & 3;
#pragma unroll
    for (int mi = 0; mi < 2; ++mi)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = wm * 32 + mi * 16 + g + h * 8;
            const int yy = ty0 + r / HT_W, xx = tx0 + r % HT_W;
            const long long row = (long long)n * a.H + yy;
#pragma unroll
            for (int ni = 0; ni < NI; ++ni) {
                const int co = co0 + wn * WN + ni * 8 + 2 * t4;
                float v0 = acc[mi][ni][2 * h], v1 = acc[mi][ni][2 * h + 1];
                if (a.bias) {
                    v0 += a.bias[co];
                    v1 += a.bias[co + 1];
                }
                if (a.relu) {
                    v0 = fmaxf(v0, 0.0f);
                    v1 = fmaxf(v1, 0.0f);
                }
                if (a.mask) {
                    const bf16* mp = a.mask + act_at(row, xx, a.moff + co, a.mC, a.W);
                    v0 = __bfloat162float(mp[0]) > 0.0f ? v0 : 0.0f;
                    v1 = __bfloat162float(mp[1]) > 0.0f ? v1 : 0.0f;
                }
                const __nv_bfloat162 o = __floats2bfloat162_rn(v0, v1);
                if (!a.up) {
                    *reinterpret_cast<__nv_bfloat162*>(a.y + act_at(row, xx, a.yoff + co, a.yC, a.W)) = o;
                } else {
#pragma unroll
                    for (int dy = 0; dy < 2; ++dy)
#pragma unroll
                        for (int dx = 0; dx < 2; ++dx)
                            *reinterpret_cast<__nv_bfloat162*>(
                                a.y + act_at(2 * row + dy, 2 * xx + dx, a.yoff + co, a.yC, 2 * a.W)) = o;
                }
            }
        }
}

// -------------------------------------------------------- weight gradient
struct WgradArgs {
    const bf16* g;  // gradient at the conv output: channels goff .. goff + Cout - 1 of a tensor of gC
    int gC, goff;
    const bf16* x;  // conv input view, Cin channels
    int xC, xoff;
    int Cout, Cin, N, H, W;
    int chunks_per_split;  // 32-pixel chunks per split (blockIdx.y)
    float* part;           // [splits][Cout][9][Cin]
    float* bpart;          // [splits][Cout]: bias gradient partials (centre-tap CTAs of ci tile 0)
};

template <int MT, int NT>
__global__ void __launch_bounds__(256) k_wgrad(WgradArgs a) {
    grid_begin();
    constexpr int LG = MT + 8, LX = NT + 8;
    __shared__ __align__(128) bf16 sG[2][32 * LG];
    __shared__ __align__(128) bf16 sX[2][32 * LX];
    constexpr int WM = MT / 16, WNW = 8 / WM;  // warp grid
    constexpr int WT = NT / WNW;               // columns per warp
    constexpr int NI = WT / 8;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int n_ci = a.Cin / NT;
    int b = blockIdx.x;
    const int tap = b % 9;
    b /= 9;
    const int cit = b % n_ci, cot = b / n_ci;
    const int co0 = cot * MT, ci0 = cit * NT;
    const int dy = tap / 3 - 1, dx = tap % 3 - 1;
    const int HW = a.H * a.W;
    const int M = a.N * HW;
    const int nchunks = (M + 31) / 32;
    const int c_begin = blockIdx.y * a.chunks_per_split;
    const int c_end = min(c_begin + a.chunks_per_split, nchunks);

    auto load = [&](int c, int s) {
        for (int qq = tid; qq < 32 * MT / 8; qq += 256) {
            const int px = qq / (MT / 8), pp = qq % (MT / 8);
            const int m = c * 32 + px;
            const bool v = m < M;
            const int mm = v ? m : 0;
            cp_async16(&sG[s][px * LG + pp * 8], a.g + act_at(mm / a.W, mm % a.W, a.goff + co0 + pp * 8, a.gC, a.W),
                       v);
        }
        for (int qq = tid; qq < 32 * NT / 8; qq += 256) {
            const int px = qq / (NT / 8), pp = qq % (NT / 8);
            const int m = c * 32 + px;
            const bool v = m < M;
            const int mm = v ? m : 0;
            const int n = mm / HW;
            const int r = mm - n * HW;
            const int yy = wrap(r / a.W + dy, a.H), xx = wrap(r % a.W + dx, a.W);
            cp_async16(&sX[s][px * LX + pp * 8],
                       a.x + act_at((long long)n * a.H + yy, xx, a.xoff + ci0 + pp * 8, a.xC, a.W), v);
        }
    };

    const int wm = warp % WM, wn = warp / WM;
    float acc[NI][4];
#pragma unroll
    for (int ni = 0; ni < NI; ++ni)
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[ni][k] = 0.0f;
    const int q = lane >> 3, rr = lane & 7;
    const bool do_bias = tap == 4 && cit == 0;
    float bsum = 0.0f;
    if (c_begin < c_end) {
        load(c_begin, 0);
        cp_async_commit();
    }
    for (int c = c_begin; c < c_end; ++c) {
        const int s = (c - c_begin) & 1;
        if (c + 1 < c_end) {
            load(c + 1, s ^ 1);
            cp_async_commit();
            cp_async_wait<1>();
        } else {
            cp_async_wait<0>();
        }
        __syncthreads();
        if (do_bias && tid < MT)
#pragma unroll 8
            for (int px = 0; px < 32; ++px) bsum += __bfloat162float(sG[s][px * LG + tid]);
#pragma unroll
        for (int kk = 0; kk < 32; kk += 16) {
            uint32_t af[4];
            // A[m = co][k = px] from sG[px][co]: transposed 8x8 loads
            ldsm_x4_t(af, &sG[s][(kk + rr + (q >> 1) * 8) * LG + wm * 16 + (q & 1) * 8]);
#pragma unroll
            for (int ni = 0; ni < NI; ++ni) {
                uint32_t b0, b1;
                ldsm_x2_t(b0, b1, &sX[s][(kk + rr + (q & 1) * 8) * LX + wn * WT + ni * 8]);
                mma_bf16(acc[ni], af, b0, b1);
            }
        }
        __syncthreads();
    }
    if (do_bias && tid < MT) a.bpart[(long long)blockIdx.y * a.Cout + co0 + tid] = bsum;
    const int g = lane >> 2, t4 = lane & 3;
    float* out = a.part + (long long)blockIdx.y * a.Cout * 9 * a.Cin;
#pragma unroll
    for (int ni = 0; ni < NI; ++ni)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int co = co0 + wm * 16 + g + h * 8;
            const int ci = ci0 + wn * WT + ni * 8 + 2 * t4;
            float* o = out + ((long long)co * 9 + tap) * a.Cin + ci;
            o[0] = acc[ni][2 * h];
            o[1] = acc[ni][2 * h + 1];
        }
}

// Weight gradient, halo-tile form (images at least 16 wide): a CTA owns a
// 32 (co) x 32 (ci) block for all nine taps and walks a range of 8 x 16
// pixel tiles; per tile it stages the output gradient (128 pixels x 32 co)
// and the 10 x 18 input halo (32 ci) once; the A fragment (gradient,
// transposed) of a 16-pixel K step is loaded once and used for all nine taps,
// whose B fragments come from the halo at the shifted pixel rows.  Warp w owns
// co rows 16 (w & 1) .. +15 and ci columns 8 (w >> 1) .. +7 of every tap.
struct WgradHaloArgs {
    const bf16* g;  // gradient at the conv output (channels goff .. of a tensor of gC)
    int gC, goff;
    const bf16* x;  // conv input view
    int xC, xoff;
    int Cout, Cin, N, H, W;
    int tiles_per_split;  // pixel tiles per split (blockIdx.y)
    float* part;          // [splits][Cout][9][Cin]
    float* bpart;         // [splits][Cout] (ci tile 0 CTAs)
};

constexpr int WH_G = HT_H * HT_W * CV_LD;       // halves per gradient stage
constexpr int WH_X = HT_HH * HT_HW * CV_LD;     // halves per halo stage
__host__ __device__ constexpr size_t wgrad_halo_smem_bytes() { return (size_t)2 * (WH_G + WH_X) * 2; }

__global__ void __launch_bounds__(256) k_wgrad_halo(WgradHaloArgs a) {
    grid_begin();
    extern __shared__ __align__(128) bf16 wh_smem[];
    bf16* sG = wh_smem;              // [2][WH_G]: [pixel][co]
    bf16* sX = wh_smem + 2 * WH_G;   // [2][WH_X]: [halo pixel][ci]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int n_ci = a.Cin / 32;
    const int cit = blockIdx.x % n_ci, cot = blockIdx.x / n_ci;
    const int co0 = cot * 32, ci0 = cit * 32;
    const int tiles_x = a.W / HT_W, tiles_y = a.H / HT_H;
    const int n_tiles = a.N * tiles_x * tiles_y;
    const int t_begin = blockIdx.y * a.tiles_per_split;
    const int t_end = min(t_begin + a.tiles_per_split, n_tiles);

    auto load_tile = [&](int tile, int s) {
        int b = tile;
        const int tx0 = (b % tiles_x) * HT_W;
        b /= tiles_x;
        const int ty0 = (b % tiles_y) * HT_H;
        const int n = b / tiles_y;
        bf16* G = sG + s * WH_G;
        for (int q = tid; q < HT_H * HT_W * 4; q += 256) {
            const int part = q / (HT_H * HT_W), r = q - part * (HT_H * HT_W);
            const long long row = (long long)n * a.H + ty0 + r / HT_W;
            cp_async16(G + r * CV_LD + part * 8, a.g + act_at(row, tx0 + (r % HT_W), a.goff + co0 + part * 8, a.gC, a.W),
                       true);
        }
        bf16* X = sX + s * WH_X;
        for (int q = tid; q < HT_HH * HT_HW * 4; q += 256) {
            const int part = q / (HT_HH * HT_HW), hp = q - part * (HT_HH * HT_HW);
            const int hy = hp / HT_HW, hx = hp - (hp / HT_HW) * HT_HW;
            const int yy = wrap(ty0 + hy - 1, a.H), xx = wrap(tx0 + hx - 1, a.W);
            cp_async16(X + hp * CV_LD + part * 8,
                       a.x + act_at((long long)n * a.H + yy, xx, a.xoff + ci0 + part * 8, a.xC, a.W), true);
        }
    };

    const int wm = warp & 1, wn = warp >> 1;
    float acc[9][4];
#pragma unroll
    for (int k = 0; k < 9; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[k][j] = 0.0f;
    const bool do_bias = cit == 0;
    float bsum = 0.0f;
    const int q = lane >> 3, rr = lane & 7;

    if (t_begin < t_end) {
        load_tile(t_begin, 0);
        cp_async_commit();
    }
    for (int tile = t_begin; tile < t_end; ++tile) {
        const int s = (tile - t_begin) & 1;
        if (tile + 1 < t_end) {
            load_tile(tile + 1, s ^ 1);
            cp_async_commit();
            cp_async_wait<1>();
        } else {
            cp_async_wait<0>();
        }
        __syncthreads();
        const bf16* G = sG + s * WH_G;
        const bf16* X = sX + s * WH_X;
        if (do_bias && tid < 32)
#pragma unroll 8
            for (int px = 0; px < HT_H * HT_W; ++px) bsum += __bfloat162float(G[px * CV_LD + tid]);
#pragma unroll 1
        for (int k0 = 0; k0 < HT_H * HT_W; k0 += 16) {
            // A[m = co][k = pixel] from G[pixel][co] (transposed 8x8 loads)
            uint32_t af[4];
            ldsm_x4_t(af, G + (k0 + rr + (q >> 1) * 8) * CV_LD + wm * 16 + (q & 1) * 8);
            // this lane's B row: pixel k0 + rr + 8 (q & 1) of the tile, at its halo position
            const int pr = k0 + rr + (q & 1) * 8;
            const int hc = (pr / HT_W + 1) * HT_HW + (pr % HT_W) + 1;
#pragma unroll
            for (int tap = 0; tap < 9; ++tap) {
                const int off = (tap / 3 - 1) * HT_HW + (tap % 3 - 1);
                uint32_t b0, b1;
                ldsm_x2_t(b0, b1, X + (hc + off) * CV_LD + wn * 8);
                mma_bf16(acc[tap], af, b0, b1);
            }
        }
        __syncthreads();
    }
    if (do_bias && tid < 32) a.bpart[(long long)blockIdx.y * a.Cout + co0 + tid] = bsum;
    const int g = lane >> 2, t4 = lane & 3;
    float* out = a.part + (long long)blockIdx.y * a.Cout * 9 * a.Cin;
#pragma unroll
    for (int tap = 0; tap < 9; ++tap)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int co = co0 + wm * 16 + g + h * 8;
            const int ci = ci0 + wn * 8 + 2 * t4;
            float* o = out + ((long long)co * 9 + tap) * a.Cin + ci;
            o[0] = acc[tap][2 * h];
            o[1] = acc[tap][2 * h + 1];
        }
}

// Sums over splits of every layer's weight- and bias-gradient partials, one launch per
// backward pass: out[i] = sum_s part[s * n + i] in a fixed order.  Each job has its own
// partials, so the sums wait until all are written (one pair of launches per layer, 28
// in all, took 206 us and their gaps at 256^2 x 16, most of it latency: 55 us now).
//  narrow (weights: many outputs, a multiple of four): 128 outputs per block, four per
//   t & 31 (with one each the launch had 62,530 blocks of two loads: 137 us), t >> 5 a
//   lane of splits (s = lane, lane + 8, ...); the 8 lane sums are added in order;
//  wide (biases, head: few outputs, many partials): one output per block, a strided
//   sum per thread and a fixed-order tree.
constexpr int SUM_MAX_JOBS = 32;
struct SumJobs {
    int count;
    int first[SUM_MAX_JOBS + 1];  // first block of each job
    const float* part[SUM_MAX_JOBS];
    float* out[SUM_MAX_JOBS];
    int n[SUM_MAX_JOBS], splits[SUM_MAX_JOBS];
    bool wide[SUM_MAX_JOBS];
    bool add(const float* p, int splits_, long long n_, bool wide_, float* o) {
        if (count == SUM_MAX_JOBS) return false;
        if (count == 0) first[0] = 0;
        part[count] = p;
        out[count] = o;
        n[count] = (int)n_;
        splits[count] = splits_;
        wide[count] = wide_;
        first[count + 1] = first[count] + (int)(wide_ ? n_ : (n_ + 127) / 128);
        ++count;
        return true;
    }
};

__global__ void __launch_bounds__(256) k_sum_splits(const __grid_constant__ SumJobs a) {
    grid_begin();
    __shared__ float4 red4[8][32];
    float* red = &red4[0][0].x;
    const int t = threadIdx.x, b = blockIdx.x;
    int k = 0;
    while (b >= a.first[k + 1]) ++k;
    const int q = b - a.first[k], n = a.n[k], splits = a.splits[k];
    const float* part = a.part[k];
    if (a.wide[k]) {
        float s = 0.0f;
        for (int c = t; c < splits; c += 256) s += part[(long long)c * n + q];
        red[t] = s;
        __syncthreads();
        for (int w = 128; w > 0; w >>= 1) {
            if (t < w) red[t] += red[t + w];
            __syncthreads();
        }
        if (t == 0) a.out[k][q] = red[0];
        return;
    }
    const int tx = t & 31, ty = t >> 5, i = q * 128 + 4 * tx;
    float4 s = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (i < n)
#pragma unroll 4
        for (int c = ty; c < splits; c += 8) {
            const float4 v = *reinterpret_cast<const float4*>(part + (long long)c * n + i);
            s.x += v.x;
            s.y += v.y;
            s.z += v.z;
            s.w += v.w;
        }
    red4[ty][tx] = s;
    __syncthreads();
    if (t < 128 && q * 128 + t < n) {
        float v = 0.0f;
#pragma unroll
        for (int c = 0; c < 8; ++c) v += red[c * 128 + t];
        a.out[k][q * 128 + t] = v;
    }
}

// ------------------------------------------------------ element-wise parts
// network input: 3 float32 planes [P][3] (pixel-major) -> BF16, 32 channels
// (zero padded); one thread per (row, channel group, x), x fastest
__global__ void k_input(const float* in, long long rows, int W, bf16* __restrict__ x0) {
    grid_begin();
    const long long total = rows * 4 * W;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(i % W);
        const long long t = i / W;
        const int g = (int)(t % 4);
        const long long p = (t / 4) * W + x;
        float f[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        if (g == 0)
#pragma unroll
            for (int c = 0; c < 3; ++c) f[c] = in[p * 3 + c];
        *reinterpret_cast<uint4*>(x0 + i * 8) = pack8(f);  // act_at(row, x, 8 g, 32, W) = 8 i
    }
}

// 2x2 average pool of a view (H, W: input size) into a dense tensor of
// N x H/2 x W/2 pixels and C channels; one thread per output (row, group, x)
__global__ void k_pool(const bf16* s, int sC, int soff, int C, int N, int H, int W,
                       bf16* __restrict__ out) {
    grid_begin();
    const int C8 = C / 8, H2 = H / 2, W2 = W / 2;
    const long long total = (long long)N * H2 * C8 * W2;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(i % W2);
        const long long t = i / W2;
        const int c8 = (int)(t % C8);
        const long long row = t / C8;  // n H2 + y
        float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
        for (int dy = 0; dy < 2; ++dy)
#pragma unroll
            for (int dx = 0; dx < 2; ++dx) {
                float f[8];
                unpack8(*reinterpret_cast<const uint4*>(s + act_at(2 * row + dy, 2 * x + dx, soff + c8 * 8, sC, W)), f);
#pragma unroll
                for (int k = 0; k < 8; ++k) acc[k] += f[k];
            }
#pragma unroll
        for (int k = 0; k < 8; ++k) acc[k] *= 0.25f;
        *reinterpret_cast<uint4*>(out + i * 8) = pack8(acc);  // act_at(row, x, 8 c8, C, W2) = 8 i
    }
}

// gradient through nearest upsampling: out (coarse, dense, C channels) at
// (y, x) = (sum of the 2x2 fine block of g) * (mask at fine (2y, 2x) > 0)
__global__ void k_up_bwd(const bf16* g, int gC, int goff, const bf16* mask, int mC,
                         int moff, int C, int N, int H, int W, bf16* __restrict__ out) {
    grid_begin();
    const int C8 = C / 8, H2 = H / 2, W2 = W / 2;
    const long long total = (long long)N * H2 * C8 * W2;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(i % W2);
        const long long t = i / W2;
        const int c8 = (int)(t % C8);
        const long long row = t / C8;  // n H2 + y
        float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
        for (int dy = 0; dy < 2; ++dy)
#pragma unroll
            for (int dx = 0; dx < 2; ++dx) {
                float f[8];
                unpack8(*reinterpret_cast<const uint4*>(g + act_at(2 * row + dy, 2 * x + dx, goff + c8 * 8, gC, W)), f);
#pragma unroll
                for (int k = 0; k < 8; ++k) acc[k] += f[k];
            }
        float mk[8];
        unpack8(*reinterpret_cast<const uint4*>(mask + act_at(2 * row, 2 * x, moff + c8 * 8, mC, W)), mk);
#pragma unroll
        for (int k = 0; k < 8; ++k) acc[k] = mk[k] > 0.0f ? acc[k] : 0.0f;
        *reinterpret_cast<uint4*>(out + i * 8) = pack8(acc);
    }
}

// skip gradient: out (fine, dense, C channels) at p =
// (gp[parent(p)] / 4 + gcat[p]) * (s[p] > 0), gp coarse dense with C channels
__global__ void k_skip_bwd(const bf16* gp, const bf16* gcat, int gC, int goff,
                           const bf16* s, int sC, int soff, int C, int N, int H, int W,
                           bf16* __restrict__ out) {
    grid_begin();
    const int C8 = C / 8;
    const long long total = (long long)N * H * C8 * W;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(i % W);
        const long long t = i / W;
        const int c8 = (int)(t % C8);
        const long long row = t / C8;  // n H + y; its parent row is row / 2 (H even)
        float a[8], b[8], m[8];
        unpack8(*reinterpret_cast<const uint4*>(gp + act_at(row / 2, x / 2, c8 * 8, C, W / 2)), a);
        unpack8(*reinterpret_cast<const uint4*>(gcat + act_at(row, x, goff + c8 * 8, gC, W)), b);
        unpack8(*reinterpret_cast<const uint4*>(s + act_at(row, x, soff + c8 * 8, sC, W)), m);
#pragma unroll
        for (int k = 0; k < 8; ++k) a[k] = m[k] > 0.0f ? 0.25f * a[k] + b[k] : 0.0f;
        *reinterpret_cast<uint4*>(out + i * 8) = pack8(a);
    }
}

// ------------------------------------------------------------------ head
// y[p][j] = sum_c Wh[j][c] h[p][c] + bh[j], j = 0, 1 (FP32 weights)
template <int C>
__global__ void k_head_fwd(const bf16* h, const float* Wh, const float* bh, long long P, int W,
                           float* __restrict__ y) {
    grid_begin();
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < P; p += (long long)gridDim.x * blockDim.x) {
        float y0 = bh[0], y1 = bh[1];
        const long long row = p / W;
        const int x = (int)(p - row * W);
#pragma unroll
        for (int c8 = 0; c8 < C / 8; ++c8) {
            float f[8];
            unpack8(*reinterpret_cast<const uint4*>(h + act_at(row, x, c8 * 8, C, W)), f);
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                y0 += Wh[c8 * 8 + k] * f[k];
                y1 += Wh[C + c8 * 8 + k] * f[k];
            }
        }
        y[p * 2] = y0;
        y[p * 2 + 1] = y1;
    }
}

// Head forward + squared error + backward over a contiguous pixel range per
// block.  gh[p][c] = (sum_j gy_j Wh[j][c]) * (h > 0), gy = 2 (y - t) / count.
// Per-block partials: pw[block][2C + 2] (dWh then dbh), pl[block] (sum of squares).
template <int C>
__global__ void __launch_bounds__(256) k_head_bwd(const bf16* h, const float* Wh, const float* bh, const float* tgt,
                                                   long long P, int W, int rows_per_block, float inv_count2,
                                                   bf16* __restrict__ gh, float* __restrict__ pw,
                                                   double* __restrict__ pl) {
    grid_begin();
    constexpr int NV = 2 * C + 2;
    __shared__ float sw[8][NV];
    __shared__ double sl[8];
    float acc[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) acc[k] = 0.0f;
    double loss = 0.0;
    const long long p0 = (long long)blockIdx.x * rows_per_block;
    const long long p1 = min(p0 + rows_per_block, P);
    for (long long p = p0 + threadIdx.x; p < p1; p += blockDim.x) {
        float hv[C];
        const long long row = p / W;
        const int x = (int)(p - row * W);
#pragma unroll
        for (int c8 = 0; c8 < C / 8; ++c8) {
            float f[8];
            unpack8(*reinterpret_cast<const uint4*>(h + act_at(row, x, c8 * 8, C, W)), f);
#pragma unroll
            for (int k = 0; k < 8; ++k) hv[c8 * 8 + k] = f[k];
        }
        float y0 = bh[0], y1 = bh[1];
#pragma unroll
        for (int c = 0; c < C; ++c) {
            y0 += Wh[c] * hv[c];
            y1 += Wh[C + c] * hv[c];
        }
        const float d0 = y0 - tgt[p * 2], d1 = y1 - tgt[p * 2 + 1];
        loss += (double)d0 * d0 + (double)d1 * d1;
        const float g0 = d0 * inv_count2, g1 = d1 * inv_count2;
        float gv[C];
#pragma unroll
        for (int c = 0; c < C; ++c) {
            gv[c] = hv[c] > 0.0f ? g0 * Wh[c] + g1 * Wh[C + c] : 0.0f;
            acc[c] += g0 * hv[c];
            acc[C + c] += g1 * hv[c];
        }
        acc[2 * C] += g0;
        acc[2 * C + 1] += g1;
#pragma unroll
        for (int c8 = 0; c8 < C / 8; ++c8) {
            float f[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) f[k] = gv[c8 * 8 + k];
            *reinterpret_cast<uint4*>(gh + act_at(row, x, c8 * 8, C, W)) = pack8(f);
        }
    }
    // warp then block reduction in a fixed order
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        float v = acc[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) sw[warp][k] = v;
    }
    for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
    if (lane == 0) sl[warp] = loss;
    __syncthreads();
    for (int k = threadIdx.x; k < NV; k += blockDim.x) {
        float v = 0.0f;
        for (int w = 0; w < 8; ++w) v += sw[w][k];
        pw[(long long)blockIdx.x * NV + k] = v;
    }
    if (threadIdx.x == 0) {
        double v = 0.0;
        for (int w = 0; w < 8; ++w) v += sl[w];
        pl[blockIdx.x] = v;
    }
}

// *out = sum of n doubles: strided per-thread sums, fixed-order tree (one block of 256)
__global__ void __launch_bounds__(256) k_sum_doubles(const double* part, int n, double* __restrict__ out) {
    grid_begin();
    __shared__ double red[256];
    double s = 0.0;
    for (int k = threadIdx.x; k < n; k += 256) s += part[k];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = red[0];
}

// ------------------------------------------------------------------ Adam
// Element (co, tap, ci) of a layer's [Cout][9][Cin] weights in the per-stage
// images of the streamed tensor-core convolution (output-channel block NB,
// 16-channel chunks): block nb, chunk c16, tap, output group (of NB / 8),
// input group (2), then the 8 x 8 core matrix (row = output channel).
__host__ __device__ __forceinline__ long long blocked_at(int co, int tap, int ci, int Cin, int NB) {
    const int nb = co / NB, cl = co % NB, c16 = ci / 16, kc = ci % 16;
    const long long o = ((((long long)nb * (Cin / 16) + c16) * 9 + tap) * (NB / 8) + cl / 8) * 2 + kc / 8;
    return o * 64 + (cl % 8) * 8 + kc % 8;
}

constexpr int AR_MAX_LAYERS = 16;
struct AdamRefreshArgs {
    float* p;
    float* m;
    float* v;
    const float* g;
    long long n;                 // parameters
    float lr, b1, b2, eps, c1, c2;
    int adam;                    // 0: only the BF16 copies of the current p
    bf16 *wb, *wt, *wbk, *wtk;   // [Cout][9][Cin], [Cin][9][Cout] (flipped taps), their stage images
    int nl;
    long long woff[AR_MAX_LAYERS], qoff[AR_MAX_LAYERS];
    int cout[AR_MAX_LAYERS], cin[AR_MAX_LAYERS];
    int nbf[AR_MAX_LAYERS], nbt[AR_MAX_LAYERS];  // stage-image blocks (0: none) of wb and wt
};

// One pass over the parameters: the Adam update (optional), then every BF16
// copy of each 3x3 weight: wb[co][tap][ci], the input-gradient form
// wt[ci][8 - tap][co] (shift_{8 - tap} = -shift_tap), and the stage images
// of both for the streamed tensor-core convolution.
__global__ void k_adam_refresh(AdamRefreshArgs a) {
    grid_begin();
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < a.n; i += (long long)gridDim.x * blockDim.x) {
        float pi = a.p[i];
        if (a.adam) {
            const float gi = a.g[i];
            const float mi = a.b1 * a.m[i] + (1.0f - a.b1) * gi;
            const float vi = a.b2 * a.v[i] + (1.0f - a.b2) * gi * gi;
            a.m[i] = mi;
            a.v[i] = vi;
            pi = pi - a.lr * (mi * a.c1) / (sqrtf(vi * a.c2) + a.eps);
            a.p[i] = pi;
        }
        for (int k = 0; k < a.nl; ++k) {
            const long long j = i - a.woff[k];
            const int Cout = a.cout[k], Cin = a.cin[k];
            if (j < 0 || j >= (long long)Cout * 9 * Cin) continue;
            const int ci = (int)(j % Cin);
            const long long r = j / Cin;
            const int tap = (int)(r % 9);
            const int co = (int)(r / 9);
            const bf16 b = __float2bfloat16_rn(pi);
            const long long q = a.qoff[k];
            a.wb[q + j] = b;
            a.wt[q + ((long long)ci * 9 + (8 - tap)) * Cout + co] = b;
            if (a.nbf[k]) a.wbk[q + blocked_at(co, tap, ci, Cin, a.nbf[k])] = b;
            if (a.nbt[k]) a.wtk[q + blocked_at(ci, 8 - tap, co, Cout, a.nbt[k])] = b;
            break;
        }
    }
}

// ------------------------------------------------------ warm-start handoff
struct WarmArgs {
    const float* pred;
    double rho_dev_scale, rho_floor, t_dev_scale;
    const double* rho0;
    const double* T0;
    double* rho;
    double* T;
    long long P;  // sites per case
};

__device__ __forceinline__ double warm_rho_hat(const WarmArgs& a, double rho0, float p) {
    return fmax(rho0 + a.rho_dev_scale * lbgb::widen(p), a.rho_floor);
}
__device__ __forceinline__ double warm_T_hat(const WarmArgs& a, double T0, float p) {
    return T0 * (1.0 + a.t_dev_scale * lbgb::widen(p));
}

constexpr int WARM_THREADS = 512;    // threads of a block
constexpr int WARM_KEEP = 12;        // sites a thread keeps in registers
constexpr int WARM_MAX_CLUSTER = 16;

// An integer that orders as the double does (min and max without the FP64 units), and back.
__device__ __forceinline__ long long order_key(double x) {
    const long long b = __double_as_longlong(x);
    return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ double of_order_key(long long k) {
    return __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffLL));
}

struct WarmShared {
    double sum[WARM_THREADS / 32][4], block_sum[4], out[4];
    long long lo[WARM_THREADS / 32], hi[WARM_THREADS / 32], block_lo, block_hi;
};

// Sums v[0..NS) (NS <= 4) and, with MINMAX, the least and greatest key over the
// cluster: lanes, warps and blocks each in a fixed order.  The first warp of each block
// then calls fin(sums, lo, hi, out[4]) and every thread returns its out: at one
// FP64 warp operation in 16 cycles, sixteen warps repeating the last additions and
// divisions cost more than the passes over the sites.
template <int NS, bool MINMAX, class Fin>
__device__ __forceinline__ void cluster_reduce(const double (&vin)[NS], long long lo, long long hi, WarmShared& sh,
                                               double (&out)[4], Fin fin) {
    namespace cg = cooperative_groups;
    static_assert(WARM_THREADS == 512 && WARM_MAX_CLUSTER == 16 && NS <= 4, "half a warp joins them");
    constexpr unsigned ALL = 0xffffffffu;
    cg::cluster_group cl = cg::this_cluster();
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    // the first two exchanges halve the values that a lane carries: six additions for
    // four sums; lanes 8 k .. 8 k + 7 then hold value k
    double v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = k < NS ? vin[k < NS ? k : 0] : 0.0;
    const bool up16 = lane & 16, up8 = lane & 8;
    double x = up16 ? v[2] : v[0];
    x += __shfl_xor_sync(ALL, up16 ? v[0] : v[2], 16);
    if (NS > 1) {
        double y = up16 ? v[3] : v[1];
        y += __shfl_xor_sync(ALL, up16 ? v[1] : v[3], 16);
        const double send = up8 ? x : y;
        x = (up8 ? y : x) + __shfl_xor_sync(ALL, send, 8);
    } else {
        x += __shfl_xor_sync(ALL, x, 8);
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(ALL, x, o);
    if ((lane & 7) == 0) sh.sum[warp][lane >> 3] = x;
    if (MINMAX) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lo = min(lo, __shfl_xor_sync(ALL, lo, o));
            hi = max(hi, __shfl_xor_sync(ALL, hi, o));
        }
        if (lane == 0) {
            sh.lo[warp] = lo;
            sh.hi[warp] = hi;
        }
    }
    __syncthreads();
    // half a warp joins the sixteen values of one sum (of the warps, then of the blocks)
    const int k = t >> 4, l = t & 15;
    auto join = [&](double a) {
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) a += __shfl_xor_sync(ALL, a, o);
        return a;
    };
    auto join_keys = [&] {
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) {
            lo = min(lo, __shfl_xor_sync(ALL, lo, o));
            hi = max(hi, __shfl_xor_sync(ALL, hi, o));
        }
    };
    if (t < 64) {
        const double a = join(sh.sum[l][k]);
        if (l == 0) sh.block_sum[k] = a;
    } else if (MINMAX && t < 96) {
        lo = sh.lo[l];
        hi = sh.hi[l];
        join_keys();
        if (t == 64) {
            sh.block_lo = lo;
            sh.block_hi = hi;
        }
    }
    cl.sync();
    const int blocks = (int)cl.num_blocks();
    if (t < 32) {
        // lanes 0 - 15: sums 0 and 2; lanes 16 - 31: sums 1 and 3
        double s[4];
#pragma unroll
        for (int q = 0; q < (NS > 2 ? 2 : 1); ++q) {
            const double a = join(l < blocks ? *cl.map_shared_rank(&sh.block_sum[2 * q + k], l) : 0.0);
            s[2 * q] = __shfl_sync(ALL, a, 0);
            s[2 * q + 1] = __shfl_sync(ALL, a, 16);
        }
        if (MINMAX) {
            const int c = l < blocks ? l : 0;
            lo = *cl.map_shared_rank(&sh.block_lo, c);
            hi = *cl.map_shared_rank(&sh.block_hi, c);
            join_keys();
        }
        double o[4] = {0.0, 0.0, 0.0, 0.0};
        fin(s, of_order_key(lo), of_order_key(hi), o);
        if (t == 0) {
#pragma unroll
            for (int q = 0; q < 4; ++q) sh.out[q] = o[q];
        }
    }
    cl.sync();  // (and no block overwrites its values before all have read them)
#pragma unroll
    for (int q = 0; q < 4; ++q) out[q] = sh.out[q];
}

// Cases of at most WARM_BLOCK_SITES sites: one block of 256 threads per case, each pass
// from the inputs.  Little shared memory and few registers, so eight blocks share an SM;
// the cluster kernel below has one block of 512 threads on an SM, whose three reductions
// alone take 25 us.  A case of 16^2 11.4 us (cluster kernel 24.6), 500 of 32^2 58 (105),
// 1000 of 32^2 98 (184); at 48^2 one case 34 (26), 1000 cases 208 (211): the line
// lies between 32^2 and 48^2.
constexpr int WARM_BLOCK_SITES = 1536;

// fixed-order reduction over a block of 256 threads (op 0: sum, -1: least, 1: greatest)
template <int NV>
__device__ __forceinline__ void warm_block_reduce(double (&v)[NV], double (*red)[256], const int (&op)[NV]) {
#pragma unroll
    for (int k = 0; k < NV; ++k) red[k][threadIdx.x] = v[k];
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w)
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                const double a = red[k][threadIdx.x], b = red[k][threadIdx.x + w];
                red[k][threadIdx.x] = op[k] == 0 ? a + b : (op[k] < 0 ? fmin(a, b) : fmax(a, b));
            }
        __syncthreads();
    }
#pragma unroll
    for (int k = 0; k < NV; ++k) v[k] = red[k][0];
    __syncthreads();
}

// The handoff of k_warm (see there).
__global__ void __launch_bounds__(256) k_warm_block(WarmArgs a) {
    __shared__ double red[5][256];
    const long long base = (long long)blockIdx.x * a.P;
    auto rho_hat = [&](long long i) { return warm_rho_hat(a, a.rho0[base + i], a.pred[2 * (base + i)]); };
    auto T_hat = [&](long long i) { return warm_T_hat(a, a.T0[base + i], a.pred[2 * (base + i) + 1]); };
    double v1[5] = {0.0, 0.0, 0.0, INFINITY, -INFINITY};
    for (long long i = threadIdx.x; i < a.P; i += 256) {
        const double r = rho_hat(i);
        v1[0] += a.rho0[base + i];
        v1[1] += r;
        v1[2] += a.rho0[base + i] * a.T0[base + i];
        v1[3] = fmin(v1[3], r);
        v1[4] = fmax(v1[4], r);
    }
    const int op1[5] = {0, 0, 0, -1, 1};
    warm_block_reduce<5>(v1, red, op1);
    const double S0 = v1[0], S1 = v1[1], E0 = v1[2], lo = v1[3], hi = v1[4];
    double v2[1] = {0.0};
    for (long long i = threadIdx.x; i < a.P; i += 256) {
        const double r = rho_hat(i);
        v2[0] += (r - lo) * (hi - r);
    }
    const int op2[1] = {0};
    warm_block_reduce<1>(v2, red, op2);
    double lam = v2[0] > 0.0 ? (S0 - S1) / v2[0] : 0.0;
    const double cap = hi > lo ? 1.0 / (hi - lo) : 1.0;
    lam = fmin(fmax(lam, -cap), cap);
    double v3[2] = {0.0, 0.0};
    for (long long i = threadIdx.x; i < a.P; i += 256) {
        const double r = rho_hat(i);
        const double r1 = r + lam * (r - lo) * (hi - r);
        v3[0] += r1;
        v3[1] += r1 * T_hat(i);
    }
    const int op3[2] = {0, 0};
    warm_block_reduce<2>(v3, red, op3);
    const double fr = S0 / v3[0], ft = E0 / (fr * v3[1]);
    for (long long i = threadIdx.x; i < a.P; i += 256) {
        const double r = rho_hat(i);
        const double t = T_hat(i);  // (read before the fields, which may be the inputs, are written)
        a.rho[base + i] = (r + lam * (r - lo) * (hi - r)) * fr;
        a.T[base + i] = t * ft;
    }
}

// One cluster of 1 - 16 blocks per case.  Mass is moved inside the interfaces with
// the weight w = (rho_hat - lo)(hi - rho_hat) (zero in both bulk phases), then a
// final scaling makes it exact; T is scaled to the initial energy.  Three
// reductions over the case, each needing the one before, bound by the FP64 units
// (18 operations per site) and, below some 4,096 sites a block, by the chain of the
// reductions: with one block per case 8 cases of 256^2 kept 8 SMs busy for 727 us; a
// cluster spreads a case over up to 16 SMs, which exchange their sums through
// distributed shared memory in the same launch, and a thread keeps rho_hat, T_hat and w
// of its first WARM_KEEP sites between the passes.  8 cases of 256^2: 46 us; 86 us with
// clusters of 16 in two rounds, w formed in each pass and every warp joining the sums.
__global__ void __launch_bounds__(WARM_THREADS) k_warm(WarmArgs a) {
    namespace cg = cooperative_groups;
    __shared__ WarmShared sh;
    cg::cluster_group cl = cg::this_cluster();
    const long long base = (long long)(blockIdx.x / cl.num_blocks()) * a.P;
    const long long first = (long long)cl.block_rank() * WARM_THREADS + threadIdx.x;
    const long long step = (long long)cl.num_blocks() * WARM_THREADS;
    // of a kept site: rho_hat (then rho1), T_hat, w
    double rk[WARM_KEEP], tk[WARM_KEEP], wk[WARM_KEEP];
    auto weight = [](double r, double lo, double hi) { return (r - lo) * (hi - r); };
    // pass 1: S0 = sum rho0, S1 = sum rho_hat, E0 = sum rho0 T0, lo, hi
    double v1[3] = {0.0, 0.0, 0.0}, out[4];
    long long klo = order_key(INFINITY), khi = order_key(-INFINITY);
    auto site = [&](long long i, double& r, double& t) {
        const double r0 = a.rho0[i], t0 = a.T0[i];
        r = warm_rho_hat(a, r0, a.pred[2 * i]);
        t = warm_T_hat(a, t0, a.pred[2 * i + 1]);
        v1[0] += r0;
        v1[1] += r;
        v1[2] += r0 * t0;
        const long long key = order_key(r);
        klo = min(klo, key);
        khi = max(khi, key);
    };
    auto again = [&](long long i, double& r, double& t) {
        r = warm_rho_hat(a, a.rho0[i], a.pred[2 * i]);
        t = warm_T_hat(a, a.T0[i], a.pred[2 * i + 1]);
    };
    const long long more = first + WARM_KEEP * step;
    double r, t;
#pragma unroll
    for (int k = 0; k < WARM_KEEP; ++k)
        if (first + k * step < a.P) site(base + first + k * step, rk[k], tk[k]);
    for (long long i = more; i < a.P; i += step) site(base + i, r, t);
    double S0 = 0.0, S1 = 0.0, E0 = 0.0;  // (the first warp's)
    cluster_reduce<3, true>(v1, klo, khi, sh, out, [&](const double* s, double least, double greatest, double* o) {
        S0 = s[0];
        S1 = s[1];
        E0 = s[2];
        o[0] = least;
        o[1] = greatest;
    });
    const double lo = out[0], hi = out[1];
    // pass 2: SW = sum w
    double v2[1] = {0.0};
#pragma unroll
    for (int k = 0; k < WARM_KEEP; ++k)
        if (first + k * step < a.P) {
            wk[k] = weight(rk[k], lo, hi);
            v2[0] += wk[k];
        }
    for (long long i = more; i < a.P; i += step) {
        again(base + i, r, t);
        v2[0] += weight(r, lo, hi);
    }
    cluster_reduce<1, false>(v2, 0, 0, sh, out, [&](const double* s, double, double, double* o) {
        const double l = s[0] > 0.0 ? (S0 - S1) / s[0] : 0.0;
        const double cap = hi > lo ? 1.0 / (hi - lo) : 1.0;
        o[0] = fmin(fmax(l, -cap), cap);
    });
    const double lam = out[0];
    // pass 3: S2 = sum rho1, Q = sum rho1 T_hat
    double v3[2] = {0.0, 0.0};
#pragma unroll
    for (int k = 0; k < WARM_KEEP; ++k)
        if (first + k * step < a.P) {
            rk[k] += lam * wk[k];
            v3[0] += rk[k];
            v3[1] += rk[k] * tk[k];
        }
    for (long long i = more; i < a.P; i += step) {
        again(base + i, r, t);
        r += lam * weight(r, lo, hi);
        v3[0] += r;
        v3[1] += r * t;
    }
    cluster_reduce<2, false>(v3, 0, 0, sh, out, [&](const double* s, double, double, double* o) {
        o[0] = S0 / s[0];
        o[1] = E0 / (o[0] * s[1]);
    });
    const double fr = out[0], ft = out[1];
#pragma unroll
    for (int k = 0; k < WARM_KEEP; ++k)
        if (first + k * step < a.P) {
            a.rho[base + first + k * step] = rk[k] * fr;
            a.T[base + first + k * step] = tk[k] * ft;
        }
    for (long long i = more; i < a.P; i += step) {
        again(base + i, r, t);
        a.rho[base + i] = (r + lam * weight(r, lo, hi)) * fr;
        a.T[base + i] = t * ft;
    }
}

}  // namespace unk
