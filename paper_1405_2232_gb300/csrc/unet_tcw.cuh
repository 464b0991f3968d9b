// unet_tcw.cuh -- weight (and bias) gradient of the 3x3 circular convolution
// on the tcgen05 tensor cores, for layers with at least 64 output channels
// (levels 1 .. 3 of the network) or 32 (level 0, XM and ROWS3 below):
//   dW[co][tap][ci] = sum_p g[p][co] x[p + shift_tap][ci],   db[co] = sum_p g[p][co]
// as one GEMM per tap with M = 128 output channels (a block; rows past Cout
// are computed and dropped), N = NBW input channels (a block) and K = pixels.
//
// A CTA owns one output-channel block, one input-channel block, one kernel
// row dy (taps 3 dy .. 3 dy + 2) and a contiguous range of image row segments
// (a split of the pixels; the splits' partial sums are reduced afterwards in
// a fixed order, as for the mma.sync kernel).  With dy fixed, every output row
// y needs exactly one input row, y + dy - 1, so a stage is
//   g: the row segment of the output gradient, MB / 8 channel groups of segw
//      pixels (16 bytes each): group j, pixel p -> j * segw * 16 + p * 16;
//   x: input row y + dy - 1, NBW / 8 channel groups of segw + 16 slots (slots
//      8 .. 8 + segw - 1, the neighbours at 7 and 8 + segw): group k, slot q ->
//      GX + (k * (segw + 16) + q) * 16.
// Each arrives as one tensor copy of all its groups; the box of x starts 8 pixels to
// the left, columns outside the image are filled with zeros, and the edge warp then
// writes the wrapped neighbours over them.  (A copy per group took about 110 cycles
// each whatever its kind, more than the MMAs of the stage: with 16 pictures of 256^2 the
// eleven layers took 768 us so and 587 now, 96 -> 32 at level 0 168 and 118, 384 -> 128 at
// level 2 97 and 66.  Now the reads of the operands, 24 MMAs in 1,400 - 1,600
// cycles, and the L2 cache, which gives each row to three kernel rows, bound it.)
// Both operands are read MN-major (8 channels of one pixel are one 16-byte
// core-matrix row; 8 pixels of a K step are 128 contiguous bytes): A = g with
// its channel groups segw * 16 bytes apart, B = x with tap dx's view starting
// at slot 7 + dx.  The three accumulators (dx = 0, 1, 2; NBW TMEM columns
// each) stay in TMEM for the CTA's whole range.
//
// With XM (layers with 32 output channels and at least 64 input channels)
// the roles of the operands swap: A = x with M = 128 input channels, B = g
// with N = NA = Cout, so the 128 MMA rows are the wider side (with M = 32
// output channels three quarters of every MMA would be empty); the
// accumulators are D[ci][co] and the partial sums are written with TMEM lane
// = input channel.
//
// With ROWS3 (32 input and 32 output channels, the full-resolution layers) the input
// rows y - 1, y, y + 1 of a stage lie one after the other, so that A's 128 rows are
// three kernel rows of 32 input channels (96 used) and one pass over the pixels
// takes all nine taps: the three layers of 16 x 256^2 took 86 us each on the mma.sync kernel,
// the training step 2,464 us with them and 2,319 so.
//
// Roles: warp 0 produces (elected lane: barrier byte count and the two tensor
// copies), warp 6 writes the wrapped neighbours and passes the stage on, warp 5
// issues the MMAs (warp-wide loop, elected lane), warps 1-4 sum g for the bias
// gradient while the MMAs run (CTAs of input block 0 and dy = 1 only; their
// arrivals release the stage together with the MMA commit) and write the
// partial sums at the end (TMEM lane = output channel).  Every wait is bounded
// (bit 6 of *err on a timeout).
#pragma once

#include "unet_tcs.cuh"  // ts_tma, ts_mma1

namespace unk {

constexpr int TW_THREADS = 224;
constexpr int TW_MMA_WARP = 5, TW_EDGE_WARP = 6;
constexpr int TW_MB = 128;

struct WgradTcArgs {
    const bf16* g;  // gradient at the conv output: channels goff .. of a tensor of gC
    int gC, goff;
    const bf16* x;  // conv input: channels xoff .. of a tensor of xC
    int xC, xoff;
    int Cout, Cin, N, H, W;
    int splits, items_per_split;  // row segments per split
    int ggroups, xgroups;         // channel groups of a stage's copies (the maps' boxes)
    float* part;                  // [splits][Cout][9][Cin]
    float* bpart;                 // [splits][Cout]
    int* err;
};

__host__ __device__ constexpr int tw_segw(int W) { return W < TC_M ? W : TC_M; }
// channel groups staged per stage: g (output channels) and x (input channels)
__host__ __device__ constexpr int tw_gplanes(int NA, bool XM) { return XM ? NA / 8 : TW_MB / 8; }
__host__ __device__ constexpr int tw_xplanes(int NA, bool XM) { return XM ? TW_MB / 8 : NA / 8; }
__host__ __device__ constexpr int tw_gbytes(int NA, bool XM, int segw) { return tw_gplanes(NA, XM) * segw * 16; }
__host__ __device__ constexpr int tw_xrow(int segw) { return segw + 2 * TC_BODY; }  // slots of an x row
__host__ __device__ constexpr int tw_xbytes(int NA, bool XM, int segw) { return tw_xplanes(NA, XM) * tw_xrow(segw) * 16; }
__host__ __device__ constexpr int tw_stage_bytes(int NA, bool XM, int segw) {
    return tw_gbytes(NA, XM, segw) + tw_xbytes(NA, XM, segw);
}
__host__ __device__ constexpr int tw_stages(int NA, bool XM, int segw) {
    return (int)((232448 - 1024 - 512) / tw_stage_bytes(NA, XM, segw)) > 6
               ? 6
               : (int)((232448 - 1024 - 512) / tw_stage_bytes(NA, XM, segw));
}
__host__ __device__ constexpr size_t tw_smem_bytes(int NA, bool XM, int segw) {
    return (size_t)tw_stages(NA, XM, segw) * tw_stage_bytes(NA, XM, segw) + 512 + 1024;
}
// input-channel block of a layer (0: not for this kernel)
__host__ __device__ constexpr int tw_block(int Cin) {
    return Cin % 128 == 0 ? 128 : (Cin % 64 == 0 ? 64 : (Cin % 32 == 0 ? 32 : 0));
}

template <int NA, bool XM, bool ROWS3 = false>
__global__ void __launch_bounds__(TW_THREADS, 1)
    k_wgrad_tc(WgradTcArgs a, const __grid_constant__ CUtensorMap gmap, const __grid_constant__ CUtensorMap xmap,
               int stages) {
    // NA: N of the MMA (input-channel block; with XM the output channels)
    constexpr int NBW = XM ? TW_MB : NA;            // input channels of a block
    constexpr int XG = tw_xplanes(NA, XM);          // input channel groups staged
    constexpr uint32_t COLS = 3 * NA <= 128 ? 128u : (3 * NA <= 256 ? 256u : 512u);
    static_assert(2 * XG <= 32, "one edge value per lane");
    static_assert(!ROWS3 || XM, "the rows stack along the 128 rows of A");
    extern __shared__ __align__(1024) uint8_t tw_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(tw_raw) + 1023) & ~uintptr_t(1023));
    const int H = a.H, W = a.W;
    const int segw = tw_segw(W);
    const int segs = W / segw;
    const int GB = tw_gbytes(NA, XM, segw);
    const int SB = GB + tw_xbytes(NA, XM, segw);
    uint8_t* sS = base;                                                     // [stages][SB]
    uint64_t* full = reinterpret_cast<uint64_t*>(sS + (size_t)stages * SB);  // [stages]
    uint64_t* empty = full + 6;                                             // [stages]
    uint64_t* ready = empty + 6;                                            // [stages]
    uint64_t* mdone = ready + 6;
    uint32_t* s_tmem = reinterpret_cast<uint32_t*>(mdone + 1);
    volatile int* s_abort = reinterpret_cast<volatile int*>(s_tmem + 1);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // unit: output block, input block, dy, split (split outermost: the CTAs
    // working on the same pixels run together)
    const int ncob = XM ? 1 : (a.Cout + TW_MB - 1) / TW_MB;
    const int ncib = ROWS3 ? 1 : (a.Cin + NBW - 1) / NBW;
    int u = blockIdx.x;
    const int cob = u % ncob;
    u /= ncob;
    const int cib = u % ncib;
    u /= ncib;
    const int dy = ROWS3 ? 0 : u % 3;
    const int split = ROWS3 ? u : u / 3;
    const int items = a.N * H * segs;
    const int it0 = split * a.items_per_split;
    const int it1 = min(it0 + a.items_per_split, items);
    const int nitems = it1 > it0 ? it1 - it0 : 0;
    const bool do_bias = ROWS3 || (cib == 0 && dy == 1);
    const int cg0 = (a.goff + cob * TW_MB) / 8;         // first g channel group of the block
    const int gvalid = XM ? a.Cout / 8 : min(TW_MB, a.Cout - cob * TW_MB) / 8;  // g groups that exist
    const int xg0 = (a.xoff + cib * NBW) / 8;
    // x groups that exist (ROWS3: those of the three rows, one after the other)
    const int xvalid = ROWS3 ? 3 * a.xgroups : min(NBW, a.Cin - cib * NBW) / 8;
    const int EDGES = 2 * xvalid;                        // wrapped neighbours per stage

    if (tid == 0) {
        for (int s = 0; s < stages; ++s) {
            tc_bar_init(&full[s], 1);
            tc_bar_init(&ready[s], 1);
            tc_bar_init(&empty[s], do_bias ? 1 + 4 : 1);
        }
        tc_bar_init(mdone, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        *s_abort = 0;
    }
    grid_wait();
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(s_tmem)),
                     "r"(COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *s_tmem;
    grid_launch();  // (after the TMEM allocation, which the next kernel's must not come before)

    if (warp == 0) {
        // ------------------------------------------------ producer
        const uint32_t bytes = (uint32_t)(a.ggroups * segw + (ROWS3 ? 3 : 1) * a.xgroups * tw_xrow(segw)) * 16;
        int s = 0;
        uint32_t ph = 0;
        int j = 0;
        for (int i = 0; i < nitems && __shfl_sync(0xffffffffu, *s_abort, 0) == 0; ++i, ++j) {
            const int item = it0 + i;
            const int seg = item % segs;
            const int row = item / segs;  // n H + y
            const int y = row % H, n = row / H;
            const int x0 = seg * segw;
            if (j >= stages && !__all_sync(0xffffffffu, tc_bar_wait(&empty[s], ph ^ 1u))) {
                if (lane == 0) {
                    *s_abort = 1;
                    if (a.err) atomicOr(a.err, 1 << 6);
                }
                break;
            }
            const uint32_t st = smem_addr(sS + (size_t)s * SB);
            const uint32_t fb = smem_addr(&full[s]);
            {
                // arm with every byte of the stage's two copies (filled columns count)
                asm volatile(
                    "{\n .reg .pred e;\n .reg .b32 el;\n elect.sync el|e, 0xffffffff;\n"
                    " @e mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n}\n" ::"r"(fb),
                    "r"(bytes)
                    : "memory");
            }
            ts_tma(&gmap, st, fb, x0 / 8, cg0, row);
#pragma unroll
            for (int r = 0; r < (ROWS3 ? 3 : 1); ++r)
                ts_tma(&xmap, st + GB + r * a.xgroups * tw_xrow(segw) * 16, fb, x0 / 8 - 1, xg0,
                       n * H + wrap(y + dy + r - 1, H));
            if (++s == stages) {
                s = 0;
                ph ^= 1u;
            }
        }
        if (lane == 0)
            for (int k = (j > stages ? j - stages : 0); k < j; ++k)
                (void)tc_bar_wait(&full[k % stages], (uint32_t)((k / stages) & 1));
        __syncwarp();
    } else if (warp == TW_MMA_WARP) {
        // ------------------------------------------------ MMA issue
        // kind::f16, D FP32, A and B BF16, both MN-major (bits 15, 16)
        constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) |
                                   ((uint32_t)(NA >> 3) << 17) | ((uint32_t)(TW_MB >> 4) << 24);
        // no-swizzle MN-major operands: the leading byte offset is the stride
        // between K groups (8 pixels: 128 bytes), the stride byte offset the
        // stride between MN groups (8 channels)
        // g: channel groups segw * 16 bytes apart
        const uint64_t dg0 = tc_mdesc(smem_addr(sS), 128, (uint32_t)(segw * 16));
        // x: channel groups one row with its halo apart
        const uint64_t dx0 = tc_mdesc(smem_addr(sS) + (uint32_t)(GB + (TC_BODY - 1) * 16), 128, (uint32_t)(tw_xrow(segw) * 16));
        const uint64_t da0 = XM ? dx0 : dg0, db0 = XM ? dg0 : dx0;
        const uint32_t ahi = (uint32_t)(da0 >> 32), bhi = (uint32_t)(db0 >> 32);
        const int ksteps = segw / 16;
        int s = 0;
        uint32_t fph = 0;
        bool ok = true;
        for (int i = 0; i < nitems && __shfl_sync(0xffffffffu, *s_abort, 0) == 0; ++i) {
            const uint32_t a_lo = (uint32_t)da0 + (uint32_t)s * (uint32_t)(SB >> 4);
            const uint32_t b_lo = (uint32_t)db0 + (uint32_t)s * (uint32_t)(SB >> 4);
            if (!__all_sync(0xffffffffu, tc_bar_wait(&ready[s], fph))) {
                ok = false;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int k = 0; k < ksteps; ++k) {
#pragma unroll
                for (int dx = 0; dx < 3; ++dx)
                    // the x view of tap dx starts dx slots further
                    ts_mma1(tmem + (uint32_t)(dx * NA), a_lo + (uint32_t)((XM ? dx : 0) + k * 16), ahi,
                            b_lo + (uint32_t)((XM ? 0 : dx) + k * 16), bhi, IDESC, (i > 0 || k > 0) ? 1u : 0u);
            }
            tc_commit_one(&empty[s]);
            if (++s == stages) {
                s = 0;
                fph ^= 1u;
            }
        }
        if (!ok && lane == 0) {
            *s_abort = 1;
            if (a.err) atomicOr(a.err, 1 << 6);
        }
        tc_commit_one(mdone);  // arrives once every MMA issued has completed
    } else if (warp == TW_EDGE_WARP) {
        // ------------------------------------------------ wrapped neighbours
        // lane: input group, side.  The values of the next EB items are in registers
        // while those of this one go into their slots, once the copy has filled these
        // with zeros.
        constexpr int EB = 4;
        const int ek = lane >> 1, eside = lane & 1;
        auto value = [&](int i) {
            uint4 v = make_uint4(0, 0, 0, 0);
            const int item = it0 + i, seg = item % segs, row = item / segs;
            if (lane < EDGES && i < nitems && seg == (eside ? segs - 1 : 0)) {
                const int r = ROWS3 ? ek / a.xgroups : 0;
                const int y = row % H, xrow = row - y + wrap(y + dy + r - 1, H);
                v = *reinterpret_cast<const uint4*>(
                    a.x + act_at(xrow, eside ? 0 : W - 1, (xg0 + ek - r * a.xgroups) * 8, a.xC, W));
            }
            return v;
        };
        uint8_t* slot = sS + GB + (ek * tw_xrow(segw) + (eside ? TC_BODY + segw : TC_BODY - 1)) * 16;
        uint4 cur[EB], nxt[EB];
#pragma unroll
        for (int t = 0; t < EB; ++t) nxt[t] = value(t);
        int s = 0;
        uint32_t fph = 0;
        bool ok = true;
        for (int i0 = 0; i0 < nitems && ok; i0 += EB) {
#pragma unroll
            for (int t = 0; t < EB; ++t) {
                cur[t] = nxt[t];
                nxt[t] = value(i0 + EB + t);
            }
#pragma unroll
            for (int t = 0; t < EB; ++t) {
                const int i = i0 + t;
                if (i >= nitems || !ok) break;
                if (!__all_sync(0xffffffffu, tc_bar_wait(&full[s], fph))) {
                    ok = false;
                    break;
                }
                if (lane < EDGES && (it0 + i) % segs == (eside ? segs - 1 : 0))
                    *reinterpret_cast<uint4*>(slot + (size_t)s * SB) = cur[t];
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) tc_bar_arrive(&ready[s]);
                if (++s == stages) {
                    s = 0;
                    fph ^= 1u;
                }
            }
            if (__any_sync(0xffffffffu, *s_abort != 0)) break;
        }
        if (!ok && lane == 0) {
            *s_abort = 1;
            if (a.err) atomicOr(a.err, 1 << 6);
        }
    } else {
        // ------------------------------------------------ warps 1-4: bias sums, then the partials
        const int q = warp & 3;  // TMEM lanes 32 q ..; bias: g groups q, q + 4, ..
        float bs[32];
#pragma unroll
        for (int k = 0; k < 32; ++k) bs[k] = 0.0f;
        if (do_bias) {
            int s = 0;
            uint32_t fph = 0;
            for (int i = 0; i < nitems; ++i) {
                if (!__all_sync(0xffffffffu, tc_bar_wait(&full[s], fph))) {
                    if (lane == 0) {
                        *s_abort = 1;
                        if (a.err) atomicOr(a.err, 1 << 6);
                    }
                    break;
                }
                const uint8_t* gst = sS + (size_t)s * SB;
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) {
                    const int k = q + 4 * jj;
                    if (k < gvalid) {
                        uint4 u[TC_M / 32];  // (segw <= 128)
#pragma unroll
                        for (int r = 0; r < TC_M / 32; ++r)
                            if (lane + 32 * r < segw)
                                u[r] = *reinterpret_cast<const uint4*>(gst + (k * segw + lane + 32 * r) * 16);
#pragma unroll
                        for (int r = 0; r < TC_M / 32; ++r)
                            if (lane + 32 * r < segw) {
                                float f[8];
                                unpack8(u[r], f);
#pragma unroll
                                for (int e = 0; e < 8; ++e) bs[jj * 8 + e] += f[e];
                            }
                    }
                }
                __syncwarp();
                if (lane == 0) tc_bar_arrive(&empty[s]);
                if (++s == stages) {
                    s = 0;
                    fph ^= 1u;
                }
                if (__any_sync(0xffffffffu, *s_abort != 0)) break;
            }
            // lane sums -> the warp's 32 channels (fixed order)
#pragma unroll
            for (int k = 0; k < 32; ++k)
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) bs[k] += __shfl_xor_sync(0xffffffffu, bs[k], o);
            const int k = q + 4 * (lane >> 3);
            if (k < gvalid) {
                const int co = cob * TW_MB + 8 * k + (lane & 7);
                float v = 0.0f;
#pragma unroll
                for (int i = 0; i < 32; ++i) v = (i == lane) ? bs[i] : v;
                a.bpart[(long long)split * a.Cout + co] = v;
            }
        }
        // wait for the last MMAs, then TMEM lane (32 q + lane) = output
        // channel (with XM: input channel)
        const bool done = __all_sync(0xffffffffu, tc_bar_wait(mdone, 0u));
        if (!done && lane == 0 && a.err) atomicOr(a.err, 1 << 6);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int col = 32 * q + lane;
        const int co = cob * TW_MB + col;
        const bool valid = col < (XM ? xvalid : gvalid) * 8 && nitems > 0 && done;
        const int r = ROWS3 ? col / a.Cin : 0;  // kernel row of this lane
        float* out = XM ? a.part + (long long)split * a.Cout * 9 * a.Cin + cib * NBW + (col - r * a.Cin)
                        : a.part + ((long long)split * a.Cout + co) * 9 * a.Cin;
#pragma unroll 1
        for (int dx = 0; dx < 3; ++dx) {
            const int tap = (dy + r) * 3 + dx;
#pragma unroll 1
            for (int cc = 0; cc < NA; cc += 32) {
                uint32_t v[32];
                const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(dx * NA + cc);
                asm volatile(
                    "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                    "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                    : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
                      "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
                      "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]),
                      "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]),
                      "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
                    : "r"(taddr));
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (valid && XM) {
                    // column j = output channel cc + j: [co][tap][ci], this lane's ci
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        out[((long long)(cc + j) * 9 + tap) * a.Cin] = __uint_as_float(v[j]);
                } else if (valid) {
                    float4* o4 = reinterpret_cast<float4*>(out + (long long)tap * a.Cin + cib * NBW + cc);
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        o4[k] = make_float4(__uint_as_float(v[4 * k]), __uint_as_float(v[4 * k + 1]),
                                            __uint_as_float(v[4 * k + 2]), __uint_as_float(v[4 * k + 3]));
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(COLS) : "memory");
}

}  // namespace unk
