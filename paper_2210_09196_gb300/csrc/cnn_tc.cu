// Forward pass of the learned estimator (four 3x3 convolutions 2 -> 32 -> 32 -> 32 -> 2 on a 2-row grid, dilated along
// the subcarriers by 1, 8, 16, 1; ReLU after the first three, the input added to the last) on the 5th-generation
// tensor cores: all four layers of a tile in one kernel, BF16 operands, FP32 accumulation in TMEM. Activations go
// through HBM only where the caller wants them (training).
//
// A tile is 256 subcarriers of one grid, both rows. Activations sit in shared memory channels-last, one 128-byte row
// of 64 values (r, ci) per subcarrier, so that a layer is, per 128 subcarriers,
//     D[x][(h, co)] = sum_kw sum_(r, ci) A[x + (kw - 1) dil][(r, ci)] B_kw[(h, co)][(r, ci)],
//     B_kw[(h, co)][(r, ci)] = W[co][ci][r - h + 1][kw]
// (every pair of rows h, r meets exactly one of the three kh): M = 128, N = 64, K = 3 x 64, K-major operands with
// 128-byte swizzling. A shift by 8 or 16 subcarriers moves the operand's start by one or two groups of 8 rows, so the
// dilated taps need no copies. The middle layers carry 94 % of the multiply-adds: 24 MMAs each per tile at 48 clocks,
// the time shared memory takes to deliver their operands. Layer 4 forms the 12 products (kw, h, co) of every
// subcarrier (N = 16), which are added up across neighbouring subcarriers through shared memory. Layer 1 (12 products
// per value) is on packed FP32 FMAs: as tensor-core sums its values round to another BF16 now and then, and one such
// step in a large activation moves the estimate by 1e-3 of its RMS. K runs over rows, taps and channels in the order
// (r, kw, ci) for the same reason.
//
// A tile has 256 - 2 * 25 = 206 outputs (the receptive field of the layers after the first is +-25); a grid of at most
// 256 subcarriers is one tile with nothing computed twice. Rows outside the grid are written as zeros, the "same"
// padding; 16 zero rows before and after the tile catch the taps that leave it.
//
// Four tiles are in flight per CTA (one CTA per SM), 128 threads each: while the products of some run, the threads of
// others turn accumulators into activations. A thread owns two subcarriers (a TMEM lane in each of the tile's two
// blocks) and all their channels. A layer's output takes the place of its input, whose products are over by then, so
// that four tiles fit in shared memory (two tiles with two buffers each: 240 us for the case below).
// Measured (GB300, 512 grids of 3276 subcarriers): 190 us, 460 TFLOP/s of the network's arithmetic; layer by layer through
// HBM, with layers 1 and 4 on FP32 FMAs, the same took 780 us. Bound by the threads' share: per tile about 10 k clocks of
// packed FMAs (layer 1), 5 k of bias, ReLU and packing, 6 k of waiting for products, four tiles overlapping.
// Every wait is bounded (2 s). After one that expired the CTA's outputs are NaN, the error bit is set where the caller has an
// error word, and the threads go on without waiting, so all barriers are met: no address depends on what a wait was for.
// MMAs in flight are drained (bounded) before TMEM is freed, on a barrier of its own: that of the products may be a phase
// behind by then, and a wait for its newest phase would pass at once.
#include "tc_common.cuh"

namespace pusch {
namespace {

using namespace tc;

constexpr int kRows = 256, kMargin = 16;         // subcarriers of a tile; zero rows before and after
constexpr int kHalo = 25;                        // 8 + 16 + 1
constexpr int kCtx = 4, kCtxThreads = 128, kThreads = kCtx * kCtxThreads;
constexpr uint32_t kBufBytes = (kRows + 2 * kMargin) * 128;
// shared memory: weights (layers 2 and 3 [3 kw][64][64], layer 4 [16][64], layer 1 FP32 [2 ci][3 kw][3 kh][32 co]), then
// per tile in flight the activations and the input rows
constexpr uint32_t kOffW2 = 0, kOffW3 = kOffW2 + 24576, kOffW4 = kOffW3 + 24576, kOffW1 = kOffW4 + 2048;
constexpr uint32_t kOffCtx = kOffW1 + 3072;
constexpr uint32_t kOffX = kBufBytes;
constexpr uint32_t kCtxBytes = (kOffX + 4 * (kRows + 8) * 4 + 1023) & ~1023u;
constexpr size_t kSmemBytes = 1024 + kOffCtx + kCtx * (size_t)kCtxBytes;
static_assert(kOffW3 % 1024 == 0 && kOffW4 % 1024 == 0 && kOffCtx % 1024 == 0 && kBufBytes % 1024 == 0, "atoms");

struct FwdArgs {
    int w, in_ld, acts_ld, tiles, tiles_per_grid, step, halo;
    long long acts_layer;    // elements between two layers of acts
    unsigned long long selftest_ns;   // not 0: every wait is on a barrier that nothing completes, with this limit
};

// Instruction descriptor of kind::f16 with BF16 A and B (format code 1), F32 accumulator, both K-major, M = 128.
constexpr uint32_t idesc_bf16(int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((128u >> 4) << 24);
}

__device__ __forceinline__ void ctx_sync(int ctx) {
    asm volatile("bar.sync %0, %1;" ::"r"(1 + ctx), "r"(kCtxThreads) : "memory");
}

// element (row, k) of a K-major operand of 64 BF16 per row with 128-byte swizzling
__device__ __forceinline__ uint32_t sw128(int row, int k) {
    return (uint32_t)row * 128u + ((uint32_t)((k >> 3) ^ (row & 7)) << 4) + (uint32_t)(k & 7) * 2u;
}
__global__ void __launch_bounds__(kThreads, 1)
cnn_fwd_kernel(FwdArgs g, const __nv_bfloat16 *__restrict__ in, const __nv_bfloat16 *__restrict__ P,
               float *__restrict__ y, __nv_bfloat16 *__restrict__ acts, uint32_t *__restrict__ err) {
    chain_wait(in, P, y, acts, err);
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bars[kCtx], bar_drain[kCtx], bar_never;
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    __shared__ __align__(16) float s_bias[3][32];
    __shared__ float s_bias4[2];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t *gb = smem_raw + (base - raw);
    const int tid = threadIdx.x, warp = tid >> 5;
    volatile int *abort = &s_abort;

    // ---------------------------------------------------------------- weights, zero margins
    for (uint32_t i = tid; i < (kOffCtx + kCtx * kCtxBytes) / 16; i += kThreads)
        reinterpret_cast<uint4 *>(gb)[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    constexpr int kP1 = 32 * 2 * 9, kP2 = 32 * 32 * 9;
    const __nv_bfloat16 *W1 = P, *W2 = W1 + kP1 + 32, *W3 = W2 + kP2 + 32, *W4 = W3 + kP2 + 32;
    auto put = [&](uint32_t off, __nv_bfloat16 v) { *reinterpret_cast<__nv_bfloat16 *>(gb + off) = v; };
    for (int i = tid; i < kP2; i += kThreads) {
        const int co = i / 288, rem = i - co * 288, ci = rem / 9, kk = rem - ci * 9, kh = kk / 3, kw = kk - kh * 3;
        const __nv_bfloat16 v2 = W2[i], v3 = W3[i];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = h + kh - 1;
            if (r < 0 || r > 1) continue;
            const uint32_t o = (uint32_t)kw * 8192u + sw128(h * 32 + co, r * 32 + ci);
            put(kOffW2 + o, v2);
            put(kOffW3 + o, v3);
        }
    }
    for (int i = tid; i < kP1; i += kThreads) {
        // layer 1: [32 co][2 ci][3 kh][3 kw]
        const int co = i / 18, rem = i - co * 18, ci = rem / 9, kk = rem - ci * 9, kh = kk / 3, kw = kk - kh * 3;
        // layer 4: [2 co][32 ci][3 kh][3 kw], operand row n = kw * 4 + h * 2 + co
        const int co4 = i / 288, rem4 = i - co4 * 288, ci4 = rem4 / 9;
        const __nv_bfloat16 v4 = W4[i];
        reinterpret_cast<float *>(gb + kOffW1)[((ci * 3 + kw) * 3 + kh) * 32 + co] = __bfloat162float(W1[i]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int kk4 = rem4 - ci4 * 9, r4 = h + kk4 / 3 - 1;
            if (r4 >= 0 && r4 <= 1) put(kOffW4 + sw128((kk4 % 3) * 4 + h * 2 + co4, r4 * 32 + ci4), v4);
        }
    }
    if (tid < 32) {
        s_bias[0][tid] = __bfloat162float(W1[kP1 + tid]);
        s_bias[1][tid] = __bfloat162float(W2[kP2 + tid]);
        s_bias[2][tid] = __bfloat162float(W3[kP2 + tid]);
        if (tid < 2) s_bias4[tid] = __bfloat162float(W4[2 * 32 * 9 + tid]);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (tid == 0) {
        for (int c = 0; c < kCtx; ++c) {
            mbar_init(smem_u32(&bars[c]), 1);
            mbar_init(smem_u32(&bar_drain[c]), 1);
        }
        mbar_init(smem_u32(&bar_never), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_abort = 0;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(kCtx * 128));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();

    const int ctx = warp >> 2, w4 = warp & 3, row = tid & (kCtxThreads - 1);   // rows row and row + 128
    const uint32_t cbase = base + kOffCtx + (uint32_t)ctx * kCtxBytes;
    uint8_t *cg = gb + kOffCtx + (size_t)ctx * kCtxBytes;
    const uint32_t tm = s_tmem + (uint32_t)ctx * 128u;                     // columns of this tile: block b at 64 b
    const uint32_t tm_own = tm + ((uint32_t)w4 << 21);
    const uint32_t bar = smem_u32(&bars[ctx]);
    uint32_t phase = 0;
    float *xs = reinterpret_cast<float *>(cg + kOffX);                      // [4 (ci, r)][kRows + 8], row i at i + 1
    float *sums = reinterpret_cast<float *>(cg + kMargin * 128);            // layer 4: [256][13], over the activations

    // operands written, accumulators read: then one lane issues the products of both 128-subcarrier blocks
    auto hand_over = [&]() {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        fence_before_sync();
        ctx_sync(ctx);
    };
    auto wait_products = [&]() {
        if ((tid & 31) == 0 && !*abort) {
            if (g.selftest_ns)
                mbar_wait_sleep(smem_u32(&bar_never), 0u, abort, err, 32, g.selftest_ns);
            else
                mbar_wait_sleep(bar, phase, abort, err, 32);
        }
        __syncwarp();
        phase ^= 1u;
        fence_after_sync();
    };
    // one of the middle layers' products: taps at x - dil, x, x + dil, weights at `wo`
    auto mma_mid = [&](uint32_t wo, int dil) {
        if (w4 == 0 && elect_one()) {
            fence_after_sync();
            const uint64_t db = smem_desc(base + wo, 0, 1024, 2);
#pragma unroll 1
            for (int b = 0; b < 2; ++b) {
                const uint64_t da = smem_desc(cbase + (uint32_t)(kMargin + b * 128) * 128u, 0, 1024, 2);
                const uint64_t sh = (uint64_t)((uint32_t)dil * 128u >> 4);
                const uint64_t a[3] = {da - sh, da, da + sh};
#pragma unroll
                for (int r = 0; r < 2; ++r)
#pragma unroll
                    for (int kw = 0; kw < 3; ++kw)
#pragma unroll
                        for (int ks = 2 * r; ks < 2 * r + 2; ++ks)
                            mma<false>(tm + (uint32_t)b * 64u, a[kw] + 2u * ks, db + 512u * kw + 2u * ks, idesc_bf16(64),
                                       (kw | ks) ? 1u : 0u);
            }
            mma_commit(bar);
        }
        __syncwarp();
    };

    // the activations of a finished layer, from shared memory (the products read them meanwhile) to global memory: 32
    // subcarriers of a channel per store (16-byte pieces of 32 channels touch 32 lines and took 2.5 times as long)
    auto store_acts = [&](int layer, int gi, int x, bool mine, int r) {
        if (!mine) return;
        const uint8_t *src = cg + (size_t)(kMargin + r) * 128;
        __nv_bfloat16 *o = acts + layer * g.acts_layer + (long long)gi * 64 * g.acts_ld + x;
#pragma unroll 2
        for (int c = 0; c < 8; ++c) {
            const uint4 v = *reinterpret_cast<const uint4 *>(src + ((c ^ ((kMargin + r) & 7)) << 4));
            const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int co = (8 * c + e) & 31, h = c >> 2;
                const uint16_t bits = (uint16_t)(u[e >> 1] >> (16 * (e & 1)));
                o[(long long)(co * 2 + h) * g.acts_ld] = __ushort_as_bfloat16(bits);
            }
        }
    };
    // this thread's input values of a tile (channel ci, row r at ci * 2 + r; subcarriers row, row + 128), and those
    // next to the tile's ends
    const __nv_bfloat16 zero = __float2bfloat16_rn(0.f);
    auto fetch = [&](int t, __nv_bfloat16 (&v)[2][4], __nv_bfloat16 (&edge)[4]) {
        const int gi = t / g.tiles_per_grid, x = (t - gi * g.tiles_per_grid) * g.step - g.halo + row;
        const bool on = t < g.tiles;
        const int xe = row == 0 ? x - 1 : x + 129;
        const bool oe = on && (row == 0 || row == kCtxThreads - 1) && xe >= 0 && xe < g.w;
        const __nv_bfloat16 *ip = in + (long long)gi * 4 * g.in_ld;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
#pragma unroll
            for (int b = 0; b < 2; ++b)
                v[b][q] = on && x + 128 * b >= 0 && x + 128 * b < g.w ? ip[(long long)q * g.in_ld + x + 128 * b] : zero;
            edge[q] = oe ? ip[(long long)q * g.in_ld + xe] : zero;
        }
    };
    // layer 1: lane (half, p) holds the weights of channels 2 p, 2 p + 1 and runs over 32 subcarriers
    const int p1 = tid & 15, row1 = w4 * 64 + 2 * (tid & 16);
    __nv_bfloat16 xv[2][4], xe[4];
    fetch(blockIdx.x + ctx * gridDim.x, xv, xe);

    for (int t = blockIdx.x + ctx * gridDim.x; t < g.tiles; t += kCtx * gridDim.x) {
        const int gi = t / g.tiles_per_grid, k = t - gi * g.tiles_per_grid;
        const int o0 = k * g.step, x = o0 - g.halo + row;
        bool inside[2], mine[2];                                            // in the grid; an output of this tile
        // ---- input rows; the next tile's are on their way meanwhile
        float res[2][4];                                                    // the residual
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const int xb = x + 128 * b;
            inside[b] = xb >= 0 && xb < g.w;
            mine[b] = inside[b] && xb >= o0 && xb < o0 + g.step;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                res[b][q] = __bfloat162float(xv[b][q]);
                xs[q * (kRows + 8) + row + 128 * b + 1] = res[b][q];
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (row == 0) xs[q * (kRows + 8)] = __bfloat162float(xe[q]);
            if (row == kCtxThreads - 1) xs[q * (kRows + 8) + kRows + 1] = __bfloat162float(xe[q]);
        }
        ctx_sync(ctx);
        fetch(t + kCtx * gridDim.x, xv, xe);
        // ---- layer 1 on packed FP32 FMAs
        {
            float2 w1[2][3][3];                                             // [ci][kw][kh]
            const float2 *wp = reinterpret_cast<const float2 *>(gb + kOffW1) + p1;
#pragma unroll
            for (int ci = 0; ci < 2; ++ci)
#pragma unroll
                for (int kw = 0; kw < 3; ++kw)
#pragma unroll
                    for (int kh = 0; kh < 3; ++kh) w1[ci][kw][kh] = wp[((ci * 3 + kw) * 3 + kh) * 16];
            const float2 b1 = *reinterpret_cast<const float2 *>(&s_bias[0][2 * p1]);
            const int x1 = o0 - g.halo + row1;
            float win[4][3];                                                // the three subcarriers around row1 + i
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                win[q][1] = xs[q * (kRows + 8) + row1];
                win[q][2] = xs[q * (kRows + 8) + row1 + 1];
            }
#pragma unroll 8
            for (int i = 0; i < 32; ++i) {
                float2 a0 = b1, a1 = b1;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    win[q][0] = win[q][1];
                    win[q][1] = win[q][2];
                    win[q][2] = xs[q * (kRows + 8) + row1 + i + 2];
                }
#pragma unroll
                for (int ci = 0; ci < 2; ++ci)
#pragma unroll
                    for (int kw = 0; kw < 3; ++kw) {
                        const float2 p0 = make_float2(win[2 * ci][kw], win[2 * ci][kw]);
                        const float2 q1 = make_float2(win[2 * ci + 1][kw], win[2 * ci + 1][kw]);
                        a0 = __ffma2_rn(w1[ci][kw][1], p0, __ffma2_rn(w1[ci][kw][2], q1, a0));
                        a1 = __ffma2_rn(w1[ci][kw][0], p0, __ffma2_rn(w1[ci][kw][1], q1, a1));
                    }
                const __nv_bfloat162 c0 = __floats2bfloat162_rn(fmaxf(a0.x, 0.f), fmaxf(a0.y, 0.f));
                const __nv_bfloat162 c1 = __floats2bfloat162_rn(fmaxf(a1.x, 0.f), fmaxf(a1.y, 0.f));
                const bool in1 = x1 + i >= 0 && x1 + i < g.w;
                *reinterpret_cast<uint32_t *>(cg + sw128(kMargin + row1 + i, 2 * p1)) =
                    in1 ? *reinterpret_cast<const uint32_t *>(&c0) : 0u;
                *reinterpret_cast<uint32_t *>(cg + sw128(kMargin + row1 + i, 32 + 2 * p1)) =
                    in1 ? *reinterpret_cast<const uint32_t *>(&c1) : 0u;
            }
        }
        hand_over();
        mma_mid(kOffW2, 8);
        if (acts) {
            store_acts(0, gi, x, mine[0], row);
            store_acts(0, gi, x + 128, mine[1], row + 128);
        }
        // ---- layers 2 and 3: bias, ReLU, BF16; then the next layer's products
#pragma unroll 1
        for (int layer = 1; layer < 3; ++layer) {
            wait_products();
            uint8_t *dst = cg + (size_t)(kMargin + row) * 128;
            const int sw = (kMargin + row) & 7;                             // the same for row + 128
#pragma unroll
            for (int bh = 0; bh < 4; ++bh) {                                // block, row h
                const int b = bh >> 1, h = bh & 1;
                float v[32];
                tmem_ld32_nowait(tm_own + 32u * bh, reinterpret_cast<uint32_t(&)[32]>(v));
                tmem_wait_ld();
                uint32_t pk[16];
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const float4 bv = *reinterpret_cast<const float4 *>(&s_bias[layer][4 * c]);
                    const __nv_bfloat162 lo = __floats2bfloat162_rn(fmaxf(v[4 * c] + bv.x, 0.f), fmaxf(v[4 * c + 1] + bv.y, 0.f));
                    const __nv_bfloat162 hi =
                        __floats2bfloat162_rn(fmaxf(v[4 * c + 2] + bv.z, 0.f), fmaxf(v[4 * c + 3] + bv.w, 0.f));
                    pk[2 * c] = inside[b] ? *reinterpret_cast<const uint32_t *>(&lo) : 0u;
                    pk[2 * c + 1] = inside[b] ? *reinterpret_cast<const uint32_t *>(&hi) : 0u;
                }
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    *reinterpret_cast<uint4 *>(dst + b * 128 * 128 + (((4 * h + c) ^ sw) << 4)) =
                        make_uint4(pk[4 * c], pk[4 * c + 1], pk[4 * c + 2], pk[4 * c + 3]);
            }
            hand_over();
            if (layer == 1) {
                mma_mid(kOffW3, 16);
            } else {
                if (w4 == 0 && elect_one()) {
                    fence_after_sync();
                    const uint64_t db = smem_desc(base + kOffW4, 0, 1024, 2);
                    for (int b = 0; b < 2; ++b) {
                        const uint64_t da = smem_desc(cbase + (uint32_t)(kMargin + b * 128) * 128u, 0, 1024, 2);
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)
                            mma<false>(tm + (uint32_t)b * 64u, da + 2u * ks, db + 2u * ks, idesc_bf16(16), ks ? 1u : 0u);
                    }
                    mma_commit(bar);
                }
                __syncwarp();
            }
            if (acts) {
                store_acts(layer, gi, x, mine[0], row);
                store_acts(layer, gi, x + 128, mine[1], row + 128);
            }
        }
        // ---- layer 4: the products (kw, h, co) of every subcarrier, added up over its neighbours
        wait_products();
        if (acts) ctx_sync(ctx);                                            // the stores have read the activations
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            uint32_t r[32];
            tmem_ld16(tm_own + 64u * b, r);
#pragma unroll
            for (int q = 0; q < 12; ++q) sums[(row + 128 * b) * 13 + q] = __uint_as_float(r[q]);
        }
        fence_before_sync();
        ctx_sync(ctx);
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            if (!mine[b]) continue;
            const int i = row + 128 * b;
            float *o = y + (long long)gi * 4 * g.w + x + 128 * b;
            const bool lost = *abort;                                       // a wait of this CTA expired
#pragma unroll
            for (int co = 0; co < 2; ++co)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float v = s_bias4[co] + sums[i * 13 + 4 + h * 2 + co];
                    if (i > 0) v += sums[(i - 1) * 13 + h * 2 + co];
                    if (i < kRows - 1) v += sums[(i + 1) * 13 + 8 + h * 2 + co];
                    o[(long long)(co * 2 + h) * g.w] = lost ? __int_as_float(0x7fffffff) : v + res[b][co * 2 + h];
                }
        }
        // (the next tile's first barrier orders these reads before the activations are written again)
    }

    // every MMA has completed: the last wait of each tile in flight covered them unless a wait expired
    if (*abort) {
        if (w4 == 0 && elect_one()) {
            mma_commit(smem_u32(&bar_drain[ctx]));
            mbar_drain(smem_u32(&bar_drain[ctx]), 0u);
        }
        __syncwarp();
    }
    fence_before_sync();
    __syncthreads();
    if (warp == 0) {
        fence_after_sync();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s_tmem), "r"(kCtx * 128));
    }
}

}  // namespace

cudaError_t launch_cnn_fwd(const __nv_bfloat16 *in, const __nv_bfloat16 *P, float *y, __nv_bfloat16 *acts, int n, int w,
                           uint32_t *err, cudaStream_t st, unsigned long long selftest_ns) {
    if (n == 0 || w == 0) return cudaSuccess;
    FwdArgs a;
    a.selftest_ns = selftest_ns;
    a.w = w;
    a.in_ld = w;
    a.acts_ld = w;
    a.acts_layer = (long long)n * 64 * w;
    const int out = kRows - 2 * kHalo;
    a.tiles_per_grid = w <= kRows ? 1 : (w + out - 1) / out;
    a.step = (w + a.tiles_per_grid - 1) / a.tiles_per_grid;
    a.halo = a.tiles_per_grid == 1 ? 0 : kHalo;
    const long long tiles = (long long)n * a.tiles_per_grid;
    if (tiles > 0x3fffffffLL) return cudaErrorInvalidConfiguration;
    a.tiles = (int)tiles;
    cudaError_t e = cudaFuncSetAttribute(cnn_fwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long long grid = tiles < sms ? tiles : sms;
    launch_chained(true, cnn_fwd_kernel, dim3((unsigned)grid), dim3(kThreads), kSmemBytes, st, a, in, P, y, acts, err);
    return cudaGetLastError();
}

}  // namespace pusch
