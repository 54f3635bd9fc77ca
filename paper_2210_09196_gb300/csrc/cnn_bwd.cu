// Backward pass of the learned estimator: the gradients of mean((y - target)^2) with respect to the packed parameters.
//
//   cnn_bwd_out   the loss and its gradient g4 = 2 (y - target) / count; layer 4's weight gradient, and its input gradient
//                 g3, masked by the activation it belongs to
//   cnn_bwd_mid   layers 3 and 2, on the tensor cores: weight gradient and masked input gradient (g2, g1)
//   cnn_bwd_in    layer 1's weight gradient
//
// Gradients stay FP32 and lie channels-last in the work buffer, [n][w][64 (row, channel)], so that a subcarrier is one
// 256-byte row for whoever writes or reads it. For the products an FP32 gradient is split into three BF16 parts, 8 bits
// of mantissa each, whose sum is the FP32 value; weights and activations are BF16 anyway. The products are exact and
// accumulate in FP32.
//
// cnn_bwd_mid, per tile of 128 subcarriers (with 16 more on either side, zeros outside the grid):
//   input gradient   D[x][(r, ci)] = sum_kw sum_(h, co) G[x - (kw - 1) dil][(h, co)] W[co][ci][r - h + 1][kw]: M = 128,
//                    N = 64, K = 3 taps x 64, for each part of G: 36 MMAs of 48 clocks. G is a K-major operand of 64
//                    values per subcarrier (128-byte swizzling); a shift by dil is an offset of whole 8-row groups. The
//                    smallest part goes first: the tensor core truncates the running sum in every step, so that only the
//                    12 steps of the largest part should meet a sum of full size (largest first: g2 off by 8.1e-7 of its
//                    norm, g1 by 1.7e-6; smallest first: 1.2e-7 and 2.0e-7).
//   weight gradient  P[(part, h, co)][(kw, r, ci)] = sum_x G_part[(h, co)][x] A[(r, ci)][x + (kw - 1) dil]: the same
//                    shared-memory rows read as MN-major operands, K = x. M = 128 holds 64 rows of zeros beside the lowest
//                    part, then the two upper parts; N = 192 holds the three taps, whose operand blocks lie dil rows
//                    apart: 16 MMAs of 80 clocks. P is formed anew in every tile and added up over the CTA's tiles in FP32
//                    in shared memory: a sum that stayed in TMEM lost some 1.1e-7 of itself per tile to the truncation
//                    (3.6e-6 at 4096 grids x 256, 1.3e-5 at 12288; now 3e-8, and the whole error is below that of rounded
//                    FP32 sums of all products).
// Two tiles are in flight per CTA (one CTA per SM), 256 threads each. Activations arrive in 2-byte loads along the
// subcarriers (the caller's layout, any width) and go to shared memory channels-last.
// Measured (GB300, a step of 1024 grids x 256): out 40, mid 93 each, in 20 us; on FP32 FMAs (weights gradient: one thread
// per channel pair) the backward pass took 4.0 ms. mid is bound by the chain load - split - products - mask - sum of a
// tile, of which two overlap (issue 28 %, shared-memory pipe 58 %); out and in by the packed FMAs.
// Every wait is bounded (2 s). After one that expired the loss and the CTA's gradients are NaN, which the layers before take
// over; the error bit is set where there is an error word; the threads go on without waiting, so all barriers are met: no
// address depends on what a wait was for. MMAs in flight are drained (bounded) before TMEM is freed, on a barrier of its
// own: those of the products may be a phase behind by then.
#include "tc_common.cuh"

namespace pusch {
namespace {

using namespace tc;

// element (row, k) of an operand of 64 BF16 (128 bytes) per row with 128-byte swizzling
__device__ __forceinline__ uint32_t sw128(int row, int k) {
    return (uint32_t)row * 128u + ((uint32_t)((k >> 3) ^ (row & 7)) << 4) + (uint32_t)(k & 7) * 2u;
}

// 32 channels (one grid row) of activations of subcarrier x -> half a shared-memory row; zeros when off
__device__ __forceinline__ void load_acts_row(const __nv_bfloat16 *a, long long ld, int x, bool on, uint8_t *buf, int row,
                                              int half) {
    uint16_t v[32];
    const __nv_bfloat16 *p = a + (long long)half * ld + x;                 // channel ci, grid row `half`
#pragma unroll
    for (int c = 0; c < 32; ++c) v[c] = on ? __bfloat16_as_ushort(__ldg(p + (long long)(2 * c) * ld)) : (uint16_t)0;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        uint32_t u[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) u[e] = (uint32_t)v[8 * c + 2 * e] | ((uint32_t)v[8 * c + 2 * e + 1] << 16);
        *reinterpret_cast<uint4 *>(buf + sw128(row, half * 32 + 8 * c)) = make_uint4(u[0], u[1], u[2], u[3]);
    }
}

struct BwdArgs {
    int w, tiles, tiles_per_grid, dil;
    int vec;                 // the work buffer is 16-byte aligned
    float scale;             // 1 / count of the mean
    unsigned long long selftest_ns;   // not 0: every wait is on a barrier that nothing completes, with this limit
};

constexpr int kTile = 128;
__device__ __forceinline__ float nan_value() { return __int_as_float(0x7fffffff); }

// the gradients' rows in the work buffer, which may be aligned to its floats only
__device__ __forceinline__ float4 load4(const float *p, int vec) {
    if (vec) return __ldg(reinterpret_cast<const float4 *>(p));
    return make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));
}
__device__ __forceinline__ float2 load2(const float *p, int vec) {
    if (vec) return __ldg(reinterpret_cast<const float2 *>(p));
    return make_float2(__ldg(p), __ldg(p + 1));
}
__device__ __forceinline__ void store4(float *p, float a, float b, float c, float d, int vec) {
    if (vec) {
        *reinterpret_cast<float4 *>(p) = make_float4(a, b, c, d);
    } else {
        p[0] = a;
        p[1] = b;
        p[2] = c;
        p[3] = d;
    }
}
__device__ __forceinline__ void store2(float *p, float a, float b, int vec) {
    if (vec) {
        *reinterpret_cast<float2 *>(p) = make_float2(a, b);
    } else {
        p[0] = a;
        p[1] = b;
    }
}

// ------------------------------------------------------------------------------------------- layers 3 and 2
constexpr int kHaloR = 16, kBufRows = kTile + 2 * kHaloR;
constexpr uint32_t kPartBytes = kBufRows * 128;
constexpr int kCtx = 2, kCtxThreads = 256, kMidThreads = kCtx * kCtxThreads;
// weights, 64 x 16 zeros, per context three parts of G and the activations, the CTA's weight gradient
constexpr uint32_t kOffZero = 24576, kZeroBytes = 16 * 128, kOffCtx = kOffZero + kZeroBytes, kCtxBytes = 4 * kPartBytes;
constexpr uint32_t kOffAcc = kOffCtx + kCtx * kCtxBytes;
constexpr size_t kMidSmem = 1024 + kOffAcc + 9 * 1024 * 4;
constexpr int kCtxCols = 256;     // TMEM: 64 columns of D, 192 of P

// kind::f16 with BF16 operands, F32 accumulator, M = 128
constexpr uint32_t idesc_bf16(int N, bool mn_major) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (mn_major ? (1u << 15) | (1u << 16) : 0u) | ((uint32_t)(N >> 3) << 17) |
           ((128u >> 4) << 24);
}

__device__ __forceinline__ void ctx_sync(int ctx) {
    asm volatile("bar.sync %0, %1;" ::"r"(1 + ctx), "r"(kCtxThreads) : "memory");
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t *>(&v);
}
// what is left of (a, b) after its BF16 part u
__device__ __forceinline__ float2 minus_bf16(float2 v, uint32_t u) {
    return make_float2(v.x - __uint_as_float(u << 16), v.y - __uint_as_float(u & 0xffff0000u));
}

// Mutual exclusion of a CTA's contexts, by one thread of each; bounded as the waits on barriers are.
__device__ __forceinline__ void lock_acquire(int *lock, volatile int *abort, uint32_t *err) {
    const uint64_t deadline = globaltimer() + kWaitNs;
    while (atomicCAS(lock, 0, 1) != 0) {
        if (*abort) break;
        if (globaltimer() > deadline) {
            *abort = 1;
            if (err) atomicOr(err, kErrTensorWait);
            break;
        }
        __nanosleep(32);
    }
    __threadfence_block();
}
__device__ __forceinline__ void lock_release(int *lock) {
    __threadfence_block();
    atomicExch(lock, 0);
}

__global__ void __launch_bounds__(kMidThreads, 1)
cnn_bwd_mid_kernel(BwdArgs g, const float *__restrict__ gout, const __nv_bfloat16 *__restrict__ acts,
                   const __nv_bfloat16 *__restrict__ W, float *__restrict__ gin, float *__restrict__ dW,
                   float *__restrict__ db, float *__restrict__ loss, uint32_t *__restrict__ err) {
    chain_wait(gout, acts, W, gin, dW, db, loss, err);
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bar_d[kCtx], bar_p[kCtx], bar_drain[kCtx], bar_never;
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort, s_lock;
    __shared__ float s_db[32];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t *gb = smem_raw + (base - raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    volatile int *abort = &s_abort;

    // B_kw[(r, ci)][(h, co)] = W[co][ci][r - h + 1][kw]; zeros beside the lowest part
    for (int i = tid; i < 32 * 32 * 9; i += kMidThreads) {
        const int co = i / 288, rem = i - co * 288, ci = rem / 9, kk = rem - ci * 9, kh = kk / 3, kw = kk - kh * 3;
        const __nv_bfloat16 v = W[i];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = h + kh - 1;
            if (r >= 0 && r <= 1)
                *reinterpret_cast<__nv_bfloat16 *>(gb + kw * 8192 + sw128(r * 32 + ci, h * 32 + co)) = v;
        }
    }
    if (tid < (int)kZeroBytes / 16) reinterpret_cast<uint4 *>(gb + kOffZero)[tid] = make_uint4(0u, 0u, 0u, 0u);
    float *acc = reinterpret_cast<float *>(gb + kOffAcc);                  // [kh * 3 + kw][ci][co]
    for (int i = tid; i < 9 * 1024; i += kMidThreads) acc[i] = 0.f;
    if (tid < 32) s_db[tid] = 0.f;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (tid == 0) {
        for (int c = 0; c < kCtx; ++c) {
            mbar_init(smem_u32(&bar_d[c]), 1);
            mbar_init(smem_u32(&bar_p[c]), 1);
            mbar_init(smem_u32(&bar_drain[c]), 1);
        }
        mbar_init(smem_u32(&bar_never), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_abort = 0;
        s_lock = 0;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(kCtx * kCtxCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();

    const int ctx = warp >> 3, w8 = warp & 7, t8 = tid & (kCtxThreads - 1);
    const uint32_t cbase = base + kOffCtx + (uint32_t)ctx * kCtxBytes;
    uint8_t *cg = gb + kOffCtx + (size_t)ctx * kCtxBytes;
    uint8_t *ca = cg + 3 * kPartBytes;                                     // activations
    const uint32_t tmD = s_tmem + (uint32_t)ctx * kCtxCols, tmP = tmD + 64u;
    const uint32_t quarter = (uint32_t)(w8 & 3) << 21;
    auto wait = [&](uint64_t *b, uint32_t ph) {
        if (lane == 0 && !*abort) {
            if (g.selftest_ns)
                mbar_wait_sleep(smem_u32(&bar_never), 0u, abort, err, 32, g.selftest_ns);
            else
                mbar_wait_sleep(smem_u32(&b[ctx]), ph, abort, err, 32);
        }
        __syncwarp();
        fence_after_sync();
    };

    // P of this context's tile -> acc, by all of the context's threads once the products have completed. A weight gets
    // terms from four lane quarters q = (part, h) and two grid rows r: in each of four phases the quarters take different
    // taps, and a quarter's two warps different r, so that no two threads add to the same word (with atomics the
    // backward pass of 1024 grids x 256 took 315 us, so it takes 254, as with one sum over all tiles).
    auto add_p = [&]() {
        if (t8 == 0) lock_acquire(&s_lock, abort, err);
        ctx_sync(ctx);
        const int q = w8 & 3, h = q & 1, r = w8 >> 2;
#pragma unroll 1
        for (int f = 0; f < 4; ++f) {
            const int kw = (q + f) & 3;
            if (kw < 3) {
                float v[32];                                               // 32 columns: tap kw, grid row r
                tmem_ld32_nowait(tmP + quarter + 64u * kw + 32u * r, reinterpret_cast<uint32_t(&)[32]>(v));
                tmem_wait_ld();
                float *o = acc + ((r - h + 1) * 3 + kw) * 1024 + lane;     // lane: co
#pragma unroll
                for (int ci = 0; ci < 32; ++ci) o[ci * 32] += v[ci];
            }
            ctx_sync(ctx);
        }
        if (t8 == 0) lock_release(&s_lock);
        fence_before_sync();
    };
    const int ch4 = t8 & 15;                                               // this thread's channels 4 ch4 .. + 3 of G
    float4 dbs = make_float4(0.f, 0.f, 0.f, 0.f);
    uint32_t done = 0;                                                     // tiles of this context so far
    for (int t = blockIdx.x + ctx * gridDim.x; t < g.tiles; t += kCtx * gridDim.x, ++done) {
        const int gi = t / g.tiles_per_grid, x0 = (t - gi * g.tiles_per_grid) * kTile;
        if (done) {                                                        // the last tile's products: its operands are free,
            wait(bar_p, (done - 1) & 1u);                                  // and (the barriers in add_p) its activations,
            add_p();                                                       // the ReLU mask, have been read by all warps
        }
        // ---- all loads of the tile at once: G rows (t8 / 16) + 16 i, activations of channels 8 w8 .. + 7 of rows
        //      32 j + lane
        const float *gp = gout + (long long)gi * g.w * 64 + 4 * ch4;
        const __nv_bfloat16 *ap =
            acts + ((long long)gi * 64 + (w8 & 3) * 16 + (w8 >> 2)) * g.w + (x0 - kHaloR + lane);
        float4 gv[kBufRows / 16];
        uint16_t av[kBufRows / 32][8];
#pragma unroll
        for (int i = 0; i < kBufRows / 16; ++i) {
            const int x = x0 - kHaloR + (t8 >> 4) + 16 * i;
            gv[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (x >= 0 && x < g.w) gv[i] = load4(gp + (long long)x * 64, g.vec);
        }
#pragma unroll
        for (int j = 0; j < kBufRows / 32; ++j) {
            const int x = x0 - kHaloR + lane + 32 * j;
            const bool on = x >= 0 && x < g.w;
#pragma unroll
            for (int c = 0; c < 8; ++c)
                av[j][c] = on ? __bfloat16_as_ushort(__ldg(ap + (long long)(2 * c) * g.w + 32 * j)) : (uint16_t)0;
        }
        // ---- G in three parts
#pragma unroll
        for (int i = 0; i < kBufRows / 16; ++i) {
            const int row = (t8 >> 4) + 16 * i;
            const float4 v = gv[i];
            if (row >= kHaloR && row < kHaloR + kTile) {
                dbs.x += v.x;
                dbs.y += v.y;
                dbs.z += v.z;
                dbs.w += v.w;
            }
            float2 a = make_float2(v.x, v.y), b = make_float2(v.z, v.w);
            uint8_t *o = cg + sw128(row, 4 * ch4);
#pragma unroll
            for (int p = 0; p < 3; ++p) {
                const uint32_t ua = pack_bf16(a.x, a.y), ub = pack_bf16(b.x, b.y);
                *reinterpret_cast<uint2 *>(o + p * kPartBytes) = make_uint2(ua, ub);
                a = minus_bf16(a, ua);
                b = minus_bf16(b, ub);
            }
        }
        // ---- activations
#pragma unroll
        for (int j = 0; j < kBufRows / 32; ++j) {
            uint32_t u[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) u[e] = (uint32_t)av[j][2 * e] | ((uint32_t)av[j][2 * e + 1] << 16);
            *reinterpret_cast<uint4 *>(ca + sw128(32 * j + lane, 8 * w8)) = make_uint4(u[0], u[1], u[2], u[3]);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        fence_before_sync();
        ctx_sync(ctx);
        if (w8 == 0 && elect_one()) {
            fence_after_sync();
            const uint64_t sh = (uint64_t)((uint32_t)g.dil * 128u >> 4);
            const uint64_t dB = smem_desc(base, 0, 1024, 2);
#pragma unroll 1
            for (int p = 2; p >= 0; --p) {                                 // smallest part first
                const uint64_t dA = smem_desc(cbase + p * kPartBytes + kHaloR * 128u, 0, 1024, 2) + sh;
#pragma unroll
                for (int kw = 0; kw < 3; ++kw)
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)
                        mma<false>(tmD, dA - kw * sh + 2u * ks, dB + 512u * kw + 2u * ks, idesc_bf16(64, false),
                                   (p < 2 || (kw | ks)) ? 1u : 0u);
            }
            mma_commit(smem_u32(&bar_d[ctx]));
            const uint64_t dG = smem_desc(cbase + kHaloR * 128u, kPartBytes, 1024, 2);
            // zeros, then the lowest part: the block of zeros is the same in every step, the distance grows
            const uint64_t dL = smem_desc(base + kOffZero, cbase + 2 * kPartBytes + kHaloR * 128u - (base + kOffZero), 1024, 2);
            const uint64_t dX = smem_desc(cbase + 3 * kPartBytes + (uint32_t)(kHaloR - g.dil) * 128u, (uint32_t)g.dil * 128u,
                                          1024, 2);
#pragma unroll 1
            for (int ks = 0; ks < kTile / 16; ++ks)
                mma<false>(tmP, dL + ((uint64_t)(128u * ks) << 16), dX + 128u * ks, idesc_bf16(192, true), ks > 0 ? 1u : 0u);
#pragma unroll 1
            for (int ks = 0; ks < kTile / 16; ++ks)
                mma<false>(tmP, dG + 128u * ks, dX + 128u * ks, idesc_bf16(192, true), 1u);
            mma_commit(smem_u32(&bar_p[ctx]));
        }
        __syncwarp();
        // ---- input gradient: masked by the activation, one subcarrier and grid row per thread
        wait(bar_d, done & 1u);
        {
            const int half = w8 >> 2, row = (w8 & 3) * 32 + lane, x = x0 + row;
            float v[32];
            tmem_ld32_nowait(tmD + quarter + 32u * half, reinterpret_cast<uint32_t(&)[32]>(v));
            tmem_wait_ld();
            float *o = gin + ((long long)gi * g.w + x) * 64 + half * 32;
            const bool lost = *abort;                                      // a wait of this CTA expired
            if (x < g.w) {
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const uint4 m = *reinterpret_cast<const uint4 *>(ca + sw128(kHaloR + row, half * 32 + 8 * c));
                    const uint32_t u[4] = {m.x, m.y, m.z, m.w};
                    float r[8];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        r[2 * e] = lost ? nan_value() : __uint_as_float(u[e] << 16) > 0.f ? v[8 * c + 2 * e] : 0.f;
                        r[2 * e + 1] = lost ? nan_value() : __uint_as_float(u[e] & 0xffff0000u) > 0.f ? v[8 * c + 2 * e + 1] : 0.f;
                    }
                    store4(o + 8 * c, r[0], r[1], r[2], r[3], g.vec);
                    store4(o + 8 * c + 4, r[4], r[5], r[6], r[7], g.vec);
                }
            }
        }
        fence_before_sync();
    }
    if (done) {
        wait(bar_p, (done - 1) & 1u);
        add_p();
        atomicAdd(&s_db[(4 * ch4) & 31], dbs.x);
        atomicAdd(&s_db[(4 * ch4 + 1) & 31], dbs.y);
        atomicAdd(&s_db[(4 * ch4 + 2) & 31], dbs.z);
        atomicAdd(&s_db[(4 * ch4 + 3) & 31], dbs.w);
    }
    __syncthreads();
    // ---- the CTA's weight gradient: one addition per weight in global memory
    for (int i = tid; i < 9 * 1024; i += kMidThreads) {
        const int co = i / 288, rem = i - co * 288, ci = rem / 9, kk = rem - ci * 9;
        atomicAdd(dW + i, *abort ? nan_value() : acc[(kk * 32 + ci) * 32 + co]);
    }
    if (tid < 32) atomicAdd(db + tid, *abort ? nan_value() : s_db[tid]);
    if (tid == 0 && loss && *abort) atomicAdd(loss, nan_value());
    if (*abort) {                                                          // MMAs of a wait that expired
        if (w8 == 0 && elect_one()) {
            mma_commit(smem_u32(&bar_drain[ctx]));
            mbar_drain(smem_u32(&bar_drain[ctx]), 0u);
        }
        __syncwarp();
    }
    __syncthreads();
    if (warp == 0) {
        fence_after_sync();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s_tmem), "r"(kCtx * kCtxCols));
    }
}

// ------------------------------------------------------------------------------------------- layers 4 and 1
// On packed FP32 FMAs: a warp takes one subcarrier at a time, its lanes the 64 (row, channel) values in pairs, so that
// rows of the channels-last gradients move as 256-byte lines; the 12 values (kw, ...) of the narrow side around the
// subcarrier are the same for all lanes and slide along.
constexpr int kEndThreads = 256, kRowsPerWarp = kTile / (kEndThreads / 32);

__device__ __forceinline__ float2 dup(float v) { return make_float2(v, v); }

// acc [12 (kw, j)][2 channels of the lane] of all warps -> red, in the gradient's order (index(ch, kw, j)), then one
// addition per weight in global memory, 32 neighbouring weights per warp (scattered, the additions of all CTAs to the
// same few lines took longer than the sums).
constexpr int kEndWeights = 32 * 2 * 9;
template <typename Index>
__device__ __forceinline__ void flush(float2 (&acc)[3][4], float *red, float *grad, Index index) {
    const int tid = threadIdx.x, lane = tid & 31;
    for (int i = tid; i < kEndWeights; i += kEndThreads) red[i] = 0.f;
    __syncthreads();
#pragma unroll
    for (int kw = 0; kw < 3; ++kw)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            atomicAdd(&red[index(2 * lane, kw, j)], acc[kw][j].x);
            atomicAdd(&red[index(2 * lane + 1, kw, j)], acc[kw][j].y);
        }
    __syncthreads();
    for (int i = tid; i < kEndWeights; i += kEndThreads) atomicAdd(grad + i, red[i]);
}

__global__ void __launch_bounds__(kEndThreads, 2)
cnn_bwd_out_kernel(BwdArgs g, const float *__restrict__ y, const float *__restrict__ tgt,
                   const __nv_bfloat16 *__restrict__ acts, const __nv_bfloat16 *__restrict__ W, float *__restrict__ gin,
                   float *__restrict__ dW, float *__restrict__ db, float *__restrict__ loss) {
    chain_wait(y, tgt, acts, W, gin, dW, db, loss);
    __shared__ __align__(16) uint8_t s_a[kTile * 128];
    __shared__ float4 s_g[kTile + 2];            // g4 (h * 2 + co) of subcarriers x0 - 1 .. x0 + kTile
    __shared__ float s_red[kEndWeights];
    __shared__ float s_sum[3];                   // loss, bias gradient
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid < 3) s_sum[tid] = 0.f;
    const int ch = 2 * lane, r = ch >> 5, ci = ch & 31;
    float2 wv[3][4], acc[3][4];
#pragma unroll
    for (int kw = 0; kw < 3; ++kw)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int h = j >> 1, co = j & 1;
            const __nv_bfloat16 *p = W + (co * 32 + ci) * 9 + (r - h + 1) * 3 + kw;
            wv[kw][j] = make_float2(__bfloat162float(p[0]), __bfloat162float(p[9]));
            acc[kw][j] = make_float2(0.f, 0.f);
        }
    float part = 0.f, b0 = 0.f, b1 = 0.f;
    for (int t = blockIdx.x; t < g.tiles; t += gridDim.x) {
        const int gi = t / g.tiles_per_grid, x0 = (t - gi * g.tiles_per_grid) * kTile;
        __syncthreads();                         // the last tile has been read
        {
            const int half = tid >> 7, row = tid & 127, x = x0 + row;
            load_acts_row(acts + (long long)gi * 64 * g.w, g.w, x, x < g.w, s_a, row, half);
        }
        if (tid < kTile + 2) {
            const int x = x0 - 1 + tid;
            float gv[4] = {0.f, 0.f, 0.f, 0.f};
            if (x >= 0 && x < g.w) {
#pragma unroll
                for (int co = 0; co < 2; ++co)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const long long o = ((long long)gi * 4 + co * 2 + h) * g.w + x;
                        const float d = y[o] - tgt[o];
                        gv[h * 2 + co] = 2.f * d * g.scale;
                        if (tid > 0 && tid <= kTile) part += d * d;
                    }
                if (tid > 0 && tid <= kTile) {
                    b0 += gv[0] + gv[2];
                    b1 += gv[1] + gv[3];
                }
            }
            s_g[tid] = make_float4(gv[0], gv[1], gv[2], gv[3]);
        }
        __syncthreads();
        const int r0 = warp * kRowsPerWarp;
        float2 win[3][4];                        // g4 at x - 1, x, x + 1
        auto fill = [&](float2 (&v)[4], int i) {
            const float4 q = s_g[i];
            v[0] = dup(q.x);
            v[1] = dup(q.y);
            v[2] = dup(q.z);
            v[3] = dup(q.w);
        };
        fill(win[1], r0);
        fill(win[2], r0 + 1);
        float *o = gin + ((long long)gi * g.w + x0 + r0) * 64 + ch;
#pragma unroll 4
        for (int i = 0; i < kRowsPerWarp; ++i) {
            if (x0 + r0 + i >= g.w) break;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                win[0][j] = win[1][j];
                win[1][j] = win[2][j];
            }
            fill(win[2], r0 + i + 2);
            const uint32_t u = *reinterpret_cast<const uint32_t *>(s_a + sw128(r0 + i, ch));
            const float2 a = make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u));
            float2 v0 = make_float2(0.f, 0.f), v1 = v0;
#pragma unroll
            for (int kw = 0; kw < 3; ++kw)       // g4 at x - (kw - 1)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float2 gg = win[2 - kw][j];
                    float2 &s = (j & 1) ? v1 : v0;
                    s = __ffma2_rn(wv[kw][j], gg, s);
                    acc[kw][j] = __ffma2_rn(a, gg, acc[kw][j]);
                }
            v0 = __fadd2_rn(v0, v1);
            store2(o + (long long)i * 64, a.x > 0.f ? v0.x : 0.f, a.y > 0.f ? v0.y : 0.f, g.vec);
        }
    }
    for (int off = 16; off > 0; off >>= 1) {
        part += __shfl_down_sync(0xffffffffu, part, off);
        b0 += __shfl_down_sync(0xffffffffu, b0, off);
        b1 += __shfl_down_sync(0xffffffffu, b1, off);
    }
    if (lane == 0) {
        atomicAdd(&s_sum[0], part);
        atomicAdd(&s_sum[1], b0);
        atomicAdd(&s_sum[2], b1);
    }
    flush(acc, s_red, dW, [](int c, int kw, int j) { return ((j & 1) * 32 + (c & 31)) * 9 + ((c >> 5) - (j >> 1) + 1) * 3 + kw; });
    if (tid == 0) {
        if (loss) atomicAdd(loss, s_sum[0] * g.scale);
        atomicAdd(db, s_sum[1]);
        atomicAdd(db + 1, s_sum[2]);
    }
}

__global__ void __launch_bounds__(kEndThreads, 3)
cnn_bwd_in_kernel(BwdArgs g, const float *__restrict__ gout, const __nv_bfloat16 *__restrict__ in,
                  float *__restrict__ dW, float *__restrict__ db) {
    chain_wait(gout, in, dW, db);
    __shared__ float4 s_x[kTile + 2];            // inputs (r * 2 + ci) of subcarriers x0 - 1 .. x0 + kTile
    __shared__ float s_red[kEndWeights];
    __shared__ float s_db[32];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid < 32) s_db[tid] = 0.f;
    float2 acc[3][4], sum = make_float2(0.f, 0.f);
#pragma unroll
    for (int kw = 0; kw < 3; ++kw)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[kw][j] = make_float2(0.f, 0.f);
    for (int t = blockIdx.x; t < g.tiles; t += gridDim.x) {
        const int gi = t / g.tiles_per_grid, x0 = (t - gi * g.tiles_per_grid) * kTile, r0 = warp * kRowsPerWarp;
        const float *gp = gout + ((long long)gi * g.w + x0 + r0) * 64 + 2 * lane;
        float2 gv[kRowsPerWarp];
#pragma unroll
        for (int i = 0; i < kRowsPerWarp; ++i)
            gv[i] = x0 + r0 + i < g.w ? load2(gp + (long long)i * 64, g.vec) : make_float2(0.f, 0.f);
        __syncthreads();                         // the last tile has been read
        if (tid < kTile + 2) {
            const int x = x0 - 1 + tid;
            float v[4] = {0.f, 0.f, 0.f, 0.f};
            if (x >= 0 && x < g.w) {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    v[j] = __bfloat162float(in[((long long)gi * 4 + (j & 1) * 2 + (j >> 1)) * g.w + x]);
            }
            s_x[tid] = make_float4(v[0], v[1], v[2], v[3]);
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kRowsPerWarp; ++i) {
            sum = __fadd2_rn(sum, gv[i]);
#pragma unroll
            for (int kw = 0; kw < 3; ++kw) {     // input at x + kw - 1
                const float4 q = s_x[r0 + i + kw];
                acc[kw][0] = __ffma2_rn(gv[i], dup(q.x), acc[kw][0]);
                acc[kw][1] = __ffma2_rn(gv[i], dup(q.y), acc[kw][1]);
                acc[kw][2] = __ffma2_rn(gv[i], dup(q.z), acc[kw][2]);
                acc[kw][3] = __ffma2_rn(gv[i], dup(q.w), acc[kw][3]);
            }
        }
    }
    atomicAdd(&s_db[(2 * lane) & 31], sum.x);
    atomicAdd(&s_db[(2 * lane + 1) & 31], sum.y);
    // channel c = (h, co), j = r * 2 + ci
    flush(acc, s_red, dW, [](int c, int kw, int j) { return ((c & 31) * 2 + (j & 1)) * 9 + ((j >> 1) - (c >> 5) + 1) * 3 + kw; });
    if (tid < 32) atomicAdd(db + tid, s_db[tid]);
}

}  // namespace

cudaError_t launch_cnn_bwd(int n, int w, const __nv_bfloat16 *x, const __nv_bfloat16 *acts, const __nv_bfloat16 *P,
                           const float *y, const float *target, float *grad, float *loss, float *work, uint32_t *err,
                           cudaStream_t st, unsigned long long selftest_ns) {
    if (n == 0 || w == 0) return cudaSuccess;
    constexpr int kO2 = 32 * 2 * 9 + 32, kO3 = kO2 + 32 * 32 * 9 + 32, kO4 = kO3 + 32 * 32 * 9 + 32;
    const size_t big = (size_t)n * 64 * w;
    float *ga = work, *gbuf = work + big;
    BwdArgs a;
    a.w = w;
    a.tiles_per_grid = (w + kTile - 1) / kTile;
    const long long tiles = (long long)n * a.tiles_per_grid;
    if (tiles > 0x3fffffffLL) return cudaErrorInvalidConfiguration;
    a.tiles = (int)tiles;
    a.dil = 0;
    a.selftest_ns = selftest_ns;
    a.vec = reinterpret_cast<uintptr_t>(work) % 16 == 0;
    a.scale = 1.f / (float)((long long)n * 4 * w);
    cudaError_t e = cudaFuncSetAttribute(cnn_bwd_mid_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMidSmem);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const unsigned one = (unsigned)(tiles < sms ? tiles : sms), two = (unsigned)(tiles < 2 * sms ? tiles : 2 * sms);
    const unsigned three = (unsigned)(tiles < 3 * sms ? tiles : 3 * sms);
    launch_chained(true, cnn_bwd_out_kernel, dim3(two), dim3(kEndThreads), 0, st, a, y, target, acts + 2 * big, P + kO4, gbuf, grad + kO4,
                                                    grad + kO4 + 2 * 32 * 9, loss);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    a.dil = 16;
    launch_chained(true, cnn_bwd_mid_kernel, dim3(one), dim3(kMidThreads), kMidSmem, st, a, gbuf, acts + big, P + kO3, ga, grad + kO3,
                                                           grad + kO3 + 32 * 32 * 9, loss, err);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    a.dil = 8;
    launch_chained(true, cnn_bwd_mid_kernel, dim3(one), dim3(kMidThreads), kMidSmem, st, a, ga, acts, P + kO2, gbuf, grad + kO2,
                                                           grad + kO2 + 32 * 32 * 9, loss, err);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    launch_chained(true, cnn_bwd_in_kernel, dim3(three), dim3(kEndThreads), 0, st, a, gbuf, x, grad, grad + 32 * 2 * 9);
    return cudaGetLastError();
}

}  // namespace pusch
