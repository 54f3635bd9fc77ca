// OFDM demodulation on the 5th-generation tensor cores (Section II: one FFT per antenna and OFDM symbol;
// Table I "OFDM dem."): the mixed form's 4096-point FFTs of FP16 time samples as two 64-point stages, each a
// tcgen05 product with the 64-point DFT matrix (FP16 operands, FP32 accumulation in TMEM), the twiddles between
// the stages applied in FP32 by the threads that read the first accumulator.
//
// The transform. With n = 64 a + m and k = k0 + 64 k1 (a, m, k0, k1 in [0, 64)), W = exp(-2 pi i / 4096) and
// w = W^64:
//   stage 1  Y[m][k0]   = W^(m k0) sum_a x[64 a + m] w^(a k0)
//   stage 2  X[k0 + 64 k1] = sum_m Y[m][k0] w^(m k1)
// Both stages multiply by the same real matrix A (128 rows (k; cos, -sin) x K = 64): a real column v gives
// sum_j v_j cos and -sum_j v_j sin for every k.
//   stage 1  B = the row as TMA loads it, read as a [64 a][128 mu] FP16 matrix, mu = 2 m + (re, im): N = mu,
//            K = a, N-major with 128-byte swizzling.
//   stage 2  B = Y, N = (k0; re, im), K = m, K-major without swizzling, written by the warps that read stage 1.
// The accumulators are read with 16x256b loads, whose lane 4 g + t holds rows g and g + 8 at columns 2 t and
// 2 t + 1 of every eight columns. A's rows are ordered so that g is k mod 8 and g + 8 the same k's sine row: a
// lane holds the four real sums of one complex output (cos and sine row x re and im column) and combines them
// itself, V = (cos re - msin im) + i (msin re + cos im). No value crosses lanes between the two products.
//   - Stage 1's lane t holds m = 4 i + t, i = 0..3 in every 16 columns pairs. Inside each K step of 16 the order of
//     K is free, so it is kappa = 4 t + i (the TMA map's dimensions and A's columns follow it): four consecutive
//     kappa of one k0 go to stage 2's operand as one 8-byte store. The padded strides of that operand (144 B
//     between core matrices along K, 1184 B between groups of eight columns) spread the stores over the banks.
//   - Stage 2's columns are ordered so that a lane's eight column groups are eight consecutive output positions
//     on a 16-byte boundary in memory and the four lanes of a row 64 consecutive bytes: position (bin + n_sc / 2)
//     mod 4096, octet e = t + 4 half. The remainder hr = (n_sc / 2 + off) mod 8, off the output's distance from a
//     16-byte boundary in values, rotates k0; only octet 0 then mixes two k1, and its first hr elements come from the
//     lanes of k1 - 1 (eight exchanges per 64 x 8 block). Where off > 0, the octets over a plane's ends are stored
//     value by value (7,168 rows into a plane 2, 4 or 8 bytes off a boundary: 70 us at most; 187, 194 and 205 us when all
//     of its values were stored singly).
// A 4096-point transform thus costs two MMA passes (8 MMAs of 128 x 128 x 16) and one pass of twiddles and
// transposition through shared memory.
//
// What bounds it: the reading warps. With the data as the MMA's A operand (a complex value's sums in two lanes) the
// LSU pipe was 67 % and issue 57 % busy: 128 lane exchanges and 51 2-byte stores per row and warp, 70.6 us for 7,168
// rows with 3276 of 4096 bins kept. Here 16 exchanges and 8 16-byte stores per row: 56.2 us (55 % of the measured copy
// rate), of which the accumulator reads are the largest part of the LSU pipe's work (1,024 of its wavefronts per row).
// Measured while unaligned outputs had a path in the same kernel, 58.6 us then: three CTAs per SM, also with a two-stage
// ring, 58.7 and 60.1 us; octet 0 stored one element at a time 108 us.
//
// Roles (persistent CTAs, four per SM, 128 TMEM columns each): warps 0-3 read the accumulators (warp q owns TMEM
// lane quarter q) and write the next operand or the output; warp 4 issues the row copies (TMA, a one-stage ring)
// and the MMAs. They hand over through mbarriers: the MMA commits signal the accumulator, the four reading
// warps' arrivals signal the second operand and the free accumulator. Every wait is bounded (2 s); on expiry
// the CTA sets the tensor-core bit (kErrTensorWait) of the error word, every role leaves its loop, the copies
// and MMAs in flight are drained (bounded) and TMEM is freed.
//
// Error: the input enters the first product exactly; the intermediate Y and the DFT matrix are rounded to FP16
// (round to nearest) and the output is stored as FP16, so the transform carries about 2^-11 relative error
// (measured against the FP64 oracle in the tests), far under the chain's -40 dB gate.
#include "tc_common.cuh"

namespace pusch {
namespace {

using namespace tc;

constexpr int kN = 4096;
constexpr int kEpiWarps = 4;
constexpr int kThreads = 32 * (kEpiWarps + 1);
constexpr int kCtasPerSm = 4;
constexpr int kTmemCols = 128;
constexpr int kStages = 1;

constexpr uint32_t kRowBytes = kN * 4;                      // one row of FP16 complex samples: 16 KB
constexpr uint32_t kOffIn = 0;                              // input ring (stage-1 B operands, 1024-aligned)
constexpr uint32_t kOffA = kOffIn + kStages * kRowBytes;    // A: [128][64] FP16, K-major, 16 KB
constexpr uint32_t kOffY = kOffA + 16384;                   // Y: stage 2's B operand [128][64] FP16, K-major
constexpr uint32_t kLboY = 144, kSboY = 1184;               // 8 core matrices of 128 B (+ 16), 16 column groups (+ 32)
constexpr uint32_t kOffTw = kOffY + 16 * kSboY;             // W^(8 m q), q < 8: [q][i / 2][t] pairs of float2, 4 KB
constexpr uint32_t kSmemUsed = kOffTw + 4096;
constexpr size_t kSmemBytes = kSmemUsed + 1024;             // + alignment of the base to 1024 B

// K order of both products: kappa = 16 s + 4 t + i stands for j = 16 s + 4 i + t
__device__ __forceinline__ int k_of(int kappa) { return (kappa & 48) | ((kappa & 3) << 2) | ((kappa >> 2) & 3); }

__device__ __forceinline__ void mma_f16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

// K-major, no swizzle: element (n, k) of an operand with `sbo` bytes per 8-row group and `lbo` bytes between
// the core matrices (8 rows x 8 FP16) along K.
__device__ __forceinline__ uint32_t kmajor_off(int n, int k, uint32_t lbo, uint32_t sbo) {
    return (uint32_t)(n >> 3) * sbo + (uint32_t)(k >> 3) * lbo + (uint32_t)(n & 7) * 16u + (uint32_t)(k & 7) * 2u;
}

// Bounded wait by one lane of the warp, the result broadcast to the warp.
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, volatile int *abort, uint32_t *err, int lane) {
    bool ok = true;
    if (lane == 0) ok = mbar_wait_sleep(bar, parity, abort, err, 32);
    return __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
}

// Accumulator rows lane .. lane + 15 (lane given in the address's upper half), 32 columns: r[4 i ..] = row g at
// columns 8 i + 2 t and + 1, then row g + 8 at the same columns (g = lane / 4, t = lane % 4).
__device__ __forceinline__ void tmem_ld_16x256_x4(uint32_t taddr, uint32_t *r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
// The registers go through the wait, so that no use of them can be scheduled before it.
__device__ __forceinline__ void tmem_wait16(uint32_t *r) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
                 :
                 : "memory");
}

// V = (cos re - msin im) + i (msin re + cos im) from a lane's four sums r = (cos re, cos im, msin re, msin im)
__device__ __forceinline__ float2 combine(const uint32_t *r) {
    return make_float2(__uint_as_float(r[0]) - __uint_as_float(r[3]), __uint_as_float(r[2]) + __uint_as_float(r[1]));
}

__device__ __forceinline__ uint32_t pack_half2(float a, float b) {
    const __half2 v = __floats2half2_rn(a, b);
    return *reinterpret_cast<const uint32_t *>(&v);
}

struct FftTcArgs {
    long long rows;
    int n_sc, pitch;
    int off;     // values from the last 16-byte boundary to the output
};

// OFF: the output is not on a 16-byte boundary (compiled apart: the stores over the planes' ends cost the aligned case 2 %)
template <bool OFF>
__global__ void __launch_bounds__(kThreads, kCtasPerSm)
fft_tc_kernel(const __grid_constant__ CUtensorMap tin, __half *__restrict__ out, const float2 *__restrict__ tw,
              FftTcArgs g, uint32_t *__restrict__ err) {
    chain_wait(out, tw, err);
    chain_go();
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bar_full[kStages];
    __shared__ __align__(8) uint64_t bar_acc;     // MMA commits: the accumulator holds a finished product
    __shared__ __align__(8) uint64_t bar_op;      // 4 warp arrivals: Y written / the accumulator read out
    __shared__ __align__(8) uint64_t bar_drain;
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    __shared__ __align__(16) uint32_t s_edge[kEpiWarps][16];   // a warp's first octet 0 and the one after its last

    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t *gbase = smem_raw + (base - raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    volatile int *abort = &s_abort;

    // ---------------------------------------------------------------- A (resident): (cos, -sin)(2 pi j k / 64)
    // from the table's w^q = W^(64 q), which go through shared memory (Y's place): with a table read for each of
    // A's entries the set-up took 10.8 k of a CTA's 117 k clocks. All table reads are issued before the first wait.
    constexpr int kTwPer = (512 + kThreads - 1) / kThreads;
    float2 w8[kTwPer], w64 = make_float2(0.f, 0.f);
    if (tid < 64) w64 = __ldg(&tw[64 * tid]);
#pragma unroll
    for (int u = 0; u < kTwPer; ++u) {
        const int e = tid + u * kThreads;
        if (e < 512) w8[u] = __ldg(&tw[8 * (e >> 6) * (e & 63)]);
    }
    float2 *sw64 = reinterpret_cast<float2 *>(gbase + kOffY);
    if (tid < 64) sw64[tid] = w64;
    // W^(8 m q), m = 4 i + t: pairs of consecutive i at [q][i / 2][t]
#pragma unroll
    for (int u = 0; u < kTwPer; ++u) {
        const int e = tid + u * kThreads, m = e & 63;
        if (e < 512)
            reinterpret_cast<float2 *>(gbase + kOffTw)[(((e >> 6) * 8 + (m >> 3)) * 4 + (m & 3)) * 2 + ((m >> 2) & 1)] =
                w8[u];
    }
    __syncthreads();
    // eight K values (one 16-byte core-matrix row) per thread and store; row n = 16 (k / 8) + 8 (cos, -sin) + k % 8
    for (int e = tid; e < 128 * 8; e += kThreads) {
        const int n = e >> 3, j0 = (e & 7) * 8, k = ((n >> 4) << 3) | (n & 7);
        __align__(16) __half v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const float2 w = sw64[(k_of(j0 + u) * k) & 63];
            v[u] = __float2half_rn((n & 8) ? w.y : w.x);     // Im W^q = -sin
        }
        *reinterpret_cast<uint4 *>(gbase + kOffA + kmajor_off(n, j0, 128, 1024)) = *reinterpret_cast<const uint4 *>(v);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) mbar_init(smem_u32(&bar_full[s]), 1);
        mbar_init(smem_u32(&bar_acc), 1);
        mbar_init(smem_u32(&bar_op), kEpiWarps);
        mbar_init(smem_u32(&bar_drain), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_abort = 0;
    }
    if (warp == kEpiWarps) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = s_tmem;
    const long long n_my = g.rows > blockIdx.x ? (g.rows - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;

    if (warp == kEpiWarps) {
        // ------------------------------------------------------------ control: row copies and MMAs
        if (elect_one()) {
            const uint32_t idesc = idesc_f16(128, 128, false, true);    // stage 1: B (the row) N-major
            const uint32_t idesc2 = idesc_f16(128, 128, false, false);
            // the time samples are read once: evict-first, so that they do not push the FFT output (the next
            // kernel's input) out of L2
            const uint64_t pol_in = l2_policy_evict_first();
            auto issue = [&](long long i) {
                const int s = (int)(i % kStages);
                const long long row = blockIdx.x + i * gridDim.x;
                const uint32_t bar = smem_u32(&bar_full[s]);
                mbar_expect_tx(bar, kRowBytes);
                for (int h = 0; h < 2; ++h)
                    tma_load_4d_hint(base + kOffIn + (uint32_t)s * kRowBytes + (uint32_t)h * 8192u, &tin, 64 * h,
                                     (int)(row * 4), bar, pol_in);
            };
            long long issued = 0;
            for (; issued < kStages && issued < n_my; ++issued) issue(issued);
            uint32_t op_phase = 0;
            long long it = 0;
            bool ok = true;
            for (; it < n_my && ok; ++it) {
                const int s = (int)(it % kStages);
                ok = mbar_wait_sleep(smem_u32(&bar_full[s]), (uint32_t)((it / kStages) & 1), abort, err, 64);
                if (ok && it > 0) {   // the reading warps have emptied the accumulator of row it - 1
                    ok = mbar_wait_sleep(smem_u32(&bar_op), op_phase, abort, err, 128);
                    op_phase ^= 1u;
                }
                if (!ok) break;
                fence_after_sync();
                const uint32_t a0 = base + kOffIn + (uint32_t)s * kRowBytes;
                for (int ks = 0; ks < 4; ++ks)
                    mma_f16(tmem, smem_desc(base + kOffA + (uint32_t)ks * 256u, 128, 1024, 0),
                            smem_desc(a0 + (uint32_t)ks * 2048u, 8192, 1024, 2), idesc, ks > 0 ? 1u : 0u);
                mma_commit(smem_u32(&bar_acc));
                // the stage-1 products have read the row: its ring slot takes a later row
                ok = mbar_wait_sleep(smem_u32(&bar_acc), 0u, abort, err, 32);
                if (!ok) break;
                if (issued < n_my) issue(issued++);
                ok = mbar_wait_sleep(smem_u32(&bar_op), op_phase, abort, err, 128);   // Y written
                op_phase ^= 1u;
                if (!ok) break;
                fence_after_sync();
                for (int ks = 0; ks < 4; ++ks)
                    mma_f16(tmem, smem_desc(base + kOffA + (uint32_t)ks * 256u, 128, 1024, 0),
                            smem_desc(base + kOffY + (uint32_t)ks * 2u * kLboY, kLboY, kSboY, 0), idesc2,
                            ks > 0 ? 1u : 0u);
                mma_commit(smem_u32(&bar_acc));
            }
            if (ok && n_my > 0) mbar_wait_sleep(smem_u32(&bar_op), op_phase, abort, err, 128);   // the last row read out
            if (*abort) {
                // drain: the row copies still in flight and every MMA issued (bounded waits)
                for (long long j = it; j < issued; ++j)
                    mbar_drain(smem_u32(&bar_full[(int)(j % kStages)]), (uint32_t)((j / kStages) & 1));
                mma_commit(smem_u32(&bar_drain));
                mbar_drain(smem_u32(&bar_drain), 0);
            }
        }
    } else {
        // ------------------------------------------------------------ accumulator readers (warp q = lane quarter)
        const int g8 = lane >> 2, t = lane & 3;
        const uint32_t tq = tmem + ((uint32_t)(32 * warp) << 16);
        // twiddles W^(m k0), k0 = 8 q + g8, m = 4 i + t: W^(m g8) here, W^(8 m q) in shared memory (exact table
        // entries both)
        float2 pw[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) pw[i] = __ldg(&tw[(4 * i + t) * g8]);
        const int h = g.n_sc >> 1, hr = (h + (OFF ? g.off : 0)) & 7, hb = h - hr;   // hb + off: a multiple of 8
        uint32_t first[4];   // the halves of octet 0's pairs that lie among its first hr elements
#pragma unroll
        for (int i = 0; i < 4; ++i) first[i] = t > 0 ? 0u : hr - 2 * i >= 2 ? 0xffffffffu : hr - 2 * i == 1 ? 0xffffu : 0u;
        // this lane's element of the warp's two edge octets: lane = [edge][plane][element]; -1: none
        const int ei = lane & 7, epos = (64 * 16 * (warp + (lane >> 4)) + hb + ei) & (kN - 1);
        const bool emine = hr > 0 && (lane < 16 ? ei >= hr : ei < hr) && epos < g.pitch;
        const int eout = emine ? epos + ((lane >> 3) & 1) * g.pitch : -1;
        uint32_t acc_phase = 0;
        for (long long it = 0; it < n_my; ++it) {
            const long long row = blockIdx.x + it * gridDim.x;
            // ---- stage-1 accumulator -> Y (twiddled, FP16)
            if (!warp_wait(smem_u32(&bar_acc), acc_phase, abort, err, lane)) break;
            acc_phase ^= 1u;
            fence_after_sync();
#pragma unroll
            for (int blk = 0; blk < 2; ++blk) {
                const int q = 2 * warp + blk;
                // the column group and pair of stage 2 that hold k0: octet e = u + 4 half, element x of position
                // k0 + hr
                const int pos = (8 * q + g8 + hr) & 63, x = pos & 7, e = pos >> 3;
                uint8_t *yp = gbase + kOffY + (uint32_t)(8 * (e >> 2) + x) * kSboY + (uint32_t)(e & 3) * 32u +
                              (uint32_t)(t >> 1) * kLboY + (uint32_t)(t & 1) * 8u;
                const float4 *bt = reinterpret_cast<const float4 *>(gbase + kOffTw) + q * 32 + t;
#pragma unroll
                for (int s = 0; s < 4; ++s) {
                    uint32_t r[16];
                    tmem_ld_16x256_x4(tq + ((uint32_t)(16 * blk) << 16) + 32u * s, r);
                    const float4 b0 = bt[8 * s], b1 = bt[8 * s + 4];
                    tmem_wait16(r);
                    const float2 y0 = cmul(cmul(combine(r), pw[4 * s]), make_float2(b0.x, b0.y));
                    const float2 y1 = cmul(cmul(combine(r + 4), pw[4 * s + 1]), make_float2(b0.z, b0.w));
                    const float2 y2 = cmul(cmul(combine(r + 8), pw[4 * s + 2]), make_float2(b1.x, b1.y));
                    const float2 y3 = cmul(cmul(combine(r + 12), pw[4 * s + 3]), make_float2(b1.z, b1.w));
                    *reinterpret_cast<uint2 *>(yp + 2 * s * kLboY) =
                        make_uint2(pack_half2(y0.x, y1.x), pack_half2(y2.x, y3.x));
                    *reinterpret_cast<uint2 *>(yp + 2 * s * kLboY + 16) =
                        make_uint2(pack_half2(y0.y, y1.y), pack_half2(y2.y, y3.y));
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bar_op));
            // ---- stage-2 accumulator -> output planes
            if (!warp_wait(smem_u32(&bar_acc), acc_phase, abort, err, lane)) break;
            acc_phase ^= 1u;
            fence_after_sync();
            __half *o = out + row * 2 * (long long)g.pitch;
            uint32_t hold[8] = {};   // lanes g8 = 0: octet 0 of the block's last k1
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int blk = c >> 1, half = c & 1, k1 = 16 * warp + 8 * blk + g8, e = t + 4 * half;
                uint32_t r[32];
                const uint32_t ta = tq + ((uint32_t)(16 * blk) << 16) + 64u * half;
                tmem_ld_16x256_x4(ta, r);
                tmem_ld_16x256_x4(ta + 32u, r + 16);
                tmem_wait16(r);
                tmem_wait16(r + 16);
                uint32_t v[8];   // the octet's pairs: re 0..3, im 4..7
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float2 a = combine(r + 8 * i), b = combine(r + 8 * i + 4);
                    v[i] = pack_half2(a.x, b.x);
                    v[4 + i] = pack_half2(a.y, b.y);
                }
                // element i of the octet goes to position a0 + i; of octet 0 the first hr one block further on
                const int a0 = (8 * e + 64 * k1 + hb) & (kN - 1);
                if (half == 0 && hr > 0) {
                    uint32_t rot[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) rot[i] = __shfl_sync(0xffffffffu, v[i], (lane + 28) & 31);
                    if (lane == 0) {   // the warp's first octet 0 (its own part) and the one after its last
                        uint4 *ed = reinterpret_cast<uint4 *>(&s_edge[warp][8 * blk]);
                        ed[0] = blk ? make_uint4(rot[0], rot[1], rot[2], rot[3]) : make_uint4(v[0], v[1], v[2], v[3]);
                        ed[1] = blk ? make_uint4(rot[4], rot[5], rot[6], rot[7]) : make_uint4(v[4], v[5], v[6], v[7]);
                    }
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const uint32_t prev = blk == 1 && g8 == 0 ? hold[i] : rot[i];
                        v[i] = (prev & first[i & 3]) | (v[i] & ~first[i & 3]);
                        if (blk == 0) hold[i] = rot[i];
                    }
                }
                const bool whole = !(c == 0 && lane == 0 && hr > 0);
                if (whole && (OFF ? a0 + 8 <= g.pitch : a0 < g.pitch)) {
                    if (a0 + 8 > g.n_sc) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const int n = g.n_sc - a0 - 2 * (i & 3);      // values left from this pair on
                            v[i] &= n >= 2 ? 0xffffffffu : n == 1 ? 0xffffu : 0u;
                        }
                    }
                    *reinterpret_cast<uint4 *>(o + a0) = make_uint4(v[0], v[1], v[2], v[3]);
                    *reinterpret_cast<uint4 *>(o + g.pitch + a0) = make_uint4(v[4], v[5], v[6], v[7]);
                } else if (OFF && whole && (a0 < g.pitch || a0 + 8 > kN)) {   // over an end of the plane
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int a = (a0 + i) & (kN - 1), sh = 16 * (i & 1);
                        if (a < g.pitch) {
                            o[a] = __ushort_as_half((unsigned short)(a < g.n_sc ? v[i >> 1] >> sh : 0u));
                            o[g.pitch + a] = __ushort_as_half((unsigned short)(a < g.n_sc ? v[4 + (i >> 1)] >> sh : 0u));
                        }
                    }
                }
            }
            __syncwarp();
            if (eout >= 0)
                o[eout] = epos < g.n_sc ? reinterpret_cast<const __half *>(s_edge[warp])[lane] : __float2half_rn(0.f);
            fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bar_op));
        }
    }

    fence_before_sync();
    __syncthreads();
    if (warp == kEpiWarps) {
        fence_after_sync();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols));
    }
}

}  // namespace

bool fft_tc_supported(const Geometry &g) {
    return g.form == PUSCH_FORM_MIXED && g.n_fft == kN && g.in_fp16 && !g.cp && !g.shift;
}

cudaError_t launch_fft_tc(const Geometry &g, long long rows, const void *in, void *out, const float2 *tw,
                          uint32_t *err, cudaStream_t st) {
    if (!fft_tc_supported(g)) return cudaErrorNotSupported;
    if (rows == 0) return cudaSuccess;
    if (rows * 64 > 0x7fffffffLL) return cudaErrorInvalidValue;     // TMA row coordinate is 32-bit
    PFN_cuTensorMapEncodeTiled_v12000 enc = encode_fn();
    if (!enc) return cudaErrorNotSupported;
    FftTcArgs a;
    CUtensorMap map;
    // [rows * 4 s][4 t][4 i][128 mu] FP16: sample j = 16 s + 4 i + t of a row's 64
    cuuint64_t dims[4] = {128, 4, 4, (cuuint64_t)(rows * 4)};
    cuuint64_t strides[3] = {1024, 256, 4096};
    cuuint32_t box[4] = {64, 4, 4, 4};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    CUresult r = enc(&map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, const_cast<void *>(in), dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
    a.off = (int)((reinterpret_cast<uintptr_t>(out) & 15) / sizeof(__half));
    auto k = a.off ? fft_tc_kernel<true> : fft_tc_kernel<false>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // kCtasPerSm resident CTAs per SM (4 x 57 KB of shared memory; 4 x 128 TMEM columns = 512). The CTAs are
    // independent, so a CTA that cannot be resident at once simply runs later.
    long long grid = (long long)sms * (g.fft_cap > 0 && g.fft_cap < kCtasPerSm ? g.fft_cap : kCtasPerSm);
    if (grid > rows) grid = rows;
    a.rows = rows;
    a.n_sc = g.n_sc;
    a.pitch = g.sc_pitch;
    launch_chained(g.chained, k, dim3((unsigned)grid), dim3(kThreads), kSmemBytes, st, map, static_cast<__half *>(out), tw, a, err);
    return cudaGetLastError();
}

}  // namespace pusch
