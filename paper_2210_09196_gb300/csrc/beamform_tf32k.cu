// Beamforming of the plain FP32 form on the 5th-generation tensor cores with three TF32 products per FP32
// product (Section II, Table I "BF": Y = W^H X per symbol).
//
// The complex product is the real GEMM of the mixed form, D[a][2b + c] = sum_k A[a][k] B[2b + c][k] with
// k = 2r + ri, A[a][2r] = Re X[r][a], A[a][2r + 1] = Im X[r][a], B[2b][2r] = Re W[r][b], B[2b][2r + 1] =
// Im W[r][b], B[2b + 1][2r] = -Im W[r][b], B[2b + 1][2r + 1] = Re W[r][b]. Every FP32 operand v is split
// into two TF32 values, hi = TF32(v) and lo = TF32(v - hi), so that hi + lo holds v to
// about 2^-23, and D = A_hi B_hi + (A_hi B_lo + A_lo B_hi) (the dropped A_lo B_lo is below 2^-22 of |A||B|).
// Infinities and NaN give what they give in FP32 arithmetic.
//
// B (hi and lo) stays in shared memory, 16 bytes per (beam row, antenna): 128 KB hold 64 antennas at 64 beams.
// So a cluster of 1, 2 or 4 CTAs shares one 128-subcarrier tile, each CTA forming the product over its own
// quarter (half, all) of the antennas, at most 64, and the partial sums meet through distributed shared memory:
// TMEM lane quarter q of the tile belongs to CTA q cluster / 4, whose epilogue warp q adds the others' partial
// rows, in rank order, and stores them. A streamed B would cost 512 KB of L2 reads per tile at 256 antennas
// (twice the samples); the exchange moves 192 KB.
//
// Accuracy. The tensor core truncates as it accumulates, an error in proportion to the number of accumulation
// steps, so the steps of one accumulator are kept few: the A_hi B_hi products of the first and of the second half
// of a CTA's antennas (at most 8 steps of K = 8 each) and the small products have an accumulator each, and the up to
// twelve accumulators of a beam are added in FP32. TMEM at 64 beams: E and O (the halves) once, the small products
// twice; E is read out while O is being formed, O while the next tile's E is.
// Norm-relative error against 64 bits: 1.8e-7 at 64 antennas, 2.0e-7 at 256 (FP32 FMAs: 2.0e-7, 4.0e-7; one
// accumulator for the big products: 3.1e-7, 3.3e-7; one for all: 9.5e-7 at 64).
//
// Warp roles (persistent CTAs, one per SM):
//   warps 0-7   load the FFT rows straight from global memory, six stages (of 8 antennas) ahead in registers (any
//               subcarrier count and alignment; a landing ring in shared memory took the room that B needs), and
//               split them into the hi and lo operands (K-major core matrices, no swizzle). One lane of warp 0
//               issues each stage's MMAs a stage later, and commits the stage back;
//   warps 8-15  epilogue (a TMEM lane quarter and half of the columns each): tcgen05.ld of the finished
//               accumulators, exchange, stores of the c64 beam rows.
// 16 warps leave 128 registers a thread: with more, the 64 columns of E that an epilogue thread holds spilled, and
// the spills, missing the little L1 beside 227 KB of shared memory, took 12 k clocks per tile.
//
// Measured (GB300, 2 slots of 256 antennas, 64 beams, 3276 subcarriers): 162 us against 671 us on FP32 FMAs; bound by
// the instructions of the warps that load and split (about 900 clocks per stage; HBM needs 440).
//
// Every wait is bounded (%globaltimer, 2 s); on expiry the CTA records a timeout in err_word bit 0, all roles
// leave their loops, MMAs in flight are drained (bounded) and TMEM is freed; the CTAs of a cluster leave together.
#include "tc_common.cuh"

namespace pusch {
namespace {

using namespace tc;

constexpr int kTileM = 128;
constexpr int kCA = 8;                  // antennas per stage
constexpr int kKC = 2 * kCA;            // K values per stage
constexpr int kMaxStages = 6;
constexpr int kMaxAnt = 64;             // antennas per CTA: 128 KB of B at 64 beams, 16 accumulation steps
constexpr int kMaxCluster = 4;
constexpr int kSmemLimit = 227 * 1024;
constexpr int kConvWarps = 8;
constexpr int kAhead = 6;               // stages loaded ahead in registers (four c64 values per lane each)
constexpr int kEpiWarps = 8;
constexpr int kThreads = 32 * (kConvWarps + kEpiWarps);
constexpr uint32_t kABytes = (uint32_t)kTileM * kKC * 4;   // one operand (hi or lo) of a stage: 8 KB
constexpr uint32_t kASbo = (uint32_t)(kKC / 4) * 128;      // bytes between 8-row groups of an A stage

struct Tf32Args {
    int n_rx, n_beams, n_sc, n_mtiles, N, n_chunks, n_stages, tmem_cols, cluster, vec4;
    uint32_t b_bytes;      // one of B's two operands (hi or lo)
    uint32_t red_off;      // offset of the exchange buffer from the aligned base
    int total_tiles;
};

struct Tf32Shared {
    uint64_t ready[kMaxStages], empty[kMaxStages];
    uint64_t efull, eempty, ofull, oempty, drain;
    uint64_t sfree[kEpiWarps];   // epilogue warp e: the owner has read what this CTA sent
    uint64_t rfull[kEpiWarps];   // epilogue warp e, in the owner: the other CTAs' partial rows have arrived
    uint32_t tmem_base;
    int abort;
};

// v = hi + lo in TF32: hi rounded to nearest (ties away from zero), lo the exact remainder, of which the tensor core
// reads the upper 11 bits of at most 12 (below 2^-23 of |v| is lost; below |v| = 2^-114, where lo leaves the normal
// range, more). hi stays finite: it is rounded from v brought to the largest magnitude that does not round to infinity,
// so that values next to FLT_MAX keep theirs in lo, and an infinity or a NaN is in lo alone and gives what it gives in
// FP32 arithmetic (as hi an infinity would meet both parts of the other operand, whose signs may differ, and its lo were
// a NaN). The limit is one instruction of some eight per value: 157.9 -> 161.7 us for the case above.
__device__ __forceinline__ void split_tf32(float x, uint32_t &hi, uint32_t &lo) {
    float c;   // x with its magnitude limited
    asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(c) : "f"(x), "f"(__uint_as_float(0x7f7fefffu)));
    hi = (__float_as_uint(c) + 0x1000u) & 0xffffe000u;
    lo = __float_as_uint(x - __uint_as_float(hi));
}

// Instruction descriptor of kind::tf32: D F32 (bits 4-5 = 1), A and B TF32 (format code 2 at bits 7-9 and
// 10-12), both K-major, N >> 3 at [17,23), M >> 4 at [24,29).
constexpr uint32_t idesc_tf32(int M, int N) {
    return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_tf32(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void tmem_ld16_nowait(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}

// A streamed load, or zero without touching memory. Written as one predicated instruction: a select after the load
// would wait for it at once, and nothing would be loaded ahead.
__device__ __forceinline__ float2 load_or_zero(const float2 *p, bool on) {
    float2 v = make_float2(0.f, 0.f);
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.u32 p, %3, 0;\n\t"
        "@p ld.global.cs.v2.f32 {%0, %1}, [%2];\n\t}"
        : "+f"(v.x), "+f"(v.y)
        : "l"(p), "r"((uint32_t)on));
    return v;
}

// ---- cluster: rank, barrier, peer addresses, remote arrivals and stores
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t peer(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void arrive_peer(uint32_t bar) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void store_peer(uint32_t addr, float4 v) {
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
}
__device__ __forceinline__ bool try_wait_cluster(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// mbar_wait for a barrier that another CTA of the cluster completes.
__device__ __forceinline__ bool wait_cluster(uint32_t bar, uint32_t parity, volatile int *abort, uint32_t *err) {
    for (int k = 0; k < kPollsPerTimer; ++k)
        if (try_wait_cluster(bar, parity)) return true;
    const uint64_t deadline = globaltimer() + kWaitNs;
    for (;;) {
        for (int k = 0; k < kPollsPerTimer; ++k)
            if (try_wait_cluster(bar, parity)) return true;
        if (*abort) return false;
        if (globaltimer() > deadline) {
            *abort = 1;
            if (err) atomicOr(err, kErrTensorWait);
            return false;
        }
    }
}

__global__ void __launch_bounds__(kThreads, 1)
beamform_tf32k_kernel(Tf32Args g, const float2 *__restrict__ freq, const float2 *__restrict__ W,
                     float2 *__restrict__ beam, uint32_t *__restrict__ err) {
    chain_wait(freq, W, beam, err);
    chain_go();
    extern __shared__ uint8_t smem_raw[];
    __shared__ Tf32Shared sh;

    const int N = g.N, C = g.cluster;
    const int Rk = g.n_chunks * kCA, K = 2 * Rk;                       // antennas / K values of one CTA
    const int rank = C > 1 ? (int)cluster_rank() : 0;
    const int r_first = rank * Rk, r_end = min(g.n_rx, r_first + Rk);  // this CTA's antennas (may be none)
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t *gbase = smem_raw + (base - raw);
    // [A ring: n_stages x (hi, lo)][B hi][B lo][exchange buffer]
    const uint32_t sA = base;
    const uint32_t sB = base + (uint32_t)g.n_stages * 2u * kABytes;
    uint8_t *gB = gbase + (size_t)g.n_stages * 2u * kABytes;
    const uint32_t b_sbo = (uint32_t)(K / 4) * 128u;                   // bytes between 8-row groups of B

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    volatile int *abort = &sh.abort;

    // ---------------------------------------------------------------- B (hi, lo) from W
    // Unit (n, kq) writes the 16-byte core-matrix row of beam row n for antennas 2 kq, 2 kq + 1 of this CTA:
    // element (n, k) at (n/8)*SBO + (k/4)*128 + (n%8)*16 + (k%4)*4; zero past the antennas and the beams.
    {
        const int units = N * (K / 4);
#pragma unroll 4
        for (int u = tid; u < units; u += kThreads) {
            const int kq = u / N, n = u - kq * N, b = n >> 1, r = r_first + 2 * kq;
            const float2 zero = make_float2(0.f, 0.f);
            const float2 w0 = r < r_end && b < g.n_beams ? __ldg(&W[(long long)r * g.n_beams + b]) : zero;
            const float2 w1 = r + 1 < r_end && b < g.n_beams ? __ldg(&W[(long long)(r + 1) * g.n_beams + b]) : zero;
            // row 2b: (Re, Im); row 2b + 1: (-Im, Re)
            const float v[4] = {(n & 1) ? -w0.y : w0.x, (n & 1) ? w0.x : w0.y, (n & 1) ? -w1.y : w1.x,
                                (n & 1) ? w1.x : w1.y};
            uint32_t hi[4], lo[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) split_tf32(v[e], hi[e], lo[e]);
            const size_t off = (size_t)(n >> 3) * b_sbo + (size_t)kq * 128 + (n & 7) * 16;
            *reinterpret_cast<uint4 *>(gB + off) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
            *reinterpret_cast<uint4 *>(gB + g.b_bytes + off) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");

    if (tid == 0) {
        for (int s = 0; s < kMaxStages; ++s) {
            mbar_init(smem_u32(&sh.ready[s]), kConvWarps);
            mbar_init(smem_u32(&sh.empty[s]), 1);
        }
        mbar_init(smem_u32(&sh.efull), 1);
        mbar_init(smem_u32(&sh.ofull), 1);
        mbar_init(smem_u32(&sh.eempty), kEpiWarps);
        mbar_init(smem_u32(&sh.oempty), kEpiWarps);
        for (int e = 0; e < kEpiWarps; ++e) {
            mbar_init(smem_u32(&sh.sfree[e]), 1);
            mbar_init(smem_u32(&sh.rfull[e]), C - 1 > 0 ? C - 1 : 1);
        }
        mbar_init(smem_u32(&sh.drain), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        sh.abort = 0;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh.tmem_base)),
                     "r"(g.tmem_cols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    if (C > 1) cluster_sync();                           // the peers' barriers exist
    const uint32_t tmem = sh.tmem_base;

    const int cl = blockIdx.x / C, ncl = gridDim.x / C;  // tiles cl, cl + ncl, ... are this cluster's
    const int n_my = g.total_tiles > cl ? (g.total_tiles - cl + ncl - 1) / ncl : 0;
    const int NS = g.n_stages, NC = g.n_chunks, NE = (NC + 1) / 2;   // stages of E; the rest go to O
    const uint32_t accE = tmem, accO = tmem + (uint32_t)N, accS = tmem + 2u * (uint32_t)N;

    if (warp >= kConvWarps) {
        // ------------------------------------------------------------------ epilogue
        const int e8 = warp - kConvWarps, q = warp & 3;           // q: the TMEM lane quarter this warp may access
        const int nch = N / 16, h0 = (nch + 1) / 2;      // 16-column chunks: h0 for the first four warps
        const int ch0 = e8 < 4 ? 0 : h0, chn = e8 < 4 ? h0 : nch - h0;
        const int own = 4 / C;                           // quarters per owner
        const int owner = q / own, ql = q - owner * own;
        const bool mine = owner == rank;
        // exchange buffer of the owner: slot (sender, owned quarter), [N / 4][32 lanes] float4
        const uint32_t slot_bytes = (uint32_t)N * 128u;
        const uint32_t red = base + g.red_off;
        uint32_t send = 0, send_bar = 0;
        if (!mine) {
            const int sidx = rank < owner ? rank : rank - 1;
            send = peer(red + (uint32_t)(sidx * own + ql) * slot_bytes, (uint32_t)owner) + (uint32_t)lane * 16u;
            send_bar = peer(smem_u32(&sh.rfull[e8]), (uint32_t)owner);
        }
        const uint32_t tq = (uint32_t)(q * 32) << 16;
        for (int i = 0; i < n_my; ++i) {
            const uint32_t ph = (uint32_t)i & 1u;
            bool okw = mbar_wait(smem_u32(&sh.efull), ph, abort, err);
            if (!__all_sync(0xFFFFFFFFu, okw)) break;    // warp-uniform: tcgen05.ld is warp-collective
            fence_after_sync();
            float v[4][16];
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (c < chn) tmem_ld16_nowait(accE + tq + (uint32_t)(16 * (ch0 + c)), reinterpret_cast<uint32_t (&)[16]>(v[c]));
            tmem_wait_ld();
            fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&sh.eempty));
            okw = mbar_wait(smem_u32(&sh.ofull), ph, abort, err);
            if (!__all_sync(0xFFFFFFFFu, okw)) break;
            fence_after_sync();
            const uint32_t tS = accS + tq + ph * (uint32_t)N;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                if (c >= chn) continue;
                const uint32_t c0 = (uint32_t)(16 * (ch0 + c));
                uint32_t rs[16], ro[16];
                tmem_ld16_nowait(tS + c0, rs);
                if (NC > 1) {
                    tmem_ld16_nowait(accO + tq + c0, ro);
                } else {
#pragma unroll
                    for (int j = 0; j < 16; ++j) ro[j] = 0u;
                }
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    v[c][j] = (v[c][j] + __uint_as_float(ro[j])) + __uint_as_float(rs[j]);
            }
            // everything is in registers: the next tiles' products may go on while the rows are exchanged and stored
            fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&sh.oempty));
            if (!mine) {
                okw = wait_cluster(smem_u32(&sh.sfree[e8]), ph ^ 1u, abort, err);   // the owner has room
                if (!__all_sync(0xFFFFFFFFu, okw)) break;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    if (c >= chn) continue;
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        store_peer(send + (uint32_t)(4 * (ch0 + c) + j) * 512u,
                                   make_float4(v[c][4 * j], v[c][4 * j + 1], v[c][4 * j + 2], v[c][4 * j + 3]));
                }
                __syncwarp();
                if (lane == 0) arrive_peer(send_bar);    // release: this warp's rows are in the owner's buffer
                continue;
            }
            if (C > 1) {
                okw = wait_cluster(smem_u32(&sh.rfull[e8]), ph, abort, err);        // the partial rows have come
                if (!__all_sync(0xFFFFFFFFu, okw)) break;
                // own partial sum + the others' in rank order
                const uint8_t *p = gbase + g.red_off + (size_t)ql * slot_bytes + (size_t)(4 * ch0) * 512 + lane * 16;
                for (int k = 0; k < C - 1; ++k, p += (size_t)own * slot_bytes) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        if (c >= chn) continue;
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const float4 x = *reinterpret_cast<const float4 *>(p + (4 * c + j) * 512);
                            v[c][4 * j] += x.x;
                            v[c][4 * j + 1] += x.y;
                            v[c][4 * j + 2] += x.z;
                            v[c][4 * j + 3] += x.w;
                        }
                    }
                }
                __syncwarp();
                if (lane == 0)
                    for (int k = 0; k < C; ++k)
                        if (k != rank) arrive_peer(peer(smem_u32(&sh.sfree[e8]), (uint32_t)k));
            }
            const int t = cl + i * ncl;
            const int row = t / g.n_mtiles, mt = t - row * g.n_mtiles;
            const int a = mt * kTileM + q * 32 + lane;
            if (a < g.n_sc) {
                float *dst = reinterpret_cast<float *>(beam + ((long long)row * g.n_sc + a) * g.n_beams) + 16 * ch0;
                const int left = 2 * g.n_beams - 16 * ch0;   // floats of the row from there on (even)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    if (c >= chn) continue;
                    if (g.vec4) {
#pragma unroll
                        for (int j = 0; j < 16; j += 4)
                            if (16 * c + j < left)
                                *reinterpret_cast<float4 *>(dst + 16 * c + j) =
                                    make_float4(v[c][j], v[c][j + 1], v[c][j + 2], v[c][j + 3]);
                    } else {
#pragma unroll
                        for (int j = 0; j < 16; j += 2)
                            if (16 * c + j < left)
                                *reinterpret_cast<float2 *>(dst + 16 * c + j) = make_float2(v[c][j], v[c][j + 1]);
                    }
                }
            }
        }
    } else {
        // ------------------------------------------------------------------ load and split into TF32 hi and lo
        // Warp w takes subcarriers 32 (w % 4) .. + 31 of antenna pairs p = w / 4 and w / 4 + 2 of each stage:
        // the values X[2p][m], X[2p + 1][m] become the core-matrix row of k = 4p .. 4p + 3 at (m/8)*512 + p*128 +
        // (m%8)*16 of the hi and the lo operand. Antennas and subcarriers past the end are zero.
        const int w8 = warp, m = (w8 & 3) * 32 + lane, p0 = w8 >> 2;
        const uint32_t moff = (uint32_t)(m >> 3) * kASbo + (uint32_t)(m & 7) * 16u;
        // next stage to load: chunk lc of tile li; src: this lane's value of antenna 2 p0 of the stage
        int li = 0, lc = 0, r = 0;
        bool on = false;
        const float2 *src = freq;
        const long long o1 = g.n_sc, o2 = 4ll * g.n_sc, o3 = 5ll * g.n_sc, step = (long long)kCA * g.n_sc;
        auto load = [&](float2 (&x)[4]) {
            if (lc == 0) {
                const int t = cl + li * ncl;
                const int row = t / g.n_mtiles, a = (t - row * g.n_mtiles) * kTileM + m;
                on = li < n_my && a < g.n_sc;
                r = r_first + 2 * p0;
                src = freq + ((long long)row * g.n_rx + r) * g.n_sc + a;
            }
            x[0] = load_or_zero(src, on && r < r_end);
            x[1] = load_or_zero(src + o1, on && r + 1 < r_end);
            x[2] = load_or_zero(src + o2, on && r + 4 < r_end);
            x[3] = load_or_zero(src + o3, on && r + 5 < r_end);
            src += step;
            r += kCA;
            if (++lc == NC) {
                lc = 0;
                ++li;
            }
        };
        // the MMAs of the next stage (tile mi, chunk mc; operand stage ms), by one lane of warp 0
        const uint32_t idesc = idesc_tf32(kTileM, N);
        // descriptors advance by byte offsets >> 4 in their low word
        const uint64_t dA = smem_desc(sA, 128, kASbo, 0), dBh = smem_desc(sB, 128, b_sbo, 0);
        const uint64_t dBl = smem_desc(sB + g.b_bytes, 128, b_sbo, 0);
        int mi = 0, mc = 0, ms = 0;
        uint32_t mph = 0;
        auto issue = [&]() -> bool {
            // E: read out of the previous tile's; O (and, with it, this tile's half of S): the previous tile's
            // epilogue is over
            if (mc == 0 && !mbar_wait(smem_u32(&sh.eempty), ((uint32_t)mi & 1u) ^ 1u, abort, err)) return false;
            if (mc == NE - 1 && !mbar_wait(smem_u32(&sh.oempty), ((uint32_t)mi & 1u) ^ 1u, abort, err)) return false;
            if (!mbar_wait(smem_u32(&sh.ready[ms]), mph, abort, err)) return false;
            fence_after_sync();
            const uint64_t ah = dA + (uint64_t)((uint32_t)ms * (2u * kABytes >> 4)), al = ah + (kABytes >> 4);
            const uint64_t bh = dBh + (uint64_t)(mc * 32), bl = dBl + (uint64_t)(mc * 32);
            const uint32_t big = mc < NE ? accE : accO, small = accS + (uint32_t)((mi & 1) * N);
            const uint32_t acc_b = (mc == 0 || mc == NE) ? 0u : 1u, acc_s = mc == 0 ? 0u : 1u;
            mma_tf32(big, ah, bh, idesc, acc_b);
            mma_tf32(small, ah, bl, idesc, acc_s);
            mma_tf32(small, al, bh, idesc, 1u);
            mma_tf32(big, ah + 16, bh + 16, idesc, 1u);
            mma_tf32(small, ah + 16, bl + 16, idesc, 1u);
            mma_tf32(small, al + 16, bh + 16, idesc, 1u);
            mma_commit(smem_u32(&sh.empty[ms]));
            if (mc == NE - 1) mma_commit(smem_u32(&sh.efull));
            if (++mc == NC) {
                mma_commit(smem_u32(&sh.ofull));
                mc = 0;
                ++mi;
            }
            if (++ms == NS) {
                ms = 0;
                mph ^= 1u;
            }
            return true;
        };
        float2 ring[kAhead][4];
#pragma unroll
        for (int d = 0; d < kAhead; ++d) load(ring[d]);
        const int total = n_my * NC;
        int s = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int g0 = 0; g0 < total && ok; g0 += kAhead) {
#pragma unroll
            for (int d = 0; d < kAhead; ++d) {
                if (g0 + d >= total || !ok) break;
                // the MMAs of the operand stage's previous use have completed
                const bool okw = mbar_wait(smem_u32(&sh.empty[s]), ph ^ 1u, abort, err);
                ok = __all_sync(0xFFFFFFFFu, okw);
                if (!ok) break;
                uint8_t *ahi = gbase + (size_t)s * 2u * kABytes + moff, *alo = ahi + kABytes;
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const float2 x0 = ring[d][2 * j], x1 = ring[d][2 * j + 1];
                    uint32_t hi[4], lo[4];
                    split_tf32(x0.x, hi[0], lo[0]);
                    split_tf32(x0.y, hi[1], lo[1]);
                    split_tf32(x1.x, hi[2], lo[2]);
                    split_tf32(x1.y, hi[3], lo[3]);
                    const uint32_t off = (uint32_t)(p0 + 2 * j) * 128u;
                    *reinterpret_cast<uint4 *>(ahi + off) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                    *reinterpret_cast<uint4 *>(alo + off) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&sh.ready[s]));
                if (++s == NS) {
                    s = 0;
                    ph ^= 1u;
                }
                load(ring[d]);
                if (w8 == 0 && g0 + d > 0) {
                    if (elect_one()) issue();            // the stage before
                    __syncwarp();
                }
            }
        }
        if (w8 == 0 && n_my > 0) {
            if (elect_one()) {
                if (ok) issue();
                // every MMA issued by this thread has completed once the drain barrier flips (bounded)
                mma_commit(smem_u32(&sh.drain));
                mbar_drain(smem_u32(&sh.drain), 0);
            }
            __syncwarp();
        }
    }

    fence_before_sync();
    __syncthreads();
    if (warp == 0) {
        fence_after_sync();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(g.tmem_cols));
    }
    if (C > 1) cluster_sync();   // no CTA leaves while a peer may still write to its shared memory
}

struct Tf32Plan {
    bool ok;
    int cluster, n_chunks, n_stages, tmem_cols, N;
    uint32_t b_bytes, red_off;
    size_t smem;
};

// The fewest CTAs per tile whose antennas number at most 64 each; then as many operand stages as the shared
// memory beside B and the exchange buffer holds.
Tf32Plan tf32_plan(const Geometry &g) {
    Tf32Plan p{};
    if (g.n_rx > kMaxAnt * kMaxCluster || g.n_beams > 64) return p;
    p.cluster = g.n_rx <= kMaxAnt ? 1 : (g.n_rx <= 2 * kMaxAnt ? 2 : 4);
    p.n_chunks = (g.n_rx + kCA * p.cluster - 1) / (kCA * p.cluster);
    p.N = (2 * g.n_beams + 15) & ~15;
    const int K = 2 * kCA * p.n_chunks;
    p.b_bytes = (uint32_t)((size_t)p.N * K * 4);
    p.tmem_cols = 64;
    while (p.tmem_cols < 4 * p.N) p.tmem_cols *= 2;      // two pairs of accumulators
    const uint32_t red = p.cluster > 1 ? (uint32_t)(p.cluster - 1) * (4 / p.cluster) * p.N * 128u : 0u;
    const long long rest = (long long)kSmemLimit - 1024 - 1024 - (long long)sizeof(Tf32Shared) - 2ll * p.b_bytes - red;
    p.n_stages = rest > 0 ? (int)(rest / (2 * kABytes)) : 0;
    if (p.n_stages > kMaxStages) p.n_stages = kMaxStages;
    p.red_off = (uint32_t)p.n_stages * 2u * kABytes + 2u * p.b_bytes;
    p.smem = 1024 + (size_t)p.red_off + red;
    p.ok = p.n_stages >= 2;
    return p;
}

}  // namespace

// By the geometry alone, never by the number of slots: a slot's values must not depend on the batch that it is in (the
// two kernels round differently). The kernel's time hardly depends on the beams (it is bound by its loading), that of the
// FP32 kernel goes with them in steps of 8, 16, 32 and 64. FP32 FMAs against this kernel, us, one slot / 12 slots:
//   more than 32 beams       32 x 33 x 101: 11 / 10;  64 x 40 x 25: 15 / 13;  256 x 64 x 333: 83 / 25 (one slot)
//   more than 64 antennas    72 x 24 x 129: 15, 35 / 12, 31;  96 x 32 x 257: 15, 48 / 14, 47;  96 x 32 x 1153: 23, 164 / 20, 131
//   33..64 antennas          64 x 24: 385 subcarriers 11, 52 / 13, 42;  513: 11, 59 / 13, 48;  641: 16, 70 / 13, 55
//   32 antennas              32 x 24: 641 subcarriers 10, 39 / 11, 35;  1025: 11, 56 / 11, 47;  2305: 15, 117 / 14, 92
// so at 17..32 beams and up to 64 antennas the line lies where one slot is about even. At 8 beams the FP32 kernel is
// faster (64 antennas, 3275 subcarriers, 8 slots: 111 against 134 us).
bool bf_tf32k_supported(const Geometry &g) {
    if (g.form != PUSCH_FORM_FP32 || !tf32_plan(g).ok || g.n_rx < 32 || g.n_beams <= 16) return false;
    return g.n_beams > 32 || g.n_rx > 64 || g.n_sc > (g.n_rx > 32 ? 512 : 1024);
}

cudaError_t launch_beamform_tf32k(const Geometry &g, int n_slots, const float2 *freq, const float2 *W, float2 *beam,
                                 uint32_t *err_word, cudaStream_t st) {
    if (n_slots == 0) return cudaSuccess;
    if (!tf32_plan(g).ok) return cudaErrorNotSupported;
    const Tf32Plan p = tf32_plan(g);
    Tf32Args a;
    a.n_rx = g.n_rx;
    a.n_beams = g.n_beams;
    a.n_sc = g.n_sc;
    a.n_mtiles = (g.n_sc + kTileM - 1) / kTileM;
    a.N = p.N;
    a.n_chunks = p.n_chunks;
    a.n_stages = p.n_stages;
    a.tmem_cols = p.tmem_cols;
    a.cluster = p.cluster;
    a.vec4 = g.n_beams % 2 == 0 && reinterpret_cast<uintptr_t>(beam) % 16 == 0;
    a.b_bytes = p.b_bytes;
    a.red_off = p.red_off;
    const long long tiles = (long long)n_slots * g.n_sym * a.n_mtiles;
    if (tiles * p.n_chunks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    a.total_tiles = (int)tiles;
    cudaError_t e = cudaFuncSetAttribute(beamform_tf32k_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.smem);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    ChainedConfig c(g.chained, dim3((unsigned)(sms / p.cluster * p.cluster)), dim3(kThreads), p.smem, st,
                    (unsigned)p.cluster);
    // as many clusters as are resident at once (36 of 4 CTAs on 152 SMs): the tiles are dealt out evenly, so a
    // cluster that had to wait for a place would double the time
    int clusters = sms;
    if (p.cluster > 1 && (e = cudaOccupancyMaxActiveClusters(&clusters, beamform_tf32k_kernel, &c.cfg)) != cudaSuccess)
        return e;
    if (clusters < 1) return cudaErrorInvalidConfiguration;
    if (clusters > tiles) clusters = (int)tiles;
    c.cfg.gridDim = dim3((unsigned)(clusters * p.cluster));
    if ((e = cudaLaunchKernelEx(&c.cfg, beamform_tf32k_kernel, a, freq, W, beam, err_word)) != cudaSuccess) return e;
    return cudaGetLastError();
}

}  // namespace pusch
