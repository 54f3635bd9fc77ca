// Gram matrix and right-hand sides of the MMSE detector (Eq. 2: G = H^H H, r_d = H^H y_d) on the tensor
// cores, one subcarrier per warp at a time: warp-level mma.sync m16n8k8 with TF32 operands and FP32
// accumulation. A subcarrier's products are 16 (or 32) rows of layers against K = 2 N_B real values, which is
// the M = 16 of this instruction shape exactly (the 5th-generation tcgen05 products start at M = 64, where one
// subcarrier would fill an eighth of the tile).
//
// The real and imaginary parts of eight beams are two K = 8 steps (16-byte loads bring two beams' both parts):
//   Re G = A_r A_r^T + A_i A_i^T                          (B = A^T: the A fragments serve as B fragments)
//   Im G = X - X^T,  X = A_r A_i^T                        (Im(conj(h_i) h_j); the difference is taken when a lane reads
//                                                          its row of G from shared memory)
//   P = A_r Y, Q = A_i Y,  Y = the 12 data symbols' re and im parts as 24 columns;  Re r_d = P[re d] + Q[im d],
//   Im r_d = P[im d] - Q[re d]
// Each of the five sums has its own accumulator: the tensor core truncates as it accumulates, which shrinks a sum by an
// amount that goes with its number of steps, and equal shrinking of G and r_d cancels in x (with Re G in one accumulator
// of twice the steps x was off by 1.8e-6 instead of 8.6e-7 for 32 layers; the interleaved embedding: 1.3e-6).
// Against the interleaved embedding (K = 2 N_B, Im G and Im r_d from rotated copies of the operands) this loads and
// splits each element once instead of twice and takes 36 products per 8 beams instead of 42 (16 layers; 32 layers, with
// the tiles of Re G above the diagonal left out: 96 instead of 132). Measured on GB300 (pusch_mmse_detect): 16 layers,
// 32 beams, 8 slots 120 -> 110 us; 32 layers, 64 beams, 2 slots 167 -> 153 us.
// FP32 accuracy from TF32 operands: every operand x is split into hi = x rounded to TF32 (10 explicit mantissa
// bits, ties away from zero, by an integer add and mask) and lo = x - hi (exact, |lo| <= 2^-11 |x|), which the
// tensor core reads truncated to TF32 (|x - hi - lo_tf32| <= 2^-21 |x|); each product is hi*hi + hi*lo + lo*hi
// (the lo*lo term, below 2^-22, dropped), accumulated small terms first. (The conversion instruction
// cvt.rna.tf32.f32 rounds the same way but measured 11 % slower here: it does not issue at the full rate.)
#pragma once

#include "detect_core.cuh"

namespace pusch {

__device__ __forceinline__ void tf32_split(float x, uint32_t &hi, uint32_t &lo) {
    hi = (__float_as_uint(x) + 0x1000u) & 0xffffe000u;   // round the magnitude at mantissa bit 13
    lo = __float_as_uint(x - __uint_as_float(hi));
}

__device__ __forceinline__ void mma_tf32_16x8x8(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// c += a b with a, b split in hi / lo parts (three products, the small ones first)
__device__ __forceinline__ void mma3_tf32(float (&c)[4], const uint32_t (&ah)[4], const uint32_t (&al)[4],
                                          uint32_t bh0, uint32_t bh1, uint32_t bl0, uint32_t bl1) {
    mma_tf32_16x8x8(c, al, bh0, bh1);
    mma_tf32_16x8x8(c, ah, bl0, bl1);
    mma_tf32_16x8x8(c, ah, bh0, bh1);
}

// G and r_d (12 data symbols) of one subcarrier by the whole warp.
//   H: the subcarrier's estimate rows (row i at H + i hs, NL rows of nb values)
//   Y: its data-symbol rows (row d at Y + d ys), overwritten by r_d: r_d[i] at Y[d ys + i]
//   Gs: (Re G[i][j] for j <= i, X[i][j]) at Gs + i (NL + 2) + j, over the estimate rows (written after every lane has
//       read them)
// Fragment layout of m16n8k8 (g = lane / 4, t = lane % 4): A rows g, g + 8 at columns t, t + 4; B column g at
// rows t, t + 4; the accumulator rows g, g + 8 at columns 2 t, 2 t + 1.
// NB = 0: the beam count nb at run time (a multiple of 4; the rest of a last step of 4 beams is zero).
template <int NL, int NB>
__device__ __forceinline__ void gram_rhs_tc(const float2 *H, int hs, float2 *Y, int ys, float2 *Gs, int lane, int nb = NB) {
    constexpr int MT = NL / 16;     // 16-row tiles of layers
    constexpr int NG = NL / 8;      // 8-column tiles of G's columns
    constexpr int GS = NL + 2;      // row stride of Gs (float2): the 16-byte row loads below spread over banks
    const int g = lane >> 2, t = lane & 3;
    float cg[MT][NG][4], ci[MT][NG][4], cx[MT][NG][4], cp[MT][3][4], cq[MT][3][4];
#pragma unroll
    for (int m = 0; m < MT; ++m) {
#pragma unroll
        for (int n = 0; n < NG; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) cg[m][n][e] = ci[m][n][e] = cx[m][n][e] = 0.f;
#pragma unroll
        for (int q = 0; q < 3; ++q)
#pragma unroll
            for (int e = 0; e < 4; ++e) cp[m][q][e] = cq[m][q][e] = 0.f;
    }
    // K index t is beam k0 + 2 t, t + 4 is beam k0 + 2 t + 1 (the order of K is free): one 16-byte load brings both
    const float2 *h0 = H + g * hs + 2 * t;
    const float2 *y0 = Y + g * ys + 2 * t, *y1 = Y + (8 + (g & 3)) * ys + 2 * t;   // columns g; 8 + g % 4 (re for g < 4, else im)
    const int n_b = NB > 0 ? NB : nb;
#pragma unroll 1
    for (int k0 = 0; k0 < n_b; k0 += 8) {
        const bool on = NB > 0 || k0 + 2 * t < n_b;
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        uint32_t rh[MT][4], rl[MT][4], ih[MT][4], il[MT][4];
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const float4 v = on ? *reinterpret_cast<const float4 *>(h0 + (16 * m + 8 * q) * hs + k0) : zero;
                tf32_split(v.x, rh[m][q], rl[m][q]);
                tf32_split(v.y, ih[m][q], il[m][q]);
                tf32_split(v.z, rh[m][q + 2], rl[m][q + 2]);
                tf32_split(v.w, ih[m][q + 2], il[m][q + 2]);
            }
        // B column tile n = rows 8 n .. 8 n + 7 of A, i.e. registers (0, 2) or (1, 3) of A tile n / 2
#pragma unroll
        for (int n = 0; n < NG; ++n) {
            const int mb = n >> 1, j0 = n & 1, j1 = j0 + 2;
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                if (mb <= m) {
                    mma3_tf32(cg[m][n], rh[m], rl[m], rh[mb][j0], rh[mb][j1], rl[mb][j0], rl[mb][j1]);
                    mma3_tf32(ci[m][n], ih[m], il[m], ih[mb][j0], ih[mb][j1], il[mb][j0], il[mb][j1]);
                }
                mma3_tf32(cx[m][n], rh[m], rl[m], ih[mb][j0], ih[mb][j1], il[mb][j0], il[mb][j1]);
            }
        }
        // right-hand sides: columns Re y_0..7; Im y_0..7; Re y_8..11 and Im y_8..11
        {
            const float4 va = on ? *reinterpret_cast<const float4 *>(y0 + k0) : zero;
            const float4 vb = on ? *reinterpret_cast<const float4 *>(y1 + k0) : zero;
            uint32_t bh[3][2], bl[3][2];
            tf32_split(va.x, bh[0][0], bl[0][0]);
            tf32_split(va.z, bh[0][1], bl[0][1]);
            tf32_split(va.y, bh[1][0], bl[1][0]);
            tf32_split(va.w, bh[1][1], bl[1][1]);
            tf32_split(g < 4 ? vb.x : vb.y, bh[2][0], bl[2][0]);
            tf32_split(g < 4 ? vb.z : vb.w, bh[2][1], bl[2][1]);
#pragma unroll
            for (int q = 0; q < 3; ++q)
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    mma3_tf32(cp[m][q], rh[m], rl[m], bh[q][0], bh[q][1], bl[q][0], bl[q][1]);
                    mma3_tf32(cq[m][q], ih[m], il[m], bh[q][0], bh[q][1], bl[q][0], bl[q][1]);
                }
        }
    }
    __syncwarp();  // every lane has read the estimate and data-symbol rows
#pragma unroll
    for (int m = 0; m < MT; ++m) {
#pragma unroll
        for (int n = 0; n < NG; ++n) {
            const int i = 16 * m + g, j = 8 * n + 2 * t;
            *reinterpret_cast<float4 *>(Gs + i * GS + j) = make_float4(
                cg[m][n][0] + ci[m][n][0], cx[m][n][0], cg[m][n][1] + ci[m][n][1], cx[m][n][1]);
            *reinterpret_cast<float4 *>(Gs + (i + 8) * GS + j) =
                make_float4(cg[m][n][2] + ci[m][n][2], cx[m][n][2], cg[m][n][3] + ci[m][n][3], cx[m][n][3]);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int c = 2 * t + (e & 1), i = 16 * m + g + 8 * (e >> 1);
            Y[c * ys + i] = make_float2(cp[m][0][e] + cq[m][1][e], cp[m][1][e] - cq[m][0][e]);
            // third tile: Re parts in the lanes t < 2, Im parts in t >= 2; the other product is two lanes away
            const float o = __shfl_xor_sync(kDetFull, cq[m][2][e], 2);
            reinterpret_cast<float *>(Y + (8 + (c & 3)) * ys + i)[t >> 1] = t < 2 ? cp[m][2][e] + o : cp[m][2][e] - o;
        }
    }
}

// Steps 2-4 of the 12-data-symbol detector for the warp's SPW = 32 / NL subcarriers: G and r_d of each on the
// tensor cores (gram_rhs_tc), then lane i of group grp takes row i of its subcarrier's G, adds the loading on
// the diagonal (identity rows past nl), and the Crout factorisation and the solves run as in detect_group.
//   Hw, Yw: the warp's estimate tiles (stride ht float2 per subcarrier, rows hs) and data-symbol rows (12 per
//   subcarrier, stride ys). Returns true when a pivot of lane i's subcarrier was not a positive finite number.
//   NB = 0: nb beams at run time (a multiple of 4; the ragged batch's segments). G overlays the estimate tile:
//   ht >= NL (NL + 2) float2.
template <int NL, int NB>
__device__ __forceinline__ bool detect_group_tc(float2 *Hw, int ht, int hs, float2 *Yw, int ys, int nl, float load,
                                                int grp, int i, int src0, int lane, float2 (&acc)[12],
                                                const float *__restrict__ sigma2 = nullptr, long long slot = 0,
                                                int nb = NB) {
    constexpr int SPW = 32 / NL, GS = NL + 2;
#pragma unroll 1
    for (int gg = 0; gg < SPW; ++gg)
        gram_rhs_tc<NL, NB>(Hw + gg * ht, hs, Yw + gg * 12 * ys, ys, Hw + gg * ht, lane, nb);
    __syncwarp();
    float2 G[NL];
    {
        // own row, and the column of X that makes Im G[i][j] = X[i][j] - X[j][i]
        const float4 *row = reinterpret_cast<const float4 *>(Hw + grp * ht + i * GS);
        const float2 *col = Hw + grp * ht + i;
#pragma unroll
        for (int j = 0; j < NL / 2; ++j) {
            const float4 v = row[j];
            G[2 * j] = make_float2(v.x, v.y - col[2 * j * GS].y);
            G[2 * j + 1] = make_float2(v.z, v.w - col[(2 * j + 1) * GS].y);
        }
    }
    if (sigma2) load += __ldg(&sigma2[slot]);
#pragma unroll
    for (int j = 0; j < NL; ++j)
        if (j == i) G[j] = (i < nl) ? make_float2(G[j].x + load, 0.f) : make_float2(1.f, 0.f);
    __syncwarp();  // every lane holds its row of G: the tile takes L
    return factor_solve_rhs_lanes<NL, 12, 12, true>(G, Yw + grp * 12 * ys, Hw + grp * ht, ys, 12, i, src0, acc);
}

}  // namespace pusch
