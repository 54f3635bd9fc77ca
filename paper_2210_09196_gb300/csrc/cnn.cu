// Learned channel-estimate denoiser: four 3x3 same-padded convolutions 2 -> 32 -> 32 -> 32 -> 2, ReLU after
// the first three, the input added to the output; the kernels are dilated along the subcarriers by 1, 8, 16, 1
// (receptive field +-26 subcarriers, several pilot spacings). Grids are [n][c][2][w]: n grids (one per slot, layer and
// beam), c channels (re, im of the estimate at the input and output), the two DMRS symbols as rows and w
// subcarriers. Weights and activations are stored as bfloat16, arithmetic and gradients are FP32, the
// optimiser keeps FP32 master weights. Parameters are packed per layer as W[co][ci][3][3] then b[co].
//
// Here: Adam, and for the receive chain the per-DMRS-symbol LS grid builder and the estimate writer with the
// pilot-residual fallback to the plain LS estimate. The forward pass is in cnn_tc.cu, the backward pass in cnn_bwd.cu.
#include <cuda_bf16.h>

#include "chest_common.cuh"

namespace pusch {
namespace {

constexpr int kCh[5] = {2, 32, 32, 32, 2};

__global__ void adam_kernel(int n, float lr, float b1, float b2, float eps, float c1, float c2, float *__restrict__ p,
                            __nv_bfloat16 *__restrict__ pb, const float *__restrict__ g, float *__restrict__ m,
                            float *__restrict__ v) {
    chain_wait(p, pb, g, m, v);
    chain_go();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = pi;
    pb[i] = __float2bfloat16_rn(pi);
}

int param_offset(int layer) {
    int off = 0;
    for (int k = 0; k < layer; ++k) off += kCh[k + 1] * kCh[k] * 9 + kCh[k + 1];
    return off;
}

}  // namespace

int cnn_param_count() { return param_offset(4); }

// Forward pass of n grids of width w (cnn_tc.cu). x: [n][2][2][w] bf16, y: [n][2][2][w] f32; acts (or NULL):
// [3][n][32][2][w] bf16, the post-ReLU activations.
cudaError_t cnn_forward(int n, int w, const __nv_bfloat16 *x, const __nv_bfloat16 *P, float *y, __nv_bfloat16 *acts,
                        cudaStream_t st, uint32_t *err, unsigned long long selftest_ns) {
    return launch_cnn_fwd(x, P, y, acts, n, w, err, st, selftest_ns);
}

// Backward pass (cnn_bwd.cu): grad (zeroed here) = d mean((y - target)^2) / d params; *loss = that mean (if loss !=
// NULL). work: 2 * n * 32 * 2 * w floats.
cudaError_t cnn_backward(int n, int w, const __nv_bfloat16 *x, const __nv_bfloat16 *acts, const __nv_bfloat16 *P,
                         const float *y, const float *target, float *grad, float *loss, float *work, cudaStream_t st,
                         unsigned long long selftest_ns) {
    cudaError_t e;
    if ((e = cudaMemsetAsync(grad, 0, sizeof(float) * cnn_param_count(), st)) != cudaSuccess) return e;
    if (loss && (e = cudaMemsetAsync(loss, 0, sizeof(float), st)) != cudaSuccess) return e;
    return launch_cnn_bwd(n, w, x, acts, P, y, target, grad, loss, work, nullptr, st, selftest_ns);
}

cudaError_t cnn_adam(int step, float lr, float b1, float b2, float eps, float *p, __nv_bfloat16 *pb, const float *g,
                     float *m, float *v, cudaStream_t st) {
    const int n = cnn_param_count();
    const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
    launch_chained(true, adam_kernel, dim3((n + 255) / 256), dim3(256), 0, st, n, lr, b1, b2, eps, c1, c2, p, pb, g, m, v);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------- receive-chain glue

namespace {

struct GridArgs {
    int n_sc, n_beams, n_layers, comb, n_sym, dmrs0, dmrs1;
    int port[32];
};

// Per-DMRS-symbol LS estimate of one (slot, layer, beam) grid, interpolated over the subcarriers:
// v_j[a] = interp(y_j[q] / p_j[q]) between the layer's pilot subcarriers (held outside them).
__device__ __forceinline__ float2 grid_value(const GridArgs &g, const float2 *y, const float2 *p, int a, int port) {
    int lo, hi;
    pilot_bracket(a, port, g.comb, g.n_sc, lo, hi);
    const float2 vlo = cmul(__ldg(&y[(long long)lo * g.n_beams]), pilot_inverse(__ldg(&p[lo])));
    if (hi == lo) return vlo;
    const float2 vhi = cmul(__ldg(&y[(long long)hi * g.n_beams]), pilot_inverse(__ldg(&p[hi])));
    return interp(vlo, vhi, interp_weight(a, lo, hi));
}

__device__ __forceinline__ float block_sum(float v, float *red) {
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    float s = 0.f;
    if (threadIdx.x < 32) {
        s = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.f;
        for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
        if (threadIdx.x == 0) red[0] = s;
    }
    __syncthreads();
    s = red[0];
    __syncthreads();
    return s;
}

// grid[gi][ch][j][a] (bf16) = v_j[a] / scale with scale = rms over the grid; gi = (slot * L + l) * B + b.
// The layer's LS values are formed once, in shared memory (n_pil of them per symbol; 0: they do not fit, and every
// subcarrier forms its own). Formed per subcarrier and pass, eight loads a beam row apart and eight reciprocals each
// bounded the kernel: one slot's estimate (512 grids of 3276, a pilot in 16) took 273 us, 245 so.
__global__ void __launch_bounds__(256)
ls_grid_kernel(GridArgs g, int smem_pilots, const float2 *__restrict__ beam, const float2 *__restrict__ pilots,
               __nv_bfloat16 *__restrict__ grid, float *__restrict__ scale) {
    chain_wait(beam, pilots, grid, scale);
    chain_go();
    __shared__ float red[32];
    extern __shared__ float2 s_ls[];             // [2][n_pil]
    const long long gi = blockIdx.x;
    const int b = (int)(gi % g.n_beams);
    const long long sl_l = gi / g.n_beams;
    const int l = (int)(sl_l % g.n_layers);
    const long long slot = sl_l / g.n_layers;
    const float2 *y0 = beam + ((slot * g.n_sym + g.dmrs0) * g.n_sc) * (long long)g.n_beams + b;
    const float2 *y1 = beam + ((slot * g.n_sym + g.dmrs1) * g.n_sc) * (long long)g.n_beams + b;
    const float2 *p0 = pilots + (slot * g.n_layers + l) * 2LL * g.n_sc;
    const float2 *p1 = p0 + g.n_sc;
    const int port = g.port[l];
    const int n_pil = smem_pilots ? (g.n_sc - 1 - port) / g.comb + 1 : 0;
    for (int k = threadIdx.x; k < n_pil; k += blockDim.x) {
        const int q = port + k * g.comb;
        s_ls[k] = cmul(__ldg(&y0[(long long)q * g.n_beams]), pilot_inverse(__ldg(&p0[q])));
        s_ls[n_pil + k] = cmul(__ldg(&y1[(long long)q * g.n_beams]), pilot_inverse(__ldg(&p1[q])));
    }
    __syncthreads();
    auto values = [&](int a, float2 &v0, float2 &v1) {
        if (n_pil == 0) {
            v0 = grid_value(g, y0, p0, a, port);
            v1 = grid_value(g, y1, p1, a, port);
            return;
        }
        const int k = a <= port ? 0 : min((a - port) / g.comb, n_pil - 1), lo = port + k * g.comb;
        v0 = s_ls[k];
        v1 = s_ls[n_pil + k];
        if (a > lo && k + 1 < n_pil) {
            const float w = interp_weight(a, lo, lo + g.comb);
            v0 = interp(v0, s_ls[k + 1], w);
            v1 = interp(v1, s_ls[n_pil + k + 1], w);
        }
    };
    float ss = 0.f;
    for (int a = threadIdx.x; a < g.n_sc; a += blockDim.x) {
        float2 v0, v1;
        values(a, v0, v1);
        // the contraction is written out: another one moves the scale by an ulp and with it a BF16 rounding now and then
        ss += fmaf(v1.y, v1.y, fmaf(v1.x, v1.x, fmaf(v0.x, v0.x, __fmul_rn(v0.y, v0.y))));
    }
    const float tot = block_sum(ss, red);
    const float sc = sqrtf(tot / (2.f * g.n_sc)) + 1e-30f;
    const float inv = 1.f / sc;
    if (threadIdx.x == 0) scale[gi] = sc;
    __nv_bfloat16 *o = grid + gi * 4LL * g.n_sc;  // [2 ch][2 rows][n_sc]
    for (int a = threadIdx.x; a < g.n_sc; a += blockDim.x) {
        float2 v0, v1;
        values(a, v0, v1);
        o[0 * g.n_sc + a] = __float2bfloat16_rn(v0.x * inv);
        o[1 * g.n_sc + a] = __float2bfloat16_rn(v1.x * inv);
        o[2 * g.n_sc + a] = __float2bfloat16_rn(v0.y * inv);
        o[3 * g.n_sc + a] = __float2bfloat16_rn(v1.y * inv);
    }
}

// Denoised estimate of grid gi: H = scale * (y_row0 + y_row1) / 2.
// Fallback test on the layer's pilots q (both DMRS symbols j, LS_j[q] = y_j[q] / p_j[q]):
//   r_cnn = mean |LS_j[q] - scale * y_row_j[q]|^2                 (how well the estimate explains the pilots)
//   r_ref = mean |LS_j[q] - (LS_j[q - comb] + LS_j[q + comb]) / 2|^2 over the inner pilots
//           (how well plain linear interpolation predicts a pilot from its neighbours), floored at sigma^2.
// r_cnn <= kappa * r_ref: the CNN estimate replaces the plain LS estimate in H_hat; otherwise the plain LS
// estimate already written there is kept (fallback). resid[gi] = r_cnn / r_ref.
__global__ void __launch_bounds__(256)
cnn_to_h_kernel(GridArgs g, float noise_var, float kappa, const float *__restrict__ y, const float *__restrict__ scale,
                const float2 *__restrict__ beam, const float2 *__restrict__ pilots, float2 *__restrict__ H,
                float *__restrict__ resid, uint8_t *__restrict__ fallback) {
    chain_wait(y, scale, beam, pilots, H, resid, fallback);
    chain_go();
    __shared__ float red[32];
    const long long gi = blockIdx.x;
    const int b = (int)(gi % g.n_beams);
    const long long sl_l = gi / g.n_beams;
    const int l = (int)(sl_l % g.n_layers);
    const long long slot = sl_l / g.n_layers;
    const float2 *y0 = beam + ((slot * g.n_sym + g.dmrs0) * g.n_sc) * (long long)g.n_beams + b;
    const float2 *y1 = beam + ((slot * g.n_sym + g.dmrs1) * g.n_sc) * (long long)g.n_beams + b;
    const float2 *p0 = pilots + (slot * g.n_layers + l) * 2LL * g.n_sc;
    const float2 *p1 = p0 + g.n_sc;
    const float *yo = y + gi * 4LL * g.n_sc;
    const float sc = scale[gi];
    const int port = g.port[l];
    const int npil = (g.n_sc - 1 - port) / g.comb + 1;
    auto ls = [&](const float2 *yy, const float2 *pp, int q) {
        return cmul(__ldg(&yy[(long long)q * g.n_beams]), pilot_inverse(__ldg(&pp[q])));
    };
    float rc = 0.f, rr = 0.f;
    for (int k = threadIdx.x; k < npil; k += blockDim.x) {
        const int q = port + k * g.comb;
        const float2 l0 = ls(y0, p0, q), l1 = ls(y1, p1, q);
        const float d0x = l0.x - sc * yo[0 * g.n_sc + q], d0y = l0.y - sc * yo[2 * g.n_sc + q];
        const float d1x = l1.x - sc * yo[1 * g.n_sc + q], d1y = l1.y - sc * yo[3 * g.n_sc + q];
        rc += d0x * d0x + d0y * d0y + d1x * d1x + d1y * d1y;
        if (k > 0 && k + 1 < npil) {
            const float2 a0 = ls(y0, p0, q - g.comb), b0 = ls(y0, p0, q + g.comb);
            const float2 a1 = ls(y1, p1, q - g.comb), b1 = ls(y1, p1, q + g.comb);
            const float e0x = l0.x - 0.5f * (a0.x + b0.x), e0y = l0.y - 0.5f * (a0.y + b0.y);
            const float e1x = l1.x - 0.5f * (a1.x + b1.x), e1y = l1.y - 0.5f * (a1.y + b1.y);
            rr += e0x * e0x + e0y * e0y + e1x * e1x + e1y * e1y;
        }
    }
    const float r_cnn = block_sum(rc, red) / (2.f * npil);
    const float r_loo = npil > 2 ? block_sum(rr, red) / (2.f * (npil - 2)) : 0.f;
    const float r_ref = fmaxf(r_loo, noise_var > 0.f ? noise_var : 1e-30f);
    const bool use_cnn = r_cnn <= kappa * r_ref;
    if (threadIdx.x == 0) {
        if (resid) resid[gi] = r_cnn / r_ref;
        if (fallback) fallback[gi] = use_cnn ? 0 : 1;
    }
    if (!use_cnn) return;
    for (int a = threadIdx.x; a < g.n_sc; a += blockDim.x) {
        const float2 h = make_float2(0.5f * sc * (yo[0 * g.n_sc + a] + yo[1 * g.n_sc + a]),
                                     0.5f * sc * (yo[2 * g.n_sc + a] + yo[3 * g.n_sc + a]));
        H[((slot * g.n_sc + a) * g.n_layers + l) * (long long)g.n_beams + b] = h;
    }
}

GridArgs grid_args(const Geometry &g) {
    GridArgs a;
    a.n_sc = g.n_sc;
    a.n_beams = g.n_beams;
    a.n_layers = g.n_layers;
    a.comb = g.comb;
    a.n_sym = g.n_sym;
    a.dmrs0 = g.dmrs0;
    a.dmrs1 = g.dmrs1;
    for (int l = 0; l < 32; ++l) a.port[l] = g.port[l];
    return a;
}

}  // namespace

cudaError_t launch_ls_grid(const Geometry &g, int n_slots, const float2 *beam, const float2 *pilots,
                           __nv_bfloat16 *grid, float *scale, cudaStream_t st) {
    const long long grids = (long long)n_slots * g.n_layers * g.n_beams;
    if (grids == 0) return cudaSuccess;
    if (grids > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    const size_t bytes = ((size_t)(g.n_sc - 1) / g.comb + 1) * 2 * sizeof(float2);   // of the port with most pilots
    const int fits = bytes <= 47 * 1024;
    launch_chained(true, ls_grid_kernel, dim3((unsigned)grids), dim3(256), fits ? bytes : 0, st, grid_args(g), fits, beam,
                   pilots, grid, scale);
    return cudaGetLastError();
}

cudaError_t launch_cnn_to_h(const Geometry &g, int n_slots, float kappa, const float *y, const float *scale,
                            const float2 *beam, const float2 *pilots, float2 *H, float *resid, uint8_t *fallback,
                            cudaStream_t st) {
    const long long grids = (long long)n_slots * g.n_layers * g.n_beams;
    if (grids == 0) return cudaSuccess;
    launch_chained(true, cnn_to_h_kernel, dim3((unsigned)grids), dim3(256), 0, st, grid_args(g), g.noise_var + g.loading, kappa, y, scale, beam,
                                                     pilots, H, resid, fallback);
    return cudaGetLastError();
}

}  // namespace pusch
