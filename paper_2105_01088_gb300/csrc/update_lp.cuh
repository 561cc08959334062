// Per-state update of App. A in the TF32 and BF16 forms: the orthogonal step
// Gamma <- R Gamma R^T, R = exp(X), X = (ds/4)[Gamma, dGamma] (Eq. ExpStep), with
// its products on the tensor cores, followed by the FP64 canonical-form
// renormalisation (Newton-Schulz polar iteration).
//
// Only small quantities pass through the low-precision products, so their
// relative rounding (2^-11 for TF32) scales the step, not the state:
//   * E = R - I by scaling and squaring in increment form: with X_s = X 2^-s,
//     E_s = X_s P_2, P_j = I + (X_s / j) P_{j+1}, P_d = I + X_s / d (Horner), and
//     each squaring E <- 2E + E E.  The recurrences run on transposes, which the
//     tensor core reads directly (a K-major operand is a row-major transpose):
//     Q_j = P_j^T = I + (1/j) Q_{j+1} X_s^T, E^T = Q_2 X_s^T, E^T <- 2 E^T + E^T E^T,
//     each product also writing its transpose.
//   * Gamma' = Gamma + F - F^T + G, F = E Gamma, G = F E^T (= E Gamma E^T), summed
//     in FP64 onto the FP64 Gamma.
// The purification then removes the purity drift of order 2^-11 ||E|| in FP64.
#pragma once
#include <cuda_bf16.h>
#include "common.cuh"
#include "update.cuh"

namespace sgs {

#define EXP_LP_DEGREE 6        // Taylor degree: ||X_s|| <= 1/8 truncates below 1e-10 relative
#define LP_NS_ITERS 3          // purity drift ~1e-3 ||E|| reaches rounding in three Newton-Schulz steps

// Partial sums of ||X||_F^2 of X = (ds/4)(Y - Y^T) (Y: [M][n][n] fp32), both entries of a pair from tiles
// K >= L staged through shared memory.  Grid (EXP_PARTX, states), 256 threads.
__global__ void __launch_bounds__(256) exp_norm_lp_kernel(const float* Y, int n, double ds, double* part) {
    __shared__ float t[32][33];
    __shared__ double red[32];
    const int mu = blockIdx.y, tiles = lower_tile_count(n), tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const float* y = Y + (size_t)mu * n * n;
    double ss = 0.0;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        int K, L;
        lower_tile(tile, K, L);
        const int k0 = K * 32, l0 = L * 32;
        for (int j = ty; j < 32; j += 8)
            t[j][tx] = (l0 + j < n && k0 + tx < n) ? y[(size_t)(l0 + j) * n + k0 + tx] : 0.0f;
        __syncthreads();
        for (int j = ty; j < 32; j += 8) {
            const int k = k0 + j, l = l0 + tx;
            if (k >= n || l >= n || k <= l) continue;
            const double v = 0.25 * ds * ((double)y[(size_t)k * n + l] - (double)t[tx][j]);
            ss = fma(2.0 * v, v, ss);
        }
        __syncthreads();
    }
    ss = block_sum(ss, red);
    if (threadIdx.x == 0) part[(size_t)mu * EXP_PARTS + blockIdx.x] = ss;
}

// X_s = 2^-s (ds/4)(Y - Y^T) with ||X_s||_F <= 1/8 and Q_d = I - X_s / d; X_s, Q: [M][n][ldp] fp32, whose
// padding columns are zero already.  Grid (CTAs, states), 256 threads.
__global__ void __launch_bounds__(256) exp_prepare_lp_kernel(const float* Y, int n, int ldp, double ds,
                                                             const double* part, float* Xs, float* Q, int* sq, int* err) {
    __shared__ float a[32][33], t[32][33];
    __shared__ double red[32];
    const int mu = blockIdx.y, tiles = lower_tile_count(n), tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const double nrm = sqrt(block_sum(threadIdx.x < EXP_PARTX ? part[(size_t)mu * EXP_PARTS + threadIdx.x] : 0.0, red));
    int s = 0;
    while (nrm * ldexp(1.0, -s) > EXP_THETA && s < 64) s++;
    if (s > EXP_MAX_SQUARINGS) {
        if (threadIdx.x == 0 && blockIdx.x == 0) atomicOr(err, SGS_DEV_EXPNORM);
        s = EXP_MAX_SQUARINGS;
    }
    if (threadIdx.x == 0 && blockIdx.x == 0) sq[mu] = s;
    const float sc = (float)(0.25 * ds * ldexp(1.0, -s));
    const float* y = Y + (size_t)mu * n * n;
    float* xs = Xs + (size_t)mu * n * ldp;
    float* q = Q + (size_t)mu * n * ldp;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        int K, L;
        lower_tile(tile, K, L);
        const int k0 = K * 32, l0 = L * 32;
        for (int j = ty; j < 32; j += 8) {
            a[j][tx] = (k0 + j < n && l0 + tx < n) ? y[(size_t)(k0 + j) * n + l0 + tx] : 0.0f;
            t[j][tx] = (l0 + j < n && k0 + tx < n) ? y[(size_t)(l0 + j) * n + k0 + tx] : 0.0f;
        }
        __syncthreads();
        for (int j = ty; j < 32; j += 8)
            for (int side = 0; side < (K == L ? 1 : 2); side++) {         // tile (K, L), and (L, K)
                const int k = (side ? l0 : k0) + j, l = (side ? k0 : l0) + tx;
                if (k >= n || l >= n) continue;
                const float v = sc * (side ? t[j][tx] - a[tx][j] : a[j][tx] - t[tx][j]);
                xs[(size_t)k * ldp + l] = v;
                q[(size_t)k * ldp + l] = (k == l ? 1.0f : 0.0f) - v * (1.0f / EXP_LP_DEGREE);
            }
        __syncthreads();
    }
}

// fp32 [count] -> tensor-core operand: kind 0 tf32 (rounded to nearest), 1 bf16, 2 tf32
// split (hi, lo)
__global__ void lp_split_kernel(const float* src, void* hi, void* lo, size_t count, int kind) {
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < count; e += (size_t)gridDim.x * blockDim.x) {
        const float x = src[e];
        if (kind == 0) {
            static_cast<float*>(hi)[e] = round_tf32(x);
        } else if (kind == 1) {
            static_cast<__nv_bfloat16*>(hi)[e] = __float2bfloat16_rn(x);
        } else {
            const float h = __uint_as_float(__float_as_uint(x) & 0xffffe000u);
            static_cast<float*>(hi)[e] = h;
            static_cast<float*>(lo)[e] = x - h;
        }
    }
}

// the same for two arrays of [M][count] whose state's flag is above cmp (the states a squaring has changed);
// grid (CTAs, M)
__global__ void lp_split2_kernel(const float* src0, void* hi0, const float* src1, void* hi1, size_t count, int kind,
                                 const int* flag, int cmp) {
    if (flag[blockIdx.y] <= cmp) return;
    const size_t off = blockIdx.y * count;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < 2 * count; e += (size_t)gridDim.x * blockDim.x) {
        const bool second = e >= count;
        const size_t o = off + (second ? e - count : e);
        const float x = (second ? src1 : src0)[o];
        void* hi = second ? hi1 : hi0;
        if (kind == 1) static_cast<__nv_bfloat16*>(hi)[o] = __float2bfloat16_rn(x);
        else static_cast<float*>(hi)[o] = round_tf32(x);
    }
}

// the operand copies [M][bytes] of states with an odd flag from odd to even (the buffer a state's last
// squaring wrote); grid (CTAs, M)
__global__ void lp_select_kernel(const uint4* odd, uint4* even, size_t words, const int* flag) {
    if ((flag[blockIdx.y] & 1) == 0) return;
    const size_t off = blockIdx.y * words;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < words; e += (size_t)gridDim.x * blockDim.x)
        even[off + e] = odd[off + e];
}

// FP64 [M][n][n] -> operand [M][n][ldp]: kind 0 tf32 (rounded), 1 bf16, 2 tf32 split (hi, lo)
__global__ void lp_from_f64_kernel(const double* src, int n, int ldp, void* hi, void* lo, int kind) {
    const int mu = blockIdx.y;
    const double* x = src + (size_t)mu * n * n;
    const size_t off = (size_t)mu * n * ldp;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < (size_t)n * ldp; e += (size_t)gridDim.x * blockDim.x) {
        const int k = (int)(e / ldp), l = (int)(e % ldp);
        const double v = l < n ? x[(size_t)k * n + l] : 0.0;
        if (kind == 1) {
            static_cast<__nv_bfloat16*>(hi)[off + e] = __float2bfloat16_rn((float)v);
        } else if (kind == 2) {
            const float f = (float)v;
            const float h = __uint_as_float(__float_as_uint(f) & 0xffffe000u);
            static_cast<float*>(hi)[off + e] = h;
            static_cast<float*>(lo)[off + e] = (float)(v - (double)h);
        } else {
            static_cast<float*>(hi)[off + e] = round_tf32((float)v);
        }
    }
}

// Gamma' = Gamma + (F - F^T) + (G - G^T)/2 in FP64; F, G: [M][n][ldp] fp32
__global__ void assemble_lp_kernel(const double* gamma, const float* F, const float* G, int n, int ldp, double* out) {
    const int mu = blockIdx.y;
    const size_t nn = (size_t)n * n, np = (size_t)n * ldp;
    const double* g = gamma + mu * nn;
    const float* f = F + mu * np;
    const float* h = G + mu * np;
    double* o = out + mu * nn;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < nn; e += (size_t)gridDim.x * blockDim.x) {
        const int k = (int)(e / n), l = (int)(e % n);
        const size_t a = (size_t)k * ldp + l, t = (size_t)l * ldp + k;
        o[e] = g[e] + ((double)f[a] - (double)f[t]) + 0.5 * ((double)h[a] - (double)h[t]);
    }
}

}  // namespace sgs
