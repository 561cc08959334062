// Per-state update of App. A: Gamma <- R Gamma R^T with R = exp(X),
// X = (ds/4)[Gamma, dGamma] (Eq. ExpStep; the factor 1/4 makes the step agree
// with Gamma + ds dGamma of Eq. RKstep to first order), followed by the
// canonical-form renormalisation (polar factor, Newton-Schulz in FP64).
//
// exp(X) by scaling and squaring: X_s = X / 2^s with ||X_s||_2 <= 1/8, the Taylor
// polynomial of degree 10 (truncation < 3e-18) evaluated by Paterson-Stockmeyer in
// blocks of three, p = B0 + B1 Y + B2 Y^2 + B3 Y^3 with Y = X_s^3 and
// B_j = sum_i X_s^i / (3j + i)!, i < 3 (five products instead of Horner's nine), then s
// squarings.  X is normal (antisymmetric), so ||X||_2 <= ||X^3||_F^(1/3), and X^3 is one of
// the polynomial's products: X^2 and X^3 are formed unscaled, s comes from ||X^3||_F, and the
// powers are scaled by powers of two (exact).  ||X||_F overestimates ||X||_2 by about
// sqrt(n) / 2 where X has no dominant directions, ||X^3||_F^(1/3) by (0.08 n)^(1/6): three
// squarings fewer at n = 2000, two and a half at 512.  The products run on the batched FP64
// GEMM; this file holds the elementwise pieces.
#pragma once
#include "common.cuh"

namespace sgs {

#define EXP_TAYLOR_DEGREE 10
#define EXP_MAX_SQUARINGS 14
#define EXP_THETA 0.125
#define EULER_NS_ITERS 6       // Newton-Schulz steps after an Euler step: singular values 1 + d with
                               // |d| <= 0.3 reach 1 to rounding (d -> -1.5 d^2 per step)

// partial sums of a state's exponential: EXP_PARTX of ||X||_F^2, then EXP_PART3 of ||X^3||_F^2
#define EXP_PARTX 128
#define EXP_PART3 64
#define EXP_PARTS (EXP_PARTX + EXP_PART3)

// X = (ds/4)(Y - Y^T) with Y = Gamma dGamma (so [Gamma, dGamma] = Y - Y^T), and partial sums of
// ||X||_F^2.  Both entries of a pair come from tiles K >= L staged through shared memory, so every read
// and write runs along rows.  Grid (EXP_PARTX, states), 256 threads.
__global__ void __launch_bounds__(256) exp_commutator_kernel(const double* Y, double* X, int n, double ds, double* part) {
    __shared__ double a[32][33], t[32][33], red[32];
    const int mu = blockIdx.y, tiles = lower_tile_count(n), tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const double* y = Y + (size_t)mu * n * n;
    double* x = X + (size_t)mu * n * n;
    double ss = 0.0;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        int K, L;
        lower_tile(tile, K, L);
        const int k0 = K * 32, l0 = L * 32;
        for (int j = ty; j < 32; j += 8) {            // a = Y[k0..][l0..], t = Y[l0..][k0..]
            a[j][tx] = (k0 + j < n && l0 + tx < n) ? y[(size_t)(k0 + j) * n + l0 + tx] : 0.0;
            t[j][tx] = (l0 + j < n && k0 + tx < n) ? y[(size_t)(l0 + j) * n + k0 + tx] : 0.0;
        }
        __syncthreads();
        for (int j = ty; j < 32; j += 8) {
            const double v = 0.25 * ds * (a[j][tx] - t[tx][j]);
            a[j][tx] = v;
            if (k0 + j > l0 + tx) ss = fma(2.0 * v, v, ss);
        }
        __syncthreads();
        store_antisym_tile(x, n, k0, l0, a);
        __syncthreads();
    }
    ss = block_sum(ss, red);
    if (threadIdx.x == 0) part[(size_t)mu * EXP_PARTS + blockIdx.x] = ss;
}

// partial sums of ||X^3||_F^2; grid (EXP_PART3, states)
__global__ void __launch_bounds__(256) exp_norm_kernel(const double* X3, int n, double* part) {
    __shared__ double red[32];
    const size_t nn = (size_t)n * n;
    const double* x = X3 + blockIdx.y * nn;
    double ss = 0.0;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < nn; e += (size_t)gridDim.x * blockDim.x)
        ss = fma(x[e], x[e], ss);
    ss = block_sum(ss, red);
    if (threadIdx.x == 0) part[(size_t)blockIdx.y * EXP_PARTS + EXP_PARTX + blockIdx.x] = ss;
}

// The squarings s of each state from ||X^3||_F; X, X^2 and X^3 scaled by 2^-s, 2^-2s, 2^-3s in place; the
// polynomial's leading block P = c1 X_s + c0 I; the state's result buffer after its s squarings, which
// alternate between even and odd (R[mu]).  ||X||_F beyond what EXP_MAX_SQUARINGS halvings bring under
// EXP_THETA is reported.
__global__ void __launch_bounds__(256) exp_scale_kernel(double* X, double* X2, double* X3, double c1, double c0, int n,
                                                        double* P, const double* part, double* even, double* odd,
                                                        double** R, int* sq, int* err) {
    __shared__ double red[32];
    const int mu = blockIdx.y;
    const size_t nn = (size_t)n * n;
    const double* p = part + (size_t)mu * EXP_PARTS;
    double v = block_sum(threadIdx.x < EXP_PART3 ? p[EXP_PARTX + threadIdx.x] : 0.0, red);
    int s = 0;                                     // v 2^-6s <= EXP_THETA^6
    while (v > 0x1p-18 && s < EXP_MAX_SQUARINGS) { v *= 0x1p-6; s++; }
    if (blockIdx.x == 0) {
        const double f = block_sum(threadIdx.x < EXP_PARTX ? p[threadIdx.x] : 0.0, red);
        if (threadIdx.x == 0) {
            const double most = EXP_THETA * (1 << EXP_MAX_SQUARINGS);
            if (f > most * most) atomicOr(err, SGS_DEV_EXPNORM);
            sq[mu] = s;
            R[mu] = ((s & 1) ? odd : even) + mu * nn;
        }
    }
    const double s1 = __hiloint2double((1023 - s) << 20, 0), s2 = __hiloint2double((1023 - 2 * s) << 20, 0),
                 s3 = __hiloint2double((1023 - 3 * s) << 20, 0);
    double *x = X + mu * nn, *x2 = X2 + mu * nn, *x3 = X3 + mu * nn, *o = P + mu * nn;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < nn; e += (size_t)gridDim.x * blockDim.x) {
        const int k = (int)(e / n), l = (int)(e % n);
        const double xs = x[e] * s1;
        o[e] = fma(c1, xs, k == l ? c0 : 0.0);
        if (s > 0) {
            x[e] = xs;
            x2[e] *= s2;
            x3[e] *= s3;
        }
    }
}

// health of an instance: out[0] = max |(Gamma^2)_kl + delta_kl| over the states (G2 holds
// Gamma^2), out[1] = number of non-finite entries of Gamma, out[2] = smallest / largest
// eigenvalue of G at the last amplitude solve (gram: the two, from gram_eig_kernel), out[3] =
// the energy of that solve
__global__ void __launch_bounds__(1024) health_kernel(const double* G2, const double* gamma, size_t count, int n,
                                                       const double* gram, const double* E, double* out) {
    __shared__ double red[32];
    double worst = 0.0, bad = 0.0;
    const size_t nn = (size_t)n * n;
    for (size_t e = threadIdx.x; e < count; e += blockDim.x) {
        const size_t w = e % nn;
        const double d = G2[e] + ((w / n) == (w % n) ? 1.0 : 0.0);
        worst = fmax(worst, fabs(d));
        if (!isfinite(gamma[e])) bad += 1.0;
        if (!isfinite(d)) worst = INFINITY;
    }
    // block max via a sum of per-warp maxima is not a max: reduce with shuffles, then shared memory
    for (int o = 16; o > 0; o >>= 1) worst = fmax(worst, __shfl_down_sync(0xffffffffu, worst, o));
    __shared__ double wmax[32];
    if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = worst;
    bad = block_sum(bad, red);
    if (threadIdx.x == 0) {
        double mx = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) mx = fmax(mx, wmax[w]);
        out[0] = mx;
        out[1] = bad;
        out[2] = gram[1] > 0.0 ? gram[0] / gram[1] : 0.0;
        out[3] = E[0];
    }
}

// out = x + a y (the Euler step of Eq. RKstep)
__global__ void axpy_kernel(const double* x, const double* y, double a, double* out, size_t count) {
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < count; e += (size_t)gridDim.x * blockDim.x)
        out[e] = x[e] + a * y[e];
}

__global__ void copy_kernel(const double* src, double* dst, size_t count) {
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < count; e += (size_t)gridDim.x * blockDim.x)
        dst[e] = src[e];
}

}  // namespace sgs
