// Renyi-2 entropy of the leading 2 N_A Majoranas (impurity + first l sites)
// of the SGS state (App. B).
//
// With the transition operator X_ab = |a><b| / <b|a>, whose two-point matrix is
// Delta^{a,b} (Sec. III B), rho_a rho_b = |G_ab|^2 X_ab, and the partial trace
// over B of an even Gaussian operator keeps the A block of its matrix.  The
// trace of two unit-trace Gaussian operators on A with matrices D1, D2 is
// 2^-N_A Pf([[D1, i 1], [-i 1, D2]]), so
//   T^{ab}_{cd} = lambda_a conj(lambda_b) lambda_c conj(lambda_d) G_ba G_dc 2^-N_A
//                 Pf([[Delta^{ab}_A, i 1], [-i 1, Delta^{cd}_A]]),
// which equals the paper's Eq. TrArho2_final term by term (checked against
// it and against Fock-space reduced density matrices) but needs no Pfaffian
// of the 4 N_B x 4 N_B matrix M_B: the pair pass already holds Delta.
// S_2 = -ln sum T (Eq. S2_SGS); T^{ab}_{cd} = T^{cd}_{ab}, so unordered pairs
// of ordered pairs (u <= v) are evaluated once.
#pragma once
#include "common.cuh"
#include "pair.cuh"
#include "pf_packed.cuh"

namespace sgs {

#define RENYI_MAX_DIM PACKED_PF_MAX     // 2 * 2 N_A <= 152 (impurity + up to 18 sites) in one CTA's shared memory

// blocks[u] = Delta^{ab}_A (complex, na2 x na2), w[u] = lambda_a conj(lambda_b) G_ba, u = a M + b
__global__ void renyi_blocks_kernel(InstDev d, const double* si, const double* imd, const double* Gm,
                                    const double* lam, const int* pair_index, int na2, double* blocks, double* w) {
    const int u = blockIdx.x;
    const int M = d.M, n = d.n;
    const int a = u / M, b = u % M;
    double* B = blocks + (size_t)u * na2 * na2 * 2;
    const double* g = d.gamma + (size_t)a * nn(d);
    int p = (a == b) ? -1 : pair_index[a * M + b];
    const double sgn = (a < b) ? 1.0 : -1.0;      // Delta^{ab} for a > b is conj(Delta^{ba})
    for (int e = threadIdx.x; e < na2 * na2; e += blockDim.x) {
        const int r = e / na2, c = e % na2;
        double re, im;
        if (p < 0) { re = g[(size_t)r * n + c]; im = 0.0; }
        else {
            re = -2.0 * si[(size_t)p * nn(d) + (size_t)r * n + c];
            im = sgn * imd[(size_t)p * nn(d) + (size_t)r * n + c];
        }
        B[2 * e] = re;
        B[2 * e + 1] = im;
    }
    if (threadIdx.x == 0) {
        cplx la = cmk(lam[2 * a], lam[2 * a + 1]), lb = cmk(lam[2 * b], lam[2 * b + 1]);
        cplx gba = cmk(Gm[2 * (b * M + a)], Gm[2 * (b * M + a) + 1]);
        cplx x = cmul(cmul(la, cconj(lb)), gba);
        w[2 * u] = x.x;
        w[2 * u + 1] = x.y;
    }
}

// One CTA per unordered pair (u <= v) of ordered pairs: the Pfaffian of Z = [[Delta_u, i 1], [-i 1, Delta_v]] in
// shared memory (pf_packed.cuh).  Entropies of 2, 7, 12 and 16 sites at 666 matrices each, with the energy they
// need: 16.4 ms with both triangles updated, the scaled row formed again for every element and a logarithm per
// step; now 5.4, of which the FP64 pipe's time for the eliminations is 3.3.
__global__ void __launch_bounds__(256) renyi_pf_kernel(const double* blocks, const double* w, long long npairs,
                                                       int na2, double log_norm, double* partial) {
    extern __shared__ double sm[];
    const int m = 2 * na2, NW = blockDim.x >> 5;
    const PackedPf pk(sm, m);
    __shared__ long long s_u, s_v;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long q0 = blockIdx.x + (long long)blockIdx.y * gridDim.x;
    if (q0 >= npairs) return;
    if (tid == 0) {             // decode q0 = v (v + 1) / 2 + u, u <= v
        long long v = (long long)((sqrt(8.0 * (double)q0 + 1.0) - 1.0) * 0.5);
        while ((v + 1) * (v + 2) / 2 <= q0) ++v;
        while (v * (v + 1) / 2 > q0) --v;
        s_v = v;
        s_u = q0 - v * (v + 1) / 2;
    }
    __syncthreads();
    const long long u = s_u, v = s_v;
    const double2* Bu = reinterpret_cast<const double2*>(blocks) + (size_t)u * na2 * na2;
    const double2* Bv = reinterpret_cast<const double2*>(blocks) + (size_t)v * na2 * na2;
    for (int i = warp; i < m - 1; i += NW)
        for (int j = i + 1 + lane; j < m; j += 32) {
            double2 z = make_double2(0.0, 0.0);
            if (j < na2) z = Bu[i * na2 + j];
            else if (i >= na2) z = Bv[(i - na2) * na2 + j - na2];
            else if (j == i + na2) z.y = 1.0;               // i 1
            pk.set(i, j, z.x, z.y);
        }
    __syncthreads();
    int e = 0;
    cplx x;
    const bool zero = packed_pfaffian(pk, x, e);
    if (tid == 0) {
        const cplx wu = cmk(w[2 * u], w[2 * u + 1]), wv = cmk(w[2 * v], w[2 * v + 1]);
        const double mag = exp(e * 0.693147180559945309417 + log_norm) * (u < v ? 2.0 : 1.0);
        x = cscale(cmul(cmul(wu, wv), x), mag);
        partial[2 * q0] = zero ? 0.0 : x.x;
        partial[2 * q0 + 1] = zero ? 0.0 : x.y;
    }
}

// Subsystems too large for one CTA's shared memory: the Pfaffians of a chunk of
// pairs go through the batched blocked Pfaffian of the pair pass.  Z_q =
// [[Delta_u, i 1], [-i 1, Delta_v]] in planes (re, im) of m x m, m = 2 na2; entries past
// the last pair get the pairing matrix J (Pf = 1) and are ignored.
__global__ void renyi_build_kernel(const double* blocks, long long q0, long long npairs, int na2, double* Y) {
    const long long q = q0 + blockIdx.x;
    const int m = 2 * na2;
    const size_t mm = (size_t)m * m;
    double* zr = Y + (size_t)blockIdx.x * 2 * mm;
    double* zi = zr + mm;
    if (q >= npairs) {
        for (size_t e = threadIdx.x; e < mm; e += blockDim.x) {
            const int r = (int)(e / m), c = (int)(e % m);
            zr[e] = (c == r + 1 && (r & 1) == 0) ? 1.0 : ((r == c + 1 && (c & 1) == 0) ? -1.0 : 0.0);
            zi[e] = 0.0;
        }
        return;
    }
    long long v = (long long)((sqrt(8.0 * (double)q + 1.0) - 1.0) * 0.5);
    while ((v + 1) * (v + 2) / 2 <= q) ++v;
    while (v * (v + 1) / 2 > q) --v;
    const long long u = q - v * (v + 1) / 2;
    const double* Bu = blocks + (size_t)u * na2 * na2 * 2;
    const double* Bv = blocks + (size_t)v * na2 * na2 * 2;
    for (size_t e = threadIdx.x; e < mm; e += blockDim.x) {
        const int r = (int)(e / m), c = (int)(e % m);
        double xr = 0.0, xi = 0.0;
        if (r < na2 && c < na2) { xr = Bu[2 * (r * na2 + c)]; xi = Bu[2 * (r * na2 + c) + 1]; }
        else if (r >= na2 && c >= na2) { xr = Bv[2 * ((r - na2) * na2 + c - na2)]; xi = Bv[2 * ((r - na2) * na2 + c - na2) + 1]; }
        else if (c == r + na2) xi = 1.0;
        else if (r == c + na2) xi = -1.0;
        zr[e] = xr;
        zi[e] = xi;
    }
}

// T of each pair of the chunk from the Pfaffian (phase, log|Pf|)
__global__ void renyi_combine_kernel(const double* logabs, const double* phase, const double* w, long long q0,
                                     long long cnt, long long npairs, double log_norm, double* partial) {
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < cnt; j += (long long)gridDim.x * blockDim.x) {
        const long long q = q0 + j;
        if (q >= npairs) continue;
        long long v = (long long)((sqrt(8.0 * (double)q + 1.0) - 1.0) * 0.5);
        while ((v + 1) * (v + 2) / 2 <= q) ++v;
        while (v * (v + 1) / 2 > q) --v;
        const long long u = q - v * (v + 1) / 2;
        double tr = 0.0, ti = 0.0;
        const double la = logabs[j];
        if (la > -1e300) {
            const cplx x = cmul(cmul(cmk(w[2 * u], w[2 * u + 1]), cmk(w[2 * v], w[2 * v + 1])),
                                cmk(phase[2 * j], phase[2 * j + 1]));
            const double mag = exp(la + log_norm) * (u < v ? 2.0 : 1.0);
            tr = x.x * mag;
            ti = x.y * mag;
        }
        partial[2 * q] = tr;
        partial[2 * q + 1] = ti;
    }
}

// deterministic sum of count complex values: block partial sums, then one block
__global__ void complex_sum_kernel(const double* in, long long count, double* out) {
    __shared__ double red[32];
    double sr = 0.0, si = 0.0;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < count; e += (long long)gridDim.x * blockDim.x) {
        sr += in[2 * e];
        si += in[2 * e + 1];
    }
    sr = block_sum(sr, red);
    si = block_sum(si, red);
    if (threadIdx.x == 0) { out[2 * blockIdx.x] = sr; out[2 * blockIdx.x + 1] = si; }
}

}  // namespace sgs
