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
#include "factor.cuh"
#include "pair.cuh"

namespace sgs {

#define RENYI_MAX_DIM 152     // 2 * 2 N_A <= 152 (impurity + up to 18 sites) in one CTA's shared memory

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

// dynamic shared memory of renyi_pf_kernel: the packed upper triangles (re, im), four vectors, and the packed
// entries' row and column
inline size_t renyi_smem(int m) {
    return (size_t)m * (m - 1) / 2 * (2 * sizeof(double) + 2) + 4 * (size_t)m * sizeof(double) + 16;
}

// One CTA per unordered pair (u <= v) of ordered pairs: complex Parlett-Reid elimination of
// Z = [[Delta_u, i 1], [-i 1, Delta_v]] in shared memory.  Z is antisymmetric: only its upper triangle is kept,
// packed by rows, so that what is live after a step is the tail of the storage and every lane of the rank-2
// update has an element (their rows and columns from a table).  The step's rows k and q = k + 1 are done after
// it, so the interchange of q and the pivot p only writes row and column p.
// Bound by the FP64 pipe: 8 FMAs per live element and step, m^3 / 12 elements in all.  2080 matrices' worth of
// the earlier form (both triangles, the scaled row formed again for every element, a logarithm per step) took
// 8.0 ms for m = 24, 64 and 104 at 666 matrices each.
__global__ void __launch_bounds__(256) renyi_pf_kernel(const double* blocks, const double* w, long long npairs,
                                                       int na2, double log_norm, double* partial) {
    extern __shared__ double sm[];
    const int m = 2 * na2, T = m * (m - 1) / 2, NT = blockDim.x, NW = NT >> 5;
    double* Zr = sm;                            // row i, column j > i at off(i) + j
    double* Zi = Zr + T;
    double* tr = Zi + T;                        // tau and u of the step
    double* ti = tr + m;
    double* ur = ti + m;
    double* ui = ur + m;
    uchar2* ij = reinterpret_cast<uchar2*>(ui + m);
    __shared__ long long red_v[8];
    __shared__ int red_i[8];
    __shared__ double s_inv[2], s_pr[RENYI_MAX_DIM / 2], s_pi[RENYI_MAX_DIM / 2];
    __shared__ long long s_u, s_v;
    __shared__ int s_flip;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    auto off = [m](int i) { return i * (2 * m - i - 1) / 2 - i - 1; };
    const long long q0 = blockIdx.x + (long long)blockIdx.y * gridDim.x;
    if (q0 >= npairs) return;
    if (tid == 0) {             // decode q0 = v (v + 1) / 2 + u, u <= v
        long long v = (long long)((sqrt(8.0 * (double)q0 + 1.0) - 1.0) * 0.5);
        while ((v + 1) * (v + 2) / 2 <= q0) ++v;
        while (v * (v + 1) / 2 > q0) --v;
        s_v = v;
        s_u = q0 - v * (v + 1) / 2;
        s_flip = 0;
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
            const int e = off(i) + j;
            Zr[e] = z.x;
            Zi[e] = z.y;
            ij[e] = make_uchar2((unsigned char)i, (unsigned char)j);
        }
    __syncthreads();
    bool zero = false;
    for (int k = 0; k < m - 1; k += 2) {
        const int q = k + 1, ok = off(k), oq = off(q);
        // the pivot: the largest entry of row k, the smaller column on a tie
        long long key = -1;
        int p = 0x7fffffff;
        for (int i = q + tid; i < m; i += NT) {
            const double x = Zr[ok + i], y = Zi[ok + i];
            const long long m2 = abs_key(fma(x, x, y * y));
            if (m2 > key) { key = m2; p = i; }
        }
        warp_argmax(key, p);
        if (lane == 0) { red_v[warp] = key; red_i[warp] = p; }
        __syncthreads();
        key = lane < NW ? red_v[lane] : -1ll;
        p = lane < NW ? red_i[lane] : 0x7fffffff;
        warp_argmax(key, p);
        if (!(key > 0 && key <= 0x7FF0000000000000ll)) { zero = true; break; }     // zero (or NaN)
        const int op = off(p);
        if (tid == NT - 1) {
            const double pr = Zr[ok + p], pi = Zi[ok + p];
            const double rm = 1.0 / fma(pr, pr, pi * pi);
            s_inv[0] = pr * rm;
            s_inv[1] = -pi * rm;
            s_pr[k >> 1] = pr;
            s_pi[k >> 1] = pi;
            if (p != q) s_flip ^= 1;
        }
        // u_i = -Z'[q][i] with the interchange of q and p: Z'[q][i] = Z[p][i] (i > p), -Z[i][p] (q < i < p),
        // -Z[q][p] (i = p); Z'[p][i] = Z[q][i], Z'[i][p] = -Z[q][i]
        for (int i = q + 1 + tid; i < m; i += NT) {
            const double zr = Zr[oq + i], zi = Zi[oq + i];
            if (i == p) {
                ur[i] = zr;
                ui[i] = zi;
            } else {
                const int e = i > p ? op + i : off(i) + p;
                const double yr = p == q ? zr : Zr[e], yi = p == q ? zi : Zi[e];
                ur[i] = i > p ? -yr : yr;
                ui[i] = i > p ? -yi : yi;
                if (p != q) {
                    Zr[e] = i > p ? zr : -zr;
                    Zi[e] = i > p ? zi : -zi;
                }
            }
        }
        __syncthreads();
        for (int i = q + 1 + tid; i < m; i += NT) {         // tau_i = Z'[k][i] / pivot
            const int e = ok + (i == p ? q : i);
            const double xr = Zr[e], xi = Zi[e], ir = s_inv[0], ii = s_inv[1];
            tr[i] = xr * ir - xi * ii;
            ti[i] = xr * ii + xi * ir;
        }
        __syncthreads();
        // Z[i][j] += tau_i u_j - u_i tau_j on the live triangle, rows k + 2 on
        for (int e = off(k + 2) + k + 3 + tid; e < T; e += NT) {
            const uchar2 x = ij[e];
            const double ar = tr[x.x], ai = ti[x.x], br = ur[x.x], bi = ui[x.x];
            const double cr = tr[x.y], ci = ti[x.y], dr = ur[x.y], di = ui[x.y];
            double r = Zr[e], s = Zi[e];
            r = fma(ar, dr, r);
            s = fma(ar, di, s);
            r = fma(-ai, di, r);
            s = fma(ai, dr, s);
            r = fma(-br, cr, r);
            s = fma(-br, ci, s);
            r = fma(bi, ci, r);
            s = fma(-bi, cr, s);
            Zr[e] = r;
            Zi[e] = s;
        }
        __syncthreads();
    }
    // the pivots' product as mantissa and exponent of two, by one warp
    if (warp == 0) {
        int e = 0;
        cplx x = cmk(1.0, 0.0);
        for (int t = lane; t < m / 2 && !zero; t += 32) {
            x = cmul(x, cmk(s_pr[t], s_pi[t]));
            const int f = min(max(2046 - max(expo_field(x.x), expo_field(x.y)), 1), 2046);
            x = cscale(x, __hiloint2double(f << 20, 0));    // 2^(f - 1023)
            e += 1023 - f;
        }
        for (int o = 16; o > 0; o >>= 1) {
            x = cmul(x, cmk(__shfl_xor_sync(0xffffffffu, x.x, o), __shfl_xor_sync(0xffffffffu, x.y, o)));
            e += __shfl_xor_sync(0xffffffffu, e, o);
        }
        if (lane == 0) {
            if (zero) x = cmk(0.0, 0.0);
            const cplx wu = cmk(w[2 * u], w[2 * u + 1]), wv = cmk(w[2 * v], w[2 * v + 1]);
            const double mag = exp(e * 0.693147180559945309417 + log_norm) * (u < v ? 2.0 : 1.0);
            x = cscale(cmul(cmul(wu, wv), x), s_flip ? -mag : mag);
            partial[2 * q0] = zero ? 0.0 : x.x;
            partial[2 * q0 + 1] = zero ? 0.0 : x.y;
        }
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
