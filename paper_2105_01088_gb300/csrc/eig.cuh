// Optimal amplitudes: lowest solution of h lambda = E G lambda (Eq. eigLambda)
// by canonical orthogonalisation, in FP64, one CTA per instance.
//
// Canonical orthogonalisation drops the eigenvalues of G below cut * max (the paper
// assumes linearly independent states).  Where none can be dropped, any X with
// X^dag G X = 1 serves, and the solve takes the direct route (amp_direct): G = U D U^dag
// with U^{-1} formed alongside, H' = D^{-1/2} U^{-1} h U^{-dag} D^{-1/2}, Householder
// reduction of H' to a real tridiagonal T, the lowest eigenvalue of T by multisection
// (32 shifts at a time, each tested for positive definiteness of T - x), its vector by
// inverse iteration, and back.  All of it sits in shared memory.  "None can be dropped" is
// decided by bounds: lambda_min >= 1 / tr(G^{-1}) and lambda_max <= tr(G), both traces at
// hand after the factorisation, so tr(G) tr(G^{-1}) < AMP_COND (1e8, four orders inside
// the cut of 1e-12) suffices.  The route is for states with order-one amplitudes: its errors are
// normwise, u |lambda|, while c_mu divides by lambda_mu, and on a G that is diagonal to rounding
// (random states: overlaps down to 1e-40) Jacobi leaves exact zeros, which freeze a state.  So
// overlaps all below AMP_SMALL, or an amplitude below AMP_SMALL times the largest, go to Jacobi.
//
// Otherwise (nearly dependent states, NaN) the solve takes amp_jacobi: the M x M Hermitian
// pair (G, h) is embedded as the real symmetric 2M x 2M pair [[Re, -Im], [Im, Re]] (every
// eigenvalue doubled; the eigenvector [x; y] maps to x + i y), and both symmetric
// eigenproblems are solved with parallel cyclic Jacobi (round-robin pairing, disjoint
// rotations applied to all rows and then all columns) on global scratch.
//
// What bounds it: one SM's FP64 pipe (two FMAs per clock, so a warp instruction every 16
// clocks) and the latency of M dependent steps.  Jacobi for both eigenproblems does about
// 8 sweeps x 2M rounds over (2M)^2 elements each; the direct route does each of its O(M^3)
// parts once, with work spread so that no FP64 instruction is repeated by several warps.
// Measured with overlapping states: a step at 2N = 244, M = 16 went from 11.7 to 7.9 ms and at
// 2N = 512, M = 32 from 104 to about 82 ms (Jacobi: 3.8 and 25 ms of them).
//
// The same kernel then forms lambda-tilde = G lambda, the decoupling
// constants c_mu (Sec. III A) and the per-(mu, beta) coefficients of
// Eq. (EOM-Gamma3): with z = conj(lt_mu) c_mu lambda_beta,
//   a1 = 2i z G_mu,beta,  a2 = 2 z G_mu,beta,  a3 = -z (h_mu,beta - E G_mu,beta).
#pragma once
#include "common.cuh"

namespace sgs {

struct AmpArgs {
    int M;
    const double* Gm;     // [M][M] complex
    const double* hm;     // [M][M] complex
    double* scratch;      // >= 6 (2M)^2 + 8 (2M) doubles
    double* E;            // [1] energy of this step
    double* lam;          // [M] complex
    double* lt;           // [M] complex
    double* coef;         // [M][M][6]
    int cmode;            // 0: c = 1/(lambda conj(lt)); 1: c = lt conj(lambda)/|lambda lt|
    double cut;
    int* err;
};

// Jacobi on the m x m symmetric A (row stride ld), accumulating V (= I on
// entry).  Returns the number of sweeps used (or -1 if not converged).
__device__ int jacobi_sym(double* A, double* V, int m, int ld, double* rc, double* rs, int* rp, int* rq,
                          double* red) {
    const int mm = (m + 1) & ~1;            // pad to even with one idle index
    const int npair = mm / 2;
    int sweeps = 0;
    for (; sweeps < 60; sweeps++) {
        double off = 0.0, dg = 0.0;
        for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
            int i = e / m, j = e % m;
            double v = A[i * ld + j];
            if (i == j) dg += v * v; else off += v * v;
        }
        off = block_sum(off, red);
        dg = block_sum(dg, red);
        if (off <= 1e-30 * dg || off < 1e-280) return sweeps;
        for (int r = 0; r < mm - 1; r++) {
            for (int i = threadIdx.x; i < npair; i += blockDim.x) {
                auto pos = [&](int j) { return j == 0 ? 0 : ((j - 1 + r) % (mm - 1)) + 1; };
                int p = pos(i), q = pos(mm - 1 - i);
                if (p > q) { int t = p; p = q; q = t; }
                double c = 1.0, s = 0.0;
                if (q < m) {
                    double apq = A[p * ld + q];
                    if (fabs(apq) > 1e-300) {
                        double th = (A[q * ld + q] - A[p * ld + p]) / (2.0 * apq);
                        double t = (th >= 0.0 ? 1.0 : -1.0) / (fabs(th) + sqrt(th * th + 1.0));
                        c = 1.0 / sqrt(t * t + 1.0);
                        s = t * c;
                    }
                } else {
                    q = -1;
                }
                rc[i] = c; rs[i] = s; rp[i] = p; rq[i] = q;
            }
            __syncthreads();
            for (int e = threadIdx.x; e < npair * m; e += blockDim.x) {
                int i = e / m, j = e % m;
                int p = rp[i], q = rq[i];
                if (q < 0 || rs[i] == 0.0) continue;
                double c = rc[i], s = rs[i];
                double ap = A[p * ld + j], aq = A[q * ld + j];
                A[p * ld + j] = c * ap - s * aq;
                A[q * ld + j] = s * ap + c * aq;
            }
            __syncthreads();
            for (int e = threadIdx.x; e < npair * m; e += blockDim.x) {
                int i = e / m, j = e % m;
                int p = rp[i], q = rq[i];
                if (q < 0 || rs[i] == 0.0) continue;
                double c = rc[i], s = rs[i];
                double ap = A[j * ld + p], aq = A[j * ld + q];
                A[j * ld + p] = c * ap - s * aq;
                A[j * ld + q] = s * ap + c * aq;
                double vp = V[j * ld + p], vq = V[j * ld + q];
                V[j * ld + p] = c * vp - s * vq;
                V[j * ld + q] = s * vp + c * vq;
            }
            __syncthreads();
            for (int i = threadIdx.x; i < npair; i += blockDim.x) {
                int p = rp[i], q = rq[i];
                if (q >= 0 && rs[i] != 0.0) { A[p * ld + q] = 0.0; A[q * ld + p] = 0.0; }
            }
            __syncthreads();
        }
    }
    return -1;
}

// the real embedding [[Re, -Im], [Im, Re]] of the M x M complex X
__device__ __forceinline__ void amp_embed(const double* X, double* R, int M) {
    const int m = 2 * M;
    for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
        const int i = e / m, j = e % m, ib = i / M, jb = j / M, x = 2 * ((i % M) * M + j % M);
        R[e] = ib == jb ? X[x] : (ib == 0 ? -X[x + 1] : X[x + 1]);
    }
}

#define AMP_THREADS 256
#define AMP_COND 1e8
#define AMP_SMALL 1e-6

// lr (2M: real and imaginary parts of a solution lambda) and E from two Jacobi eigenproblems on
// the real embedding; false if nothing is kept of G.  scratch: 6 (2M)^2 + 8 (2M) doubles (global);
// its first (2M)^2 hold the diagonalised embedding of G afterwards
__device__ __noinline__ bool amp_jacobi(const AmpArgs& a, double* lr, double& E) {
    __shared__ double rc[SGS_MAX_RANK + 1], rs[SGS_MAX_RANK + 1];
    __shared__ int rp[SGS_MAX_RANK + 1], rq[SGS_MAX_RANK + 1];
    __shared__ double red[32];
    __shared__ int s_keep[2 * SGS_MAX_RANK];
    __shared__ int s_nkeep, s_jmin;

    const int M = a.M, m = 2 * M, ld = m;
    double* GR = a.scratch;
    double* V1 = GR + m * m;
    double* HR = V1 + m * m;
    double* XR = HR + m * m;
    double* TM = XR + m * m;
    double* V2 = TM + m * m;

    amp_embed(a.Gm, GR, M);
    amp_embed(a.hm, HR, M);
    for (int e = threadIdx.x; e < m * m; e += blockDim.x) V1[e] = (e / m == e % m) ? 1.0 : 0.0;
    __syncthreads();
    int sw = jacobi_sym(GR, V1, m, ld, rc, rs, rp, rq, red);
    if (threadIdx.x == 0) {
        if (sw < 0) atomicOr(a.err, SGS_DEV_EIG);
        double wmax = 0.0;
        for (int j = 0; j < m; j++) wmax = fmax(wmax, GR[j * ld + j]);
        int nk = 0;
        for (int j = 0; j < m; j++)
            if (GR[j * ld + j] > a.cut * wmax) s_keep[nk++] = j;
        s_nkeep = nk;
        if (nk == 0) atomicOr(a.err, SGS_DEV_EIG);
    }
    __syncthreads();
    const int K = s_nkeep;
    if (K == 0) return false;
    // XR = V1[:, keep] / sqrt(w)
    for (int e = threadIdx.x; e < m * K; e += blockDim.x) {
        int i = e / K, t = e % K;
        int j = s_keep[t];
        XR[i * ld + t] = V1[i * ld + j] / sqrt(GR[j * ld + j]);
    }
    __syncthreads();
    // TM = HR XR (m x K), then H' = XR^T TM (K x K) into V1's storage
    for (int e = threadIdx.x; e < m * K; e += blockDim.x) {
        int i = e / K, t = e % K;
        double v = 0.0;
        for (int j = 0; j < m; j++) v += HR[i * ld + j] * XR[j * ld + t];
        TM[i * ld + t] = v;
    }
    __syncthreads();
    double* Hp = V1;
    for (int e = threadIdx.x; e < K * K; e += blockDim.x) {
        int s = e / K, t = e % K;
        double v = 0.0;
        for (int i = 0; i < m; i++) v += XR[i * ld + s] * TM[i * ld + t];
        Hp[s * ld + t] = v;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < K * K; e += blockDim.x) {
        int s = e / K, t = e % K;
        if (s < t) {
            double v = 0.5 * (Hp[s * ld + t] + Hp[t * ld + s]);
            Hp[s * ld + t] = v;
            Hp[t * ld + s] = v;
        }
        V2[s * ld + t] = (s == t) ? 1.0 : 0.0;
    }
    __syncthreads();
    sw = jacobi_sym(Hp, V2, K, ld, rc, rs, rp, rq, red);
    if (threadIdx.x == 0) {
        if (sw < 0) atomicOr(a.err, SGS_DEV_EIG);
        int jm = 0;
        for (int j = 1; j < K; j++)
            if (Hp[j * ld + j] < Hp[jm * ld + jm]) jm = j;
        s_jmin = jm;
    }
    __syncthreads();
    E = Hp[s_jmin * ld + s_jmin];
    // lambda_R = XR u
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        double v = 0.0;
        for (int t = 0; t < K; t++) v += XR[i * ld + t] * V2[t * ld + s_jmin];
        lr[i] = v;
    }
    __syncthreads();
    return true;
}

// (a, b) += (x, y) (u, v) and (a, b) -= (x, y) (u, v), complex
__device__ __forceinline__ void cfma(cplx& a, cplx x, cplx u) {
    a.x = fma(x.x, u.x, a.x);
    a.x = fma(-x.y, u.y, a.x);
    a.y = fma(x.x, u.y, a.y);
    a.y = fma(x.y, u.x, a.y);
}

__device__ __forceinline__ double warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// T - x positive definite (T real symmetric tridiagonal: diagonal d, off-diagonal e with squares
// e2): every leading principal minor positive, by the minors' three-term recurrence; the pair of
// minors is rescaled by a power of two every four rows, so it neither over- nor underflows for T of magnitude
// 2^-150 .. 2^150 (the caller scales others)
__device__ __forceinline__ bool amp_posdef(const double* d, const double* e2, int M, double x) {
    double p0 = 1.0, p1 = d[0] - x;
    bool ok = p1 > 0.0;
    for (int i = 1; i < M; i++) {
        const double p2 = fma(d[i] - x, p1, -e2[i - 1] * p0);
        p0 = p1;
        p1 = p2;
        ok = ok && p1 > 0.0;
        if ((i & 3) == 0) {
            const int ex = max((__double2hiint(p0) >> 20) & 0x7ff, (__double2hiint(p1) >> 20) & 0x7ff);
            const int f = min(max(2046 - ex, 1), 2046);          // 2^(1023 - ex)
            const double sc = __hiloint2double(f << 20, 0);
            p0 *= sc;
            p1 *= sc;
        }
    }
    return ok;
}

// a Hermitian matrix reduced to a real symmetric tridiagonal T (diagonal d, off-diagonal e with squares e2)
struct AmpTri {
    double d[SGS_MAX_RANK], e[SGS_MAX_RANK], e2[SGS_MAX_RANK];
    cplx v[SGS_MAX_RANK], w[SGS_MAX_RANK], tau[SGS_MAX_RANK], part[AMP_THREADS / 32][SGS_MAX_RANK];
};

// The reduction of B (M x M, row stride ld, overwritten) by the whole block; the reflectors' vectors into the columns
// of V (may be nullptr)
__device__ __forceinline__ void amp_reduce(cplx* V, cplx* B, int M, int ld, AmpTri& t) {
    constexpr int NW = AMP_THREADS / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // Householder reduction: reflector k = 1 - tau v v^dag (v_{k+1} = 1) makes column k (beta, 0, ..)
    // with real beta; A <- A - v w^dag - w v^dag, w = p - (tau/2) (p^dag v) v, p = tau A v
    for (int k = 0; k + 1 < M; k++) {
        if (warp == 0) {
            double xn = 0.0;
            for (int i = k + 2 + lane; i < M; i += 32) xn += cabs2(B[i * ld + k]);
            xn = warp_sum(xn);
            const cplx al = B[(k + 1) * ld + k];
            cplx tau = cmk(0.0, 0.0), sc = cmk(0.0, 0.0);
            double beta = al.x;
            if (xn > 0.0 || al.y != 0.0) {
                beta = sqrt(cabs2(al) + xn);
                if (al.x >= 0.0) beta = -beta;
                const double rb = 1.0 / beta;
                tau = cmk((beta - al.x) * rb, -al.y * rb);
                const cplx q = cmk(al.x - beta, al.y);
                sc = cscale(cconj(q), 1.0 / cabs2(q));
            }
            for (int i = k + 1 + lane; i < M; i += 32) {
                const cplx v = i == k + 1 ? cmk(1.0, 0.0) : cmul(B[i * ld + k], sc);
                t.v[i] = v;
                if (V) V[i * ld + k] = v;       // kept for the back transformation
            }
            if (lane == 0) { t.tau[k] = tau; t.e[k] = beta; t.e2[k] = beta * beta; }
        }
        __syncthreads();
        // A v: lanes over rows, the columns shared out among the warps
        for (int i = k + 1 + lane; i < M; i += 32) {
            cplx p = cmk(0.0, 0.0);
            for (int j = k + 1 + warp; j < M; j += NW) cfma(p, B[i * ld + j], t.v[j]);
            t.part[warp][i] = p;
        }
        __syncthreads();
        if (warp == 0) {
            const cplx tau = t.tau[k];
            double dr = 0.0, di = 0.0;
            for (int i = k + 1 + lane; i < M; i += 32) {
                cplx p = t.part[0][i];
                for (int w = 1; w < NW; w++) p = cadd(p, t.part[w][i]);
                p = cmul(tau, p);
                t.w[i] = p;
                const cplx x = cmul(cconj(p), t.v[i]);
                dr += x.x;
                di += x.y;
            }
            const cplx f = cscale(cmul(tau, cmk(warp_sum(dr), warp_sum(di))), -0.5);
            for (int i = k + 1 + lane; i < M; i += 32) {
                cplx w = t.w[i];
                cfma(w, f, t.v[i]);
                t.w[i] = w;
            }
        }
        __syncthreads();
        for (int i = k + 1 + warp; i < M; i += NW) {
            const cplx vi = cscale(t.v[i], -1.0), wi = cscale(t.w[i], -1.0);
            for (int j = k + 1 + lane; j <= i; j += 32) {
                cplx x = B[i * ld + j];
                cfma(x, vi, cconj(t.w[j]));
                cfma(x, wi, cconj(t.v[j]));
                if (i == j) x.y = 0.0;
                B[i * ld + j] = x;
                B[j * ld + i] = cconj(x);
            }
        }
        __syncthreads();
    }
    for (int i = tid; i < M; i += AMP_THREADS) t.d[i] = B[i * ld + i].x;
    __syncthreads();
}

// The lowest eigenvalue of T between lo and hi, by one warp: T is scaled to order one first where its magnitude is
// extreme (by 2^(f - 1023), f returned); top bounds |T|, nan: T is not finite
__device__ __forceinline__ int amp_lowest(AmpTri& t, int M, double& lo, double& hi, double& top, bool& nan) {
    const int lane = threadIdx.x & 31;
    // T of extreme magnitude (energies in units far from its own): to order one by a power of two, exact
    int ex = 0;
    for (int i = lane; i < M; i += 32) {
        ex = max(ex, (__double2hiint(t.d[i]) >> 20) & 0x7ff);
        if (i + 1 < M) ex = max(ex, (__double2hiint(t.e[i]) >> 20) & 0x7ff);
    }
    ex = __reduce_max_sync(0xffffffffu, ex);
    const int f = ex > 0 && (ex < 1023 - 150 || ex > 1023 + 150) ? min(max(2046 - ex, 1), 2045) : 1023;
    if (f != 1023) {
        const double sc = __hiloint2double(f << 20, 0);
        for (int i = lane; i < M; i += 32) {
            t.d[i] *= sc;
            if (i + 1 < M) {
                t.e[i] *= sc;
                t.e2[i] = t.e[i] * t.e[i];
            }
        }
        __syncwarp();
    }
    // lo, hi bracket the lowest eigenvalue: Gershgorin below, the smallest diagonal entry above
    lo = hi = INFINITY;
    top = 0.0;
    nan = false;
    for (int i = lane; i < M; i += 32) {
        const double r = (i > 0 ? fabs(t.e[i - 1]) : 0.0) + (i + 1 < M ? fabs(t.e[i]) : 0.0);
        lo = fmin(lo, t.d[i] - r);
        hi = fmin(hi, t.d[i]);
        top = fmax(top, fabs(t.d[i]) + r);
        nan = nan || !isfinite(t.d[i] + r);
    }
    nan = __any_sync(0xffffffffu, nan);                  // (fmin and fmax drop a NaN)
    for (int o = 16; o > 0; o >>= 1) {
        lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmin(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        top = fmax(top, __shfl_xor_sync(0xffffffffu, top, o));
    }
    const double ulp = 2.220446049250313e-16;
    lo -= 4.0 * ulp * top;
    for (int it = 0; it < 14 && hi - lo > ulp * fmax(fabs(lo), fabs(hi)); it++) {
        const double x = fma(hi - lo, (lane + 1) * (1.0 / 33.0), lo);
        const unsigned pd = __ballot_sync(0xffffffffu, amp_posdef(t.d, t.e2, M, x));
        const int n = __ffs(~pd) - 1;                    // shifts 0 .. n - 1 lie below (n = -1: all)
        const double below = __shfl_sync(0xffffffffu, x, n > 0 ? n - 1 : (n < 0 ? 31 : 0));
        const double above = __shfl_sync(0xffffffffu, x, n < 0 ? 31 : n);
        if (n != 0) lo = below;
        if (n >= 0) hi = above;
    }
    return f;
}

// The direct route: lr and E as amp_jacobi gives them, up to lambda's scale and phase.  Returns false
// (nothing decided) where a pivot is not positive, tr(G) tr(G^{-1}) >= AMP_COND, or overlaps or amplitudes
// are small (AMP_SMALL).  M <= SGS_MAX_RANK;
// sm: 3 M (M + 1) complex.  Threads: AMP_THREADS, warp w taking rows w, w + 8, ...; odd row strides keep
// both row and column walks free of bank conflicts.
__device__ __noinline__ bool amp_direct(const AmpArgs& a, cplx* sm, double* lr, double& E) {
    constexpr int NW = AMP_THREADS / 32, MR = SGS_MAX_RANK;
    __shared__ AmpTri t;
    __shared__ double s_rcp[MR], red[32], s_E;
    __shared__ int s_bad;
    const int M = a.M, ld = M + 1, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    cplx* A = sm;                   // G, then U^{-1} h
    cplx* W = A + M * ld;           // U^{-1} (unit lower triangular)
    cplx* B = W + M * ld;           // h, then H', then T and the reflectors
    double trg = 0.0;
    // |G_ij| >= AMP_SMALL somewhere off the diagonal, on the high words (an FP64 compare costs a warp 64 clocks)
    const int least = __double2hiint(AMP_SMALL);
    int overlap = M == 1;
    for (int i = warp; i < M; i += NW)
        for (int j = lane; j < M; j += 32) {
            const int e = 2 * (i * M + j);
            if (i != j && (int)(max(__double2hiint(a.Gm[e]) & 0x7fffffff, __double2hiint(a.Gm[e + 1]) & 0x7fffffff)) >= least)
                overlap = 1;
            A[i * ld + j] = cmk(a.Gm[e], a.Gm[e + 1]);
            B[i * ld + j] = cmk(a.hm[e], a.hm[e + 1]);
            W[i * ld + j] = cmk(i == j ? 1.0 : 0.0, 0.0);
            if (i == j) trg += a.Gm[e];
        }
    if (tid == 0) {
        const double d = a.Gm[0];
        s_bad = !(d > 0.0);
        t.d[0] = d;
        s_rcp[0] = 1.0 / d;
    }
    if (!__syncthreads_or(overlap)) return false;
    trg = block_sum(trg, red);
    // step k: rows i > k lose l times row k, l = A_ik / d_k: the trailing lower triangle of G and
    // the columns j <= k of U^{-1}.  Column and row k are not written in step k; the thread that
    // completes the next pivot also forms its reciprocal, so one barrier per step is enough.
    for (int k = 0; k + 1 < M; k++) {
        const double rk = s_rcp[k];
        for (int i = k + 1 + warp; i < M; i += NW) {
            const cplx l = cscale(A[i * ld + k], -rk);
            for (int j = lane; j <= i; j += 32) {
                if (j <= k) {
                    cplx x = W[i * ld + j];
                    cfma(x, l, W[k * ld + j]);
                    W[i * ld + j] = x;
                } else {
                    cplx x = A[i * ld + j];
                    cfma(x, l, cconj(A[j * ld + k]));
                    A[i * ld + j] = x;
                    if (i == k + 1) {
                        if (!(x.x > 0.0)) s_bad = 1;
                        t.d[i] = x.x;
                        s_rcp[i] = 1.0 / x.x;
                    }
                }
            }
        }
        __syncthreads();
    }
    double tri = 0.0;               // tr(G^{-1}) = sum_ij |U^{-1}_ij|^2 / d_i
    for (int i = warp; i < M; i += NW)
        for (int j = lane; j <= i; j += 32) tri += cabs2(W[i * ld + j]) * s_rcp[i];
    tri = block_sum(tri, red);
    if (s_bad || !(trg * tri < AMP_COND)) return false;
    if (tid < M) s_rcp[tid] = 1.0 / sqrt(t.d[tid]);          // D^{-1/2}
    // A <- U^{-1} h, then H' = D^{-1/2} A U^{-dag} D^{-1/2} (lower part, mirrored) into B
    for (int i = warp; i < M; i += NW)
        for (int j = lane; j < M; j += 32) {
            cplx x = cmk(0.0, 0.0);
            for (int k = 0; k <= i; k++) cfma(x, W[i * ld + k], B[k * ld + j]);
            A[i * ld + j] = x;
        }
    __syncthreads();
    for (int i = warp; i < M; i += NW)
        for (int j = lane; j <= i; j += 32) {
            cplx x = cmk(0.0, 0.0);
            for (int k = 0; k <= j; k++) cfma(x, A[i * ld + k], cconj(W[j * ld + k]));
            x = cscale(x, s_rcp[i] * s_rcp[j]);
            if (i == j) x.y = 0.0;
            B[i * ld + j] = x;
            B[j * ld + i] = cconj(x);
        }
    __syncthreads();
    amp_reduce(A, B, M, ld, t);
    if (warp == 0) {
        double lo, hi, top;
        bool nan;
        const int f = amp_lowest(t, M, lo, hi, top, nan);
        const double ulp = 2.220446049250313e-16;
        // inverse iteration at a shift just below the eigenvalue, where T - x is positive definite and
        // its factorisation needs no pivoting; each pass cuts the other components by about
        // 16 ulp top / gap
        if (lane == 0) {
            s_E = nan ? __longlong_as_double(0x7ff8000000000000ll) : 0.5 * (lo + hi) * __hiloint2double((2046 - f) << 20, 0);
            const double x = lo - 16.0 * ulp * top, least = ulp * top + 1e-300;
            double* q = reinterpret_cast<double*>(t.part);             // 1 / pivots
            double* l = q + MR;                                        // multipliers
            double* z = l + MR;
            double r = 1.0 / fmax(t.d[0] - x, least);
            q[0] = r;
            for (int i = 1; i < M; i++) {
                l[i] = t.e[i - 1] * r;
                r = 1.0 / fmax(fma(-t.e[i - 1], l[i], t.d[i] - x), least);
                q[i] = r;
            }
            for (int i = 0; i < M; i++) z[i] = 1.0 + 0.125 * (i % 5);
            for (int it = 0; it < 3; it++) {
                for (int i = 1; i < M; i++) z[i] = fma(-l[i], z[i - 1], z[i]);
                z[M - 1] *= q[M - 1];
                double big = fabs(z[M - 1]);
                for (int i = M - 2; i >= 0; i--) {
                    z[i] = fma(-l[i + 1], z[i + 1], z[i] * q[i]);
                    big = fmax(big, fabs(z[i]));
                }
                const int ex = (__double2hiint(big) >> 20) & 0x7ff;    // to order one by a power of two
                const double sc = __hiloint2double(min(max(2046 - ex, 1), 2046) << 20, 0);
                for (int i = 0; i < M; i++) z[i] *= sc;
            }
        }
        __syncwarp();
        // y = H_0 H_1 ... H_{M-2} z, then D^{-1/2} y
        const double* z = reinterpret_cast<double*>(t.part) + 2 * MR;
        cplx y[2];
        for (int u = 0; u < 2; u++) y[u] = cmk(lane + 32 * u < M ? z[lane + 32 * u] : 0.0, 0.0);
        for (int k = M - 2; k >= 0; k--) {
            double dr = 0.0, di = 0.0;
            cplx v[2];
            for (int u = 0; u < 2; u++) {
                const int i = lane + 32 * u;
                v[u] = (i > k && i < M) ? A[i * ld + k] : cmk(0.0, 0.0);
                const cplx x = cmul(cconj(v[u]), y[u]);
                dr += x.x;
                di += x.y;
            }
            const cplx f = cscale(cmul(t.tau[k], cmk(warp_sum(dr), warp_sum(di))), -1.0);
            for (int u = 0; u < 2; u++) cfma(y[u], f, v[u]);
        }
        for (int u = 0; u < 2; u++)
            if (lane + 32 * u < M) t.w[lane + 32 * u] = cscale(y[u], s_rcp[lane + 32 * u]);
    }
    __syncthreads();
    // lambda = U^{-dag} D^{-1/2} y
    for (int j = tid; j < M; j += AMP_THREADS) {
        cplx x = cmk(0.0, 0.0);
        for (int i = j; i < M; i++) cfma(x, cconj(W[i * ld + j]), t.w[i]);
        lr[j] = x.x;
        lr[M + j] = x.y;
    }
    E = s_E;
    if (tid == 0 && !isfinite(s_E)) atomicOr(a.err, SGS_DEV_EIG);
    __syncthreads();
    // every |lambda_j| at least AMP_SMALL times the largest (the larger part of each, on the high words)
    int mine = 0x7fffffff, most = 0;
    for (int j = lane; j < M; j += 32) {
        const int x = max(__double2hiint(lr[j]) & 0x7fffffff, __double2hiint(lr[M + j]) & 0x7fffffff);
        mine = min(mine, x);
        most = max(most, x);
    }
    mine = __reduce_min_sync(0xffffffffu, mine);
    most = __reduce_max_sync(0xffffffffu, most);
    return !(most - mine > __double2hiint(1.0) - least);
}

// where in scratch the solve marks its route (0: Jacobi, 1: direct; 2: gram_eig_kernel has run since), before the two
// values of gram_eig_kernel
__host__ __device__ inline size_t gram_mark(int M) { return 6 * (size_t)(2 * M) * (2 * M) + 2 * M; }

// dynamic shared memory of amp_solve_kernel
inline size_t amp_smem(int M) { return 3 * (size_t)M * (M + 1) * sizeof(cplx); }

__global__ void __launch_bounds__(AMP_THREADS) amp_solve_kernel(AmpArgs a) {
    extern __shared__ double amp_sm[];
    __shared__ double lr[2 * SGS_MAX_RANK], red[32];
    __shared__ cplx s_lam[SGS_MAX_RANK], s_lt[SGS_MAX_RANK], s_w[SGS_MAX_RANK];
    __shared__ cplx s_ph;
    const int M = a.M, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const double* G = a.Gm;
    const double* h = a.hm;
    double E = 0.0;
    const bool direct = amp_direct(a, reinterpret_cast<cplx*>(amp_sm), lr, E);
    if (tid == 0) a.scratch[gram_mark(M)] = direct ? 1.0 : 0.0;
    if (direct) {
        amp_embed(G, a.scratch, M);          // for gram_eig_kernel
    } else {
        __syncthreads();
        if (!amp_jacobi(a, lr, E)) return;
    }
    // normalisation lambda^dag G lambda = 1 and the phase convention; lambda-tilde = G lambda
    double nrm = 0.0;
    for (int i = warp; i < M; i += AMP_THREADS / 32) {
        cplx x = cmk(0.0, 0.0);
        for (int j = lane; j < M; j += 32)
            cfma(x, cmk(G[2 * (i * M + j)], G[2 * (i * M + j) + 1]), cmk(lr[j], lr[M + j]));
        x.x = warp_sum(x.x);
        x.y = warp_sum(x.y);
        if (lane == 0) {
            s_lt[i] = x;
            nrm += lr[i] * x.x + lr[M + i] * x.y;
        }
    }
    nrm = block_sum(nrm, red);
    if (tid == 0) {
        const double sc = 1.0 / sqrt(nrm);
        if (!(nrm > 0.0) || !isfinite(nrm)) atomicOr(a.err, SGS_DEV_EIG);
        int jb = 0;
        double best = -1.0;
        for (int i = 0; i < M; i++) {
            const double m2 = lr[i] * lr[i] + lr[M + i] * lr[M + i];
            if (m2 > best * (1.0 + 1e-12)) { best = m2; jb = i; }
        }
        const double pr = lr[jb], pi = lr[M + jb];
        const double pm = sqrt(pr * pr + pi * pi);
        s_ph = cmk(pr / pm * sc, -pi / pm * sc);   // times conj(lambda_j)/|lambda_j| and the norm
        a.E[0] = E;
    }
    __syncthreads();
    for (int i = tid; i < M; i += AMP_THREADS) {
        const cplx l = cmul(cmk(lr[i], lr[M + i]), s_ph), t = cmul(s_lt[i], s_ph);
        s_lam[i] = l;
        a.lam[2 * i] = l.x;
        a.lam[2 * i + 1] = l.y;
        a.lt[2 * i] = t.x;
        a.lt[2 * i + 1] = t.y;
        const cplx zz = cmul(l, cconj(t));          // lambda_mu conj(lt_mu)
        const double az = sqrt(cabs2(zz));
        cplx c = cmk(0.0, 0.0);
        if (az >= 1e-300) c = (a.cmode == 0) ? cdiv(cmk(1.0, 0.0), zz) : cscale(cconj(zz), 1.0 / az);
        s_w[i] = cmul(cconj(t), c);
    }
    __syncthreads();
    for (int mu = warp; mu < M; mu += AMP_THREADS / 32)
        for (int be = lane; be < M; be += 32) {
            const int e = mu * M + be;
            const cplx z = cmul(s_w[mu], s_lam[be]);
            const cplx g = cmk(G[2 * e], G[2 * e + 1]), hh = cmk(h[2 * e], h[2 * e + 1]);
            const cplx zg = cmul(z, g);
            const cplx a3 = cscale(cmul(z, csub(hh, cscale(g, E))), -1.0);
            double* co = a.coef + (size_t)e * 6;
            co[0] = -2.0 * zg.y; co[1] = 2.0 * zg.x; co[2] = 2.0 * zg.x; co[3] = 2.0 * zg.y; co[4] = a3.x; co[5] = a3.y;
        }
}

// dynamic shared memory of gram_eig_kernel
inline size_t gram_smem(int M) { return (size_t)M * (M + 1) * sizeof(cplx); }

// The smallest and the largest eigenvalue of G of the last amplitude solve, for the health report: after a Jacobi
// solve they are on its diagonal, after the direct route (which leaves the embedding of G in scratch) they come from
// the tridiagonal form by multisection, as the energy does.  Jacobi for them took about half of what the direct route
// saves a step.  They go to scratch behind the solve's mark, which then says that they are there.
__global__ void __launch_bounds__(AMP_THREADS) gram_eig_kernel(double* scratch, int M) {
    extern __shared__ double amp_sm[];
    __shared__ AmpTri t;
    cplx* B = reinterpret_cast<cplx*>(amp_sm);
    const int m = 2 * M, ld = M + 1, tid = threadIdx.x;
    double* mark = scratch + gram_mark(M);
    const double route = *mark;
    if (route == 2.0) return;
    __syncthreads();
    if (tid == 0) *mark = 2.0;
    if (route != 1.0) {
        if (tid == 0) {
            double lo = INFINITY, hi = 0.0;
            for (int j = 0; j < m; j++) {
                lo = fmin(lo, scratch[(size_t)j * m + j]);
                hi = fmax(hi, scratch[(size_t)j * m + j]);
            }
            mark[1] = lo;
            mark[2] = hi;
        }
        return;
    }
    for (int e = tid; e < M * M; e += AMP_THREADS) {
        const int i = e / M, j = e % M;
        B[i * ld + j] = cmk(scratch[(size_t)i * m + j], scratch[(size_t)(i + M) * m + j]);
    }
    __syncthreads();
    amp_reduce(nullptr, B, M, ld, t);
    if (tid < 32) {
        double lo, hi, top, low;
        bool nan;
        amp_lowest(t, M, lo, hi, top, nan);
        low = 0.5 * (lo + hi);
        __syncwarp();
        for (int i = tid; i < M; i += 32) t.d[i] = -t.d[i];         // the largest of T: the lowest of -T
        __syncwarp();
        amp_lowest(t, M, lo, hi, top, nan);
        if (tid == 0) {
            mark[1] = low;
            mark[2] = -0.5 * (lo + hi);
        }
    }
}

}  // namespace sgs
