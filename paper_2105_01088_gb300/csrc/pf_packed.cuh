// Pfaffian of one complex antisymmetric matrix of up to PACKED_PF_MAX rows by a CTA, in shared memory:
// Parlett-Reid elimination with pivoting on the upper triangle.
//
// The triangle is packed by rows, so that what is live after a step is the tail of the storage and every
// lane of the rank-2 update has an element (rows and columns from a table).  The step's rows k and q = k + 1
// are done after it, so the interchange of q and the pivot p only writes row and column p.
// Bound by the FP64 pipe: 8 FMAs per live element and step, m^3 / 12 elements in all.
#pragma once
#include "common.cuh"
#include "factor.cuh"
#include "pair.cuh"

namespace sgs {

#define PACKED_PF_MAX 152

// dynamic shared memory: the packed triangles (re, im), four vectors, the entries' row and column
inline size_t packed_pf_smem(int m) {
    return (size_t)m * (m - 1) / 2 * (2 * sizeof(double) + 2) + 4 * (size_t)m * sizeof(double) + 16;
}

struct PackedPf {
    int m, T;
    double *Zr, *Zi;                            // row i, column j > i at off(i) + j
    double *tr, *ti, *ur, *ui;                  // tau and u of the step
    uchar2* ij;
    __device__ PackedPf(double* sm, int m_) : m(m_), T(m_ * (m_ - 1) / 2) {
        Zr = sm;
        Zi = Zr + T;
        tr = Zi + T;
        ti = tr + m;
        ur = ti + m;
        ui = ur + m;
        ij = reinterpret_cast<uchar2*>(ui + m);
    }
    __device__ __forceinline__ int off(int i) const { return i * (2 * m - i - 1) / 2 - i - 1; }
    __device__ __forceinline__ void set(int i, int j, double re, double im) const {
        const int e = off(i) + j;
        Zr[e] = re;
        Zi[e] = im;
        ij[e] = make_uchar2((unsigned char)i, (unsigned char)j);
    }
};

// The elimination, by all threads (the matrix set and synchronised; at most 256).  Returns whether the
// Pfaffian is zero; else it is x 2^e, |x| of order one, in every lane of warp 0.
__device__ __forceinline__ bool packed_pfaffian(const PackedPf& P, cplx& x, int& e) {
    __shared__ long long red_v[8];
    __shared__ int red_i[8];
    __shared__ double s_inv[2], s_pr[PACKED_PF_MAX / 2], s_pi[PACKED_PF_MAX / 2];
    __shared__ int s_flip;
    const int m = P.m, T = P.T, NT = blockDim.x, NW = NT >> 5;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    double *Zr = P.Zr, *Zi = P.Zi, *tr = P.tr, *ti = P.ti, *ur = P.ur, *ui = P.ui;
    const uchar2* ij = P.ij;
    if (tid == NT - 1) s_flip = 0;
    for (int k = 0; k < m - 1; k += 2) {
        const int q = k + 1, ok = P.off(k), oq = P.off(q);
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
        if (!(key > 0 && key <= 0x7FF0000000000000ll)) return true;     // zero (or NaN)
        const int op = P.off(p);
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
                const int e = i > p ? op + i : P.off(i) + p;
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
        for (int e = P.off(k + 2) + k + 3 + tid; e < T; e += NT) {
            const uchar2 at = ij[e];
            const double ar = tr[at.x], ai = ti[at.x], br = ur[at.x], bi = ui[at.x];
            const double cr = tr[at.y], ci = ti[at.y], dr = ur[at.y], di = ui[at.y];
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
        e = 0;
        x = cmk(1.0, 0.0);
        for (int t = lane; t < m / 2; t += 32) {
            x = cmul(x, cmk(s_pr[t], s_pi[t]));
            const int f = min(max(2046 - max(expo_field(x.x), expo_field(x.y)), 1), 2046);
            x = cscale(x, __hiloint2double(f << 20, 0));    // 2^(f - 1023)
            e += 1023 - f;
        }
        for (int o = 16; o > 0; o >>= 1) {
            x = cmul(x, cmk(__shfl_xor_sync(0xffffffffu, x.x, o), __shfl_xor_sync(0xffffffffu, x.y, o)));
            e += __shfl_xor_sync(0xffffffffu, e, o);
        }
        if (s_flip) x = cscale(x, -1.0);
    }
    return false;
}

// The phase Pfaffians Pf(Gamma_0 + Delta^{a,b}) of small matrices, a CTA each, straight from S^{-1} and
// Im Delta: no planes, panels, packed operands and trailing updates.  Bound by the elimination's steps at small n
// (about 1.2 us each: the pivot's search, the interchange, tau) and by the FP64 pipe above n of about 100.
__global__ void __launch_bounds__(256) pf_small_kernel(InstDev d, const double* si, const double* imd, double* logabs,
                                                       double* phase, int* err) {
    extern __shared__ double sm[];
    const int n = d.n, q = blockIdx.x, p = d.pf_pair[q];
    const PackedPf pk(sm, n);
    const double* s = si + (size_t)p * nn(d);
    const double* im = imd + (size_t)p * nn(d);
    const int lane = threadIdx.x & 31, NW = blockDim.x >> 5;
    for (int i = threadIdx.x >> 5; i < n - 1; i += NW)
        for (int j = i + 1 + lane; j < n; j += 32) {
            const size_t e = (size_t)i * n + j;
            pk.set(i, j, d.gamma[e] - 2.0 * s[e], im[e]);
        }
    __syncthreads();
    int e = 0;
    cplx x;
    const bool zero = packed_pfaffian(pk, x, e);
    if (threadIdx.x != 0) return;
    if (zero) {
        atomicOr(err, SGS_DEV_PF_ZERO);
        logabs[q] = -INFINITY;
        phase[2 * q] = 1.0;
        phase[2 * q + 1] = 0.0;
        return;
    }
    const double am = sqrt(cabs2(x));
    logabs[q] = fma((double)e, 0.693147180559945309417, log(am));
    phase[2 * q] = x.x / am;
    phase[2 * q + 1] = x.y / am;
}

}  // namespace sgs
