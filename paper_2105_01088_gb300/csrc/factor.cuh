// Batched FP64 factorisations of the pair matrices.
//
//  * Gauss-Jordan inverse with partial pivoting of S = Gamma_a + Gamma_b
//    (Eq. def-delta-matrix needs S^{-1}; |Pf S| = |det S|^{1/2} gives the
//    overlap magnitude of Sec. II B).  Blocked: a panel kernel eliminates b
//    columns of every matrix (one CTA per matrix, panel in shared memory),
//    then one batched product applies the delayed rank-b update to the
//    rest of each matrix.
//  * Complex Pfaffian of Y = Gamma_0 + Delta^{a,b} (the phase of the overlap
//    in the reference gauge of Sec. II B) by Parlett-Reid elimination with
//    pivoting, blocked the same way: the panel kernel performs b elimination
//    steps, materialising the two columns each step needs from the stored
//    matrix (its upper triangle, the only part kept current) plus the pending
//    rank-2 updates, and the rank-2b trailing update is a batch of two real
//    products per matrix (real and imaginary parts, k = 4b).
//
// Both panels have a second form, a cluster of 2 to 8 CTAs per matrix, for batches that leave
// SMs idle with one CTA per matrix: each CTA keeps its share of the rows in shared memory, and
// what every row needs (pivot candidates and their rows) is pushed to all CTAs of the cluster
// through distributed shared memory before a cluster barrier.
#pragma once
#include <cooperative_groups.h>
#include <algorithm>
#include "common.cuh"
#include "oz_digits.cuh"

namespace sgs {

// ---------------------------------------------------------------- Gauss-Jordan

#define GJ_MAX_PANEL 64       // widest Gauss-Jordan panel

struct GJPanelArgs {
    double* const* W;        // [batch] n x n working matrices (row-major)
    double* const* T;        // [batch] bb x n copy of the panel rows (update operand), or nullptr
    int* piv;                // [batch][n]
    double* logdet;          // [batch] log|det S|
    double* dsign;           // [batch] sign(det S)
    int* err;                // error word (SGS_DEV_SINGULAR)
    int n, k0, bb;
    double tiny;             // a pivot of magnitude <= tiny counts as singular
};

// bf16 digits of four values into w (w[i][0] | w[i][1] << 32: the four digits of slice i), zero
// where E = 0 or the value is absent (present[u] false)
__device__ __forceinline__ void oz_digits4(const double (&v)[4], const bool (&present)[4], int E, unsigned (&w)[OZ_S][2]) {
#pragma unroll
    for (int u = 0; u < 4; u++) {
        float f[OZ_S];
        if (E > 0 && present[u]) oz_digit_floats((unsigned long long)__double_as_longlong(v[u]), E, f);
        else {
#pragma unroll
            for (int i = 0; i < OZ_S; i++) f[i] = 0.0f;
        }
#pragma unroll
        for (int i = 0; i < OZ_S; i++) {
            const unsigned h = __float_as_uint(f[i]) >> 16;
            if (u & 1) w[i][u >> 1] |= h << 16;
            else w[i][u >> 1] = h;
        }
    }
}

// Products of many pivots are kept as a mantissa and an exponent of two, so that the logarithm, the
// square root and the divisions (hundreds of clocks each on this part's FP64 pipe) are taken once per
// matrix instead of once per pivot.  x scaled by a power of two to magnitude 1 .. 2 by its bits, the
// exponent added to e; zero, infinities and NaN are left as they are (a subnormal is scaled up first: a
// product of two of them would vanish)
__device__ __forceinline__ double pow2_split(double x, int& e) {
    int f = (__double2hiint(x) >> 20) & 0x7ff;
    if (f == 0 && (__double_as_longlong(x) << 1) != 0) {
        x *= 0x1p54;
        e -= 54;
        f = (__double2hiint(x) >> 20) & 0x7ff;
    }
    const bool ok = f > 0 && f < 2047;
    e += ok ? f - 1023 : 0;
    return ok ? __hiloint2double(__double2hiint(x) - ((f - 1023) << 20), __double2loint(x)) : x;
}
__device__ __forceinline__ int expo_field(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// det += the panel's pivots (|pivot_j| in pabs, signs in sign), by one warp: logdet[b] holds the
// product's exponent and dsign[b] its signed mantissa until the last panel, which leaves log|det| and
// the sign.  singular: log|det| becomes -infinity
__device__ void gj_det(const GJPanelArgs& a, int b, const double* pabs, bool negative, bool singular) {
    const int lane = threadIdx.x & 31;
    int e = 0;
    double m = 1.0;
    for (int j = lane; j < a.bb; j += 32) m *= pow2_split(pabs[j], e);
    for (int o = 16; o > 0; o >>= 1) {
        m *= __shfl_xor_sync(0xffffffffu, m, o);
        e += __shfl_xor_sync(0xffffffffu, e, o);
    }
    if (lane != 0) return;
    const double m0 = a.k0 == 0 ? 1.0 : a.dsign[b];
    double ex = a.k0 == 0 ? 0.0 : a.logdet[b];
    m = pow2_split(m * m0, e);
    ex = singular ? -INFINITY : ex + e;
    if (negative) m = -m;
    if (a.k0 + a.bb == a.n) {
        a.logdet[b] = fma(ex, 0.693147180559945309417, log(fabs(m)));
        a.dsign[b] = m < 0.0 ? -1.0 : 1.0;
    } else {
        a.logdet[b] = ex;
        a.dsign[b] = m;
    }
}

// The panel's row interchanges (c <-> p, in order) as one permutation of the rows they touch: row
// rows[e] receives the old row src[e], e < nr.  Adds one interchange, by one warp (the searches as
// ballots); returns the new nr
__device__ __forceinline__ int gj_list_add(int c, int p, int* rows, int* src, int nr) {
    if (p == c) return nr;
    const int lane = threadIdx.x & 31;
    unsigned mc = 0, mp = 0;
    for (int e0 = 0; e0 < nr; e0 += 32) {
        const int e = e0 + lane;
        const int r = e < nr ? rows[e] : -1;
        const unsigned bc = __ballot_sync(0xffffffffu, r == c), bp = __ballot_sync(0xffffffffu, r == p);
        if (!mc && bc) mc = (unsigned)(e0 + __ffs(bc));       // 1 + index
        if (!mp && bp) mp = (unsigned)(e0 + __ffs(bp));
    }
    int ic = (int)mc - 1, ip = (int)mp - 1;
    if (ic < 0) { if (lane == 0) { rows[nr] = c; src[nr] = c; } ic = nr++; }
    if (ip < 0) { if (lane == 0) { rows[nr] = p; src[nr] = p; } ip = nr++; }
    __syncwarp();
    if (lane == 0) {
        const int t = src[ic];
        src[ic] = src[ip];
        src[ip] = t;
    }
    __syncwarp();
    return nr;
}

// The panel columns k0 .. k0 + bb - 1 of rows r0 .. r0 + rn - 1 of W into panel (row stride ps) or back:
// 16 lanes per row up to 16 columns, else a warp
template <bool STORE>
__device__ __forceinline__ void gj_panel_copy(double* W, double* panel, int n, int k0, int bb, int ps, int r0, int rn) {
    const int lg = bb <= 16 ? 4 : 5, q0 = threadIdx.x & ((1 << lg) - 1);
    double* w = W + (size_t)r0 * n + k0;
#pragma unroll 4
    for (int r = threadIdx.x >> lg; r < rn; r += blockDim.x >> lg)
        for (int q = q0; q < bb; q += 1 << lg) {
            if (STORE) w[(size_t)r * n + q] = panel[r * ps + q];
            else panel[r * ps + q] = w[(size_t)r * n + q];
        }
}

// The end of a Gauss-Jordan panel: its row interchanges (s_rows, s_src, nr) applied to columns c0 .. c1 - 1
// of W other than the panel's, staged through stage[0 .. cap), a block of columns at a time; the update
// operand T of those columns (the pivot rows, panel columns zeroed), if asked for.
template <int LOADS>
__device__ void gj_panel_finish(const GJPanelArgs& a, double* W, int b, double* stage, int cap, const int* s_rows,
                                const int* s_src, int nr, int c0, int c1) {
    const int n = a.n, k0 = a.k0, bb = a.bb;
    // a warp per row, lanes along the columns, LOADS loads in flight per lane
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (nr > 0) {
        const int qc = min(c1 - c0, cap / nr);
        for (int q0 = c0; q0 < c1; q0 += qc) {
            const int qn = min(qc, c1 - q0);
            for (int e = warp; e < nr; e += nw) {
                const double* src = W + (size_t)s_src[e] * n + q0;
#pragma unroll LOADS
                for (int x = lane; x < qn; x += 32)
                    if ((unsigned)(q0 + x - k0) >= (unsigned)bb) stage[e * qn + x] = src[x];
            }
            __syncthreads();
            for (int e = warp; e < nr; e += nw) {
                double* dst = W + (size_t)s_rows[e] * n + q0;
#pragma unroll LOADS
                for (int x = lane; x < qn; x += 32)
                    if ((unsigned)(q0 + x - k0) >= (unsigned)bb) dst[x] = stage[e * qn + x];
            }
            __syncthreads();
        }
    }
    if (a.T) {
        double* T = a.T[b];
        for (int e = threadIdx.x; e < bb * (c1 - c0); e += blockDim.x) {
            const int r = e / (c1 - c0), q = c0 + e % (c1 - c0);
            T[(size_t)r * n + q] = (q >= k0 && q < k0 + bb) ? 0.0 : W[(size_t)(k0 + r) * n + q];
        }
    }
}

// largest key (>= -1) of a warp and, among equal keys, the smallest index, in every lane: three 32-bit
// warp reductions
__device__ __forceinline__ void warp_argmax(long long& key, int& idx) {
    const unsigned full = 0xffffffffu;
    const unsigned long long u = (unsigned long long)(key + 1);
    const unsigned hi = (unsigned)(u >> 32), mh = __reduce_max_sync(full, hi);
    const unsigned lo = hi == mh ? (unsigned)u : 0u, ml = __reduce_max_sync(full, lo);
    const unsigned ix = (hi == mh && lo == ml) ? (unsigned)idx : 0x7fffffffu;
    idx = (int)__reduce_min_sync(full, ix);
    key = (long long)(((unsigned long long)mh << 32) | ml) - 1;
}

// One CTA per matrix, CTAS of them on an SM.  Four (32 registers a thread) make up to 608 matrices one wave: at two, 400
// inverses of 64 x 64 took 767 us, at four 602.  Batches of one wave at two take the form with 56 registers: 16 inverses
// of 64 x 64 379 us against 397, 64 of 200 x 200 2768 against 2831.
template <int CTAS>
__global__ void __launch_bounds__(512, CTAS) gj_panel_kernel(GJPanelArgs a) {
    extern __shared__ double sm[];
    const int ps = a.bb + 1;                   // odd row stride: column walks hit distinct banks
    double* panel = sm;                        // n x ps
    double* rowc = panel + (size_t)a.n * ps;   // bb
    __shared__ double red_v[32];
    __shared__ int red_i[32];
    __shared__ int s_piv[GJ_MAX_PANEL], s_rows[2 * GJ_MAX_PANEL], s_src[2 * GJ_MAX_PANEL], s_nr, s_neg, s_sing;
    __shared__ double s_pabs[GJ_MAX_PANEL], s_inv;

    const int b = blockIdx.x, n = a.n, k0 = a.k0, bb = a.bb;
    double* W = a.W[b];
    int* piv = a.piv + (size_t)b * n;

    gj_panel_copy<false>(W, panel, n, k0, bb, ps, 0, n);
    if (threadIdx.x == 0) s_neg = s_sing = 0;
    __syncthreads();

    for (int j = 0; j < bb; j++) {
        const int c = k0 + j;
        long long best = -1;
        int bi = 0x7fffffff;
        for (int r = c + threadIdx.x; r < n; r += blockDim.x) {
            const long long v = abs_key(panel[r * ps + j]);
            if (v > best) { best = v; bi = r; }
        }
        double mv;
        int p;
        block_argmax(best < 0 ? -1.0 : __longlong_as_double(best), bi, red_v, red_i, mv, p);
        if (!(mv > a.tiny)) {          // singular (or NaN): flag, keep going with p = c
            if (threadIdx.x == 0) { atomicOr(a.err, SGS_DEV_SINGULAR); s_sing = 1; }
            p = c;
        }
        // rows c and p: interchanged now in the panel; on the other columns of W the panel's
        // interchanges are applied together after the panel (nothing reads them before)
        if (p != c) {
            for (int q = threadIdx.x; q < bb; q += blockDim.x) {
                double t = panel[c * ps + q];
                panel[c * ps + q] = panel[p * ps + q];
                panel[p * ps + q] = t;
            }
        }
        if (threadIdx.x == 0) { piv[c] = p; s_piv[j] = p; }
        __syncthreads();
        // warp 0 forms the pivot's reciprocal once (an FP64 division is many instructions on this
        // part's FP64 pipe) and the scaled pivot row; |pivot| is kept and the logarithms are summed
        // after the panel
        if (threadIdx.x < 32) {
            double pv = panel[c * ps + j];
            const bool sing = !(mv > a.tiny);
            if (sing) pv = 1.0;
            double inv = 0.0;
            if (threadIdx.x == 0) {
                inv = 1.0 / pv;
                s_inv = inv;
                s_pabs[j] = sing ? 1.0 : fabs(pv);
                s_neg ^= (pv < 0.0) != (p != c);
            }
            inv = __shfl_sync(0xffffffffu, inv, 0);
            for (int q = threadIdx.x; q < bb; q += 32) rowc[q] = (q == j) ? inv : panel[c * ps + q] * inv;
        }
        __syncthreads();
        const double inv = s_inv;
        for (int q = threadIdx.x; q < bb; q += blockDim.x) panel[c * ps + q] = rowc[q];
        for (int r = threadIdx.x; r < n; r += blockDim.x) {
            if (r == c) continue;
            double f = panel[r * ps + j];
            if (abs_key(f) != 0) {               // an integer test: no FP64 compare
                for (int q = 0; q < bb; q++)
                    if (q != j) panel[r * ps + q] -= f * rowc[q];
            }
            panel[r * ps + j] = -f * inv;
        }
        __syncthreads();
    }

    gj_panel_copy<true>(W, panel, n, k0, bb, ps, 0, n);
    __syncthreads();
    if (threadIdx.x < 32) {
        int nr = 0;
        for (int j = 0; j < bb; j++) nr = gj_list_add(k0 + j, s_piv[j], s_rows, s_src, nr);
        if (threadIdx.x == 0) s_nr = nr;
    } else if (threadIdx.x < 64) {
        gj_det(a, b, s_pabs, s_neg != 0, s_sing != 0);
    }
    __syncthreads();
    gj_panel_finish<CTAS == 2 ? 8 : 4>(a, W, b, panel, n * ps, s_rows, s_src, s_nr, 0, n);
}

// The panel by a cluster of C CTAs per matrix (grid batch x C): CTA r holds rows r ch .. r ch + ch - 1 of
// the panel in shared memory, G = 2^lg threads per row (each taking every G-th column), and one
// more warp for what is not per row.  Per column: each CTA's pivot candidate (the largest entry of its
// rows from the diagonal on) with its row and reciprocal, and the diagonal's row from its owner, go to
// every CTA before one cluster barrier; then each CTA knows the pivot row, interchanges what it holds of
// the two rows and eliminates.  The slots alternate between two buffers, so that one barrier per column
// is enough.  The arithmetic is the one-CTA form's operation by operation, so the bits are too: the form
// chosen for a batch does not show in its results.  The interchanges of the other columns are shared out by columns.
// Bound by the latency of a column: reduction, push, cluster barrier (about 1300 clocks with the remote
// stores), a few FP64 instructions at 64 clocks each.  Comparisons and conversions stay on integers (an
// FP64 one by every warp costs 19 clocks per warp of the SM's FP64 pipe).
#define GJC_STAGE 4096        // doubles of shared memory at least (staging of the interchanges)
__global__ void __launch_bounds__(288) gj_cluster_kernel(GJPanelArgs a, int C, int ch, int lg) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ double sm[];
    const int n = a.n, k0 = a.k0, bb = a.bb, ps = bb + 1;
    const int rank = blockIdx.x % C, b = blockIdx.x / C;
    const int r0 = rank * ch, rn = max(0, min(ch, n - r0));        // own rows
    // slots[2][C + 1][bb + 3]: a candidate's row, its value, 1 / value and row index; slot C the
    // diagonal's row
    const int sl = bb + 3, NT = blockDim.x, NW = (NT >> 5) - 1;    // NW warps of rows
    double* slots = sm;
    double* panel = slots + 2 * (C + 1) * sl;
    __shared__ long long red_v[8];
    __shared__ int red_i[8];
    __shared__ int s_rows[2 * GJ_MAX_PANEL], s_src[2 * GJ_MAX_PANEL], s_nr;
    __shared__ double s_pabs[GJ_MAX_PANEL], rowc[GJ_MAX_PANEL];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, G = 1 << lg, g = tid & (G - 1), RP = (32 * NW) >> lg;
    const bool extra = warp == NW;
    const long long tiny_key = abs_key(a.tiny);
    double* W = a.W[b];
    gj_panel_copy<false>(W, panel, n, k0, bb, ps, r0, rn);
    int nr = 0, neg = 0, singular = 0;     // the extra warp's: interchanges listed, the determinant's sign
    cluster.sync();                        // every CTA of the cluster has started; the panel is in place
    for (int j = 0; j < bb; j++) {
        const int c = k0 + j;
        double* slot = slots + (j & 1) * (C + 1) * sl;
        // candidate of this CTA: the largest magnitude at or below the diagonal, smaller row on a tie
        long long key = -1;
        int idx = 0x7fffffff;
        if (!extra) {
            if (g == 0)
                for (int r = (tid >> lg); r < rn; r += RP)
                    if (r0 + r >= c) {
                        const long long v = abs_key(panel[r * ps + j]);
                        if (v > key) { key = v; idx = r0 + r; }
                    }
            warp_argmax(key, idx);
            if (lane == 0) { red_v[warp] = key; red_i[warp] = idx; }
        }
        __syncthreads();
        key = lane < NW ? red_v[lane] : -1ll;
        idx = lane < NW ? red_i[lane] : 0x7fffffff;
        warp_argmax(key, idx);
        const bool have = key >= 0;
        if (extra) {                       // the value, its reciprocal and row
            const double v = have ? panel[(idx - r0) * ps + j] : 0.0;
            const double inv = 1.0 / v;
            if (lane < C) {
                double* to = cluster.map_shared_rank(slot, lane) + rank * sl + bb;
                to[0] = v;
                to[1] = inv;
                reinterpret_cast<long long*>(to)[2] = have ? idx : -1;
            }
        } else {                           // half a warp per destination up to 16 columns, else a warp
            const int half = bb <= 16, wd = half ? 16 : 32, l = lane & (wd - 1);
            const bool diag = c >= r0 && c < r0 + rn;
            for (int d = half ? 2 * warp + (lane >> 4) : warp; d < C; d += NW << half) {
                double* to = cluster.map_shared_rank(slot, d);
                for (int q = l; q < bb; q += wd) {
                    if (have) to[rank * sl + q] = panel[(idx - r0) * ps + q];
                    if (diag) to[C * sl + q] = panel[(c - r0) * ps + q];
                }
            }
        }
        cluster.sync();
        // the pivot: the largest candidate, on a tie the smaller row (lower ranks hold smaller rows)
        int w = lane;
        key = -1;
        if (lane < C && (int)reinterpret_cast<const long long*>(slot)[lane * sl + bb + 2] >= 0)
            key = abs_key(slot[lane * sl + bb]);
        warp_argmax(key, w);
        // singular (or NaN): flag, keep going with p = c and pivot 1
        const bool sing = !(key > tiny_key && key <= 0x7FF0000000000000ll);
        if (sing) w = 0;
        const int p = sing ? c : (int)reinterpret_cast<const long long*>(slot)[w * sl + bb + 2];
        const double* crow = slot + C * sl;
        const double* prow = sing ? crow : slot + w * sl;
        const double inv = sing ? 1.0 : slot[w * sl + bb + 1];
        if (extra)                         // the scaled pivot row
            for (int q = lane; q < bb; q += 32) rowc[q] = q == j ? inv : prow[q] * inv;
        __syncthreads();
        if (extra) {
            if (c >= r0 && c < r0 + rn)    // it takes the diagonal's row
                for (int q = lane; q < bb; q += 32) panel[(c - r0) * ps + q] = rowc[q];
            nr = gj_list_add(c, p, s_rows, s_src, nr);
            if (rank == 0) {
                const double pv = sing ? 1.0 : slot[w * sl + bb];
                neg ^= (__double2hiint(pv) < 0) != (p != c);
                singular |= sing;
                if (lane == 0) {
                    a.piv[(size_t)b * n + c] = p;
                    s_pabs[j] = fabs(pv);
                    if (sing) atomicOr(a.err, SGS_DEV_SINGULAR);
                }
            }
        } else {
            for (int rb = 0; rb < rn; rb += RP) {
                const int r = rb + (tid >> lg), i = r0 + r;
                const bool act = r < rn && i != c, sw = i == p;
                const double* x = sw ? crow : panel + r * ps;
                const double f = act ? x[j] : 0.0;
                __syncwarp();
                if (act) {
                    double* y = panel + r * ps;
                    if (abs_key(f) != 0) {
#pragma unroll 4
                        for (int q = g; q < bb; q += G) y[q] = fma(-f, rowc[q], x[q]);
                    } else if (sw) {
                        for (int q = g; q < bb; q += G) y[q] = x[q];
                    }
                    if (g == (j & (G - 1))) y[j] = -f * inv;
                }
                __syncwarp();
            }
        }
    }
    __syncthreads();
    gj_panel_copy<true>(W, panel, n, k0, bb, ps, r0, rn);
    if (extra && lane == 0) s_nr = nr;
    cluster.sync();        // no CTA's slots are written any more; W's panel columns are not read below
    if (extra && rank == 0) {
        __syncwarp();
        gj_det(a, b, s_pabs, neg != 0, singular != 0);
    }
    const int cw = (n + C - 1) / C, c0 = min(n, rank * cw), c1 = min(n, c0 + cw);
    gj_panel_finish<8>(a, W, b, sm, GJC_STAGE, s_rows, s_src, s_nr, c0, c1);
}

// shared memory of gj_cluster_kernel (bytes)
inline size_t gjc_smem(int bb, int C, int ch) {
    return std::max((size_t)2 * (C + 1) * (bb + 3) + (size_t)ch * (bb + 1), (size_t)GJC_STAGE) * sizeof(double);
}

// Rows p0 .. p0 + K - 1, columns t0 .. t0 + w - 1 of every W into T (K x w, row stride w):
// the pivot rows of the target columns of a delayed Gauss-Jordan update, taken before the
// update overwrites them.  Reads and writes run along the rows.
__global__ void gj_gather_rows_kernel(double* const* W, double* const* T, int n, int p0, int K, int t0, int w) {
    const double* src = W[blockIdx.y];
    double* dst = T[blockIdx.y];
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < (size_t)K * w;
         e += (size_t)gridDim.x * blockDim.x) {
        const int k = (int)(e / w), q = (int)(e % w);
        dst[e] = src[(size_t)(p0 + k) * n + t0 + q];
    }
}

// Both operands of a Gauss-Jordan update of small K and w (both <= 64), written directly as the
// slices the emulated product reads: A = columns p0 .. p0 + K - 1 of W (rows of K values;
// [batch][OZ_S][mp][kp], planes in oz_plane order, exponent fields [batch][mp]) and B = rows
// p0 .. p0 + K - 1 of the target columns t0 .. t0 + w - 1, op(B) column j (the K entries of
// column t0 + j) as row j ([batch][OZ_S][np][kp], natural plane order, exponent fields
// [batch][np]).  Padding rows and columns K .. kp - 1 get zero digits, as the slicers write
// them.  Grid (mp / GJ_SLICE_ROWS + 1, batch): a block of A rows per CTA, four consecutive
// columns of one row per thread; the last CTA of each matrix takes B.  One launch instead of
// the pivot-row gather and two slicing launches.
#define GJ_SLICE_ROWS 64
__global__ void __launch_bounds__(256) gj_update_slice_kernel(double* const* W, int n, int p0, int K, int t0, int w,
                                                              uint16_t* sa, int* ea, int mp, uint16_t* sb, int* eb,
                                                              int np, int kp) {
    __shared__ double tile[64][65];              // B: tile[j][k]
    __shared__ int s_e[64];
    const int b = blockIdx.y;
    const double* src = W[b];
    const int c4 = kp >> 2;
    for (int j = threadIdx.x; j < 64; j += blockDim.x) s_e[j] = 0;
    if (blockIdx.x < gridDim.x - 1) {
        const int r0 = blockIdx.x * GJ_SLICE_ROWS;
        __syncthreads();
        for (int e = threadIdx.x; e < GJ_SLICE_ROWS * c4; e += blockDim.x) {
            const int rr = e / c4, c = 4 * (e % c4), r = r0 + rr;
            int ef = 0;
            if (r < n)
                for (int u = 0; u < 4 && c + u < K; u++)
                    ef = max(ef, oz_expo_field((unsigned long long)__double_as_longlong(src[(size_t)r * n + p0 + c + u])));
            if (ef) atomicMax(&s_e[rr], ef);
        }
        __syncthreads();
        for (int e = threadIdx.x; e < GJ_SLICE_ROWS * c4; e += blockDim.x) {
            const int rr = e / c4, c = 4 * (e % c4), r = r0 + rr;
            if (r >= mp) continue;
            const int ef = s_e[rr];
            if (c == 0 && r < n) ea[(size_t)b * mp + r] = ef;
            double v[4];
            bool pr[4];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                pr[u] = r < n && c + u < K;
                v[u] = pr[u] ? src[(size_t)r * n + p0 + c + u] : 0.0;
            }
            unsigned wd[OZ_S][2];
            oz_digits4(v, pr, ef, wd);
#pragma unroll
            for (int i = 0; i < OZ_S; i++)
                *reinterpret_cast<unsigned long long*>(sa + (((size_t)b * OZ_S + oz_plane(i)) * mp + r) * kp + c) =
                    (unsigned long long)wd[i][0] | ((unsigned long long)wd[i][1] << 32);
        }
        return;
    }
    for (int e = threadIdx.x; e < K * w; e += blockDim.x) {
        const int k = e / w, j = e % w;           // along the rows of W
        tile[j][k] = src[(size_t)(p0 + k) * n + t0 + j];
    }
    __syncthreads();
    for (int j = threadIdx.x; j < w; j += blockDim.x) {
        int ef = 0;
        for (int k = 0; k < K; k++) ef = max(ef, oz_expo_field((unsigned long long)__double_as_longlong(tile[j][k])));
        s_e[j] = ef;
        eb[(size_t)b * np + j] = ef;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < np * c4; e += blockDim.x) {
        const int j = e / c4, c = 4 * (e % c4);
        double v[4];
        bool pr[4];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            pr[u] = j < w && c + u < K;
            v[u] = pr[u] ? tile[j][c + u] : 0.0;
        }
        unsigned wd[OZ_S][2];
        oz_digits4(v, pr, j < w ? s_e[j] : 0, wd);
#pragma unroll
        for (int i = 0; i < OZ_S; i++)
            *reinterpret_cast<unsigned long long*>(sb + (((size_t)b * OZ_S + i) * np + j) * kp + c) =
                (unsigned long long)wd[i][0] | ((unsigned long long)wd[i][1] << 32);
    }
}

// A delayed Gauss-Jordan update of small work on the FP64 pipe, in place: columns t0 .. t0 + w - 1 of every
// W take W[:, t] += W[:, p0 .. p0 + K - 1] T with T = their rows p0 .. p0 + K - 1 before the update, which
// are replaced by the product.  A CTA takes WT columns whole (so no other CTA reads the rows it replaces):
// T in shared memory, a thread per row.  Grid (ceil(w / WT), batch); K <= GJ_SMALL_K.  One launch, where
// the emulated form takes a slicing launch and a product tile's fixed time.
#define GJ_SMALL_K 64
template <int WT>
__global__ void __launch_bounds__(256) gj_update_small_kernel(double* const* W, int n, int p0, int K, int t0, int w) {
    __shared__ double T[GJ_SMALL_K][WT];
    double* a = W[blockIdx.y];
    const int c0 = t0 + blockIdx.x * WT, cn = min(WT, t0 + w - c0);
    for (int e = threadIdx.x; e < K * WT; e += blockDim.x) {
        const int k = e / WT, q = e % WT;
        T[k][q] = q < cn ? a[(size_t)(p0 + k) * n + c0 + q] : 0.0;
    }
    __syncthreads();
    for (int r = threadIdx.x; r < n; r += blockDim.x) {
        const double* x = a + (size_t)r * n + p0;
        double* y = a + (size_t)r * n + c0;
        const bool pivot = r >= p0 && r < p0 + K;
        double acc[WT];
#pragma unroll
        for (int q = 0; q < WT; q++) acc[q] = (pivot || q >= cn) ? 0.0 : y[q];
#pragma unroll 8
        for (int k = 0; k < K; k++) {
            const double v = x[k];
#pragma unroll
            for (int q = 0; q < WT; q++) acc[q] = fma(v, T[k][q], acc[q]);
        }
#pragma unroll
        for (int q = 0; q < WT; q++)
            if (q < cn) y[q] = acc[q];
    }
}

// Undo the row interchanges of Gauss-Jordan: inverse = X P, i.e. the column
// interchanges applied in reverse order.  perm[c] = source column of column c.
// One block per matrix: the pivots and the permutation in shared memory (2 n ints of dynamic
// shared memory), the serial interchanges by one thread there.
__global__ void gj_perm_kernel(const int* piv, int* perm, int n, int batch) {
    extern __shared__ int gj_pm[];
    int* pm = gj_pm;
    int* pv = gj_pm + n;
    const int b = blockIdx.x;
    if (b >= batch) return;
    for (int c = threadIdx.x; c < n; c += blockDim.x) {
        pm[c] = c;
        pv[c] = piv[(size_t)b * n + c];
    }
    __syncthreads();
    if (threadIdx.x == 0)
        for (int j = n - 1; j >= 0; j--) {
            const int p = pv[j];
            if (p != j) { const int t = pm[j]; pm[j] = pm[p]; pm[p] = t; }
        }
    __syncthreads();
    for (int c = threadIdx.x; c < n; c += blockDim.x) perm[(size_t)b * n + c] = pm[c];
}

__global__ void gj_gather_kernel(double* const* W, double* const* out, const int* perm, int n) {
    const int b = blockIdx.y;
    const int* pm = perm + (size_t)b * n;
    const double* src = W[b];
    double* dst = out[b];
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < (size_t)n * n;
         e += (size_t)gridDim.x * blockDim.x) {
        int r = (int)(e / n), c = (int)(e % n);
        dst[e] = src[(size_t)r * n + pm[c]];
    }
}

// ---------------------------------------------------------------- Pfaffian

struct PfPanelArgs {
    double* const* Y;        // [batch] planes: Re (n x n) then Im (n x n), antisymmetric
    double* const* TU;       // [batch] 4 x bs x n scratch: Tr, Ti, Ur, Ui (row t = step, contiguous in i)
    double* const* PA;       // [batch] packs, 4 blocks n x 4*bsmax apart:
                             //   A_re=[Tr,-Ti,-Ur,Ui] B_re=[Ur,Ui,Tr,Ti] A_im=[Tr,Ti,-Ur,-Ui] B_im=[Ui,Ur,Ti,Tr]
    double* logabs;          // [batch]
    double* phase;           // [batch][2]
    int* err;
    int n, k0, bs;           // bs = elimination steps in this panel
    int bsmax;               // pack blocks are n x 4*bsmax apart (row stride 4*bs)
    // emulated trailing update: with sa set the panel writes the update's operands as the
    // slices and exponent fields the product reads (entries 2 b, 2 b + 1: the real and
    // imaginary parts of matrix b; m = n - k0 - 2 bs rows, K = 4 bs; A slices [entry][OZ_S]
    // [mp][4 bs] in oz_plane order, B slices [entry][OZ_S][np][4 bs], exponents [entry][mp]
    // and [entry][np]) instead of the FP64 packs
    uint16_t* sa;
    uint16_t* sb;
    int* ea;
    int* eb;
    int mp, np;
};

#define PF_MAX_PANEL 32       // widest Pfaffian panel (column pairs)

// four digits per plane (w[i][0] | w[i][1] << 32: columns col .. col + 3 of slice i) into a slice
// batch [entry][OZ_S][rp][kk], planes in oz_plane order (inter, A operands) or natural order
__device__ __forceinline__ void pf_put_digits(uint16_t* base, int rp, int entry, int row, int kk, int col, bool inter,
                                              const unsigned (&w)[OZ_S][2]) {
#pragma unroll
    for (int i = 0; i < OZ_S; i++) {
        const int pl = inter ? oz_plane(i) : i;
        __stcs(reinterpret_cast<unsigned long long*>(base + (((size_t)entry * OZ_S + pl) * rp + row) * kk + col),
               (unsigned long long)w[i][0] | ((unsigned long long)w[i][1] << 32));
    }
}

// One pending rank-2 term of the panel on element (i, k): v += T[i][t] U[k][t] - U[i][t] T[k][t]
// (complex), as four FMAs per component (FP64 issues at a small fraction of the other
// pipes' rates on this part, so the count of FP64 instructions sets the panel's time).
// rowTU holds row k's T and U entries: Tr, Ti, Ur, Ui at offsets 0, bs, 2 bs, 3 bs.
__device__ __forceinline__ void pf_pending(double& vr, double& vi, double tr, double ti, double ur, double ui,
                                           const double* rowTU, int bs, int t) {
    const double Tkr = rowTU[t], Tki = rowTU[bs + t], Ukr = rowTU[2 * bs + t], Uki = rowTU[3 * bs + t];
    vr = fma(tr, Ukr, vr);
    vr = fma(-ti, Uki, vr);
    vr = fma(-ur, Tkr, vr);
    vr = fma(ui, Tki, vr);
    vi = fma(tr, Uki, vi);
    vi = fma(ti, Ukr, vi);
    vi = fma(-ur, Tki, vi);
    vi = fma(-ui, Tkr, vi);
}

// The Pfaffian's product takes the panel's pivots (pr, pi; left out where ok is 0), by one warp: phase[b]
// holds the product's mantissa (magnitude of order one) and logabs[b] its exponent of two until the last
// panel, which leaves the unit phase and log|Pf|.  flip: the panel made an odd number of interchanges
__device__ void pf_product(const PfPanelArgs& a, int b, const double* pr, const double* pi, const int* ok, bool flip) {
    const int lane = threadIdx.x & 31;
    int e = 0;
    cplx m = cmk(1.0, 0.0);
    const bool have = lane < a.bs, good = have && ok[lane];
    if (good) {
        const int f = max(expo_field(pr[lane]), expo_field(pi[lane]));
        const double sc = __hiloint2double(min(max(2046 - f, 1), 2046) << 20, 0);      // 2^(1023 - f)
        m = cmk(pr[lane] * sc, pi[lane] * sc);
        e = 2046 - min(max(2046 - f, 1), 2046) - 1023;
    }
    const bool zero = __any_sync(0xffffffffu, have && !good);
    for (int o = 16; o > 0; o >>= 1) {
        m = cmul(m, cmk(__shfl_xor_sync(0xffffffffu, m.x, o), __shfl_xor_sync(0xffffffffu, m.y, o)));
        e += __shfl_xor_sync(0xffffffffu, e, o);
    }
    if (lane != 0) return;
    double ex = a.k0 == 0 ? 0.0 : a.logabs[b];
    if (a.k0 != 0) m = cmul(m, cmk(a.phase[2 * b], a.phase[2 * b + 1]));
    const int f = max(expo_field(m.x), expo_field(m.y));
    const double sc = __hiloint2double(min(max(2046 - f, 1), 2046) << 20, 0);
    m = cscale(m, flip ? -sc : sc);
    e += 2046 - min(max(2046 - f, 1), 2046) - 1023;
    ex = zero ? -INFINITY : ex + e;
    if (a.k0 + 2 * a.bs >= a.n) {
        const double am = sqrt(cabs2(m));
        ex = fma(ex, 0.693147180559945309417, log(am));
        m = cscale(m, 1.0 / am);
    }
    a.logabs[b] = ex;
    a.phase[2 * b] = m.x;
    a.phase[2 * b + 1] = m.y;
}

// Columns of the antisymmetric Y are read as negated rows (coalesced); the
// pending rank-2 updates of the panel are added on the fly.  Launched with
// PF_PANEL_THREADS threads: four CTAs fit an SM (registers and shared memory),
// so up to 608 matrices run in one wave on 152 SMs.
#define PF_PANEL_THREADS 256
__global__ void __launch_bounds__(PF_PANEL_THREADS, 4) pf_panel_kernel(PfPanelArgs a) {
    extern __shared__ double sm[];
    const int n = a.n, k0 = a.k0, bs = a.bs;
    double* ckr = sm;            // current column k (real)
    double* cki = ckr + n;
    double* c1r = cki + n;       // current column k+1
    double* c1i = c1r + n;
    double* rowTU = c1i + n;     // 4 x bs: T/U entries of the row being materialised
    __shared__ double red_v[32];
    __shared__ int red_i[32];
    __shared__ double s_ir, s_ii;
    __shared__ double s_pvr[PF_MAX_PANEL], s_pvi[PF_MAX_PANEL];
    __shared__ int s_pok[PF_MAX_PANEL], s_flip;

    const int b = blockIdx.x;
    double* Yr = a.Y[b];
    double* Yi = Yr + (size_t)n * n;
    double* Tr = a.TU[b];                  // Tr[t * n + i]
    double* Ti = Tr + (size_t)n * bs;
    double* Ur = Ti + (size_t)n * bs;
    double* Ui = Ur + (size_t)n * bs;

    if (threadIdx.x == 0) s_flip = 0;

    for (int s = 0; s < bs; s++) {
        const int k = k0 + 2 * s;
        for (int t = threadIdx.x; t < s; t += blockDim.x) {
            rowTU[t] = Tr[(size_t)t * n + k];
            rowTU[bs + t] = Ti[(size_t)t * n + k];
            rowTU[2 * bs + t] = Ur[(size_t)t * n + k];
            rowTU[3 * bs + t] = Ui[(size_t)t * n + k];
        }
        __syncthreads();
        // current column k: -Y[k][i] + sum_t (T[i][t] U[k][t] - U[i][t] T[k][t])
        long long best = -1;
        int bi = 0x7fffffff;
        for (int i = k + 1 + threadIdx.x; i < n; i += blockDim.x) {
            double vr = -Yr[(size_t)k * n + i], vi = -Yi[(size_t)k * n + i];
            for (int t = 0; t < s; t++)
                pf_pending(vr, vi, Tr[(size_t)t * n + i], Ti[(size_t)t * n + i], Ur[(size_t)t * n + i],
                           Ui[(size_t)t * n + i], rowTU, bs, t);
            ckr[i] = vr;
            cki[i] = vi;
            const long long m2 = abs_key(fma(vr, vr, vi * vi));
            if (m2 > best) { best = m2; bi = i; }
        }
        double mv;
        int p;
        block_argmax(best < 0 ? -1.0 : __longlong_as_double(best), bi, red_v, red_i, mv, p);
        if (!(mv > 0.0)) {
            if (threadIdx.x == 0) atomicOr(a.err, SGS_DEV_PF_ZERO);
            p = k + 1;
        }
        if (p != k + 1) {
            const int q = k + 1;
            // symmetric interchange q <-> p on the upper triangle of the live part, the only part the
            // panels read (row k is done: its entries are in ckr, cki); the trailing update reads its
            // Cin there too (cin_trans), so the lower triangle is left stale.  With q < p:
            //   row entries beyond p:    Y[q][j] <-> Y[p][j]                       (j > p)
            //   between q and p:         Y'[q][c] = -Y[c][p], Y'[c][p] = -Y[q][c]  (q < c < p)
            //   the pair:                Y'[q][p] = -Y[q][p]
            for (int j = p + 1 + threadIdx.x; j < n; j += blockDim.x) {
                double t;
                t = Yr[(size_t)q * n + j]; Yr[(size_t)q * n + j] = Yr[(size_t)p * n + j]; Yr[(size_t)p * n + j] = t;
                t = Yi[(size_t)q * n + j]; Yi[(size_t)q * n + j] = Yi[(size_t)p * n + j]; Yi[(size_t)p * n + j] = t;
            }
            for (int c = q + 1 + threadIdx.x; c < p; c += blockDim.x) {
                const double ar = Yr[(size_t)q * n + c], ai = Yi[(size_t)q * n + c];
                Yr[(size_t)q * n + c] = -Yr[(size_t)c * n + p];
                Yi[(size_t)q * n + c] = -Yi[(size_t)c * n + p];
                Yr[(size_t)c * n + p] = -ar;
                Yi[(size_t)c * n + p] = -ai;
            }
            if (threadIdx.x == 0) {
                Yr[(size_t)q * n + p] = -Yr[(size_t)q * n + p];
                Yi[(size_t)q * n + p] = -Yi[(size_t)q * n + p];
            }
            for (int t = threadIdx.x; t < s; t += blockDim.x) {
                double x;
                x = Tr[(size_t)t * n + q]; Tr[(size_t)t * n + q] = Tr[(size_t)t * n + p]; Tr[(size_t)t * n + p] = x;
                x = Ti[(size_t)t * n + q]; Ti[(size_t)t * n + q] = Ti[(size_t)t * n + p]; Ti[(size_t)t * n + p] = x;
                x = Ur[(size_t)t * n + q]; Ur[(size_t)t * n + q] = Ur[(size_t)t * n + p]; Ur[(size_t)t * n + p] = x;
                x = Ui[(size_t)t * n + q]; Ui[(size_t)t * n + q] = Ui[(size_t)t * n + p]; Ui[(size_t)t * n + p] = x;
            }
            if (threadIdx.x == 0) {
                double x = ckr[q]; ckr[q] = ckr[p]; ckr[p] = x;
                x = cki[q]; cki[q] = cki[p]; cki[p] = x;
                s_flip ^= 1;      // a row/column interchange flips the sign (applied after the panel)
            }
        }
        __syncthreads();
        for (int t = threadIdx.x; t < s; t += blockDim.x) {
            rowTU[t] = Tr[(size_t)t * n + k + 1];
            rowTU[bs + t] = Ti[(size_t)t * n + k + 1];
            rowTU[2 * bs + t] = Ur[(size_t)t * n + k + 1];
            rowTU[3 * bs + t] = Ui[(size_t)t * n + k + 1];
        }
        __syncthreads();
        // current column k+1 (rows >= k+2): -Y[k+1][i] + pending
        for (int i = k + 2 + threadIdx.x; i < n; i += blockDim.x) {
            double vr = -Yr[(size_t)(k + 1) * n + i], vi = -Yi[(size_t)(k + 1) * n + i];
            for (int t = 0; t < s; t++)
                pf_pending(vr, vi, Tr[(size_t)t * n + i], Ti[(size_t)t * n + i], Ur[(size_t)t * n + i],
                           Ui[(size_t)t * n + i], rowTU, bs, t);
            c1r[i] = vr;
            c1i[i] = vi;
        }
        // pivot Y[k][k+1] = -Y[k+1][k]: thread 0 forms 1/pivot once (an FP64 division is many
        // instructions on this part's FP64 pipe) and keeps the pivot, whose logarithm and unit
        // phase are accumulated after the panel in the same order
        if (threadIdx.x == 0) {
            double pr = -ckr[k + 1], pi = -cki[k + 1];
            const bool ok = mv > 0.0;
            if (!ok) { pr = 1.0; pi = 0.0; }
            const double pm2 = pr * pr + pi * pi;
            s_ir = pr / pm2;
            s_ii = -pi / pm2;
            s_pvr[s] = pr;
            s_pvi[s] = pi;
            s_pok[s] = ok ? 1 : 0;
        }
        __syncthreads();
        // tau = (row k)/pivot = -(column k)/pivot, u = column k+1; zero above k+2
        const double ir = s_ir, ii = s_ii;   // 1/pivot
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            double tr = 0.0, ti = 0.0, ur = 0.0, ui = 0.0;
            if (i >= k + 2) {
                const double xr = -ckr[i], xi = -cki[i];
                tr = xr * ir - xi * ii;
                ti = xr * ii + xi * ir;
                ur = c1r[i];
                ui = c1i[i];
            }
            Tr[(size_t)s * n + i] = tr;
            Ti[(size_t)s * n + i] = ti;
            Ur[(size_t)s * n + i] = ur;
            Ui[(size_t)s * n + i] = ui;
        }
        __syncthreads();
    }

    // packs for the trailing update (rows >= k0 + 2 bs are the only ones used)
    const int e0 = k0 + 2 * bs;
    const int kk = 4 * bs;
    double* PAre = a.PA[b];
    const size_t blk = (size_t)n * 4 * a.bsmax;
    double* PBre = PAre + blk;
    double* PAim = PBre + blk;
    double* PBim = PAim + blk;
    // rows are staged through the column buffers (4 n doubles, free now), R rows at a time
    // with an odd row stride: T/U read along i and the packs written along their rows,
    // both coalesced, with streaming stores (the packs are read once, by the next kernel,
    // and should not push the T/U vectors of CTAs still in their panel out of L2)
    const bool sliced = a.sa != nullptr;
    __shared__ int s_E[32];
    int R = n / bs - 1;
    if (R < 1) R = 1;
    if (sliced && R > 32) R = 32;
    const int rs = R | 1;                       // 4 bs rs <= 4 n
    double* stg = sm;
    for (int i0 = e0; i0 < n; i0 += R) {
        const int rn = min(R, n - i0);
        __syncthreads();
        for (int e = threadIdx.x; e < 4 * bs * rn; e += blockDim.x) {
            const int r = e % rn, qt = e / rn;  // qt = plane * bs + t; planes Tr, Ti, Ur, Ui
            stg[qt * rs + r] = Tr[(size_t)(qt / bs) * n * bs + (size_t)(qt % bs) * n + i0 + r];
        }
        __syncthreads();
        if (!sliced) {
            for (int e = threadIdx.x; e < rn * kk; e += blockDim.x) {
                const int r = e / kk, c = e % kk, blk = c / bs, t = c % bs;
                const double* v = stg + r;      // v[(plane * bs + t) * rs]: plane 0 Tr, 1 Ti, 2 Ur, 3 Ui
                const size_t o = (size_t)(i0 + r) * kk + c;
                // A_re = [Tr, -Ti, -Ur, Ui], B_re = [Ur, Ui, Tr, Ti], A_im = [Tr, Ti, -Ur, -Ui], B_im = [Ui, Ur, Ti, Tr]
                const double x = v[(blk * bs + t) * rs];
                __stcs(PAre + o, (blk == 1 || blk == 2) ? -x : x);
                __stcs(PAim + o, blk >= 2 ? -x : x);
                __stcs(PBre + o, v[(((blk + 2) & 3) * bs + t) * rs]);
                __stcs(PBim + o, v[((3 - blk) * bs + t) * rs]);
            }
            continue;
        }
        // slices: every pack row is a signed permutation of the same 4 bs values, so the four
        // packs share the row's exponent field (the largest of them), one warp per row
        for (int r = threadIdx.x >> 5; r < rn; r += blockDim.x >> 5) {
            int ef = 0;
            for (int q = threadIdx.x & 31; q < kk; q += 32)
                ef = max(ef, oz_expo_field((unsigned long long)__double_as_longlong(stg[q * rs + r])));
            for (int w = 16; w > 0; w >>= 1) ef = max(ef, __shfl_xor_sync(0xffffffffu, ef, w));
            if ((threadIdx.x & 31) == 0) {
                s_E[r] = ef;
                const int row = i0 + r - e0;
                a.ea[(size_t)(2 * b) * a.mp + row] = ef;
                a.ea[(size_t)(2 * b + 1) * a.mp + row] = ef;
                a.eb[(size_t)(2 * b) * a.np + row] = ef;
                a.eb[(size_t)(2 * b + 1) * a.np + row] = ef;
            }
        }
        __syncthreads();
        // digits of four consecutive values t .. t + 3 of one source plane (Tr, Ti, Ur, Ui) of one
        // row per thread, once per sign the packs take them with (as the slicers write them: one
        // 8-byte word of four bf16 per plane).  Plane src sits in block src of A_re = [Tr, -Ti,
        // -Ur, Ui] and A_im = [Tr, Ti, -Ur, -Ui], block (src + 2) & 3 of B_re = [Ur, Ui, Tr, Ti]
        // and block 3 - src of B_im = [Ui, Ur, Ti, Tr]
        const int t4n = bs >> 2;
        for (int e = threadIdx.x; e < rn * 4 * t4n; e += blockDim.x) {
            const int t = 4 * (e % t4n), src = (e / t4n) & 3, r = e / (4 * t4n);
            const int E = s_E[r], row = i0 + r - e0;
            const bool nre = src == 1 || src == 2, nim = src >= 2;
#pragma unroll 1
            for (int sg = 0; sg < 2; sg++) {
                if (sg == 1 && !nre && !nim) break;
                unsigned w[OZ_S][2];
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    const double x = stg[(src * bs + t + u) * rs + r];
                    float f[OZ_S];
                    if (E > 0) oz_digit_floats((unsigned long long)__double_as_longlong(sg ? -x : x), E, f);
                    else {
#pragma unroll
                        for (int i = 0; i < OZ_S; i++) f[i] = 0.0f;
                    }
#pragma unroll
                    for (int i = 0; i < OZ_S; i++) {
                        const unsigned h = __float_as_uint(f[i]) >> 16;
                        if (u & 1) w[i][u >> 1] |= h << 16;
                        else w[i][u >> 1] = h;
                    }
                }
                // pk 0, 1: A_re, A_im (block src, the sign they take); 2, 3: B_re, B_im (positive)
#pragma unroll 1
                for (int pk = 0; pk < 4; pk++) {
                    const bool take = pk == 0 ? nre == (sg == 1) : pk == 1 ? nim == (sg == 1) : sg == 0;
                    if (!take) continue;
                    const int blk = pk < 2 ? src : pk == 2 ? ((src + 2) & 3) : 3 - src;
                    pf_put_digits(pk < 2 ? a.sa : a.sb, pk < 2 ? a.mp : a.np, 2 * b + (pk & 1), row, kk, blk * bs + t,
                                  pk < 2, w);
                }
            }
        }
    }
    if (sliced && e0 < n) {
        // zero digits on the padding rows m .. mp - 1 (A) and m .. np - 1 (B), as the slicers write
        const int m = n - e0, c4n = kk >> 2;
        const int za = (a.mp - m) * c4n, zb = (a.np - m) * c4n;
        for (int e = threadIdx.x; e < 2 * OZ_S * (za + zb); e += blockDim.x) {
            const int ep = e / (OZ_S * (za + zb)), x = e % (OZ_S * (za + zb));
            const int pl = x / (za + zb), y = x % (za + zb);
            const bool isA = y < za;
            const int z = isA ? y : y - za, row = m + z / c4n, c = 4 * (z % c4n);
            uint16_t* base = isA ? a.sa : a.sb;
            const int rp = isA ? a.mp : a.np;
            __stcs(reinterpret_cast<unsigned long long*>(base + (((size_t)(2 * b + ep) * OZ_S + pl) * rp + row) * kk + c),
                   0ull);
        }
    }
    if (threadIdx.x < 32) pf_product(a, b, s_pvr, s_pvi, s_pok, s_flip != 0);
}

// The digits of four values of one row for the packs' slices: plane src (Tr, Ti, Ur, Ui) of the
// row, columns t .. t + 3, into A_re, A_im (block src, the sign they take), B_re and B_im; E the
// row's exponent field, row counted from the trailing block's first (see pf_panel_kernel)
__device__ __forceinline__ void pf_slice4(const PfPanelArgs& a, int b, const double (&x)[4], int E, int src, int t,
                                          int row) {
    const int bs = a.bs, kk = 4 * bs;
    const bool nre = src == 1 || src == 2, nim = src >= 2, all[4] = {true, true, true, true};
#pragma unroll 1
    for (int sg = 0; sg < 2; sg++) {
        if (sg == 1 && !nre && !nim) break;
        const double v[4] = {sg ? -x[0] : x[0], sg ? -x[1] : x[1], sg ? -x[2] : x[2], sg ? -x[3] : x[3]};
        unsigned w[OZ_S][2];
        oz_digits4(v, all, E, w);
#pragma unroll 1
        for (int pk = 0; pk < 4; pk++) {
            const bool take = pk == 0 ? nre == (sg == 1) : pk == 1 ? nim == (sg == 1) : sg == 0;
            if (!take) continue;
            const int blk = pk < 2 ? src : pk == 2 ? ((src + 2) & 3) : 3 - src;
            pf_put_digits(pk < 2 ? a.sa : a.sb, pk < 2 ? a.mp : a.np, 2 * b + (pk & 1), row, kk, blk * bs + t, pk < 2,
                          w);
        }
    }
}

// The panel by a cluster of C CTAs per matrix (grid batch x C): CTA r holds the T and
// U entries of rows k0 + r ch .. of the live part in shared memory (TU[plane][step][row]), G = 2^lg threads
// per row sharing out the pending terms, and one more warp for what is not per row.  Per step, with k and q = k + 1 the step's rows:
//   * column k of the own rows; the CTA's pivot candidate with its T/U entries goes to every CTA, column k's
//     entry of row q too; cluster barrier;
//   * every CTA knows p and, with row p's T/U entries, forms column q of its rows from row p of Y (the
//     interchange of q and p: row q is done after this step, so only row p's new entries are stored, and
//     the row that takes q's place takes its T/U entries); T and U of this step;
//   * rows k + 2 and k + 3's T/U entries go to every CTA; cluster barrier.
// Y's entry (x, i), x < i, is written and read by different CTAs in different steps, ordered by the cluster
// barriers; its loads bypass L1.
// Bound by the latency of a step (two cluster barriers of about 900 clocks with their pushes, the
// reductions, an L2 access) and the FP64 pipe's 19 clocks per warp instruction, where the one-CTA form
// reads every pending term from L2 or DRAM and has one SM's FP64 pipe.
__global__ void __launch_bounds__(288) pf_cluster_kernel(PfPanelArgs a, int C, int ch, int lg) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ double sm[];
    const int NT = blockDim.x, NW = (NT >> 5) - 1;              // NW warps of rows
    const int n = a.n, k0 = a.k0, bs = a.bs, chs = ch | 1;
    const int rank = blockIdx.x % C, b = blockIdx.x / C;
    const int r0 = k0 + rank * ch, rn = max(0, min(ch, n - r0));       // own rows
    const int sl = 4 * bs + 4;                  // a slot: T/U entries, key, row, column k's entry (re, im)
    double* TU = sm;                            // [4][bs][chs]
    double* ck = TU + 4 * bs * chs;             // [2][chs] column k
    double* yq = ck + 2 * chs;                  // [2][chs] row q of Y
    double* rowK = yq + 2 * chs;                // [2][4 bs] row k's T/U entries (two steps' buffers)
    double* rowQ = rowK + 8 * bs;               // [2][4 bs] row q's
    double* slots = rowQ + 8 * bs;              // [C][sl]
    double* qck = slots + C * sl;               // [2] column k's entry of row q
    __shared__ long long red_v[8];
    __shared__ int red_i[8];
    __shared__ double s_inv[2], s_pvr[PF_MAX_PANEL], s_pvi[PF_MAX_PANEL];
    __shared__ int s_pok[PF_MAX_PANEL], s_flip;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, G = 1 << lg, g = tid & (G - 1), RP = (32 * NW) >> lg;
    const bool extra = warp == NW;
    double* Yr = a.Y[b];
    double* Yi = Yr + (size_t)n * n;
    const int pl = bs * chs;                    // plane stride of TU
    if (tid == 0) s_flip = 0;
    cluster.sync();                             // every CTA of the cluster has started

    for (int s = 0; s < bs; s++) {
        const int k = k0 + 2 * s, q = k + 1, par = s & 1;
        const double* rk = rowK + par * 4 * bs;
        const double* rq = rowQ + par * 4 * bs;
        // column k of the own rows: -Y[k][i] + pending
        long long key = -1;
        int idx = 0x7fffffff;
        for (int rb = 0; rb < rn && !extra; rb += RP) {
            const int r = rb + (tid >> lg), i = r0 + r;
            const bool act = r < rn && i > k;
            double y0 = 0.0, y1 = 0.0, z0 = 0.0, z1 = 0.0, vr = 0.0, vi = 0.0;
            if (act && g == 0) {
                y0 = __ldcg(Yr + (size_t)k * n + i);
                y1 = __ldcg(Yi + (size_t)k * n + i);
                if (i > q) { z0 = __ldcg(Yr + (size_t)q * n + i); z1 = __ldcg(Yi + (size_t)q * n + i); }
            }
            if (act)
                for (int t = g; t < s; t += G) {
                    const double* x = TU + t * chs + r;
                    pf_pending(vr, vi, x[0], x[pl], x[2 * pl], x[3 * pl], rk, bs, t);
                }
            for (int o = 1; o < G; o <<= 1) {
                vr += __shfl_xor_sync(0xffffffffu, vr, o);
                vi += __shfl_xor_sync(0xffffffffu, vi, o);
            }
            if (act && g == 0) {
                vr -= y0;
                vi -= y1;
                ck[r] = vr;
                ck[chs + r] = vi;
                yq[r] = z0;
                yq[chs + r] = z1;
                const long long m2 = abs_key(fma(vr, vr, vi * vi));
                if (m2 > key) { key = m2; idx = i; }
            }
        }
        if (!extra) {
            warp_argmax(key, idx);
            if (lane == 0) { red_v[warp] = key; red_i[warp] = idx; }
        }
        __syncthreads();
        key = lane < NW ? red_v[lane] : -1ll;
        idx = lane < NW ? red_i[lane] : 0x7fffffff;
        warp_argmax(key, idx);
        const bool have = key >= 0;
        // a warp per destination; the entries of steps not yet taken go along, unread
        for (int d = warp; d < C; d += NW + 1) {
            double* to = cluster.map_shared_rank(slots, d) + rank * sl;
            if (have) {
                if (s > 0)
                    for (int o = lane; o < 4 * bs; o += 32) to[o] = TU[o * chs + idx - r0];
                if (lane < 2) to[4 * bs + 2 + lane] = ck[lane * chs + idx - r0];
            }
            if (lane >= 2 && lane < 4)
                reinterpret_cast<long long*>(to)[4 * bs + lane - 2] = lane == 2 ? key : (have ? idx : -1);
            if (q >= r0 && q < r0 + rn && lane >= 4 && lane < 6)
                cluster.map_shared_rank(qck, d)[lane - 4] = ck[(lane - 4) * chs + q - r0];
        }
        cluster.sync();
        // the pivot: the largest candidate, on a tie the smaller row (lower ranks hold smaller rows)
        int w = lane;
        key = -1;
        const long long* meta = reinterpret_cast<const long long*>(slots) + 4 * bs;
        if (lane < C && (int)meta[lane * sl + 1] >= 0) key = meta[lane * sl];
        warp_argmax(key, w);
        const bool ok = key > 0 && key <= 0x7FF0000000000000ll;        // > 0 and not NaN, on the bits
        if (!ok) w = 0;
        const int p = ok ? (int)meta[w * sl + 1] : q;
        const double* rp = p == q ? rq : slots + w * sl;
        if (extra && lane == 0) {
            // pivot Y[k][q] = -(column k's entry of row p), its reciprocal and the records for the phase
            double pr = p == q ? -qck[0] : -slots[w * sl + 4 * bs + 2];
            double pi = p == q ? -qck[1] : -slots[w * sl + 4 * bs + 3];
            if (!ok) { pr = 1.0; pi = 0.0; }
            const double rm = 1.0 / fma(pr, pr, pi * pi);
            s_inv[0] = pr * rm;
            s_inv[1] = -pi * rm;
            s_pvr[s] = pr;
            s_pvi[s] = pi;
            s_pok[s] = ok ? 1 : 0;
            if (p != q) s_flip ^= 1;
            if (!ok && rank == 0) atomicOr(a.err, SGS_DEV_PF_ZERO);
        }
        // column q of the own rows, after the interchange of q and p: -Y'[q][i] + pending.  With q < p:
        // Y'[q][i] = Y[p][i] (i > p), -Y[i][p] (q < i < p), -Y[q][p] (i = p); row p takes row q's place
        double* ur = TU + 2 * pl + s * chs;
        double* ui = ur + pl;
        for (int rb = 0; rb < rn && !extra; rb += RP) {
            const int r = rb + (tid >> lg), i = r0 + r;
            const bool act = r < rn && i > q, sw = i == p && p != q;
            double y0 = 0.0, y1 = 0.0, vr = 0.0, vi = 0.0;
            if (act && g == 0) {
                if (i == p) {
                    y0 = -yq[r];
                    y1 = -yq[chs + r];
                } else {
                    const size_t o = i > p ? (size_t)p * n + i : (size_t)i * n + p;
                    y0 = __ldcg(Yr + o);
                    y1 = __ldcg(Yi + o);
                    if (i < p) { y0 = -y0; y1 = -y1; }
                }
            }
            if (act)
                for (int t = g; t < s; t += G) {
                    const double* x = sw ? rq + t : TU + t * chs + r;
                    const int st = sw ? bs : pl;
                    pf_pending(vr, vi, x[0], x[st], x[2 * st], x[3 * st], rp, bs, t);
                }
            if (act && sw)                      // row p's T/U entries from here on (step s's follow)
                for (int o = g; o < 4 * bs; o += G) TU[o * chs + r] = rq[o];
            __syncwarp();
            for (int o = 1; o < G; o <<= 1) {
                vr += __shfl_xor_sync(0xffffffffu, vr, o);
                vi += __shfl_xor_sync(0xffffffffu, vi, o);
            }
            if (act && g == 0) {
                ur[r] = vr - y0;
                ui[r] = vi - y1;
                if (p != q && i != p) {         // Y'[p][i] = Y[q][i] (i > p), Y'[i][p] = -Y[q][i] (i < p)
                    const double z0 = yq[r], z1 = yq[chs + r];
                    const size_t o = i > p ? (size_t)p * n + i : (size_t)i * n + p;
                    Yr[o] = i > p ? z0 : -z0;
                    Yi[o] = i > p ? z1 : -z1;
                }
                if (sw) { ck[r] = qck[0]; ck[chs + r] = qck[1]; }
            }
        }
        __syncthreads();
        // tau = (row k) / pivot = -(column k) / pivot (q < i), zero above
        {
            const double ir = s_inv[0], ii = s_inv[1];
            double* tr = TU + s * chs;
            double* ti = tr + pl;
            for (int r = tid; r < rn; r += NT) {
                const bool act = r0 + r > q;
                const double xr = act ? -ck[r] : 0.0, xi = act ? -ck[chs + r] : 0.0;
                tr[r] = xr * ir - xi * ii;
                ti[r] = xr * ii + xi * ir;
            }
        }
        __syncthreads();
        if (s + 1 < bs) {
            for (int u = 0; u < 2; u++) {               // rows k + 2 and k + 3, from their owners
                const int i = k + 2 + u;
                if (i < r0 || i >= r0 + rn) continue;
                double* mine = (u ? rowQ : rowK) + (par ^ 1) * 4 * bs;
                for (int d = warp; d < C; d += NW + 1) {
                    double* to = cluster.map_shared_rank(mine, d);
                    for (int o = lane; o < 4 * bs; o += 32) to[o] = TU[o * chs + i - r0];
                }
            }
        }
        cluster.sync();
    }

    // packs for the trailing update, own rows from e0 on (pf_panel_kernel's layout)
    const int e0 = k0 + 2 * bs, kk = 4 * bs;
    const int ra = max(0, e0 - r0);                     // first own row of the trailing block
    const int cnt = max(0, rn - ra);
    if (a.sa == nullptr) {
        double* PAre = a.PA[b];
        const size_t blk = (size_t)n * 4 * a.bsmax;
        for (int e = tid; e < cnt * kk; e += NT) {
            const int r = ra + e / kk, c = e % kk, bq = c / bs, t = c % bs;
            const double* v = TU + t * chs + r;         // v[plane * pl]
            const size_t o = (size_t)(r0 + r) * kk + c;
            const double x = v[bq * pl];
            __stcs(PAre + o, (bq == 1 || bq == 2) ? -x : x);
            __stcs(PAre + 2 * blk + o, bq >= 2 ? -x : x);
            __stcs(PAre + blk + o, v[((bq + 2) & 3) * pl]);
            __stcs(PAre + 3 * blk + o, v[(3 - bq) * pl]);
        }
    } else {
        int* s_E = reinterpret_cast<int*>(ck);          // the rows' exponent fields
        for (int r = ra + tid; r < rn; r += NT) {
            int ef = 0;
            for (int x = 0; x < kk; x++)
                ef = max(ef, oz_expo_field((unsigned long long)__double_as_longlong(TU[x * chs + r])));
            s_E[r] = ef;
            const int row = r0 + r - e0;
            a.ea[(size_t)(2 * b) * a.mp + row] = ef;
            a.ea[(size_t)(2 * b + 1) * a.mp + row] = ef;
            a.eb[(size_t)(2 * b) * a.np + row] = ef;
            a.eb[(size_t)(2 * b + 1) * a.np + row] = ef;
        }
        __syncthreads();
        const int t4n = bs >> 2;
        for (int e = tid; e < cnt * 4 * t4n; e += NT) {
            const int t = 4 * (e % t4n), src = (e / t4n) & 3, r = ra + e / (4 * t4n);
            const double* v = TU + src * pl + t * chs + r;
            const double x[4] = {v[0], v[chs], v[2 * chs], v[3 * chs]};
            pf_slice4(a, b, x, s_E[r], src, t, r0 + r - e0);
        }
        // zero digits on the padding rows m .. mp - 1 (A) and m .. np - 1 (B), shared out over the cluster
        const int m = n - e0, c4n = kk >> 2;
        const int za = (a.mp - m) * c4n, zb = (a.np - m) * c4n;
        for (int e = rank * NT + tid; e < 2 * OZ_S * (za + zb); e += C * NT) {
            const int ep = e / (OZ_S * (za + zb)), x = e % (OZ_S * (za + zb));
            const int plane = x / (za + zb), y = x % (za + zb);
            const bool isA = y < za;
            const int z = isA ? y : y - za, row = m + z / c4n, c = 4 * (z % c4n);
            uint16_t* base = isA ? a.sa : a.sb;
            const int rp = isA ? a.mp : a.np;
            __stcs(reinterpret_cast<unsigned long long*>(base + (((size_t)(2 * b + ep) * OZ_S + plane) * rp + row) * kk + c),
                   0ull);
        }
    }
    if (extra && rank == 0) pf_product(a, b, s_pvr, s_pvi, s_pok, s_flip != 0);
}

// shared memory of pf_cluster_kernel (bytes)
inline size_t pfc_smem(int bs, int C, int ch) {
    return ((size_t)(4 * bs + 4) * (ch | 1) + 16 * (size_t)bs + (size_t)C * (4 * bs + 4) + 2) * sizeof(double);
}

}  // namespace sgs
