// Batched FP64 GEMM emulated on the bf16 tensor cores (tcgen05 kind::f16) by
// splitting both operands into integer slices (the Ozaki scheme: Ozaki, Ogita,
// Oishi and Rump, Numer. Algorithms 59 (2012); its tensor-core forms by Mukunoki
// et al. and Ootomo et al.).  GB300's FP64 pipe issues about 1.25 TFLOP/s while
// its bf16 tensor cores issue over 2 PFLOP/s, so the products of the step run
// here when the emulated path is selected.  The error bound is normwise per row
// of op(A) and column of op(B) (the error budget below), not elementwise like
// that of the FP64 FMA kernel.
//
// Slicing.  Every row r of op(A) (K-major) gets the exponent field E_r of its
// largest element, so |a_rk| < 2^(E_r - 1022).  The element is rounded to the
// signed integer X = a_rk 2^(56 - (E_r - 1022)) (|X| < 2^56) and written as
// eight balanced base-128 digits, most significant first:
//     X = sum_{i=0..7} t_i 2^(7 (7 - i)),  |t_0| <= 128, |t_i| <= 64 (i >= 1),
// so a_rk = 2^(E_r - 1022) sum_i t_i 2^(-7 (i + 1)) up to 2^-57 of the row's
// scale.  Each digit is a bf16 (at most 8 significant bits: exact).  Columns of
// op(B) are sliced the same way.  The digit extraction is integer arithmetic on
// the IEEE bit pattern (FP64 arithmetic is the scarce resource here).
//
// Products.  The slice products t_i(A) t_j(B) with i + j <= 7 (36 of the 64)
// are accumulated into eight fp32 TMEM accumulators, one per group G = i + j
// (weight 2^(-7 (G + 2))).  Each product term is an integer of magnitude at
// most 2^14 (i = j = 0), 2^13 (one index 0) or 2^12, so over a K chunk of 512
// the sums of groups G <= 5 stay within 2^24 and are exact in fp32; groups 6
// and 7 may round, by at most 2^-47 of the output scale, below FP64's own
// rounding of a 512-term dot product.  K beyond 512 runs as further launches
// that add onto the output (one FP64 rounding per chunk).  The dropped products
// (i + j >= 8) weigh at most 2^-63 per term.
//
// Combination.  The eight group sums are converted to integers and combined
// exactly, hi = sum_{G<4} v_G 2^(7 (3 - G)), lo = sum_{G>=4} v_G 2^(7 (7 - G)),
// V = hi 2^28 + lo = H 2^28 + L (0 <= L < 2^28); V is rounded once to 53 bits
// and given the exponent E_r + F_c - 2107 (plus that of alpha when alpha is a
// power of two, else one multiplication), all in straight-line integer
// arithmetic on the bit pattern.  The GemmBatch epilogue (beta Cin, beta2 Cin2,
// diag, FULL / SKEW / GJ modes, pass-through of inactive batch entries) is
// applied as in gemm_f64, with no FP64 instruction beyond the additions the
// epilogue terms need (FP64 issues at a small fraction of the integer rate).
//
// Kernels per batch chunk: exponents and slices of op(A) and op(B), one pass
// over each (a warp per row where the operand's K rows are contiguous and long,
// else a block of whole rows at a time through shared memory), then the product
// kernel.  It takes 128 x 32 output tiles with CTAs of 10 warps (256 TMEM
// columns, 97 KB of shared memory), two to an SM, or, for K > 224, 128 x 64 tiles with
// one CTA of 18 warps an SM (all of its TMEM, 225 KB), which load 3/5 of the bytes per
// output.  Each CTA runs over every (grid)-th tile, so that CTAs side by side work on
// tiles side by side and share their slices in L2 (consecutive tiles per CTA read them
// from DRAM: 1.5 to 2.3 ms where this order took 0.86).  In the kernel:
//   * one producer lane loads, per 64-element K slab, the eight B slices as one
//     TMA box and the A slices in pairs (one 32 KB box per pair of
//     adjacent planes) through a ring, 128-byte swizzle, zero fill beyond K;
//     a B buffer is reloaded once its slab's MMAs have released it, and
//     the next tile's first slabs load during this tile's epilogue;
//   * one warp issues, per A slice and K16 step, one MMA of N up to 256 (wide tiles:
//     two above that) covering all the products of that slice (the B slices and the
//     groups they feed are adjacent) into the eight accumulators;
//   * the epilogue warps read the tile's Cin terms while the MMAs run, drain TMEM,
//     combine, and write the output from their registers; the next tile's MMAs start
//     when TMEM is drained (wide tiles: when the exact sums are in registers, before
//     they are rounded and stored).
// Per 128 x 64 outputs of an SM, K = 16 / 64 / 256 / 512: one tile per CTA (set-up, first
// loads and last stores exposed) 11.7, 13.4, - and 36.2 us; CTAs over many tiles 9.0,
// 11.8, 20.3 and 34.1; MMAs issued by a converged warp 17.6 and 30.8; wide tiles 15.7
// and 25.8.  What bounds it: wide tiles at K = 512 the MMAs, 40000 clocks of 46000 (36900 at
// full rate; the drain takes 5500); narrow tiles at K = 512 the loads (25.2 without them); at
// small K the integer work of the combination, about 150 instructions per output.
// Every mbarrier wait is bounded; on a timeout the launch records
// SGS_DEV_TC_TIMEOUT in the error word, waits (bounded) for its loads and MMAs
// in flight, frees TMEM and returns.
#pragma once
#include "gemm_f64.cuh"
#include "gemm_tma.cuh"
#include "oz_digits.cuh"
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>

namespace sgs {

#define OZ_G 8                // accumulator groups G = i + j <= 7
#define OZ_BM 128
#define OZ_KS 64              // K elements of one 128-byte slab row
#define OZ_KC 512             // K per exactly accumulated chunk
#define OZ_UNIT 2             // A slices per TMA box (one ring slot)
#define OZ_SLAB_A (OZ_BM * 128)

// Kernel shapes: BN output columns per tile (TMEM: 8 BN columns), EPIW epilogue warps, RING A-ring depth
// (units), BBUF B buffers, CTAS CTAs per SM.  A 128 x 64 tile takes all of an SM's TMEM and shared memory.
template <int BN, int EPIW, int RING, int BBUF, int CTAS> struct OzCfg {
    static constexpr int SLAB_B = BN * 128;
    static constexpr int SMEM = BBUF * OZ_S * SLAB_B + RING * OZ_UNIT * OZ_SLAB_A + 1024;
    static constexpr int THREADS = 32 * (EPIW + 2);
};
#define OZ_WIDE 64, 16, 3, 2, 1
#define OZ_NARROW 32, 8, 2, 1, 2
// 128 x 16 tiles for products of at most 16 output columns (the Gauss-Jordan leaf updates):
// half the epilogue of a 128 x 32 tile whose other half would be discarded
#define OZ_NARROW16 16, 8, 2, 1, 2

// device scratch of one owner (an instance, or a temporary context): slices and
// exponent fields of one batch chunk
struct OzBuf {
    uint8_t* base = nullptr;
    size_t bytes = 0;
    bool small_fma = false;        // products of small work run on the FP64 pipe (small_product)
};

// K-major operand rows as seen by the slicer: element (r, k) of op(X) is
// X[b][off + r * ld + k] (strided = 0) or X[b][off + k * ld + r] (strided = 1),
// plus s2 times the same element of X2 when X2 is given
struct OzOperand {
    const double* const* X;
    const double* const* X2;
    double s2;
    long long off;
    int ld, strided;
    int rows, k;              // K-major rows and K
    int rows_pad, kp;         // padded rows (a multiple of the tile) and row pitch (a multiple of 8)
    int b0;                   // first batch entry of the chunk
    const int* active; int active_cmp;
    int* expo;                // [chunk][rows_pad] exponent fields
    uint16_t* slices;         // [chunk][OZ_S][rows_pad][kp] bf16 digits (planes)
    int interleave;           // 1: slice i in plane oz_plane(i) (A operands), 0: plane i (B operands)
    int rb;                   // rows of a block (oz_block_slice_kernel)
};



// element (r, k) of op(X) as its bit pattern (plus s2 times the same element of X2, the one
// FP64 operation of the slicers)
__device__ __forceinline__ unsigned long long oz_load(const OzOperand& o, const double* x, const double* x2, int r,
                                                      int k) {
    const long long off = o.strided ? (long long)k * o.ld + r : (long long)r * o.ld + k;
    if (x2) return (unsigned long long)__double_as_longlong(fma(o.s2, x2[off], x[off]));
    return reinterpret_cast<const unsigned long long*>(x)[off];
}

__device__ __forceinline__ bool oz_active(const int* flag, int cmp, int b) {
    return flag == nullptr || flag[b] > cmp;
}



// the eight planes of four consecutive k of row r starting at k (k + 3 < kp; entries at or
// beyond o.k are zero digits, which the tensor map never reads): per plane one 8-byte word
// of four bf16, the high halves of the digits' floats
__device__ __forceinline__ void oz_store4(const OzOperand& o, int bl, int r, int k, const unsigned long long (&v)[4],
                                          int E) {
    float f[4][OZ_S];
#pragma unroll
    for (int u = 0; u < 4; u++) {
        if (E > 0 && k + u < o.k) oz_digit_floats(v[u], E, f[u]);
        else {
#pragma unroll
            for (int i = 0; i < OZ_S; i++) f[u][i] = 0.0f;
        }
    }
#pragma unroll
    for (int i = 0; i < OZ_S; i++) {
        const int pl = o.interleave ? oz_plane(i) : i;
        const unsigned lo = __byte_perm(__float_as_uint(f[0][i]), __float_as_uint(f[1][i]), 0x7632);
        const unsigned hi = __byte_perm(__float_as_uint(f[2][i]), __float_as_uint(f[3][i]), 0x7632);
        *reinterpret_cast<unsigned long long*>(o.slices + (((size_t)bl * OZ_S + pl) * o.rows_pad + r) * o.kp + k) =
            (unsigned long long)lo | ((unsigned long long)hi << 32);
    }
}

// Rows of a block of the one-pass slicer: rb K-major rows of kp doubles in shared memory
// (at most OZ_BLK_BYTES), rb a power of two in 16 .. 128
#define OZ_BLK_BYTES (68 * 1024)
__host__ __device__ __forceinline__ int oz_block_rows(int kp) {
    int rb = 128;
    while (rb > 16 && (size_t)rb * (kp + 1) * 8 > OZ_BLK_BYTES) rb >>= 1;
    return rb;
}

// Slices of an operand whose K-major rows are strided, or contiguous and short (K <= 512):
// a block takes rb rows whole into shared memory (loads coalesced along r for a strided
// operand, along k for a contiguous one), reduces every row's exponent field there and writes
// the digits, one pass over the operand; rows in [rows, rows_pad) get zero digits
__global__ void __launch_bounds__(256) oz_block_slice_kernel(OzOperand o) {
    extern __shared__ unsigned long long oz_blk[];
    __shared__ int s_e[128];
    const int bl = blockIdx.y, b = o.b0 + bl;
    if (!oz_active(o.active, o.active_cmp, b)) return;
    const double* x = o.X[b] + o.off;
    const double* x2 = o.X2 ? o.X2[b] + o.off : nullptr;
    const int kp = o.kp, ts = kp + 1, rb = o.rb, r0 = blockIdx.x * rb;
    const int total = rb * kp;
    if (o.strided) {
        // element idx: k = idx / rb, row idx % rb (rb consecutive doubles of one k)
        const int sh = __ffs(rb) - 1;
#pragma unroll 8
        for (int idx = threadIdx.x; idx < total; idx += 256) {
            const int k = idx >> sh, rr = idx & (rb - 1), r = r0 + rr;
            oz_blk[rr * ts + k] = (r < o.rows && k < o.k) ? oz_load(o, x, x2, r, k) : 0ull;
        }
    } else {
        // element idx: row idx / kp, k = idx % kp, stepped without divisions
        const int dr = 256 / kp, dk = 256 - dr * kp;
        int rr = threadIdx.x / kp, k = threadIdx.x - rr * kp;
#pragma unroll 8
        for (int idx = threadIdx.x; idx < total; idx += 256) {
            const int r = r0 + rr;
            oz_blk[rr * ts + k] = (r < o.rows && k < o.k) ? oz_load(o, x, x2, r, k) : 0ull;
            rr += dr;
            k += dk;
            if (k >= kp) { k -= kp; rr++; }
        }
    }
    __syncthreads();
    {   // exponent fields: 256 / rb consecutive threads per row, reduced by shuffles
        const int tpr = 256 / rb, rr = threadIdx.x / tpr, q = threadIdx.x - rr * tpr, r = r0 + rr;
        int e = 0;
        for (int k = q; k < o.k; k += tpr) e = max(e, oz_expo_field(oz_blk[rr * ts + k]));
        for (int w = tpr >> 1; w > 0; w >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, w));
        if (q == 0) {
            s_e[rr] = r < o.rows ? e : 0;
            if (r < o.rows) o.expo[(size_t)bl * o.rows_pad + r] = e;
        }
    }
    __syncthreads();
    // digits, four consecutive k per step (kp is a multiple of 8)
    const int cpr = kp >> 2;
    const int dr = 256 / cpr, dc = 256 - dr * cpr;
    int rr = threadIdx.x / cpr, c = threadIdx.x - rr * cpr;
    for (int idx = threadIdx.x; idx < rb * cpr; idx += 256) {
        const int r = r0 + rr, k = 4 * c;
        if (r < o.rows_pad) {
            const unsigned long long* t = oz_blk + rr * ts + k;
            const unsigned long long v[4] = {t[0], t[1], t[2], t[3]};
            oz_store4(o, bl, r, k, v, s_e[rr]);
        }
        rr += dr;
        c += dc;
        if (c >= cpr) { c -= cpr; rr++; }
    }
}

// four doubles' bits at a 32-byte boundary, as one access
__device__ __forceinline__ void oz_ld4(unsigned long long (&x)[4], const double* p) {
    asm volatile("ld.global.v4.b64 {%0,%1,%2,%3}, [%4];" : "=l"(x[0]), "=l"(x[1]), "=l"(x[2]), "=l"(x[3]) : "l"(p));
}
__device__ __forceinline__ void oz_st4(unsigned long long* p, const unsigned long long (&x)[4]) {
    asm volatile("st.global.v4.b64 [%0], {%1,%2,%3,%4};" :: "l"(p), "l"(x[0]), "l"(x[1]), "l"(x[2]), "l"(x[3]) : "memory");
}

// contiguous rows (K <= 128 S): one warp per row takes the row into registers, reduces the
// exponent field and writes the digits, four k per lane per step (one pass over the operand)
// Bound by memory: 496 operands of 512^2 (3.1 GB) 636 us with 8-byte loads at a stride of 32, 517 with 32-byte ones.
template <int S>
__global__ void __launch_bounds__(256) oz_row_slice_kernel(OzOperand o) {
    const int bl = blockIdx.y, b = o.b0 + bl;
    if (!oz_active(o.active, o.active_cmp, b)) return;
    const int r = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (r >= o.rows_pad) return;
    const double* x = o.X[b] + o.off;
    const double* x2 = o.X2 ? o.X2[b] + o.off : nullptr;
    unsigned long long v[S][4];          // k = 4 lane + 128 s + u
    const bool wide = (((uintptr_t)x | (uintptr_t)x2 | ((uintptr_t)o.ld * 8)) & 31) == 0;      // rows on 32 bytes
#pragma unroll
    for (int s = 0; s < S; s++) {
        const int k = 128 * s + 4 * lane;
        if (wide && r < o.rows && k + 3 < o.k) {
            oz_ld4(v[s], x + (size_t)r * o.ld + k);
        } else {
#pragma unroll
            for (int u = 0; u < 4; u++)
                v[s][u] = (r < o.rows && k + u < o.k) ? oz_load(o, x, x2, r, k + u) : 0ull;
        }
    }
    if (wide && x2) {
#pragma unroll
        for (int s = 0; s < S; s++) {
            const int k = 128 * s + 4 * lane;
            if (r < o.rows && k + 3 < o.k) {
                unsigned long long w[4];
                oz_ld4(w, x2 + (size_t)r * o.ld + k);
#pragma unroll
                for (int u = 0; u < 4; u++)
                    v[s][u] = (unsigned long long)__double_as_longlong(
                        fma(o.s2, __longlong_as_double((long long)w[u]), __longlong_as_double((long long)v[s][u])));
            }
        }
    }
    int e = 0;
#pragma unroll
    for (int s = 0; s < S; s++)
#pragma unroll
        for (int u = 0; u < 4; u++) e = max(e, oz_expo_field(v[s][u]));
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0 && r < o.rows) o.expo[(size_t)bl * o.rows_pad + r] = e;
#pragma unroll
    for (int s = 0; s < S; s++) {
        const int k = 128 * s + 4 * lane;
        if (k < o.kp) oz_store4(o, bl, r, k, v[s], r < o.rows ? e : 0);
    }
}

struct OzGemm {
    CUtensorMap ta, tb;       // slices: 3-D [chunk * 8][rows_pad][k] bf16, box 64 x rows x 1
    GemmBatch g;              // sizes, output and epilogue fields (batch index = b0 + local)
    int b0;
    int tiles, total;         // tiles per batch entry and of the launch
    int m_pad, n_pad;
    const int* ea; const int* eb;
    int* err;
    int alpha_pow2;           // alpha = +-2^alpha_e (no per-batch factor): folded into the exponent
    int alpha_e, alpha_neg;
};

__device__ __forceinline__ void oz_tma_load(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
                 :: "r"(dst), "l"(map), "r"(x), "r"(y), "r"(z), "r"(bar) : "memory");
}

// The eight group sums (integers held exactly in fp32, or rounded to even integers for
// the two lowest groups) of output column j, combined exactly into V = H 2^28 + L with
// 0 <= L < 2^28: hi = sum_{G<4} v_G 2^(7 (3 - G)) and lo = sum_{G>=4} v_G 2^(7 (7 - G))
// (|hi|, |lo| < 2^46, each a chain of 32 x 32 -> 64-bit multiply-adds), V = hi 2^28 + lo,
// H = hi + floor(lo / 2^28), L = lo mod 2^28.
__device__ __forceinline__ void oz_combine(const uint32_t (&u)[OZ_G][4], int j, long long& H, unsigned& L) {
    int v[OZ_G];
#pragma unroll
    for (int G = 0; G < OZ_G; G++) v[G] = __float2int_rn(__uint_as_float(u[G][j]));
    const long long hi = (long long)v[0] * (1 << 21) + (long long)v[1] * (1 << 14) + (long long)v[2] * 128 + v[3];
    const long long lo = (long long)v[4] * (1 << 21) + (long long)v[5] * (1 << 14) + (long long)v[6] * 128 + v[7];
    H = hi + (lo >> 28);
    L = (unsigned)lo & 0xFFFFFFFu;
}
// The bit pattern of (-1)^neg V 2^e as a double, V = H 2^28 + L (|H| < 2^47, 0 <= L < 2^28), rounded once to
// 53 bits (to nearest, ties to even) in integer arithmetic: |V| = Hm 2^28 + Lm is
// left-justified into one 64-bit word N (bits shifted out are kept as a sticky flag), N is
// rounded at its bit 11, and the biased exponent is added onto the rounded significand (a
// carry out of the significand moves into the exponent by itself).  Results beyond the
// normal range become infinities, and below it subnormals (q rounded once more).  The code
// is straight-line: both justifications of N (|V| of more or fewer than 64 bits), the case
// |V| < 2^28 and the range ends are computed with shift amounts kept in range and selected,
// with no branch and no FP64 instruction, so that the eight columns a thread combines
// interleave.
__device__ __forceinline__ unsigned long long oz_to_double_bits(long long H, unsigned L, int e, bool neg) {
    const bool sv = H < 0;
    const unsigned long long Hm = sv ? (unsigned long long)(L ? ~H : -H) : (unsigned long long)H;
    const unsigned Lm = sv ? ((0x10000000u - L) & 0xFFFFFFFu) : L;
    // |V| >= 2^28: from Hm's leading bit (lzh in 17 .. 63)
    const int lzh = __clzll((long long)Hm) & 63;               // Hm = 0: 0, and unused
    const bool right = lzh < 28;                               // Lm loses 28 - lzh bits
    const unsigned long long low = right ? (unsigned long long)(Lm >> (right ? 28 - lzh : 0))
                                         : (unsigned long long)Lm << (right ? 0 : lzh - 28);
    const unsigned long long NH = (Hm << lzh) | low;
    const unsigned stH = right ? (Lm << ((lzh + 4) & 31)) : 0u;
    // |V| < 2^28: from Lm's
    const int lzl = __clz((int)Lm);                            // Lm = 0: 32 (V = 0, handled below)
    const unsigned long long NL = (unsigned long long)Lm << ((lzl + 32) & 63);
    const bool hz = Hm == 0ull;
    const unsigned long long N = hz ? NL : NH;
    const unsigned sticky = hz ? 0u : stH;
    const int P = hz ? 31 - lzl : 91 - lzh;                    // leading bit of |V|
    unsigned long long q = N >> 11;
    const unsigned rest = (unsigned)(N & 0x3FFull) | sticky;
    q += ((N >> 10) & 1ull) & ((rest != 0u ? 1ull : 0ull) | (q & 1ull));
    const int be = P + e + 1023;
    const unsigned long long sbit = (unsigned long long)(sv != neg) << 63;
    unsigned long long bits = sbit + ((unsigned long long)(be - 1) << 52) + q;   // be <= 2046: a carry out of
    bits = be > 2046 ? (sbit | 0x7FF0000000000000ull) : bits;                  // q overflows to infinity
    // subnormal: q 2^(be - 1) in units of 2^-1074, q rounded once more to nearest even
    const int sh = min(max(1 - be, 1), 63);
    const unsigned long long ms = q >> sh, rem = q & ((1ull << sh) - 1ull), half = 1ull << (sh - 1);
    const unsigned long long msub = (1 - be < 64) ? ms + ((rem > half || (rem == half && (ms & 1ull))) ? 1ull : 0ull)
                                                  : 0ull;
    bits = be < 1 ? (sbit | msub) : bits;                      // msub = 2^52: the smallest normal, exactly
    return (Hm | Lm) ? bits : 0ull;
}

// oz_to_double_bits where the result is known to be a normal number (biased exponent P + e + 1023 in
// 1 .. 2046 for every leading-bit position P of |V| that can occur, 0 .. 74): the same bits, without
// the selects of the range ends
__device__ __forceinline__ unsigned long long oz_to_double_bits_normal(long long H, unsigned L, int e, bool neg) {
    const bool sv = H < 0;
    const unsigned long long Hm = sv ? (unsigned long long)(L ? ~H : -H) : (unsigned long long)H;
    const unsigned Lm = sv ? ((0x10000000u - L) & 0xFFFFFFFu) : L;
    const int lzh = __clzll((long long)Hm) & 63;
    const bool right = lzh < 28;
    const unsigned long long low = right ? (unsigned long long)(Lm >> (right ? 28 - lzh : 0))
                                         : (unsigned long long)Lm << (right ? 0 : lzh - 28);
    const unsigned long long NH = (Hm << lzh) | low;
    const unsigned stH = right ? (Lm << ((lzh + 4) & 31)) : 0u;
    const int lzl = __clz((int)Lm);
    const unsigned long long NL = (unsigned long long)Lm << ((lzl + 32) & 63);
    const bool hz = Hm == 0ull;
    const unsigned long long N = hz ? NL : NH;
    const unsigned sticky = hz ? 0u : stH;
    const int P = hz ? 31 - lzl : 91 - lzh;
    unsigned long long q = N >> 11;
    const unsigned rest = (unsigned)(N & 0x3FFull) | sticky;
    q += ((N >> 10) & 1ull) & ((rest != 0u ? 1ull : 0ull) | (q & 1ull));
    const unsigned long long sbit = (unsigned long long)(sv != neg) << 63;
    const unsigned long long bits = sbit + ((unsigned long long)(P + e + 1022) << 52) + q;
    return (Hm | Lm) ? bits : 0ull;
}

// Output tile x of a batch entry: tile row tm (128 rows) and tile column tn (BN columns); an antisymmetric
// result has the tiles that hold an element on or below the diagonal
template <int BN>
__device__ __forceinline__ void oz_tile(const GemmBatch& g, int x, int& m0, int& n0) {
    const int tnn = (g.n + BN - 1) / BN;
    int tm = 0, tn = x;
    if (g.mode == GEMM_SKEW) {
        for (int cnt; tn >= (cnt = min((tm + 1) * (OZ_BM / BN), tnn)); tm++) tn -= cnt;
    } else {
        tm = x / tnn;
        tn = x - tm * tnn;
    }
    m0 = tm * OZ_BM;
    n0 = tn * BN;
}

template <int BN, int EPIW, int RING, int BBUF, int CTAS>
__global__ void __launch_bounds__(32 * (EPIW + 2), CTAS) oz_gemm_kernel(const __grid_constant__ OzGemm p) {
    constexpr int SLAB_B = BN * 128, NU = OZ_S / OZ_UNIT;
    constexpr bool HOLD = CTAS == 1;             // a tile's sums are taken to registers before they are rounded
    constexpr uint32_t TCOLS = 8u * BN;          // TMEM columns: eight groups of BN
    extern __shared__ uint8_t oz_smem_raw[];
    __shared__ uint64_t bfull[BBUF], bempty[BBUF], afull[RING], aempty[RING], tfull, tempty, done;
    __shared__ uint32_t tmem_base;
    __shared__ int skip, abort_flag;

    const GemmBatch& g = p.g;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int t0 = blockIdx.x, t1 = p.total, dt = gridDim.x;
    // tile t's batch entry, whether it computes, and (inactive entries left alone) whether it does anything
    auto entry = [&](int t) { return p.b0 + t / p.tiles; };
    auto is_active = [&](int t) { return oz_active(g.active_flag, g.active_cmp, entry(t)); };
    if (g.skip_inactive) {
        bool any = false;
        for (int t = t0; t < t1; t += dt) any = any || is_active(t);
        if (!any) return;
    }
    if (tid == 0) skip = (*(volatile int*)p.err & SGS_DEV_TC_TIMEOUT) != 0;
    __syncthreads();
    if (skip) return;
    const int nslab = (g.k + OZ_KS - 1) / OZ_KS;      // k <= OZ_KC (the host splits K)

    const uint32_t raw = smem_u32(oz_smem_raw);
    const uint32_t sbase = (raw + 1023u) & ~1023u;
    auto sA = [&](int slot) { return sbase + (uint32_t)BBUF * OZ_S * SLAB_B + (uint32_t)slot * (OZ_UNIT * OZ_SLAB_A); };

    if (warp == EPIW + 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(&tmem_base)), "r"(TCOLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        auto init = [](uint64_t& bar, int count) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(smem_u32(&bar)), "r"(count));
        };
        for (int s = 0; s < BBUF; s++) {
            init(bfull[s], 1);
            init(bempty[s], 1);
        }
        for (int s = 0; s < RING; s++) {
            init(afull[s], 1);
            init(aempty[s], 1);
        }
        init(tfull, 1);
        init(tempty, EPIW);
        init(done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;");
        abort_flag = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = tmem_base;

    // A CTA takes its tiles one after the other: the producer runs ahead into the next tile's slabs as the
    // MMAs release the buffers, and the MMAs of the next tile start when the epilogue warps have drained
    // TMEM, so the loads (and most of the MMAs of the SM's other CTA) run during an epilogue.
    if (warp == EPIW) {
        if (lane == 0) {            // producer
            // one TMA box per B slab (the eight slices, 8 BN rows; one buffer, reloaded once the previous
            // slab's MMAs have released it) and per A unit (two slices, 32 KB)
            int nb = 0, q = 0;      // B slabs and A units issued
            bool ok = true;
            for (int t = t0; t < t1 && ok; t += dt) {
                if (!is_active(t)) continue;
                const int bl = t / p.tiles;
                int m0, n0;
                oz_tile<BN>(g, t - bl * p.tiles, m0, n0);
                for (int s = 0; s < nslab && ok; s++) {
                    const int bb = nb % BBUF;
                    if (nb >= BBUF && !mbar_wait_or_abort(smem_u32(&bempty[bb]), (uint32_t)((nb / BBUF - 1) & 1), p.err)) {
                        ok = false;
                        break;
                    }
                    mbar_expect_tx(smem_u32(&bfull[bb]), (uint32_t)(OZ_S * SLAB_B));
                    oz_tma_load(sbase + (uint32_t)(bb * OZ_S * SLAB_B), &p.tb, s * OZ_KS, n0, bl * OZ_S, smem_u32(&bfull[bb]));
                    nb++;
                    for (int u = 0; u < NU; u++) {
                        const int slot = q % RING;
                        if (q >= RING &&
                            !mbar_wait_or_abort(smem_u32(&aempty[slot]), (uint32_t)(((q / RING) - 1) & 1), p.err)) {
                            ok = false;
                            break;
                        }
                        mbar_expect_tx(smem_u32(&afull[slot]), (uint32_t)(OZ_UNIT * OZ_SLAB_A));
                        oz_tma_load(sA(slot), &p.ta, s * OZ_KS, m0, bl * OZ_S + OZ_UNIT * u, smem_u32(&afull[slot]));
                        q++;
                    }
                    if (*(volatile int*)&abort_flag) ok = false;
                }
            }
            if (!ok) abort_flag = 1;
            // every load issued has landed before the CTA can leave
            for (int x = (nb > BBUF ? nb - BBUF : 0); x < nb; x++)
                mbar_wait(smem_u32(&bfull[x % BBUF]), (uint32_t)((x / BBUF) & 1), p.err);
            for (int x = (q > RING ? q - RING : 0); x < q; x++)
                mbar_wait(smem_u32(&afull[x % RING]), (uint32_t)((x / RING) & 1), p.err);
        }
    } else if (warp == EPIW + 1) {
        // MMA issuer: the whole warp runs the loop converged and one lane issues.  Issued behind a branch on the
        // lane an MMA took 177 clocks (its operands moved to uniform registers one by one), more than the 144 its
        // tensor work averages for the two CTAs of an SM.
        constexpr int MAXB = 256 / BN;             // B slices per MMA (N <= 256)
        const uint32_t el = tc_elect(), tm = __shfl_sync(0xffffffffu, tmem, 0);
        // descriptors of slot 0 / slice 0; other slots and slices offset the 16-byte address field
        const uint64_t dA0 = tma_smem_desc(sA(0)), dB0 = tma_smem_desc(sbase);
        auto wait = [&](uint64_t& bar, int phase) {
            return __all_sync(0xffffffffu, mbar_wait_or_abort(smem_u32(&bar), (uint32_t)(phase & 1), p.err)) != 0;
        };
        int nb = 0, q = 0, nt = 0;                 // slabs, units and tiles taken
        bool ok = true;
        for (int t = t0; t < t1 && ok; t += dt) {
            if (!__any_sync(0xffffffffu, is_active(t))) continue;
            if (nt > 0 && !wait(tempty, nt - 1)) { ok = false; break; }       // the accumulators have been drained
            nt++;
            for (int s = 0; s < nslab && ok; s++, nb++) {
                const int bb = nb % BBUF;
                if (!wait(bfull[bb], nb / BBUF)) { ok = false; break; }
                const int nk16 = (min(OZ_KS, g.k - s * OZ_KS) + 15) / 16;
                const uint64_t db = dB0 + (uint64_t)((bb * OZ_S * SLAB_B) >> 4);
#pragma unroll
                for (int u = 0; u < NU; u++, q++) {
                    const int slot = q % RING;
                    if (!wait(afull[slot], q / RING)) { ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
                    for (int h = 0; h < OZ_UNIT; h++) {
                        const int i = oz_order(OZ_UNIT * u + h);
                        const uint64_t da = dA0 + (uint64_t)(((slot * OZ_UNIT + h) * OZ_SLAB_A) >> 4);
                        // the first slice (i = 0, taken first) opens every group's accumulator
                        const bool open = s == 0 && u == 0 && h == 0;
                        // products (i, j), j = 0 .. 7 - i, land in groups i .. 7: adjacent BN-column
                        // accumulators, and the B slices j are adjacent BN-row blocks in shared
                        // memory, so one MMA of N = BN (8 - i) covers them; more than 256 columns
                        // are two MMAs of about half the slices each
                        const int n1 = OZ_S - i <= MAXB ? OZ_S - i : (OZ_S - i + 1) / 2, n2 = OZ_S - i - n1;
                        const uint32_t acc = tm + (uint32_t)(i * BN);
#pragma unroll
                        for (int kk = 0; kk < OZ_KS / 16; kk++) {
                            if (kk >= nk16) break;
                            const uint32_t on = open && kk == 0 ? 0u : 1u;
                            tc_mma_bf16_elect(acc, da + 2 * kk, db + 2 * kk, tc_idesc(TC_BF16, BN * n1), on, el);
                            if (n2 > 0)
                                tc_mma_bf16_elect(acc + (uint32_t)(n1 * BN), da + 2 * kk,
                                                  db + (uint64_t)((n1 * SLAB_B) >> 4) + 2 * kk,
                                                  tc_idesc(TC_BF16, BN * n2), on, el);
                        }
                    }
                    tc_commit_elect(smem_u32(&aempty[slot]), el);
                }
                if (!ok) break;
                tc_commit_elect(smem_u32(&bempty[bb]), el);
                if (s == nslab - 1) tc_commit_elect(smem_u32(&tfull), el);
                if (__any_sync(0xffffffffu, *(volatile int*)&abort_flag)) ok = false;
            }
        }
        if (!ok && lane == 0) abort_flag = 1;
        // every MMA issued has completed before TMEM is freed
        tc_commit_elect(smem_u32(&done), el);
        mbar_wait(smem_u32(&done), 0u, p.err);
        __syncwarp();
    } else {
        // epilogue: warps 0 .. EPIW - 1.  Warp w has TMEM lanes 32 (w % 4) .. 32 (w % 4) + 31, an output row per
        // thread, and the columns of part w / 4, four at a time: a sector of the row.  Results go from the
        // registers to memory: a row's four columns are one 32-byte access per lane, the mirrored block of an
        // antisymmetric result and a transposed Cin run along the lanes.  Every element is read and written by
        // the one thread that computes it (Cin may be C itself).
        constexpr int PCOLS = BN / (EPIW / 4), PASSES = PCOLS / 4;
        static_assert(PCOLS % 4 == 0, "four-column passes");
        const int lq = warp & 3, part = warp >> 2;          // lane quarter, column part
        int nt = 0;                                         // tiles drained
        bool ok = true;
        for (int t = t0; t < t1 && ok; t += dt) {
        const bool active = is_active(t);
        if (!active && g.skip_inactive) continue;
        const int bl = t / p.tiles, b = p.b0 + bl;
        int m0, n0;
        oz_tile<BN>(g, t - bl * p.tiles, m0, n0);
        const double* Cinb = g.Cin ? g.Cin[b] + g.offCin : nullptr;
        const double* Cin2b = g.Cin2 ? g.Cin2[b] + g.offCin : nullptr;
        double* Cb = g.C[b] + g.offC;
        const bool skew = g.mode == GEMM_SKEW, gj = g.mode == GEMM_GJ;
        const int row = m0 + lq * 32 + lane, cp0 = n0 + part * PCOLS;
        const bool use_cin = Cinb && (!active || g.beta != 0.0);
        const bool ct = g.cin_trans != 0;
        // in-place update: C = Cin + A B, or the sign of a transposed Cin flipped by an integer XOR; a
        // Gauss-Jordan update's pivot rows take the product alone
        const bool cin_neg = active && ct && g.beta == -1.0;
        const bool plain = active && p.alpha_pow2 && !Cin2b && (!use_cin || g.beta == 1.0 || cin_neg);
        const bool drop_cin = active && gj && !g.gj_acc && row >= g.gj_k0 && row < g.gj_k0 + g.gj_b;
        const unsigned long long cin_sign = cin_neg ? 0x8000000000000000ull : 0ull;
        // 32-byte (or 16-byte) accesses along the rows where every row starts on one
        auto align_of = [&](const double* x, int ld) {
            const uintptr_t a = reinterpret_cast<uintptr_t>(x + cp0) | ((uintptr_t)ld * 8);
            return (a & 31) == 0 ? 32 : (a & 15) == 0 ? 16 : 8;
        };
        const int al_in = use_cin && !ct ? align_of(Cinb, g.ldcin) : 8, al_out = align_of(Cb, g.ldc);
        // Cin's four elements of columns c .. c + 3 of this row
        auto load_cin = [&](unsigned long long (&x)[4], int c) {
            if (!use_cin || drop_cin || row >= g.m || (skew && row < c)) {
                x[0] = x[1] = x[2] = x[3] = 0ull;
                return;
            }
            const double* s = Cinb + (ct ? (long long)c * g.ldcin + row : (long long)row * g.ldcin + c);
            if (al_in == 32 && c + 3 < g.n) {
                oz_ld4(x, s);
            } else if (al_in == 16 && c + 3 < g.n) {
                const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(s), d = *reinterpret_cast<const ulonglong2*>(s + 2);
                x[0] = a.x; x[1] = a.y; x[2] = d.x; x[3] = d.y;
            } else {
#pragma unroll
                for (int j = 0; j < 4; j++)
                    x[j] = c + j < g.n ? reinterpret_cast<const unsigned long long*>(s)[ct ? (long long)j * g.ldcin : j] : 0ull;
            }
        };
        unsigned long long ci[4], cn[4];
        load_cin(ci, cp0);                                   // in flight while the MMAs run
        const int er = (active && row < g.m) ? p.ea[(size_t)bl * p.m_pad + row] : 0;
        // the exponent fields of this part's columns, one per lane
        const int fe = (active && lane < PCOLS && cp0 + lane < g.n) ? p.eb[(size_t)bl * p.n_pad + cp0 + lane] : 0;
        if (active) {
            if (lane == 0) ok = mbar_wait_or_abort(smem_u32(&tfull), (uint32_t)(nt & 1), p.err);
            ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
            nt++;
        }
        if (ok) {
            asm volatile("tcgen05.fence::after_thread_sync;");
            const double alpha = g.alpha * (g.alpha_b ? g.alpha_b[b] : 1.0);
            const int ae = p.alpha_pow2 ? p.alpha_e : 0;
            const bool an = p.alpha_pow2 && p.alpha_neg;
            // every result of this warp's rows is a normal number: with e = er + fc - 2107 + ae and
            // the leading bit P of |V| in 0 .. 74, the biased exponent P + e + 1023 stays in 1 .. 2046
            // (rows or columns with a zero exponent field give zeros either way); then the
            // combination takes the form without the range-end selects (the same bits)
            const int fcmin = __reduce_min_sync(0xffffffffu, fe > 0 ? fe : 4096);
            const int fcmax = __reduce_max_sync(0xffffffffu, fe);
            const bool row_normal = er == 0 || fcmax == 0 ||
                                    (er + fcmin - 2107 + ae + 1023 >= 1 && er + fcmax - 2107 + ae + 1023 + 74 <= 2046);
            const bool fast = __all_sync(0xffffffffu, row_normal);
            // this warp has read its accumulators: the next tile's MMAs may start
            bool held = active;
            auto release = [&] {
                held = false;
                asm volatile("tcgen05.fence::before_thread_sync;");
                __syncwarp();
                if (lane == 0)
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(smem_u32(&tempty)) : "memory");
            };
            // the group sums of columns cl .. cl + 3 of this thread's row
            auto load_sums = [&](uint32_t (&u)[OZ_G][4], int cl) {
#pragma unroll
                for (int G = 0; G < OZ_G; G++) {
                    const uint32_t ta = tmem + ((uint32_t)(lq * 32) << 16) + (uint32_t)(G * BN + cl);
                    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                                 : "=r"(u[G][0]), "=r"(u[G][1]), "=r"(u[G][2]), "=r"(u[G][3])
                                 : "r"(ta));
                }
            };
            // columns c0 .. c0 + 3 and on have no element of this warp's rows (warp-uniform)
            auto beyond = [&](int c0) { return c0 >= g.n || (skew && m0 + lq * 32 + 31 < c0); };
            // one CTA per SM: the sums of all columns first, so that the next tile's MMAs run during the rounding
            // and the stores (the pass loop below takes entries 0 .. 3 and moves the others down)
            long long hh[HOLD ? PCOLS : 4];
            unsigned hl[HOLD ? PCOLS : 4];
            if constexpr (HOLD) {
                if (active) {
#pragma unroll
                    for (int pass = 0; pass < PASSES; pass++) {
                        const int cl = part * PCOLS + 4 * pass;
                        if (!beyond(n0 + cl)) {
                            uint32_t u[OZ_G][4];
                            load_sums(u, cl);
                            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                            for (int j = 0; j < 4; j++) oz_combine(u, j, hh[4 * pass + j], hl[4 * pass + j]);
                        }
                    }
                    release();
                }
            }
#pragma unroll 1
            for (int pass = 0; pass < PASSES; pass++) {
                const int cl = part * PCOLS + 4 * pass, c0 = n0 + cl;
                if (beyond(c0)) break;
                unsigned long long t[4] = {0ull, 0ull, 0ull, 0ull};
                if (active) {
                    uint32_t u[OZ_G][4];
                    if constexpr (!HOLD) load_sums(u, cl);
                    if (pass + 1 < PASSES) load_cin(cn, c0 + 4);
                    if constexpr (!HOLD) {
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                        if (pass == PASSES - 1) release();
#pragma unroll
                        for (int j = 0; j < 4; j++) oz_combine(u, j, hh[j], hl[j]);
                    }
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        // computed for every column and selected (no branch between the columns)
                        const int fc = __shfl_sync(0xffffffffu, fe, 4 * pass + j);
                        const unsigned long long v = fast ? oz_to_double_bits_normal(hh[j], hl[j], er + fc - 2107 + ae, an)
                                                          : oz_to_double_bits(hh[j], hl[j], er + fc - 2107 + ae, an);
                        t[j] = (er > 0 && fc > 0) ? v : 0ull;
                    }
                    if constexpr (HOLD) {
#pragma unroll
                        for (int j = 0; j + 4 < PCOLS; j++) {
                            hh[j] = hh[j + 4];
                            hl[j] = hl[j + 4];
                        }
                    }
                } else if (pass + 1 < PASSES) {
                    load_cin(cn, c0 + 4);
                }
                // The common forms issue no FP64 instruction beyond the one addition an update needs (FP64
                // issues at a small fraction of the integer rate on this part)
                if (plain) {
                    if (use_cin && !drop_cin) {
#pragma unroll
                        for (int j = 0; j < 4; j++)
                            t[j] = (unsigned long long)__double_as_longlong(
                                __longlong_as_double((long long)(ci[j] ^ cin_sign)) + __longlong_as_double((long long)t[j]));
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        double v = 0.0;
                        if (use_cin && !drop_cin) {
                            v = __longlong_as_double((long long)ci[j]);
                            if (active && g.beta != 1.0) v *= g.beta;
                        }
                        if (active) {
                            if (Cin2b && row < g.m && c0 + j < g.n)
                                v = fma(g.beta2, Cin2b[(long long)row * g.ldcin + c0 + j], v);
                            double x = __longlong_as_double((long long)t[j]);
                            if (!p.alpha_pow2) x *= alpha;
                            v += x;
                        }
                        t[j] = (unsigned long long)__double_as_longlong(v);
                    }
                }
                if (active && g.diag != 0.0 && !skew && __any_sync(0xffffffffu, row >= c0 && row < c0 + 4)) {
#pragma unroll
                    for (int j = 0; j < 4; j++)
                        if (row == c0 + j)
                            t[j] = (unsigned long long)__double_as_longlong(__longlong_as_double((long long)t[j]) + g.diag);
                }
                if (row < g.m) {
                    unsigned long long* d = reinterpret_cast<unsigned long long*>(Cb + (long long)row * g.ldc + c0);
                    const bool panel = gj && g.gj_cols;       // columns gj_k0 .. gj_k0 + gj_b - 1 are not written
                    if (!panel && c0 + 3 < g.n && (!skew || row > c0 + 3)) {
                        if (al_out == 32) oz_st4(d, t);
                        else if (al_out == 16) {
                            reinterpret_cast<ulonglong2*>(d)[0] = make_ulonglong2(t[0], t[1]);
                            reinterpret_cast<ulonglong2*>(d)[1] = make_ulonglong2(t[2], t[3]);
                        } else {
#pragma unroll
                            for (int j = 0; j < 4; j++) d[j] = t[j];
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < 4; j++) {
                            const int c = c0 + j;
                            if (c >= g.n || (skew && row < c) || (panel && c >= g.gj_k0 && c < g.gj_k0 + g.gj_b)) continue;
                            d[j] = (skew && row == c) ? 0ull : t[j];
                        }
                    }
                    if (skew) {                               // mirrored block: C[c][r] = -C[r][c] below the diagonal
#pragma unroll
                        for (int j = 0; j < 4; j++)
                            if (c0 + j < g.n && row > c0 + j)
                                reinterpret_cast<unsigned long long*>(Cb)[(long long)(c0 + j) * g.ldc + row] =
                                    t[j] ^ 0x8000000000000000ull;
                    }
                }
#pragma unroll
                for (int j = 0; j < 4; j++) ci[j] = cn[j];
            }
            if (held) release();
        } else if (lane == 0) {
            abort_flag = 1;
        }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == EPIW + 1) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(TCOLS));
    }
}

// ---------------------------------------------------------------- host side

inline size_t oz_round(size_t x, size_t a) { return (x + a - 1) / a * a; }

// scratch bytes of one batch entry of an m x n x k product (slices and exponent fields)
inline size_t oz_entry_bytes(int m, int n, int k) {
    const size_t kp = oz_round((size_t)k, 8), mp = oz_round((size_t)m, OZ_BM), np = oz_round((size_t)n, 64);
    return (size_t)OZ_S * 2 * (mp + np) * kp + 4 * (mp + np);
}

// Tensor map of a slice batch [nmat][rows_pad][kp] bf16 with x extent k (zero fill beyond),
// box 64 x box_rows x 1 (128-byte rows, 128-byte swizzle)
inline bool make_slice_map(CUtensorMap* map, const void* base, int k, int kp, int rows_pad, int nmat, int box_rows,
                           int box_planes) {
    TmaEncodeFn fn = tma_encode_fn();
    if (!fn || !base || ((uintptr_t)base & 15) || (kp & 7)) return false;
    const cuuint64_t dims[3] = {(cuuint64_t)k, (cuuint64_t)rows_pad, (cuuint64_t)nmat};
    const cuuint64_t strides[2] = {(cuuint64_t)kp * 2, (cuuint64_t)kp * rows_pad * 2};
    const cuuint32_t box[3] = {(cuuint32_t)OZ_KS, (cuuint32_t)box_rows, (cuuint32_t)box_planes};
    const cuuint32_t estr[3] = {1u, 1u, 1u};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// exponents and slices of one operand, one pass: contiguous rows a warp per row in registers, the others
// (strided, or of a few dozen entries) a block of rows at a time through shared memory, with smaller blocks
// (down to the 16 rows of a 128-byte line) where there would be fewer than two per SM.  A 244 x 244 operand of
// 16 states took 13.7 us by blocks of 32 rows.
inline int oz_sms();
inline bool oz_row_pass(const OzOperand& o) { return !o.strided && o.k >= 64 && o.k <= OZ_KC; }
inline size_t oz_block_smem(int rb, int kp) { return (size_t)rb * (kp + 1) * 8; }
inline void oz_prepare(OzOperand o, int bc, cudaStream_t st) {
    if (oz_row_pass(o)) {
        const dim3 grid((o.rows_pad + 7) / 8, bc);
        if (o.k <= 128) oz_row_slice_kernel<1><<<grid, 256, 0, st>>>(o);
        else if (o.k <= 256) oz_row_slice_kernel<2><<<grid, 256, 0, st>>>(o);
        else oz_row_slice_kernel<4><<<grid, 256, 0, st>>>(o);
    } else {
        o.rb = oz_block_rows(o.kp);
        while (o.rb > 16 && (long long)((o.rows_pad + o.rb - 1) / o.rb) * bc < 2 * oz_sms()) o.rb >>= 1;
        oz_block_slice_kernel<<<dim3((o.rows_pad + o.rb - 1) / o.rb, bc), 256, oz_block_smem(o.rb, o.kp), st>>>(o);
    }
}

// number of output tiles of one batch entry (tile width bn)
inline int oz_tiles(const GemmBatch& g, int bn) {
    const int tmn = (g.m + OZ_BM - 1) / OZ_BM, tnn = (g.n + bn - 1) / bn;
    if (g.mode != GEMM_SKEW) return tmn * tnn;
    int t = 0;
    for (int tm = 0; tm < tmn; tm++) t += std::min((tm + 1) * (OZ_BM / bn), tnn);
    return t;
}

// launches of one product, for launch accounting
inline int oz_launches(const GemmBatch& g, const OzBuf& buf) {
    if (g.batch <= 0 || g.m <= 0 || g.n <= 0 || g.k <= 0 || !buf.base) return 1;
    int total = 0;
    for (int k0 = 0; k0 < g.k; k0 += OZ_KC) {
        const size_t per = oz_entry_bytes(g.m, g.n, std::min(OZ_KC, g.k - k0));
        const size_t chunk = std::min<size_t>(g.batch, buf.bytes > 8192 ? (buf.bytes - 8192) / per : 0);
        if (chunk == 0) return 1;
        // per batch chunk: one slicing launch per operand and the product
        total += 3 * (int)((g.batch + chunk - 1) / chunk);
    }
    return total;
}

// where the slices and exponent fields of a batch chunk of bc entries of an m x n x k product
// lie in the scratch: A slices [bc][OZ_S][mp][kp] (planes in oz_plane order), B slices
// [bc][OZ_S][np][kp] (natural order), exponent fields [bc][mp] and [bc][np]
struct OzLayout {
    uint16_t* as;
    uint16_t* bs;
    int* ea;
    int* eb;
    int mp, np, kp;
};
inline OzLayout oz_layout(int m, int n, int k, const OzBuf& buf, int bc) {
    OzLayout L;
    L.kp = (int)oz_round(k, 8);
    L.mp = (int)oz_round(m, OZ_BM);
    L.np = (int)oz_round(n, 64);
    const size_t sa = (size_t)OZ_S * L.mp * L.kp * 2, sb = (size_t)OZ_S * L.np * L.kp * 2;
    L.as = reinterpret_cast<uint16_t*>(buf.base);
    L.bs = reinterpret_cast<uint16_t*>(buf.base + oz_round((size_t)bc * sa, 1024));
    L.ea = reinterpret_cast<int*>(reinterpret_cast<uint8_t*>(L.bs) + oz_round((size_t)bc * sb, 1024));
    L.eb = L.ea + oz_round((size_t)bc * L.mp, 64);
    return L;
}

// batch entries of one K chunk (k <= OZ_KC) whose slices fit the scratch at once
inline int oz_chunk_entries(const GemmBatch& g, const OzBuf& buf) {
    const size_t per = oz_entry_bytes(g.m, g.n, g.k);
    return (int)std::min<size_t>(g.batch, buf.bytes > 8192 ? (buf.bytes - 8192) / per : 0);
}

// SMs of the current device
inline int oz_sms() {
    static std::atomic<int> known[64];
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 1;
    if ((n = known[dev].load(std::memory_order_relaxed)) > 0) return n;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) return 1;
    known[dev].store(n, std::memory_order_relaxed);
    return n;
}

// Tile width of a product: OZ_NARROW16's, OZ_NARROW's, or OZ_WIDE's for long sums with enough tiles that a last
// partial round of whole SMs costs less than the wide tile gains.  Narrow / wide, us: 105 antisymmetric products of
// 804^2 at K = 512 1162 / 945, at 292 1057 / 810; 45 of 388^2 at 388 201 / 164; general 512^2 at K = 512: 160 wide
// tiles 58 / 64, 192 61 / 64, 256 72 / 65, 320 99 / 90.  The two cross where a sum has 15 steps of 16 (K > 224).  190
// pairs' V = D W (general) and X = V D (antisymmetric), n = K, with their slicing:
//   K    160          192          208          224          228          236          240          256
//   V    206 / 228    231 / 235    287 / 288    292 / 291    363 / 315    328 / 296    321 / 294    315 / 291
//   X    201 / 222    222 / 227    261 / 272    266 / 276    319 / 290    289 / 279    286 / 278    282 / 277
// Gauss-Jordan updates at K = 128 (120 of 512 x 128) 96 / 131; at K = 240 (120 of 472 x 232, the whole inverse) 7062 / 7005.
inline int oz_width(const GemmBatch& g, int bc) {
    if (g.n <= 16) return 16;
    return g.k > 224 && (long long)oz_tiles(g, 64) * bc * 2 >= 3 * oz_sms() ? 64 : 32;
}

// the product kernel on slices in place (layout L) for batch entries b0 .. b0 + bc - 1;
// b_rows: B's slices are its rows (an antisymmetric B), so alpha changes sign
inline cudaError_t oz_product(const GemmBatch& g, const OzLayout& L, int b0, int bc, bool b_rows, int* err,
                              cudaStream_t st) {
    const int bn = oz_width(g, bc);
    OzGemm p;
    std::memset(&p, 0, sizeof(p));
    if (!make_slice_map(&p.ta, L.as, g.k, L.kp, L.mp, bc * OZ_S, OZ_BM, OZ_UNIT) ||
        !make_slice_map(&p.tb, L.bs, g.k, L.kp, L.np, bc * OZ_S, bn, OZ_S))
        return cudaErrorInvalidValue;
    p.g = g; p.b0 = b0; p.m_pad = L.mp; p.n_pad = L.np; p.ea = L.ea; p.eb = L.eb; p.err = err;
    if (b_rows) p.g.alpha = -g.alpha;
    int ex = 0;
    const double fr = std::frexp(p.g.alpha, &ex);
    if (!g.alpha_b && (fr == 0.5 || fr == -0.5)) {
        p.alpha_pow2 = 1; p.alpha_e = ex - 1; p.alpha_neg = p.g.alpha < 0.0;
    }
    p.tiles = oz_tiles(g, bn);
    p.total = p.tiles * bc;
    // two CTAs per SM and no more: with a few CTAs over, those few run their tiles after all others
    const unsigned grid = (unsigned)std::min(p.total, (bn == 64 ? 1 : 2) * oz_sms());
    if (bn == 64)
        oz_gemm_kernel<OZ_WIDE><<<grid, OzCfg<OZ_WIDE>::THREADS, OzCfg<OZ_WIDE>::SMEM, st>>>(p);
    else if (bn == 16)
        oz_gemm_kernel<OZ_NARROW16><<<grid, OzCfg<OZ_NARROW16>::THREADS, OzCfg<OZ_NARROW16>::SMEM, st>>>(p);
    else
        oz_gemm_kernel<OZ_NARROW><<<grid, OzCfg<OZ_NARROW>::THREADS, OzCfg<OZ_NARROW>::SMEM, st>>>(p);
    return cudaGetLastError();
}

// one K chunk (k <= OZ_KC) of the emulated product, in batch chunks that fit the scratch
inline cudaError_t gemm_oz_chunk(const GemmBatch& g, const OzBuf& buf, int* err, cudaStream_t st) {
    const int chunk = oz_chunk_entries(g, buf);
    if (chunk <= 0) return gemm_f64(g, st);
    for (int b0 = 0; b0 < g.batch; b0 += chunk) {
        const int bc = std::min(chunk, g.batch - b0);
        const OzLayout L = oz_layout(g.m, g.n, g.k, buf, bc);
        OzOperand oa{g.A, g.A2, g.sA2, g.offA, g.lda, g.transA ? 1 : 0, g.m, g.k, L.mp, L.kp, b0,
                     g.active_flag, g.active_cmp, L.ea, L.as, 1, 0};
        // an antisymmetric B (not transposed): its K-major columns are its rows negated, so the
        // rows are sliced (contiguous, one pass) and alpha changes sign
        const bool b_rows = g.b_antisym && !g.transB;
        OzOperand ob{g.B, g.B2, g.sB2, b_rows ? g.offBr : g.offB, g.ldb, (g.transB || b_rows) ? 0 : 1, g.n, g.k, L.np,
                     L.kp, b0, g.active_flag, g.active_cmp, L.eb, L.bs, 0, 0};
        oz_prepare(oa, bc, st);
        oz_prepare(ob, bc, st);
        const cudaError_t e = oz_product(g, L, b0, bc, b_rows, err, st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// The product on operands a producer kernel has already sliced into buf (layout oz_layout of
// the whole batch): k <= OZ_KC, every entry in one chunk (oz_chunk_entries(g, buf) == batch)
inline cudaError_t gemm_oz_presliced(const GemmBatch& g, const OzBuf& buf, int* err, cudaStream_t st) {
    if (g.batch <= 0 || g.m <= 0 || g.n <= 0) return cudaSuccess;
    if (g.k <= 0 || g.k > OZ_KC || !buf.base || !err || oz_chunk_entries(g, buf) < g.batch ||
        (g.mode == GEMM_SKEW && g.m != g.n))
        return cudaErrorInvalidValue;
    return oz_product(g, oz_layout(g.m, g.n, g.k, buf, g.batch), 0, g.batch, g.b_antisym && !g.transB, err, st);
}

// the emulated product; K beyond OZ_KC runs as further launches that add onto C (the
// chunks' sums are FP64 roundings).  Falls back to gemm_f64 where there is nothing to
// slice or no scratch for one batch entry.  err: the owner's device error word.
inline cudaError_t gemm_oz(const GemmBatch& g, const OzBuf& buf, int* err, cudaStream_t st) {
    if (g.batch <= 0 || g.m <= 0 || g.n <= 0) return cudaSuccess;
    if (g.k <= 0 || !buf.base || !err) return gemm_f64(g, st);
    if (g.mode == GEMM_SKEW && g.m != g.n) return cudaErrorInvalidValue;
    if (oz_entry_bytes(g.m, g.n, std::min(g.k, OZ_KC)) + 8192 > buf.bytes) return gemm_f64(g, st);
    for (int k0 = 0; k0 < g.k; k0 += OZ_KC) {
        GemmBatch h = g;
        h.k = std::min(OZ_KC, g.k - k0);
        h.offA += g.transA ? (long long)k0 * g.lda : k0;
        h.offBr = g.offB + k0;                         // the K range within B's rows (antisymmetric B)
        h.offB += g.transB ? k0 : (long long)k0 * g.ldb;
        if (k0 > 0) {
            h.Cin = (const double* const*)g.C; h.offCin = g.offC; h.ldcin = g.ldc; h.beta = 1.0;
            h.Cin2 = nullptr; h.beta2 = 0.0; h.diag = 0.0;
            h.gj_acc = 1;          // a Gauss-Jordan update's pivot rows hold the first chunk's product now
        }
        const cudaError_t e = gemm_oz_chunk(h, buf, err, st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace sgs
