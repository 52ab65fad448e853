// slices.cuh -- FP64 operands of the Form as exact BF16 digit slices: the format that
// the Solve writes and the tensor-core FP64 Form (form.cu) reads.
//
// S = W21 L21^T in FP64 accuracy on tensor cores that multiply BF16 and add in
// FP32: the error-free splitting of Ozaki, Ogita, Oishi and Rump ("Error-free
// transformations of matrix multiplication by using fast routines of matrix
// multiplication and its applications", 2012), with integer digits.  Every row
// of an operand is scaled by a power of two 2^-E (E: |x| < 2^E over the row)
// to 62-bit integers X, rounded to nearest, and X is written in eight balanced
// base-256 digits, X = sum_s d_s 256^(7-s), |d_0| <= 64, -128 <= d_s <= 127: small
// integers, exact in BF16.  A product of digits is at most 2^14, and a sum over K
// <= 256 pivots of up to four such products (five for the sums that matter at
// 2^-40) stays below 2^24: exact in FP32.
//
// Columns: pivot k scales column k of W21 by d_k against L21, so before the
// rows are scaled W's column k is multiplied by 2^-c_k and L's by 2^c_k with
// 2^c_k about |d_k|^(1/2) (their products are unchanged): both operands then
// look like L |D|^(1/2), whose rows do not mix the scales of the pivots.
//
// Accuracy: cutting X and dropping the digit products with s + t > 7 costs an
// entry of S at most e 2^-59, and rounding the two lowest sums to whole units 2^-(53+f)
// with f = 6, 5, 4, 3, 2 for e <= 16, 32, 64, 128, 256, both times the two rows' scales
// 2^(E_i + E_j): together less than 1.1 e 2^-59 2^(E_i + E_j).  (Past 128 pivots
// the sums of g = 5 are exact only below 2^24; their digits would have to lie within
// a tenth of their extremes in nearly all pivots to pass it.)  FP64
// multiply-adds may lose e 2^-53 (|W21||L21|^T)_ij.  So digits serve an entry as well when
//     P_ij = sum_k |w_ik| |l_jk| / 2^(E_i + E_j) >= 2^-7
// (then they lose less than (2 e + 8) 2^-53 (|W21||L21|^T)_ij at the very most, and
// in the mean what FP64 multiply-adds lose), that is unless the two rows are
// large in different pivots.  The Form makes sure of that before it uses them, for 4 x 4
// entries at a time, from a lower bound of P_ij: the sum over the least entries of
// four rows each (the groups' bounds, written here).  Where that falls short
// although the rows have pivots in common, the entry's own result may still bound P_ij
// from below; where that falls short too, or a row holds an Inf or NaN, the entry is
// taken by FP64 multiply-adds.  (Two blocks of rows, each large in columns where the
// other is 2^-40 of its scale, lost 26 bits between them while rows were
// compared within their tile only.)  Random rows pass the first test from about 8 pivots
// on; of the 4 x 4 blocks of 36^3 multifrontal fronts one in 80 does not, and of their
// entries one in 1400 passes neither.
//
// Layout (what a bulk copy puts into shared memory as the MMA reads it): W in
// blocks of 128 rows, L in blocks of 64, the last of either as long as its rows, rounded
// up to 8; per row block and block of 32 pivots
// the eight slices one after another, each rows x 64 bytes, K-major with the
// 64-byte swizzle (16-byte chunk c of row r at c ^ ((r >> 1) & 3)).
#pragma once

#include "ctp_internal.cuh"

namespace ctp {

__device__ __forceinline__ unsigned hi_word(double x) { return (unsigned)__double2hiint(x); }
__device__ __forceinline__ int biased_exp(double x) { return (int)((hi_word(x) >> 20) & 0x7ffu); }

// c_k of pivot k from the stored D^-1 (its slots are D's): minus half the exponent of
// the largest entry of D^-1 in the pivot's row.  A zero pivot has no part in S
// (its column of L21 is zero): kSliceSkip, its entries count as zero.
constexpr short kSliceSkip = 32767;
__device__ __forceinline__ int slice_col_exp(const int32_t *__restrict__ piv, const double *__restrict__ Dinv, int k) {
    const int kd = piv[k];
    if (kd == CTP_PIVKIND_ZERO) return kSliceSkip;
    int e = biased_exp(Dinv[2 * k]);
    if (kd == CTP_PIVKIND_2X2_FIRST) e = max(e, biased_exp(Dinv[2 * k + 1]));
    if (kd == CTP_PIVKIND_2X2_SECOND) e = max(e, biased_exp(Dinv[2 * k - 1]));
    return (e == 0 || e == 0x7ff) ? 0 : -((e - 1023) >> 1);
}

// Exponent of |x| 2^sh, as the least E with |x| 2^sh < 2^E (kExpZero for 0,
// kExpNonfinite for Inf and NaN).
__device__ __forceinline__ int slice_exp(double x, int sh) {
    const int e = biased_exp(x);
    if (e == 0x7ff) return kExpNonfinite;
    if (e == 0) {
        const unsigned long long f = (unsigned long long)__double_as_longlong(x) & 0xFFFFFFFFFFFFFull;
        return f == 0ull ? kExpZero : -1010 - __clzll((long long)f) + sh;
    }
    return e - 1022 + sh;
}

// The 62-bit integer nearest x 2^sh 2^(62-E), plus 0x80 in every byte: byte s
// (from the top) minus 128 is then the balanced digit d_s.  low: a lower bound of
// |x| 2^(sh - E) < 1 as FP16 bits, 0 below 2^-14.
__device__ __forceinline__ unsigned long long slice_digits(double x, int sh, int E, unsigned &low) {
    const int e = biased_exp(x);
    const unsigned long long f = (unsigned long long)__double_as_longlong(x) & 0xFFFFFFFFFFFFFull;
    const unsigned long long t = (e ? (f | 0x10000000000000ull) : f) << 9;  // 62 bits, value t 2^(max(e,1)-1084)
    const int q = E - ((e ? e : 1) - 1022 + sh);                            // >= 0 but for subnormals
    low = e && q <= 13 ? (unsigned)(14 - q) << 10 | ((hi_word(x) >> 10) & 0x3FFu) : 0u;
    unsigned long long X;
    if (q <= 0)
        X = t << (-q & 63);
    else
        X = q < 64 ? ((t >> (q - 1)) + 1) >> 1 : 0ull;
    if ((long long)__double_as_longlong(x) < 0) X = 0ull - X;
    return X + 0x8080808080808080ull;
}

// digits s of two values as two BF16 (the first in the low half): bytes to
// floats by the mantissa trick, exact, upper halves kept
__device__ __forceinline__ uint32_t slice_pair(unsigned long long y0, unsigned long long y1, int s) {
    const unsigned sel = 0x7540u + (unsigned)((7 - s) & 3);  // byte of the word, then 0x4B0000..
    const unsigned w0 = s < 4 ? (unsigned)(y0 >> 32) : (unsigned)y0, w1 = s < 4 ? (unsigned)(y1 >> 32) : (unsigned)y1;
    const float f0 = __uint_as_float(__byte_perm(w0, 0x4B000000u, sel)) - 8388736.0f;
    const float f1 = __uint_as_float(__byte_perm(w1, 0x4B000000u, sel)) - 8388736.0f;
    return __byte_perm(__float_as_uint(f0), __float_as_uint(f1), 0x7632);
}

// The slices of a tile of 32 rows, by a CTA of kWarps warps: columns k < e of the
// tile in xs ([k][33], rows row0 .. row0 + nrows of the operand), column k times
// 2^(sgn * cexp[k]); the operand's `rows` in blocks of kBlk.  Zeros from e to the
// next multiple of 16 (the MMA reads no further).  grp: per block of rows and chunk of 8
// columns the groups' FP16 lower bounds of their rows' entries, 16 bytes each; -0
// where all four rows hold zeros.  red: kWarps * 32 ints, rexp: 32 ints of
// shared memory.  Two CTA barriers; xs is only read.
template <int kBlk, int kWarps>
__device__ __forceinline__ void write_slices(const double *xs, int e, int64_t row0, int nrows, const short *cexp,
                                             int sgn, unsigned char *__restrict__ img, int32_t *__restrict__ rowexp,
                                             uint16_t *__restrict__ grp, int kb, int64_t rows, int *red, int *rexp) {
    constexpr int LDX = 33;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int E = kExpZero;
    for (int k = w; k < e; k += kWarps)
        if (cexp[k] != kSliceSkip) E = max(E, slice_exp(xs[k * LDX + lane], sgn * cexp[k]));
    red[w * 32 + lane] = E;
    __syncthreads();
    if (w == 0) {
#pragma unroll
        for (int q = 1; q < kWarps; q++) E = max(E, red[q * 32 + lane]);
        rexp[lane] = E;
        if (lane < nrows) rowexp[row0 + lane] = E;
    }
    __syncthreads();
    // the block of the tile's rows (a tile lies in one)
    const int64_t blk0 = row0 / kBlk * kBlk;
    const int len = (int)min((int64_t)kBlk, slice_rows(rows - blk0)), at = (int)(row0 - blk0);
    img += (size_t)blk0 * kb * (kSlices * 64);
    grp += blk0 / kGroup * kb * kSliceK;
    const int e16 = (e + 15) & ~15, nkb = (e + kSliceK - 1) / kSliceK;
    // an item: 8 rows by the four 16-byte chunks of a K block, a lane per (row, chunk)
    for (int it = w; it < 4 * nkb; it += kWarps) {
        const int kblk = it >> 2, r = (it & 3) * 8 + (lane >> 2), c = lane & 3, k0 = kblk * kSliceK + c * 8;
        if ((it & 3) * 8 >= nrows) continue;  // the whole warp
        const bool on = r < nrows && k0 < e16;
        const int Er = rexp[r];
        unsigned long long y[8];
        unsigned low[4], some = 0u;  // FP16 pairs; which columns hold an entry
#pragma unroll
        for (int j = 0; j < 8; j++) {
            const bool in = k0 + j < e && cexp[k0 + j] != kSliceSkip;
            unsigned h = 0u;
            y[j] = 0x8080808080808080ull;
            if (in && Er < kExpNonfinite) {
                const double x = xs[(k0 + j) * LDX + r];
                y[j] = slice_digits(x, sgn * cexp[k0 + j], Er, h);
                if (Er == kExpZero) h = 0x3C00u;  // a zero row lowers nothing
                some |= (((unsigned long long)__double_as_longlong(x) << 1) != 0ull ? 1u : 0u) << j;
            } else if (in) {
                h = 0x3C00u;  // nor does one with an Inf or NaN, whose entries are known by its exponent
            }
            low[j >> 1] = (j & 1) ? low[j >> 1] | (h << 16) : h;
        }
#pragma unroll
        for (int o = 4; o <= 8; o <<= 1) {
            some |= __shfl_xor_sync(0xffffffffu, some, o);
#pragma unroll
            for (int q = 0; q < 4; q++) low[q] = __vminu2(low[q], __shfl_xor_sync(0xffffffffu, low[q], o));
        }
        if (!on) continue;
        const int rb = at + r;
        if (r % kGroup == 0) {
#pragma unroll
            for (int j = 0; j < 8; j++)
                if (!((some >> j) & 1u)) low[j >> 1] = (j & 1) ? (low[j >> 1] & 0xFFFFu) | 0x80000000u : (low[j >> 1] & 0xFFFF0000u) | 0x8000u;
            *reinterpret_cast<uint4 *>(grp + ((kblk * 4 + c) * (len / kGroup) + rb / kGroup) * 8) =
                make_uint4(low[0], low[1], low[2], low[3]);
        }
        unsigned char *dst = img + (kblk * kSlices * len + rb) * 64 + ((c ^ ((rb >> 1) & 3)) << 4);
#pragma unroll
        for (int s = 0; s < kSlices; s++) {
            uint4 v;
            v.x = slice_pair(y[0], y[1], s);
            v.y = slice_pair(y[2], y[3], s);
            v.z = slice_pair(y[4], y[5], s);
            v.w = slice_pair(y[6], y[7], s);
            *reinterpret_cast<uint4 *>(dst + s * len * 64) = v;
        }
    }
}
}  // namespace ctp
