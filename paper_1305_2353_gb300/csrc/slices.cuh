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
// Accuracy: a digit product with s + t > 7 is dropped and X is cut at 2^-62, in
// all about 2^-62 e^(1/2) of the two rows' scales 2^(E_i + E_j): less than the
// rounding of e FP64 multiply-adds wherever the large entries of one row meet
// entries of the other that are not much below its own largest, as they do in
// random data and under the growth of the pivots' columns, which all rows share.
// A row is marked, by kExpWide added to its exponent, when none of its entries
// does -- in no column is its entry, relative to its scale, times the typical
// entry (the geometric mean of the nonzero ones of the tile's 32 rows, relative
// to theirs) above 2^-kWideBits -- or when it holds an Inf or NaN, and the Form
// takes its entries of S by FP64 multiply-adds.  (Entries scattered over 2^40
// lost up to 8 bits without the mark.)
//
// Layout (what a bulk copy puts into shared memory as the MMA reads it): W in
// blocks of 128 rows, L in blocks of 64; per row block and block of 32 pivots
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
constexpr int kWideBits = 5;
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
// (from the top) minus 128 is then the balanced digit d_s.
__device__ __forceinline__ unsigned long long slice_digits(double x, int sh, int E) {
    const int e = biased_exp(x);
    const unsigned long long f = (unsigned long long)__double_as_longlong(x) & 0xFFFFFFFFFFFFFull;
    const unsigned long long t = (e ? (f | 0x10000000000000ull) : f) << 9;  // 62 bits, value t 2^(max(e,1)-1084)
    const int q = E - ((e ? e : 1) - 1022 + sh);                            // >= 0 but for subnormals
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
// 2^(sgn * cexp[k]); kBlk rows per block of the image.  Zeros from e to the
// next multiple of 16 (the MMA reads no further).  red: 2 * kWarps * 32 ints,
// rexp: 32 ints of shared memory.  Three CTA barriers; xs is only read.
template <int kBlk, int kWarps>
__device__ __forceinline__ void write_slices(const double *xs, int e, int64_t row0, int nrows, const short *cexp,
                                             int sgn, unsigned char *__restrict__ img, int32_t *__restrict__ rowexp,
                                             int kb, int *red, int *rexp) {
    constexpr int LDX = 33;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int E = kExpZero;
    for (int k = w; k < e; k += kWarps)
        if (cexp[k] != kSliceSkip) E = max(E, slice_exp(xs[k * LDX + lane], sgn * cexp[k]));
    red[w * 32 + lane] = E;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kWarps; q++) E = max(E, red[q * 32 + lane]);
    int best = kExpZero;  // the row's best column: log2 of its entry times the typical one
    for (int k = w; k < e; k += kWarps) {
        if (cexp[k] == kSliceSkip) continue;
        const int x = slice_exp(xs[k * LDX + lane], sgn * cexp[k]);
        const bool in = x > kExpZero && x < kExpNonfinite;
        const int cnt = __popc(__ballot_sync(0xffffffffu, in));
        const int sum = __reduce_add_sync(0xffffffffu, in ? E - x : 0);
        if (in) best = max(best, x - E - sum / cnt);
    }
    red[(kWarps + w) * 32 + lane] = best;
    __syncthreads();
    if (w == 0) {
#pragma unroll
        for (int q = 1; q < kWarps; q++) best = max(best, red[(kWarps + q) * 32 + lane]);
        rexp[lane] = E;
        const bool wide = E >= kExpNonfinite || (E > kExpZero && best < -kWideBits);
        if (lane < nrows) rowexp[row0 + lane] = wide ? E + kExpWide : E;
    }
    __syncthreads();
    const int e16 = (e + 15) & ~15, nkb = (e + kSliceK - 1) / kSliceK;
    // an item: 8 rows by the four 16-byte chunks of a K block, a lane per (row, chunk)
    for (int it = w; it < 4 * nkb; it += kWarps) {
        const int kblk = it >> 2, r = (it & 3) * 8 + (lane >> 2), c = lane & 3, k0 = kblk * kSliceK + c * 8;
        if (r >= nrows || k0 >= e16) continue;
        const int Er = rexp[r];
        unsigned long long y[8];
#pragma unroll
        for (int j = 0; j < 8; j++) {
            const bool in = k0 + j < e && cexp[k0 + j] != kSliceSkip && Er < kExpNonfinite;
            y[j] = in ? slice_digits(xs[(k0 + j) * LDX + r], sgn * cexp[k0 + j], Er) : 0x8080808080808080ull;
        }
        const int64_t row = row0 + r;
        const int rb = (int)(row % kBlk);
        unsigned char *dst = img + ((size_t)(row / kBlk) * kb + kblk) * ((size_t)kSlices * kBlk * 64) + rb * 64 +
                             ((c ^ ((rb >> 1) & 3)) << 4);
#pragma unroll
        for (int s = 0; s < kSlices; s++) {
            uint4 v;
            v.x = slice_pair(y[0], y[1], s);
            v.y = slice_pair(y[2], y[3], s);
            v.z = slice_pair(y[4], y[5], s);
            v.w = slice_pair(y[6], y[7], s);
            *reinterpret_cast<uint4 *>(dst + (size_t)s * kBlk * 64) = v;
        }
    }
}
}  // namespace ctp
