// solve.cu -- K5: the Solve task L21 = A21 P^T (D11 L11^T)^{-1} (Section 1 task
// list; Figure 4.1 (d),(e)) fused with the update of the delayed columns, in FP64.
//
// Every A21 row is independent: with x = A21(i, perm) the permuted row,
//   Y  = x_e L11^{-T}          (forward substitution, right-looking by column),
//   x_d <- x_d - Y L_d^T        (delayed columns: L_d are the delayed rows of L),
//   L21(i,:) = Y D11^{-1}       (1x1 and 2x2 blocks; zero pivots give 0).
// A CTA owns a tile of kRows consecutive rows; the tile is gathered through the
// permutation with coalesced loads into shared memory (padded [p][kRows+1]),
// eliminated in place, and written back in place (L21 in the first e columns,
// the updated delayed columns after them).  The operands of the Form step, Y =
// L21 D11 and L21, are also written to the workspace in the Form's own format: BF16
// pieces for the mixed-precision Forms, exact digit slices (slices.cuh) for the
// FP64 one.  Arithmetic is O(p^2) FP64 FMAs per row
// and the GB300 FP64 pipe is the bound: eight warps share each row tile (each
// updates every eighth column) so that every FP64 pipe of the SM has work.
#include <cuda_bf16.h>

#include "ctp_internal.cuh"
#include "slices.cuh"

namespace ctp {

namespace {

constexpr int kRows = 32;   // rows per tile (one per lane)
constexpr int kWarps = 8;   // warps per CTA: warp w updates the columns k = w (mod 8)

// The BF16 pieces of the first e columns of a tile's rows (in xs) into the
// K-major operand copy B (row brow of B is the tile's first row), each
// piece rounding what the previous ones left (lo_off elements apart), and
// zeros from e to Kz.  Every thread of the CTA takes (row, column pair) items
// of the real columns, so that lanes do not idle on the zero tail (the
// conversions cost about a nanosecond per value per SM).
__device__ __forceinline__ void write_pieces(__nv_bfloat16 *__restrict__ B, int64_t brow, int rows, int Kp, int e,
                                             int Kz, int pieces, int64_t lo_off, const double *xs) {
    constexpr int LDX = kRows + 1;
    const int eh = (e + 1) >> 1, zn = (Kz >> 1) - eh;
    for (int t = threadIdx.x; t < rows * eh; t += blockDim.x) {
        const int rr = t / eh, k = 2 * (t - rr * eh);
        __nv_bfloat162 *dst = reinterpret_cast<__nv_bfloat162 *>(B + (brow + rr) * Kp) + (k >> 1);
        const double v0 = xs[k * LDX + rr];
        const double v1 = k + 1 < e ? xs[(k + 1) * LDX + rr] : 0.0;
        __nv_bfloat162 b;
        b.x = __double2bfloat16(v0);
        b.y = __double2bfloat16(v1);
        dst[0] = b;
        double r0 = v0 - (double)__bfloat162float(b.x);
        double r1 = v1 - (double)__bfloat162float(b.y);
        for (int pc = 1; pc < pieces; pc++) {
            __nv_bfloat162 l;
            l.x = __double2bfloat16(r0);
            l.y = __double2bfloat16(r1);
            dst[pc * (lo_off / 2)] = l;
            r0 -= (double)__bfloat162float(l.x);
            r1 -= (double)__bfloat162float(l.y);
        }
    }
    if (zn <= 0) return;
    const __nv_bfloat162 z = __floats2bfloat162_rn(0.0f, 0.0f);
    for (int t = threadIdx.x; t < rows * zn; t += blockDim.x) {
        const int rr = t / zn, k2 = eh + (t - rr * zn);
        __nv_bfloat162 *dst = reinterpret_cast<__nv_bfloat162 *>(B + (brow + rr) * Kp) + k2;
        for (int pc = 0; pc < pieces; pc++) dst[pc * (lo_off / 2)] = z;
    }
}

// What a pass over a tile does.  A whole Solve in one pass updates every later
// column with every y_j in FP64: p^2/2 multiply-adds per row on a pipe of 2 per
// clock and SM (n = 200000, p = e = 256: 12.9 ms, 0.8 of that pipe).  The blocked
// Solve (3.10 ms: 1.9 ms in the diagonal blocks, 0.95 in the updates, the rest moving
// and scaling columns) keeps only the 32-column diagonal blocks of
// that and leaves the rest -- columns times y's block by block -- to the
// tensor cores, as products of exact digit slices (k_update in form.cu):
//   kFirst  gather through perm, eliminate the first block inside itself, write
//           the row in pivot order and the block's slices (large Solves move the
//           columns in a pass of their own instead);
//   kNext   the same for block blk (its columns are in place by now);
//   kTail   after the last block's update: the rest of the elimination, if blocks
//           were left out, then the outputs as in a whole pass.
enum { kWhole, kFirst, kNext, kTail };
struct SolvePass {
    int mode;
    int blk;      // kNext: the block; kTail: how many blocks are done
    SliceBuf yb;  // slices of the block's y (kFirst, kNext)
};

// Right-looking substitution over a tile of 32 rows: for each eliminated
// position j, every warp reads y_j of its lane's row and updates its share of
// the later columns (four independent updates in flight per warp); a CTA
// barrier separates consecutive pivots.  The outputs are computed in shared
// memory without a register copy, so that a CTA needs few
// registers and as many CTAs fit on an SM as its shared memory allows (three at
// p = 256, more for narrower fronts): enough warps for all four FP64 pipes.
// kPlain: a whole pass that writes no slices, in 40 registers without a spill (20000 fronts
// of 24 x 8: 145 -> 125 us).  One tile of RT rows: 32, a lane per row, or fewer, with the lanes of a warp on several
// columns (small supernodes, so that more SMs have a tile).  brow0: row of this front's first A21 row in the BF16
// operand copies (0 for a single supernode; the stacked offset in a batch).
// pieces > 1: also write the further BF16 pieces of the split operands (piece
// k rounds what pieces 0..k-1 left), lo_off elements apart.  sb: the slices of
// the FP64 Form (sb.W null: none).
template <int RT, bool kPlain>
__device__ __forceinline__ void solve_tile(const SolvePass &ps_, double *__restrict__ A, int64_t n, int p, int64_t lda,
                                           const int32_t *__restrict__ perm,
                                           const int32_t *__restrict__ piv,
                                           const double *__restrict__ Dinv, int e, double *__restrict__ W21,
                                           const SliceBuf &sb_,
                                           __nv_bfloat16 *__restrict__ Wb,
                                           __nv_bfloat16 *__restrict__ Lb, int Kp, int64_t brow0,
                                           int64_t lo_off, int pieces, int64_t tile, double *xs) {
    constexpr int LDX = kRows + 1, SUB = kRows / RT, CW = kWarps * SUB;
    const SolvePass ps = kPlain ? SolvePass{kWhole, 0, {}} : ps_;
    const SliceBuf sb = kPlain ? SliceBuf{} : sb_;
    const int64_t m = n - p;
    const int64_t row0 = tile * RT;
    const int r = (threadIdx.x & 31) % RT, w = (threadIdx.x >> 5) * SUB + (threadIdx.x & 31) / RT;
    const int64_t row = row0 + r;
    const bool valid = row < m;
    double *A21 = A + p;
    const bool part = ps.mode == kFirst || ps.mode == kNext;
    // pivots j0..j1-1 update columns below ku; xs holds columns c0..c1-1
    const int c0 = ps.mode == kNext ? ps.blk * kSliceK : 0;
    const int j0 = ps.mode == kTail ? min(ps.blk * kSliceK, e) : c0;
    const int j1 = part ? min(c0 + kSliceK, e) : e;
    const int ku = part ? min(c0 + kSliceK, p) : p;
    const int c1 = ps.mode == kNext ? ku : (ps.mode == kTail && j0 == e ? e : p);
    if (ps.mode == kNext && c0 >= e) return;  // the whole CTA

    // gather x = A21(rows, perm): each warp reads 32 consecutive rows of a column
    // (eight columns' loads in flight per warp)
#pragma unroll 1
    for (int k0 = c0 + w; k0 < c1; k0 += 8 * CW) {
        double v[8];
#pragma unroll
        for (int q = 0; q < 8; q++) {
            const int k = k0 + q * CW;
            v[q] = 0.0;
            if (k < c1 && valid) v[q] = A21[(int64_t)(ps.mode <= kFirst ? perm[k] : k) * lda + row];
        }
#pragma unroll
        for (int q = 0; q < 8; q++)
            if (k0 + q * CW < c1) {
                xs[(k0 + q * CW - c0) * LDX + r] = v[q];
#pragma unroll
                for (int z = RT; z < kRows; z += RT) xs[(k0 + q * CW - c0) * LDX + z + r] = 0.0;  // no such rows
            }
    }
    __syncthreads();

    for (int j = j0; j < j1;) {
        const int kd = piv[j];
        if (kd == CTP_PIVKIND_2X2_FIRST && j + 1 < j1) {
            const double y0 = xs[(j - c0) * LDX + r], y1 = xs[(j + 1 - c0) * LDX + r];
            const double *l0 = A + (int64_t)j * lda, *l1 = A + (int64_t)(j + 1) * lda;
#pragma unroll 4
            for (int k = j + 2 + w; k < ku; k += CW)
                xs[(k - c0) * LDX + r] -= y0 * __ldg(l0 + k) + y1 * __ldg(l1 + k);
            j += 2;
        } else {
            // (a 2x2 pair that a block boundary cuts: its first column has nothing left
            // to update in its block, its second is a column like any other)
            if (kd == CTP_PIVKIND_1X1 || kd == CTP_PIVKIND_2X2_SECOND) {
                const double y0 = xs[(j - c0) * LDX + r];
                const double *l0 = A + (int64_t)j * lda;
#pragma unroll 4
                for (int k = j + 1 + w; k < ku; k += CW) xs[(k - c0) * LDX + r] -= y0 * __ldg(l0 + k);
            }
            j += 1;  // zero pivots have an all-zero L column
        }
        __syncthreads();
    }

    const int tile_rows = m - row0 < RT ? (int)(m - row0) : RT;
    __shared__ short cexp[kMaxP];
    __shared__ int red[kWarps * 32], rexp[32];
    if (part) {
        if (c0 + kSliceK < p) {  // columns are left to update
            for (int k = c0 + threadIdx.x; k < j1; k += blockDim.x) cexp[k - c0] = (short)slice_col_exp(piv, Dinv, k);
            __syncthreads();
            write_slices<kWRows, kWarps>(xs, j1 - c0, row0, tile_rows, cexp, -1, ps.yb.W, ps.yb.ew, ps.yb.gw,
                                         ps.yb.kb, m, red, rexp);
        }
        if (valid)
            for (int k = c0 + w; k < c1; k += CW) A21[(int64_t)k * lda + row] = xs[(k - c0) * LDX + r];
        return;
    }

    // the Form's copies of Y = W21.  BF16 pieces: row-major, K contiguous,
    // zero from e to the end of e's last 64-wide K block (the Form reads no
    // further; a batch's rows are 256 wide whatever the front's p)
    const int Kz = min(Kp, (e + 63) / 64 * 64);
    if (sb.W != nullptr) {
        for (int k = threadIdx.x; k < e; k += blockDim.x) cexp[k] = (short)slice_col_exp(piv, Dinv, k);
        __syncthreads();
        write_slices<kWRows, kWarps>(xs, e, row0, tile_rows, cexp, -1, sb.W, sb.ew, sb.gw, sb.kb, m, red, rexp);
    }
    if (W21 != nullptr && valid)
        for (int k = w; k < e; k += CW) W21[(int64_t)k * m + row] = xs[k * LDX + r];
    if (Wb != nullptr) write_pieces(Wb, brow0 + row0, tile_rows, Kp, e, Kz, pieces, lo_off, xs);
    __syncthreads();
    // L21 = Y D11^{-1} in place (1x1 and 2x2 blocks; zero pivots give 0), written
    // back with the delayed columns as they are
    for (int k = w; k < c1; k += CW) {
        const int kd = k < e ? piv[k] : CTP_PIVKIND_DELAYED;
        if (kd == CTP_PIVKIND_2X2_SECOND) continue;  // with its first column
        double out = xs[k * LDX + r];
        if (kd == CTP_PIVKIND_2X2_FIRST) {
            const double y0 = out, y1 = xs[(k + 1) * LDX + r];
            out = __fma_rn(y1, Dinv[2 * k + 1], y0 * Dinv[2 * k]);
            const double o1 = __fma_rn(y1, Dinv[2 * k + 2], y0 * Dinv[2 * k + 1]);
            xs[(k + 1) * LDX + r] = o1;
            if (valid) A21[(int64_t)(k + 1) * lda + row] = o1;
        } else if (kd == CTP_PIVKIND_1X1) {
            out *= Dinv[2 * k];
        } else if (kd == CTP_PIVKIND_ZERO) {
            out = 0.0;
        }
        if (kd != CTP_PIVKIND_DELAYED) xs[k * LDX + r] = out;
        if (valid) A21[(int64_t)k * lda + row] = out;
    }
    if (Lb == nullptr && sb.L == nullptr) return;
    __syncthreads();
    // the Form's copies of L21
    if (sb.L != nullptr)
        write_slices<kLRows, kWarps>(xs, e, row0, tile_rows, cexp, 1, sb.L, sb.el, sb.gl, sb.kb, m, red, rexp);
    if (Lb != nullptr) write_pieces(Lb, brow0 + row0, tile_rows, Kp, e, Kz, pieces, lo_off, xs);
}

template <int RT, bool kPlain>
__global__ void __launch_bounds__(kRows * kWarps, 6)
    k_solve_fp64(SolvePass ps, double *__restrict__ A, int64_t n, int p, int64_t lda,
                 const int32_t *__restrict__ perm, const int32_t *__restrict__ piv,
                 const double *__restrict__ Dinv, const int32_t *__restrict__ nelim_p,
                 double *W21, SliceBuf sb, __nv_bfloat16 *__restrict__ Wb, __nv_bfloat16 *__restrict__ Lb, int Kp,
                 int64_t lo_off, int pieces) {
    extern __shared__ __align__(16) double xs[];  // [columns][kRows+1]
    solve_tile<RT, kPlain>(ps, A, n, p, lda, perm, piv, Dinv, *nelim_p, W21, sb, Wb, Lb, Kp, 0, lo_off, pieces, blockIdx.x, xs);
}

// Batched: CTA b takes work item b = (front, RT-row tile of its A21): the
// front is item_front[b], the tile item_tile[b].
template <int RT, bool kPlain>
__global__ void __launch_bounds__(kRows * kWarps, kPlain ? 6 : 5)
    k_solve_batch(int mode, const ctp_front *__restrict__ fronts, const BFront *__restrict__ tab, char *ws,
                  const int *__restrict__ item_front, const int *__restrict__ item_tile, BatchOpts o,
                  __nv_bfloat16 *__restrict__ Wb, __nv_bfloat16 *__restrict__ Lb) {
    extern __shared__ __align__(16) double xs[];
    const int f = item_front[blockIdx.x];
    const ctp_front fr = fronts[f];
    const BFront bt = tab[f];
    const BSection sec = bsection(bt.n, bt.p, o);
    char *base = ws + bt.ws;
    SliceBuf sb = {};
    double *W21 = nullptr;
    if (o.smode != CTP_S_NONE && o.prec == CTP_FP64) {
        if (kPlain || form_small(bt.m))
            W21 = reinterpret_cast<double *>(base + sec.W21);
        else
            sb = bsection_slices(base, sec, bt.p);
    }
    SolvePass ps = {mode, mode == kTail ? 1 : 0, {}};
    if (mode == kFirst) ps.yb = bsection_block(base, sec);
    solve_tile<RT, kPlain>(ps, fr.A, bt.n, bt.p, fr.lda, fr.perm, fr.piv, reinterpret_cast<const double *>(base + sec.Dinv),
               *fr.nelim, W21, sb, Wb, Lb, kBatchKp, bt.row0, o.lo_off, o.pieces,
               item_tile[blockIdx.x], xs);
}

// The columns of A21 into pivot order, in place: a tile of 32 rows by all columns per
// CTA; columns that stay are left alone.
__global__ void __launch_bounds__(kRows * kWarps, 6)
    k_move_columns(double *__restrict__ A21, int64_t m, int p, int64_t lda, const int32_t *__restrict__ perm) {
    extern __shared__ __align__(16) double xs[];  // [p][kRows]
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t row = (int64_t)blockIdx.x * kRows + lane;
    const bool valid = row < m;
#pragma unroll 1
    for (int k0 = w; k0 < p; k0 += 8 * kWarps) {
        double v[8];
#pragma unroll
        for (int q = 0; q < 8; q++) {
            const int k = k0 + q * kWarps;
            v[q] = 0.0;
            if (k < p && valid && perm[k] != k) v[q] = A21[(int64_t)perm[k] * lda + row];
        }
#pragma unroll
        for (int q = 0; q < 8; q++)
            if (k0 + q * kWarps < p) xs[(k0 + q * kWarps) * kRows + lane] = v[q];
    }
    __syncthreads();
    if (!valid) return;
    for (int k = w; k < p; k += kWarps)
        if (perm[k] != k) A21[(int64_t)k * lda + row] = xs[k * kRows + lane];
}

// L21 = Y D11^{-1} in place, as solve_tile's tail computes it: a thread per row and 16
// columns (and the second of a 2x2 pair that begins with the last of them).
constexpr int kScaleCols = 16, kScaleRows = 256;
__global__ void __launch_bounds__(kScaleRows)
    k_scale_columns(double *__restrict__ A21, int64_t m, int64_t lda, const int32_t *__restrict__ piv,
                    const double *__restrict__ Dinv, const int32_t *__restrict__ nelim_p) {
    const int e = *nelim_p, k0 = blockIdx.y * kScaleCols;
    const int64_t row = (int64_t)blockIdx.x * kScaleRows + threadIdx.x;
    if (k0 >= e || row >= m) return;
    double *x = A21 + (int64_t)k0 * lda + row;
    const int cnt = min(kScaleCols, e - k0);
    double v[kScaleCols + 1];
#pragma unroll
    for (int q = 0; q < kScaleCols; q++) v[q] = q < cnt ? x[q * lda] : 0.0;
    v[kScaleCols] = cnt == kScaleCols && piv[k0 + cnt - 1] == CTP_PIVKIND_2X2_FIRST ? x[kScaleCols * lda] : 0.0;
#pragma unroll
    for (int q = 0; q < kScaleCols; q++) {
        if (q >= cnt) break;
        const int k = k0 + q, kd = piv[k];
        if (kd == CTP_PIVKIND_1X1) {
            x[q * lda] = v[q] * Dinv[2 * k];
        } else if (kd == CTP_PIVKIND_2X2_FIRST) {
            x[q * lda] = __fma_rn(v[q + 1], Dinv[2 * k + 1], v[q] * Dinv[2 * k]);
            x[(q + 1) * lda] = __fma_rn(v[q + 1], Dinv[2 * k + 2], v[q] * Dinv[2 * k + 1]);
        } else if (kd == CTP_PIVKIND_ZERO) {
            x[q * lda] = 0.0;
        }
    }
}

// Slices of L11's rows below block blk, columns of the block: what the block's y
// are multiplied with.  One 32-row tile (rows r0.. in pivot order) per CTA; row r
// is row r - 32 (blk + 1) of the image.
__device__ __forceinline__ void l11_tile(const double *__restrict__ A, int64_t lda, int p, int blk, int r0,
                                         const int32_t *__restrict__ piv, const double *__restrict__ Dinv, int e,
                                         const SliceBuf &lb) {
    constexpr int LDX = kRows + 1;
    __shared__ double xs[kSliceK * LDX];
    __shared__ short cexp[kSliceK];
    __shared__ int red[kWarps * 32], rexp[32];
    const int c0 = blk * kSliceK, cnt = min(kSliceK, e - c0), first = c0 + kSliceK;
    if (cnt <= 0 || r0 < first || r0 >= p) return;  // the whole CTA
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, r = r0 + lane;
    for (int k = threadIdx.x; k < cnt; k += kRows * kWarps) cexp[k] = (short)slice_col_exp(piv, Dinv, c0 + k);
    for (int k = w; k < cnt; k += kWarps) {
        const int c = c0 + k;
        const bool d21 = r == c + 1 && piv[c] == CTP_PIVKIND_2X2_FIRST;  // that slot holds D
        xs[k * LDX + lane] = (r < p && !d21) ? A[(int64_t)c * lda + r] : 0.0;
    }
    __syncthreads();
    write_slices<kLRows, kWarps>(xs, cnt, r0 - first, min(kRows, p - r0), cexp, 1, lb.L, lb.el, lb.gl, lb.kb, p - first,
                                 red, rexp);
}
__global__ void __launch_bounds__(kRows * kWarps, 6)
    k_l11_slices(const double *__restrict__ A, int64_t lda, int p, const int32_t *__restrict__ piv,
                 const double *__restrict__ Dinv, const int32_t *__restrict__ nelim, SliceBuf lb, size_t blk_bytes,
                 size_t grp_elems) {
    lb.L += blockIdx.y * blk_bytes;
    lb.el += blockIdx.y * kMaxP;
    lb.gl += blockIdx.y * grp_elems;
    l11_tile(A, lda, p, blockIdx.y, blockIdx.x * kRows, piv, Dinv, *nelim, lb);
}
__global__ void __launch_bounds__(kRows * kWarps, 6)
    k_l11_slices_batch(const ctp_front *__restrict__ fronts, const BFront *__restrict__ tab, char *ws,
                       const int *__restrict__ list, BatchOpts o) {
    const int f = list[blockIdx.x];
    const ctp_front fr = fronts[f];
    const BFront bt = tab[f];
    if (!front_blocked(bt.m, bt.p, o)) return;  // no room for slices in its section
    const BSection sec = bsection(bt.n, bt.p, o);
    char *base = ws + bt.ws;
    l11_tile(fr.A, fr.lda, bt.p, 0, (blockIdx.y + 1) * kRows, fr.piv,
             reinterpret_cast<const double *>(base + sec.Dinv), *fr.nelim, bsection_block(base, sec));
}

}  // namespace

// How many 32-column blocks the blocked Solve of an m x p supernode takes, 0 for a
// whole pass.  Blocked, a Solve is 2 + 2 blocks launches (e is not known on the
// host; blocks past it exit at once, about 2 us each).  Strict and single-row
// pivoting accept few columns (12 of 256 on random data, 30 in large
// multifrontal panels): one block, and what it leaves goes with the tail.
// Measured, whole / blocked, all columns accepted: p = 256 from m = 344 on (498 /
// 313 us; n = 200000: 12869 / 3413); p = 160, m = 240: 254 / 205; p = 128, m = 1372:
// 170 / 164; p = 96, m = 2904: 108 / 117, m = 11904: 160 / 133; p = 64, m = 11936: 84 / 88,
// m = 23936: 113 / 104.  A dozen accepted: p = 192, m = 208: 45 / 43; p = 160, m =
// 2840: 41 / 41, m = 11840: 70 / 53; p = 128, m = 5872: 41 / 43, m = 11872: 57 / 53; p = 96, m
// = 11904: 43 / 49; p = 64, m = 23936: 41 / 53, m = 99936: 149 / 131.
int solve_blocks(int64_t m, int p, int pivot) {
    if (p <= kSliceK || m <= 0) return 0;
    const double right = (double)m * (p - kSliceK);  // entries the first block's update touches
    if (pivot == CTP_PIV_STRICT || pivot == CTP_PIV_SINGLE_ROW)
        return p > 176 || right >= (p > 96 ? 1e6 : 2.5e6) ? 1 : 0;
    return p > 128 || right * (p - kSliceK) >= 1.6e7 ? (p + kSliceK - 1) / kSliceK : 0;
}

// Rows per tile of a Solve with this many 32-row tiles: few tiles leave SMs idle, and
// one tile per SM waits for its own chain of pivots, so they get 16 or 8 rows, up
// to two tiles per SM.  Whole passes with 32 rows / with this rule, all columns accepted: n = 500,
// p = 64: 61 / 45 us; n = 1000, p = 96: 113 / 70; n = 2000, p = 64: 61 / 45; n = 3500, p = 64: 61 / 49;
// n = 9000, p = 64: 68 / 65; a dozen accepted: n = 2400, p = 96: 29 / 18; n = 2600, p = 64: 24 / 20.
// Blocked ones (up to one tile per SM, their passes are short): p = 256, n = 600: 314 /
// 271; n = 1500: 334 / 277; n = 5000: 334 / 314; p = 160, n = 2400: 203 / 170.
int solve_rows(int64_t tiles, bool blocked, int num_sms) {
    const int64_t sms = blocked ? num_sms : 2 * (int64_t)num_sms;
    return tiles > sms ? kRows : (2 * tiles > sms ? kRows / 2 : kRows / 4);
}

// Entries of A21 from which a blocked Solve (p > 64) moves the columns, and scales them
// when nothing else is left to do, in passes of their own: two launches more, but
// the first block's elimination keeps eight CTAs per SM instead of three and the
// scaling streams.  Together / apart, all columns accepted: n = 200000, p = 256: 3442 /
// 3062 us (n = 24000: 547 / 510, 12000: 400 / 402), p = 128, n = 50000: 457 / 436 (24000: 232
// / 238); a dozen accepted: p = 256, n = 200000: 567 / 444 (24000: 92 / 92, 12000: 61 / 68), p = 64,
// n = 100000: 133 / 137.
constexpr int64_t kApart = 6000000;

cudaError_t launch_solve_fp64(double *A, int64_t n, int p, int64_t lda, const int32_t *perm,
                              const int32_t *piv, const double *Dinv, const int32_t *nelim,
                              double *W21, const SliceBuf &sb, const SliceBuf &blk, int blocks, void *Wb, void *Lb, int Kp,
                              int64_t lo_off, int pieces, TileMarks *marks, int32_t *info, int num_sms, cudaStream_t st) {
    const int64_t m = n - p;
    if (m <= 0) return cudaSuccess;
    const size_t smem_p = sizeof(double) * (size_t)p * (kRows + 1);
    const int rt = solve_rows((m + kRows - 1) / kRows, blocks > 0, num_sms);
    const bool plain = blocks == 0 && sb.W == nullptr;
    auto *k = plain ? (rt == kRows       ? k_solve_fp64<kRows, true>
                       : rt == kRows / 2 ? k_solve_fp64<kRows / 2, true>
                                         : k_solve_fp64<kRows / 4, true>)
                    : (rt == kRows       ? k_solve_fp64<kRows, false>
                       : rt == kRows / 2 ? k_solve_fp64<kRows / 2, false>
                                         : k_solve_fp64<kRows / 4, false>);
    cudaError_t err = smem_at_least((const void *)k, smem_p);
    if (err != cudaSuccess) return err;
    const unsigned grid = (unsigned)((m + rt - 1) / rt);
    auto pass = [&](int mode, int b, int cols) {
        const SolvePass ps = {mode, b, blk};
        k<<<grid, kRows * kWarps, sizeof(double) * (size_t)cols * (kRows + 1), st>>>(
            ps, A, n, p, lda, perm, piv, Dinv, nelim, W21, sb, (__nv_bfloat16 *)Wb, (__nv_bfloat16 *)Lb, Kp, lo_off, pieces);
        return cudaGetLastError();
    };
    if (blocks == 0) return pass(kWhole, 0, p);
    const size_t lbytes = slice_bytes(p, kSliceK), gelems = slice_g_bytes(p, kSliceK) / sizeof(uint16_t);
    if (p > kSliceK) {
        const int nb = blocks < (p - 1) / kSliceK ? blocks : (p - 1) / kSliceK;  // the last block has nothing below
        k_l11_slices<<<dim3((unsigned)((p + kRows - 1) / kRows), (unsigned)nb), kRows * kWarps, 0, st>>>(
            A, lda, p, piv, Dinv, nelim, blk, lbytes, gelems);
        err = cudaGetLastError();
        if (err != cudaSuccess) return err;
    }
    const bool apart = p > 64 && m * p >= kApart;
    if (apart) {
        const size_t smem = sizeof(double) * (size_t)p * kRows;
        if ((err = smem_at_least((const void *)k_move_columns, smem)) != cudaSuccess) return err;
        k_move_columns<<<grid, kRows * kWarps, smem, st>>>(A + p, m, p, lda, perm);
        if ((err = cudaGetLastError()) != cudaSuccess) return err;
    }
    for (int b = 0; b < blocks; b++) {
        err = b == 0 && !apart ? pass(kFirst, 0, p) : pass(kNext, b, kSliceK);
        if (err != cudaSuccess) return err;
        if ((b + 1) * kSliceK >= p) break;
        SliceBuf u = blk;
        u.L += b * lbytes;
        u.el += b * kMaxP;
        u.gl += b * gelems;
        err = launch_update(u, A, lda, p, m, b, piv, nelim, marks, info, num_sms, st);
        if (err != cudaSuccess) return err;
    }
    if (apart && blocks * kSliceK >= p && W21 == nullptr && sb.W == nullptr && sb.L == nullptr && Wb == nullptr && Lb == nullptr) {
        k_scale_columns<<<dim3((unsigned)((m + kScaleRows - 1) / kScaleRows),
                               (unsigned)((p + kScaleCols - 1) / kScaleCols)),
                          kScaleRows, 0, st>>>(A + p, m, lda, piv, Dinv, nelim);
        return cudaGetLastError();
    }
    return pass(kTail, blocks, p);
}

static decltype(&k_solve_batch<kRows, false>) solve_batch_kernel(int rows, bool plain) {
    if (plain)
        return rows == kRows       ? k_solve_batch<kRows, true>
               : rows == kRows / 2 ? k_solve_batch<kRows / 2, true>
                                   : k_solve_batch<kRows / 4, true>;
    return rows == kRows       ? k_solve_batch<kRows, false>
           : rows == kRows / 2 ? k_solve_batch<kRows / 2, false>
                               : k_solve_batch<kRows / 4, false>;
}

cudaError_t launch_solve_batch(const ctp_front *fronts, const BFront *tab, char *ws,
                               const int *item_front, int64_t items, int rows, bool plain, BatchOpts o, void *Wb, void *Lb,
                               int pmax, cudaStream_t st, const int *item_tile) {
    if (items == 0) return cudaSuccess;
    const size_t smem = sizeof(double) * (size_t)pmax * (kRows + 1);
    auto *k = solve_batch_kernel(rows, plain);
    cudaError_t err = smem_at_least((const void *)k, smem);
    if (err != cudaSuccess) return err;
    k<<<(unsigned)items, kRows * kWarps, smem, st>>>(
        kWhole, fronts, tab, ws, item_front, item_tile, o, (__nv_bfloat16 *)Wb, (__nv_bfloat16 *)Lb);
    return cudaGetLastError();
}

cudaError_t launch_solve_batch_blocked(const ctp_front *fronts, const BFront *tab, char *ws, const int *list,
                                       int count, const int *item_front, const int *item_tile, int64_t items,
                                       int rows, const int *uitem, const int *utile, int64_t uitems, BatchOpts o, void *Wb,
                                       void *Lb, int pmax, TileMarks *marks, int32_t *info, int num_sms,
                                       cudaStream_t st) {
    if (items == 0) return cudaSuccess;
    const size_t smem = sizeof(double) * (size_t)pmax * (kRows + 1);
    auto *k = solve_batch_kernel(rows, false);
    cudaError_t err = smem_at_least((const void *)k, smem);
    if (err != cudaSuccess) return err;
    if (pmax > kSliceK) {
        const unsigned tiles = (unsigned)((pmax - 1) / kRows);  // 32-row tiles below the first block
        k_l11_slices_batch<<<dim3((unsigned)count, tiles), kRows * kWarps, 0, st>>>(fronts, tab, ws, list, o);
        if ((err = cudaGetLastError()) != cudaSuccess) return err;
    }
    k<<<(unsigned)items, kRows * kWarps, smem, st>>>(
        kFirst, fronts, tab, ws, item_front, item_tile, o, (__nv_bfloat16 *)Wb, (__nv_bfloat16 *)Lb);
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
    err = launch_update_batch(fronts, tab, ws, uitem, utile, uitems, o, marks, info, num_sms, st);
    if (err != cudaSuccess) return err;
    k<<<(unsigned)items, kRows * kWarps, smem, st>>>(
        kTail, fronts, tab, ws, item_front, item_tile, o, (__nv_bfloat16 *)Wb, (__nv_bfloat16 *)Lb);
    return cudaGetLastError();
}

}  // namespace ctp
