// system.cu -- solving a complete system with the supernodes' factors, the FP64
// residual, the backward error of Section 7 and the kernels iterative
// refinement needs.
//
// The factors are a list of fronts in elimination order (a chain or an assembly
// tree, children first).  Front f has n_f rows named by the variable indices
// rows[0..n_f) (rows[0..p) are its fully-summed variables in the order they had
// before pivoting, so front row q < p holds variable rows[perm[q]] afterwards)
// and stores, in ctp_factor_supernode's in-place layout, the unit lower
// factor L (columns 0..e-1), D (1x1 and 2x2 blocks; the (q+1, q) slot of a
// 2x2 block holds D, not L).  With P M P^T = L D L^T the solve is
//   forward   for f in order:   y = L11^{-1} b_f,  b_rest -= L_rest y,  z = D^{-1} y
//   backward  for f reversed:   x_f = L11^{-T} (z - L_rest^T x_rest)
// (Section 1's factorization applied front by front).  Right-hand sides are the
// columns of an N x nrhs column-major array X, solved in place.
#include "ctp_internal.cuh"

namespace ctp {

namespace {

constexpr int kTh = 256;   // threads of every kernel here
constexpr int kS = 8;      // pivots per step of the triangular solves
constexpr int kAhead = 4;  // steps whose entries of L11 are loaded ahead
constexpr int kRows = 32;  // rows below the pivots per tile of the updates

__device__ __forceinline__ int front_var(const ctp_sfront &f, int64_t r) {
    return r < f.p ? f.rows[f.perm[r]] : f.rows[r];
}

// The triangular solves are a chain of as many dependent FP64 multiply-adds as
// pivots; the arithmetic of one right-hand side is a few microseconds of one
// SM's FP64 pipe.  So every right-hand side has a CTA, and thread t keeps row (or column)
// t's value in a register.  Eight pivots at a time the warp that holds them solves among
// itself by shuffles and publishes the values; after one barrier the other
// warps apply them while the owner goes on.  A thread reads its entries of L11
// straight from memory, 32 columns ahead.  Fronts of 256 pivots and 2000 rows and less
// with four right-hand sides, triangular solve and update together: forward 233 us ->
// 41, backward 300 -> 42 (one CTA for all right-hand sides, two barriers per pivot,
// 256 rows per CTA of the updates before).

// Forward step of one front: gather, unit-lower solve with L11, keep y for the
// update of the rows below, scatter z = D^{-1} y.
__global__ void __launch_bounds__(kTh) k_sys_fwd_tri(ctp_sfront f, double *X, int64_t ldx, double *Y) {
    __shared__ double y[kMaxP];
    __shared__ int pv[kMaxP];
    const int e = *f.nelim, t = threadIdx.x, warp = t >> 5;
    X += (int64_t)blockIdx.x * ldx;
    const double *row = f.L + t;
    double l[kAhead][kS];  // L(t, k) of the next steps' columns k
#pragma unroll
    for (int s = 0; s < kAhead; s++)
#pragma unroll
        for (int j = 0; j < kS; j++) l[s][j] = (t < e && kS * s + j < t) ? row[(int64_t)(kS * s + j) * f.ldl] : 0.0;
    int var = 0;
    double v = 0.0;
    if (t < e) {
        var = f.rows[f.perm[t]];
        pv[t] = f.piv[t];
        v = X[var];
    }
    __syncthreads();
    // columns before `mine` act on this row: not the first column of its own 2x2 block,
    // where the (t, t-1) slot holds D
    const int mine = t >= e ? 0 : t - (t > 0 && pv[t - 1] == CTP_PIVKIND_2X2_FIRST);
    for (int k0 = 0; k0 < e; k0 += kS * kAhead) {
#pragma unroll
        for (int s = 0; s < kAhead; s++) {
            const int k = k0 + kS * s;
            if (k < e) {
                if (warp == k >> 5) {
#pragma unroll
                    for (int j = 0; j < kS; j++) {
                        const double x = __shfl_sync(0xffffffffu, v, (k + j) & 31);
                        if (k + j < mine) v -= l[s][j] * x;
                    }
                    if (t >= k && t < min(k + kS, e)) y[t] = v;
                }
                __syncthreads();
                if (warp > k >> 5 && t < e) {
                    double s0 = 0.0, s1 = 0.0;
#pragma unroll
                    for (int j = 0; j < kS; j += 2) {
                        s0 += l[s][j] * y[k + j];
                        if (k + j + 1 < mine) s1 += l[s][j + 1] * y[k + j + 1];
                    }
                    v -= s0 + s1;
                }
                const int kn = k + kS * kAhead;
#pragma unroll
                for (int j = 0; j < kS; j++) l[s][j] = (t < e && kn + j < t) ? row[(int64_t)(kn + j) * f.ldl] : 0.0;
            }
        }
    }
    if (t >= e) return;
    Y[(int64_t)blockIdx.x * kMaxP + t] = v;
    // D solve: 1x1, 2x2, zero pivot -> 0
    const int k = pv[t];
    double z = 0.0;
    if (k == CTP_PIVKIND_1X1) {
        z = v / f.D[2 * t];
    } else if (k == CTP_PIVKIND_2X2_FIRST || k == CTP_PIVKIND_2X2_SECOND) {
        const int a = (k == CTP_PIVKIND_2X2_FIRST) ? t : t - 1;
        const double d11 = f.D[2 * a], d21 = f.D[2 * a + 1], d22 = f.D[2 * a + 2];
        const double y0 = y[a], y1 = y[a + 1], det = d11 * d22 - d21 * d21;
        z = (k == CTP_PIVKIND_2X2_FIRST) ? (d22 * y0 - d21 * y1) / det : (d11 * y1 - d21 * y0) / det;
    }
    X[var] = z;
}

// Rows below the pivots: b(var(r)) -= L(r, 0:e) y for 32 rows and RB right-hand
// sides per CTA; warp w takes every eighth column.
template <int RB>
__global__ void __launch_bounds__(kTh) k_sys_fwd_upd(ctp_sfront f, double *X, int64_t ldx, int nrhs,
                                                     const double *Y, unsigned tiles) {
    constexpr int W = kTh / 32;
    __shared__ double ys[kMaxP][RB], red[W][RB][kRows];
    const int e = *f.nelim, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r0 = blockIdx.x / tiles * RB, nr = min(RB, nrhs - r0);
    const int64_t base = e + (int64_t)(blockIdx.x % tiles) * kRows, row = base + lane;
    if (base >= f.n) return;  // the whole CTA
    for (int idx = threadIdx.x; idx < RB * e; idx += kTh) {
        const int r = idx / e, q = idx - r * e;
        ys[q][r] = r < nr ? Y[(int64_t)(r0 + r) * kMaxP + q] : 0.0;
    }
    __syncthreads();
    const double *lp = f.L + row;
    double acc[RB];
#pragma unroll
    for (int r = 0; r < RB; r++) acc[r] = 0.0;
#pragma unroll 8
    for (int j = w; j < e; j += W) {
        const double l = row < f.n ? lp[(int64_t)j * f.ldl] : 0.0;
#pragma unroll
        for (int r = 0; r < RB; r++) acc[r] += l * ys[j][r];
    }
#pragma unroll
    for (int r = 0; r < RB; r++) red[w][r][lane] = acc[r];
    __syncthreads();
    for (int idx = threadIdx.x; idx < nr * kRows; idx += kTh) {
        const int r = idx / kRows, q = idx % kRows;
        const int64_t i = base + q;
        if (i >= f.n) continue;
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < W; k++) s += red[k][r][q];
        X[(int64_t)(r0 + r) * ldx + front_var(f, i)] -= s;
    }
}

// Backward step, part 1: per chunk of `chunk` rows below the pivots (a multiple of
// 32), part[c][r][j] = sum over the chunk's rows of L(row, j) x(var(row), r).
// A thread per column, so that nothing is summed across lanes (the exchanges of a lane
// per row cost more FP64 additions than the products); a column's 32 rows are
// whole sectors, which the L1 keeps between the loads.
template <int RB>
__global__ void __launch_bounds__(kTh) k_sys_bwd_part(ctp_sfront f, const double *X, int64_t ldx, int nrhs,
                                                      int chunk, double *part, unsigned chunks) {
    __shared__ double xs[kRows][RB];
    const int e = *f.nelim, t = threadIdx.x;
    const int r0 = blockIdx.x / chunks * RB, nr = min(RB, nrhs - r0);
    const unsigned c0 = blockIdx.x % chunks;
    const int64_t base = e + (int64_t)c0 * chunk, end = min((int64_t)f.n, base + chunk);
    if (base >= f.n) return;  // the whole CTA
    const double *col = f.L + (int64_t)t * f.ldl;
    double acc[RB];
#pragma unroll
    for (int r = 0; r < RB; r++) acc[r] = 0.0;
    for (int64_t b0 = base; b0 < end; b0 += kRows) {
        double l[kRows];
#pragma unroll
        for (int q = 0; q < kRows; q++) l[q] = (t < e && b0 + q < end) ? col[b0 + q] : 0.0;
        __syncthreads();
        for (int idx = t; idx < kRows * RB; idx += kTh) {
            const int q = idx % kRows, r = idx / kRows;
            const bool in = b0 + q < end && r < nr;
            xs[q][r] = in ? X[(int64_t)(r0 + r) * ldx + front_var(f, b0 + q)] : 0.0;
        }
        __syncthreads();
        if ((t & ~31) >= e) continue;  // the whole warp
#pragma unroll
        for (int q = 0; q < kRows; q++)
#pragma unroll
            for (int r = 0; r < RB; r++) acc[r] += l[q] * xs[q][r];
    }
    if (t >= e) return;
#pragma unroll
    for (int r = 0; r < RB; r++)
        if (r < nr) part[((int64_t)c0 * nrhs + r0 + r) * kMaxP + t] = acc[r];
}

// Backward step, part 2: z = x(piv vars) - sum of the chunk partials, then
// L11^T x = z, eight pivots at a time from the last, thread t with column t of L11.
__global__ void __launch_bounds__(kTh) k_sys_bwd_tri(ctp_sfront f, double *X, int64_t ldx, int nrhs, int chunk,
                                                     const double *part) {
    __shared__ double x[kMaxP];
    const int e = *f.nelim, t = threadIdx.x, warp = t >> 5;
    const int64_t nch = (f.n - e + chunk - 1) / chunk;
    X += (int64_t)blockIdx.x * ldx;
    part += (int64_t)blockIdx.x * kMaxP;
    const double *col = f.L + (int64_t)t * f.ldl;
    const int top = (e + kS - 1) / kS - 1;  // the last step's index
    double l[kAhead][kS];                   // L(k, t) of the next steps' rows k
#pragma unroll
    for (int s = 0; s < kAhead; s++)
#pragma unroll
        for (int j = 0; j < kS; j++) {
            const int i = kS * (top - s) + j;
            l[s][j] = (i > t && i < e) ? col[i] : 0.0;
        }
    int var = 0;
    double v = 0.0;
    int last = kMaxP;  // rows after `last` act on this column: not the second of its own
                       // 2x2 block, where the (t+1, t) slot holds D
    if (t < e) {
        var = f.rows[f.perm[t]];
        last = t + (f.piv[t] == CTP_PIVKIND_2X2_FIRST);
        double s0 = 0.0, s1 = 0.0;
        int64_t c = 0;
#pragma unroll 4
        for (; c + 1 < nch; c += 2) {
            s0 += part[c * nrhs * kMaxP + t];
            s1 += part[(c + 1) * nrhs * kMaxP + t];
        }
        if (c < nch) s0 += part[c * nrhs * kMaxP + t];
        v = X[var] - (s0 + s1);
    }
    for (int g = top; g >= 0; g -= kAhead) {
#pragma unroll
        for (int s = 0; s < kAhead; s++) {
            const int k = kS * (g - s);
            if (k >= 0) {
                if (warp == k >> 5) {
#pragma unroll
                    for (int j = kS - 1; j >= 0; j--) {
                        const double xj = __shfl_sync(0xffffffffu, v, (k + j) & 31);
                        if (k + j > last && k + j < e) v -= l[s][j] * xj;
                    }
                    if (t >= k && t < k + kS) x[t] = t < e ? v : 0.0;
                }
                __syncthreads();
                if (warp < k >> 5) {
                    double s0 = 0.0, s1 = 0.0;
#pragma unroll
                    for (int j = 0; j < kS; j += 2) {
                        if (k + j > last && k + j < e) s0 += l[s][j] * x[k + j];
                        if (k + j + 1 < e) s1 += l[s][j + 1] * x[k + j + 1];
                    }
                    v -= s0 + s1;
                }
#pragma unroll
                for (int j = 0; j < kS; j++) {
                    const int i = k - kS * kAhead + j;
                    l[s][j] = i > t ? col[i] : 0.0;
                }
            }
        }
    }
    if (t < e) X[var] = v;
}

// R -= M X (kAbs = false) or R += |M| 1 (kAbs = true: the row sums of |M|),
// M symmetric with its lower triangle stored (column-major, ldm), one 64 x 64
// tile of the lower block triangle per CTA; both the tile and its transpose
// contribute, accumulated with FP64 atomics.
constexpr int kRT = 64;
template <bool kAbs>
__global__ void __launch_bounds__(kTh) k_symv(int64_t N, const double *__restrict__ M, int64_t ldm,
                                              int nrhs, const double *__restrict__ X, int64_t ldx,
                                              double *R, int64_t ldr) {
    __shared__ double a[kRT][kRT + 1];
    __shared__ double xi[kRT], xj[kRT];
    const int64_t b = blockIdx.x;
    int64_t ti = (int64_t)((sqrt(8.0 * (double)b + 1.0) - 1.0) * 0.5);
    while ((ti + 1) * (ti + 2) / 2 <= b) ti++;
    while (ti * (ti + 1) / 2 > b) ti--;
    const int64_t tj = b - ti * (ti + 1) / 2;
    const int64_t i0 = ti * kRT, j0 = tj * kRT;
    const bool diag = ti == tj;
    for (int idx = threadIdx.x; idx < kRT * kRT; idx += kTh) {
        const int ii = idx % kRT, jj = idx / kRT;
        const int64_t gi = i0 + ii, gj = j0 + jj;
        double v = (gi < N && gj < N && (!diag || ii >= jj)) ? M[gj * ldm + gi] : 0.0;
        a[ii][jj] = kAbs ? fabs(v) : v;
    }
    const int nr = kAbs ? 1 : nrhs;
    for (int r = 0; r < nr; r++) {
        __syncthreads();
        if (threadIdx.x < kRT) {
            const int64_t g = j0 + threadIdx.x;
            xj[threadIdx.x] = kAbs ? 1.0 : (g < N ? X[(int64_t)r * ldx + g] : 0.0);
        } else if (threadIdx.x < 2 * kRT) {
            const int64_t g = i0 + threadIdx.x - kRT;
            xi[threadIdx.x - kRT] = kAbs ? 1.0 : (g < N ? X[(int64_t)r * ldx + g] : 0.0);
        }
        __syncthreads();
        if (threadIdx.x < kRT) {
            const int ii = threadIdx.x;
            double s = 0.0;
            for (int jj = 0; jj < kRT; jj++) s += a[ii][jj] * xj[jj];
            if (i0 + ii < N) atomicAdd(R + (int64_t)r * ldr + i0 + ii, kAbs ? s : -s);
        } else if (threadIdx.x < 2 * kRT) {
            const int jj = threadIdx.x - kRT;
            double s = 0.0;
            for (int ii = 0; ii < kRT; ii++)
                if (!diag || ii > jj) s += a[ii][jj] * xi[ii];
            if (j0 + jj < N) atomicAdd(R + (int64_t)r * ldr + j0 + jj, kAbs ? s : -s);
        }
    }
}

__device__ __forceinline__ void atomic_max_nonneg(double *addr, double v) {
    // non-negative doubles order like their bit patterns
    atomicMax(reinterpret_cast<unsigned long long *>(addr), (unsigned long long)__double_as_longlong(v));
}

// mx[3 r + 0..2] = max |R(:, r)|, max |X(:, r)|, max |B(:, r)|; mx[3 nrhs] = max row sum.
__global__ void __launch_bounds__(kTh) k_maxabs(int64_t N, int nrhs, const double *R, int64_t ldr,
                                                const double *X, int64_t ldx, const double *B,
                                                int64_t ldb, const double *rowsum, double *mx) {
    const int r = blockIdx.y;
    double m0 = 0.0, m1 = 0.0, m2 = 0.0, m3 = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * kTh + threadIdx.x; i < N; i += (int64_t)gridDim.x * kTh) {
        m0 = fmax(m0, fabs(R[(int64_t)r * ldr + i]));
        m1 = fmax(m1, fabs(X[(int64_t)r * ldx + i]));
        m2 = fmax(m2, fabs(B[(int64_t)r * ldb + i]));
        if (r == 0 && rowsum != nullptr) m3 = fmax(m3, rowsum[i]);
    }
    for (int o = 16; o > 0; o >>= 1) {
        m0 = fmax(m0, __shfl_xor_sync(0xffffffffu, m0, o));
        m1 = fmax(m1, __shfl_xor_sync(0xffffffffu, m1, o));
        m2 = fmax(m2, __shfl_xor_sync(0xffffffffu, m2, o));
        m3 = fmax(m3, __shfl_xor_sync(0xffffffffu, m3, o));
    }
    if ((threadIdx.x & 31) == 0) {
        atomic_max_nonneg(mx + 3 * r + 0, m0);
        atomic_max_nonneg(mx + 3 * r + 1, m1);
        atomic_max_nonneg(mx + 3 * r + 2, m2);
        if (r == 0 && rowsum != nullptr) atomic_max_nonneg(mx + 3 * nrhs, m3);
    }
}

// berr[r] = ||R||_inf / (||M||_inf ||X||_inf + ||B||_inf)   (Section 7)
__global__ void k_berr(int nrhs, const double *mx, double *berr) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= nrhs) return;
    const double den = mx[3 * nrhs] * mx[3 * r + 1] + mx[3 * r + 2];
    berr[r] = den > 0.0 ? mx[3 * r] / den : 0.0;
}

// X(:, r) += Dx(:, r)
__global__ void k_axpy(int64_t N, int nrhs, double *X, int64_t ldx, const double *Dx, int64_t ldd) {
    const int r = blockIdx.y;
    for (int64_t i = (int64_t)blockIdx.x * kTh + threadIdx.x; i < N; i += (int64_t)gridDim.x * kTh)
        X[(int64_t)r * ldx + i] += Dx[(int64_t)r * ldd + i];
}

// Gradient of a loss through x = M^{-1} b with respect to the stored lower
// triangle of the symmetric M (each stored off-diagonal entry stands for both
// m_ij and m_ji): dL/dm_ij = -sum_r (g_ir x_jr + g_jr x_ir) for i > j and
// -sum_r g_ir x_ir on the diagonal, with g = M^{-T} dL/dx.  Dense form: the lower
// triangle of an N x N column-major output (strict upper triangle zeroed).
__global__ void __launch_bounds__(kTh) k_sym_grad_dense(int64_t N, int nrhs, const double *__restrict__ G,
                                                        int64_t ldg, const double *__restrict__ X,
                                                        int64_t ldx, double *__restrict__ out,
                                                        int64_t ldo) {
    for (int64_t j = blockIdx.y; j < N; j += gridDim.y)
    for (int64_t i = (int64_t)blockIdx.x * kTh + threadIdx.x; i < N; i += (int64_t)gridDim.x * kTh) {
        double s = 0.0;
        if (i > j) {
            for (int r = 0; r < nrhs; r++)
                s += G[(int64_t)r * ldg + i] * X[(int64_t)r * ldx + j] +
                     G[(int64_t)r * ldg + j] * X[(int64_t)r * ldx + i];
        } else if (i == j) {
            for (int r = 0; r < nrhs; r++) s += G[(int64_t)r * ldg + i] * X[(int64_t)r * ldx + i];
        }
        out[j * ldo + i] = -s;
    }
}

// The same restricted to a pattern of stored entries (row[k], col[k]), any order;
// an entry with row == col is a diagonal entry, otherwise it stands for both
// (row, col) and (col, row).
__global__ void __launch_bounds__(kTh) k_sym_grad_pattern(int64_t nnz, const int32_t *__restrict__ row,
                                                          const int32_t *__restrict__ col, int nrhs,
                                                          const double *__restrict__ G, int64_t ldg,
                                                          const double *__restrict__ X, int64_t ldx,
                                                          double *__restrict__ out) {
    for (int64_t k = (int64_t)blockIdx.x * kTh + threadIdx.x; k < nnz; k += (int64_t)gridDim.x * kTh) {
        const int64_t i = row[k], j = col[k];
        double s = 0.0;
        // the same expressions as the dense kernel, so both round alike
        if (i != j) {
            for (int r = 0; r < nrhs; r++)
                s += G[(int64_t)r * ldg + i] * X[(int64_t)r * ldx + j] +
                     G[(int64_t)r * ldg + j] * X[(int64_t)r * ldx + i];
        } else {
            for (int r = 0; r < nrhs; r++) s += G[(int64_t)r * ldg + i] * X[(int64_t)r * ldx + i];
        }
        out[k] = -s;
    }
}

// R -= A X for a symmetric A given by its lower triangle in compressed columns
// (kAbs: R += |A| 1, the row sums of |A|).  A column's entries update R(i) (atomics)
// and their transposes accumulate into R(j).  G lanes share a column, eight right-hand
// sides at a time, by the columns' mean length: a lane's chain of atomics stays short, and
// few entries do not idle a warp.  One lane for the columns of meshes, whose
// neighbours' X(i) and R(i) are neighbours in memory; more where the matrix has few
// columns.  Columns of more than kLong entries a lane are shared by the warp.
// Measured, 16 right-hand sides, rows at random: a warp per column / a lane per column / this
// rule: N = 2000, 40 a column 46 / 167 / 45 us; N = 20000, 70 279 / 821 / 211; N =
// 200000, 6 1674 / 156 / 178, 20 1693 / 564 / 544, 60 2530 / 1739 / 1565.  At most 16
// entries a lane (8: 521 and 1592 us for the last two, but 22% slower on bands).
constexpr int kLong = 64, kSpmvPer = 16;
constexpr int64_t kSpmvFill = 152 * 512;
template <bool kAbs>
__global__ void __launch_bounds__(kTh) k_spmv_csc(int64_t N, const int64_t *__restrict__ colptr,
                                                  const int32_t *__restrict__ rowind,
                                                  const double *__restrict__ val, int nrhs,
                                                  const double *__restrict__ X, int64_t ldx, double *R,
                                                  int64_t ldr) {
    constexpr int NR = kAbs ? 1 : 8;
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (kTh / 32);
    const int64_t per = (colptr[N] - colptr[0] + N - 1) / N;
    int G = 1;
    while (G < 32 && (G * kSpmvPer < per || (G < per && N * G < kSpmvFill))) G *= 2;
    const int sub = lane & (G - 1), wc = 32 / G;
    for (int64_t j0 = wc * ((int64_t)blockIdx.x * (kTh / 32) + (threadIdx.x >> 5)); j0 < N; j0 += wc * warps) {
        const int64_t j = j0 + lane / G;
        const int64_t q0 = j < N ? colptr[j] : 0, q1 = j < N ? colptr[j + 1] : 0;
        const bool lng = G < 32 && q1 - q0 > kLong * G;
        const unsigned longs = __ballot_sync(0xffffffffu, lng && sub == 0);
        const int nr = kAbs ? 1 : nrhs;
        for (int r0 = 0; r0 < nr; r0 += NR) {
            const int ng = min(NR, nr - r0);
            const double *Xr = X + (int64_t)r0 * ldx;
            double *Rr = R + (int64_t)r0 * ldr;
            double xj[NR], t[NR];
#pragma unroll
            for (int r = 0; r < NR; r++) {
                xj[r] = kAbs ? 1.0 : (r < ng && q1 > q0 ? Xr[r * ldx + j] : 0.0);
                t[r] = 0.0;
            }
            if (!lng)
                for (int64_t q = q0 + sub; q < q1; q += G) {
                    const int64_t i = rowind[q];
                    const double a = kAbs ? fabs(val[q]) : val[q];
#pragma unroll
                    for (int r = 0; r < NR; r++) {
                        if (r >= ng) break;
                        if (i == j) {
                            t[r] += a * xj[r];
                        } else {
                            atomicAdd(Rr + r * ldr + i, kAbs ? a : -a * xj[r]);
                            t[r] += a * (kAbs ? 1.0 : Xr[r * ldx + i]);
                        }
                    }
                }
            for (int o = G >> 1; o > 0; o >>= 1)
#pragma unroll
                for (int r = 0; r < NR; r++)
                    if (r < ng) t[r] += __shfl_xor_sync(0xffffffffu, t[r], o);
            if (!lng && q1 > q0 && sub == 0) {
#pragma unroll
                for (int r = 0; r < NR; r++)
                    if (r < ng) atomicAdd(Rr + r * ldr + j, kAbs ? t[r] : -t[r]);
            }
            for (unsigned b = longs; b; b &= b - 1) {
                const int l = __ffs(b) - 1;
                const int64_t jl = j0 + l / G, a0 = __shfl_sync(0xffffffffu, q0, l), a1 = __shfl_sync(0xffffffffu, q1, l);
                for (int r = 0; r < ng; r++) {
                    const double x = kAbs ? 1.0 : Xr[r * ldx + jl];
                    double s = 0.0;
                    for (int64_t q = a0 + lane; q < a1; q += 32) {
                        const int64_t i = rowind[q];
                        const double a = kAbs ? fabs(val[q]) : val[q];
                        if (i == jl) {
                            s += a * x;
                        } else {
                            atomicAdd(Rr + r * ldr + i, kAbs ? a : -a * x);
                            s += a * (kAbs ? 1.0 : Xr[r * ldx + i]);
                        }
                    }
                    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                    if (lane == 0) atomicAdd(Rr + r * ldr + jl, kAbs ? s : -s);
                }
            }
        }
    }
}

inline unsigned blocks_for(int64_t n) { return (unsigned)((n + kTh - 1) / kTh); }

// Rows per chunk of the backward sums: enough chunks for the SMs, not so many that
// the one CTA per right-hand side is long in adding them up.
int bwd_chunk(int64_t n) {
    const int64_t c = (n + kRows * 152 - 1) / (kRows * 152) * kRows;
    return (int)(c < kRows ? kRows : c);
}

// Right-hand sides per CTA of the updates: as few as leave at most two CTAs per
// SM (a front's tiles alone do not fill the chip, and a CTA's time is its FP64 work).
int rhs_per_cta(unsigned tiles, int nrhs) {
    int rb = 1;
    while (rb < 8 && rb < nrhs && (int64_t)tiles * ((nrhs + rb - 1) / rb) > 304) rb *= 2;
    return rb;
}

}  // namespace

size_t sys_solve_ws_bytes(int64_t nmax, int nrhs) {
    // a front of n <= nmax rows has at most 152 chunks of at least kRows rows
    const int64_t nch = nmax < kRows * 152 ? (nmax + kRows - 1) / kRows : 152;
    return align256(sizeof(double) * (size_t)kMaxP * nrhs) +
           align256(sizeof(double) * (size_t)nch * nrhs * kMaxP);
}

cudaError_t launch_sys_forward(const ctp_sfront &f, double *X, int64_t ldx, int nrhs, void *ws,
                               cudaStream_t st) {
    double *Y = (double *)ws;
    k_sys_fwd_tri<<<(unsigned)nrhs, kTh, 0, st>>>(f, X, ldx, Y);
    const unsigned tiles = (unsigned)((f.n + kRows - 1) / kRows);
    if (tiles > 0) {
        const int rb = rhs_per_cta(tiles, nrhs);
        const unsigned grid = tiles * (unsigned)((nrhs + rb - 1) / rb);
        switch (rb) {
        case 1: k_sys_fwd_upd<1><<<grid, kTh, 0, st>>>(f, X, ldx, nrhs, Y, tiles); break;
        case 2: k_sys_fwd_upd<2><<<grid, kTh, 0, st>>>(f, X, ldx, nrhs, Y, tiles); break;
        case 4: k_sys_fwd_upd<4><<<grid, kTh, 0, st>>>(f, X, ldx, nrhs, Y, tiles); break;
        default: k_sys_fwd_upd<8><<<grid, kTh, 0, st>>>(f, X, ldx, nrhs, Y, tiles); break;
        }
    }
    return cudaGetLastError();
}

cudaError_t launch_sys_backward(const ctp_sfront &f, double *X, int64_t ldx, int nrhs, void *ws,
                                cudaStream_t st) {
    double *part = (double *)((char *)ws + align256(sizeof(double) * (size_t)kMaxP * nrhs));
    const int chunk = bwd_chunk(f.n);
    const unsigned chunks = (unsigned)((f.n + chunk - 1) / chunk);  // upper bound on those below the pivots
    if (chunks > 0) {
        const int rb = rhs_per_cta(chunks, nrhs);
        const unsigned grid = chunks * (unsigned)((nrhs + rb - 1) / rb);
        switch (rb) {
        case 1: k_sys_bwd_part<1><<<grid, kTh, 0, st>>>(f, X, ldx, nrhs, chunk, part, chunks); break;
        case 2: k_sys_bwd_part<2><<<grid, kTh, 0, st>>>(f, X, ldx, nrhs, chunk, part, chunks); break;
        case 4: k_sys_bwd_part<4><<<grid, kTh, 0, st>>>(f, X, ldx, nrhs, chunk, part, chunks); break;
        default: k_sys_bwd_part<8><<<grid, kTh, 0, st>>>(f, X, ldx, nrhs, chunk, part, chunks); break;
        }
    }
    k_sys_bwd_tri<<<(unsigned)nrhs, kTh, 0, st>>>(f, X, ldx, nrhs, chunk, part);
    return cudaGetLastError();
}

cudaError_t launch_symv_residual(int64_t N, const double *M, int64_t ldm, int nrhs, const double *X,
                                 int64_t ldx, double *R, int64_t ldr, cudaStream_t st) {
    const int64_t nt = (N + kRT - 1) / kRT;
    const int64_t tiles = nt * (nt + 1) / 2;
    if (tiles == 0) return cudaSuccess;
    if (tiles > 0x7fffffffLL) return cudaErrorInvalidValue;
    k_symv<false><<<(unsigned)tiles, kTh, 0, st>>>(N, M, ldm, nrhs, X, ldx, R, ldr);
    return cudaGetLastError();
}

cudaError_t launch_abs_rowsum(int64_t N, const double *M, int64_t ldm, double *rowsum,
                              cudaStream_t st) {
    const int64_t nt = (N + kRT - 1) / kRT;
    const int64_t tiles = nt * (nt + 1) / 2;
    if (tiles == 0) return cudaSuccess;
    if (tiles > 0x7fffffffLL) return cudaErrorInvalidValue;
    k_symv<true><<<(unsigned)tiles, kTh, 0, st>>>(N, M, ldm, 1, nullptr, 0, rowsum, N);
    return cudaGetLastError();
}

cudaError_t launch_backward_error(int64_t N, int nrhs, const double *R, int64_t ldr, const double *X,
                                  int64_t ldx, const double *B, int64_t ldb, const double *rowsum,
                                  double *mx, double *berr, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(mx, 0, sizeof(double) * (3 * (size_t)nrhs + 1), st);
    if (e != cudaSuccess) return e;
    const unsigned gx = (unsigned)(N < 1 ? 1 : ((N + kTh - 1) / kTh < 304 ? (N + kTh - 1) / kTh : 304));
    k_maxabs<<<dim3(gx, nrhs), kTh, 0, st>>>(N, nrhs, R, ldr, X, ldx, B, ldb, rowsum, mx);
    k_berr<<<(nrhs + 127) / 128, 128, 0, st>>>(nrhs, mx, berr);
    return cudaGetLastError();
}

cudaError_t launch_axpy(int64_t N, int nrhs, double *X, int64_t ldx, const double *Dx, int64_t ldd,
                        cudaStream_t st) {
    if (N == 0 || nrhs == 0) return cudaSuccess;
    const unsigned gx = (unsigned)((N + kTh - 1) / kTh < 1216 ? (N + kTh - 1) / kTh : 1216);
    k_axpy<<<dim3(gx, nrhs), kTh, 0, st>>>(N, nrhs, X, ldx, Dx, ldd);
    return cudaGetLastError();
}

cudaError_t launch_sym_grad_dense(int64_t N, int nrhs, const double *G, int64_t ldg, const double *X,
                                  int64_t ldx, double *out, int64_t ldo, cudaStream_t st) {
    if (N == 0) return cudaSuccess;
    const unsigned gx = blocks_for(N) < 64 ? blocks_for(N) : 64;
    const unsigned gy = N < 65535 ? (unsigned)N : 65535u;
    k_sym_grad_dense<<<dim3(gx, gy), kTh, 0, st>>>(N, nrhs, G, ldg, X, ldx, out, ldo);
    return cudaGetLastError();
}

cudaError_t launch_sym_grad_pattern(int64_t nnz, const int32_t *row, const int32_t *col, int nrhs,
                                    const double *G, int64_t ldg, const double *X, int64_t ldx,
                                    double *out, cudaStream_t st) {
    if (nnz == 0) return cudaSuccess;
    const unsigned g = blocks_for(nnz) < 4096 ? blocks_for(nnz) : 4096;
    k_sym_grad_pattern<<<g, kTh, 0, st>>>(nnz, row, col, nrhs, G, ldg, X, ldx, out);
    return cudaGetLastError();
}

cudaError_t launch_spmv_csc_residual(int64_t N, const int64_t *colptr, const int32_t *rowind,
                                     const double *val, int nrhs, const double *X, int64_t ldx, double *R,
                                     int64_t ldr, cudaStream_t st) {
    const int64_t g = (N + 7) / 8 < 152 * 8 ? (N + 7) / 8 : 152 * 8;
    k_spmv_csc<false><<<(unsigned)g, kTh, 0, st>>>(N, colptr, rowind, val, nrhs, X, ldx, R, ldr);
    return cudaGetLastError();
}

cudaError_t launch_spmv_csc_abs_rowsum(int64_t N, const int64_t *colptr, const int32_t *rowind,
                                       const double *val, double *rowsum, cudaStream_t st) {
    const int64_t g = (N + 7) / 8 < 152 * 8 ? (N + 7) / 8 : 152 * 8;
    k_spmv_csc<true><<<(unsigned)g, kTh, 0, st>>>(N, colptr, rowind, val, 1, nullptr, 0, rowsum, N);
    return cudaGetLastError();
}

}  // namespace ctp
