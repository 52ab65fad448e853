// form.cu -- K6 (FP64): the Form task S = L21 D11 L21^T = W21 L21^T (Section 1
// task list), lower triangle only, in FP64 on the tensor cores.
//
// GB300's FP64 pipe gives 1.26 TFLOP/s, its BF16 tensor cores about 1700, and a
// product of two FP64 matrices is 36 exact BF16 products: the operands come as
// eight digit slices each (slices.cuh), the products d_s d_t' of slices with
// g = s + t <= 7 are summed per g in FP32 without rounding, and the epilogue
// adds the eight sums, which are integers, in 64-bit integer arithmetic and
// rounds once to FP64.  slices.cuh says what this loses (less than the rounding
// of FP64 multiply-adds) and which rows it is not good enough for: those are
// marked, and the epilogue takes their entries by FP64 multiply-adds.
//
// Kernel: persistent, one CTA per SM, tiles of 128 rows x 64 columns.
//   warp 0      producer: bulk copies of K blocks of 32 pivots (W 64 KB, L 32 KB:
//               all slices, already in the MMA's layout) through a ring of two
//               stages.
//   warp 1      MMA issuer: the slices of L lie one after another, so slice s of W
//               against slices 0..7-s of L is one operand of 64 (8 - s) rows and
//               its results land in the accumulators of g = s..7 (64 TMEM
//               columns each, all 512 in use): twelve MMAs of N <= 256 per
//               16 pivots for all 36 products.
//   warps 2-17  epilogue: a thread holds 16 columns of one row of S as 64-bit
//               integers; the accumulators are handed back as soon as they have
//               been added up, and rounding and stores overlap the next tile.
// Bound: tensor pipe for e from about 100 on, S traffic and the epilogue's integer
// instructions below.  FP64 multiply-adds ran at 0.99 of the FP64 pipe's rate.
// Every mbarrier wait is bounded; on timeout the kernel records CTP_ETIMEOUT,
// waits (bounded) for its copies in flight, frees its tensor memory and returns.
#include "slices.cuh"
#include "tc_common.cuh"

namespace ctp {

using namespace tc;

namespace {

constexpr int kBM = kWRows, kBN = kLRows;
constexpr int kEpiWarps = 16, kThreads = 32 * (2 + kEpiWarps);
constexpr int kCols = kBN / (kEpiWarps / 4);  // columns of S per epilogue thread
constexpr int kStages = 2;
constexpr uint32_t kStageBytes = kWBlock + kLBlock;
constexpr size_t kSmem = kStages * (size_t)kStageBytes + 1024;
constexpr int kPanel = 8;  // column blocks of a panel of the walk

struct Bars {
    unsigned long long full[kStages], empty[kStages], acc_full, acc_empty;
    uint32_t tmem_base;
    int abort;
};

// K-major operand with the 64-byte swizzle: rows of 64 bytes, groups of 8 rows 512
// bytes apart
__device__ __forceinline__ uint64_t sdesc64(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(512 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)4 << 61;
    return d;
}

__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, unsigned long long *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void tmem_ld16_nowait(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}

struct Tile {
    int ti, tj, e;
    int64_t m, lds, ldl;
    SliceBuf sb;
    const double *L21, *D;
    const int32_t *piv;
    void *S;
};

struct Work {
    // one supernode
    SliceBuf sb;
    int64_t m, lds, ldl;
    const double *L21, *D;
    const int32_t *piv, *nelim;
    void *S;
    // a batch (fronts != nullptr): item t is tile item_tile[t] of front
    // item_front[t], or without item_tile the item's place among the front's
    // consecutive items
    const ctp_front *fronts;
    const BFront *tab;
    char *ws;
    const int *item_front, *item_tile;
    BatchOpts o;
    int64_t count;  // items, or slots of the walk
};

// The walk over one supernode's tiles: panels of kPanel column blocks, inside a
// panel the row blocks one after another, inside a row block its column blocks.
// The tiles that run at one time then share a few W and L blocks, and W is read
// from HBM once per panel (512 columns of S), not per column block.  Slots above
// the diagonal are skipped.
__host__ __device__ inline int64_t slots_before(int64_t P, int64_t nM) {
    return kPanel * (P * nM - (kPanel / 2) * (P * (P - 1) / 2));
}
__host__ __device__ inline int64_t walk_slots(int64_t m) {
    const int64_t nM = (m + kBM - 1) / kBM, nN = (m + kBN - 1) / kBN;
    return slots_before((nN + kPanel - 1) / kPanel, nM);
}

// The k-th tile of this CTA; false past the end.  ti < 0: a slot without a tile.
__device__ __forceinline__ bool tile_at(const Work &w, int64_t k, Tile &x) {
    const int64_t t = blockIdx.x + k * (int64_t)gridDim.x;
    if (t >= w.count) return false;
    if (w.fronts != nullptr) {
        const int f = w.item_front[t];
        const BFront b = w.tab[f];
        const int64_t q = w.item_tile != nullptr ? (int64_t)w.item_tile[t] : t - b.f0;
        // row block i has 2 (i + 1) tiles, i (i + 1) precede it
        int64_t i = (int64_t)((sqrtf(4.0f * (float)q + 1.0f) - 1.0f) * 0.5f);
        while ((i + 1) * (i + 2) <= q) i++;
        while (i * (i + 1) > q) i--;
        x.ti = (int)i;
        x.tj = (int)(q - i * (i + 1));
        ctp_options oo;
        oo.pivot = w.o.pivot;
        oo.smode = w.o.smode;
        oo.prec = w.o.prec;
        const BSection sec = bsection(b.n, b.p, &oo);
        x.sb = bsection_slices(w.ws + b.ws, sec, b.p);
        const ctp_front &fr = w.fronts[f];
        x.m = b.m;
        x.e = *fr.nelim;
        x.L21 = fr.A + b.p;
        x.ldl = fr.lda;
        x.D = fr.D;
        x.piv = fr.piv;
        x.S = fr.S;
        x.lds = fr.lds;
        return true;
    }
    x.sb = w.sb;
    x.m = w.m;
    x.e = *w.nelim;
    x.L21 = w.L21;
    x.ldl = w.ldl;
    x.D = w.D;
    x.piv = w.piv;
    x.S = w.S;
    x.lds = w.lds;
    const int64_t nM = (w.m + kBM - 1) / kBM, nN = (w.m + kBN - 1) / kBN;
    int64_t lo = 0, hi = (nN + kPanel - 1) / kPanel;
    while (hi - lo > 1) {
        const int64_t mid = (lo + hi) >> 1;
        if (slots_before(mid, nM) <= t)
            lo = mid;
        else
            hi = mid;
    }
    const int64_t r = t - slots_before(lo, nM);
    const int64_t ti = lo * (kPanel / 2) + r / kPanel, tj = lo * kPanel + r % kPanel;
    x.tj = (int)tj;
    x.ti = (tj < nN && tj <= 2 * ti + 1) ? (int)ti : -1;
    return true;
}

// V = 0, or V 2^ex outside the normal range of FP64
__device__ __noinline__ double to_fp64_rare(long long V, int ex) {
    return V == 0 ? 0.0 : scalbn((double)V, ex);
}
// V 2^ex rounded to nearest even, in integer instructions (the FP64 pipe takes
// about 20 cycles per warp instruction and SM)
__device__ __forceinline__ double to_fp64(long long V, int ex) {
    const unsigned long long a = V < 0 ? 0ull - (unsigned long long)V : (unsigned long long)V;
    const int lz = __clzll((long long)a) & 63;
    const unsigned long long n = a << lz;
    unsigned long long mant = n >> 11;
    mant += ((n >> 10) & 1u) & (((n & 0x3FFull) != 0ull ? 1u : 0u) | (unsigned)(mant & 1u));
    const int be = 63 - lz + ex + 1022;  // biased exponent - 1: the hidden bit adds the 1
    if ((unsigned)be >= 2045u || V == 0) return to_fp64_rare(V, ex);
    const unsigned long long bits = ((unsigned long long)be << 52) + mant;
    return __longlong_as_double((long long)(bits | ((unsigned long long)V & 0x8000000000000000ull)));
}

// Entries (i, j..j+7) of S by FP64 multiply-adds over the stored L21 and D11 (i < m;
// columns past i count as 0): the marked rows' path.
__device__ __noinline__ void plain_entries(const double *L21, int64_t ldl, const double *D, const int32_t *piv, int e,
                                          int64_t i, int64_t j, double (&acc)[8]) {
#pragma unroll
    for (int c = 0; c < 8; c++) acc[c] = 0.0;
    for (int k = 0; k < e; k++) {
        const int kd = piv[k];
        if (kd == CTP_PIVKIND_ZERO) continue;
        const double *col = L21 + (int64_t)k * ldl;
        double w = col[i] * D[2 * k];
        if (kd == CTP_PIVKIND_2X2_FIRST) w = fma(col[i + ldl], D[2 * k + 1], w);
        if (kd == CTP_PIVKIND_2X2_SECOND) w = fma(col[i - ldl], D[2 * k - 1], w);
#pragma unroll
        for (int c = 0; c < 8; c++)
            if (j + c <= i) acc[c] = fma(w, col[j + c], acc[c]);
    }
}

// kMode: ctp_smode of S
template <int kMode>
__global__ void __launch_bounds__(kThreads, 1) k_form_fp64(const Work wk, int32_t *__restrict__ info) {
    using OutT = typename std::conditional<kMode == CTP_S_FP32 || kMode == CTP_S_FP32_PACKED, float, double>::type;
    constexpr bool kPacked = kMode == CTP_S_FP64_PACKED || kMode == CTP_S_FP32_PACKED;
    constexpr bool kSub = kMode == CTP_S_FP64_SUB;
    extern __shared__ unsigned char smraw[];
    __shared__ Bars bars;
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; s++) {
            mbar_init(&bars.full[s], 1);
            mbar_init(&bars.empty[s], 1);
        }
        mbar_init(&bars.acc_full, 1);
        mbar_init(&bars.acc_empty, kEpiWarps);
        bars.abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc(&bars.tmem_base, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = bars.tmem_base;

    if (warp == 0) {
        // ---------------- producer
        if (lane == 0) {
            int stage = 0, issued = 0;
            uint32_t phase = 0;
            Tile x;
            bool ok = true;
            for (int64_t k = 0; ok && tile_at(wk, k, x); k++) {
                if (x.ti < 0) continue;
                // rows of the tile in use, in groups of 8
                const uint32_t rw = (uint32_t)(min((int64_t)kBM, x.m - (int64_t)x.ti * kBM) + 7) & ~7u;
                const uint32_t rl = (uint32_t)(min((int64_t)kBN, x.m - (int64_t)x.tj * kBN) + 7) & ~7u;
                const int KB = (x.e + kSliceK - 1) / kSliceK;
                const unsigned char *srcW = x.sb.W + (size_t)x.ti * x.sb.kb * kWBlock;
                const unsigned char *srcL = x.sb.L + (size_t)x.tj * x.sb.kb * kLBlock;
                for (int kb = 0; kb < KB; kb++) {
                    if (!mbar_wait(&bars.empty[stage], phase ^ 1u, &bars.abort)) {
                        ok = false;
                        break;
                    }
                    uint8_t *dW = smem + (size_t)stage * kStageBytes, *dL = dW + kWBlock;
                    mbar_expect_tx(&bars.full[stage], kSlices * 64 * (rw + rl));
                    if (rw == kBM)
                        bulk_load(dW, srcW + (size_t)kb * kWBlock, kWBlock, &bars.full[stage]);
                    else
                        for (int s = 0; s < kSlices; s++)
                            bulk_load(dW + s * kWSlice, srcW + (size_t)kb * kWBlock + s * kWSlice, rw * 64,
                                      &bars.full[stage]);
                    if (rl == kBN)
                        bulk_load(dL, srcL + (size_t)kb * kLBlock, kLBlock, &bars.full[stage]);
                    else
                        for (int s = 0; s < kSlices; s++)
                            bulk_load(dL + s * kLSlice, srcL + (size_t)kb * kLBlock + s * kLSlice, rl * 64,
                                      &bars.full[stage]);
                    issued++;
                    if (++stage == kStages) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
            }
            if (!ok) atomicExch(&bars.abort, 1);
            if (*(volatile int *)&bars.abort) {
                // no CTA leaves with copies in flight: the last one of each stage
                int never = 0;
                for (int b = 0; b < kStages && b < issued; b++) {
                    const int i = issued - 1 - b;
                    mbar_wait(&bars.full[i % kStages], (uint32_t)(i / kStages) & 1u, &never);
                }
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0, accphase = 0;
            Tile x;
            bool ok = true;
            for (int64_t k = 0; ok && tile_at(wk, k, x); k++) {
                if (x.ti < 0) continue;
                if (!mbar_wait(&bars.acc_empty, accphase ^ 1u, &bars.abort)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const int KB = (x.e + kSliceK - 1) / kSliceK;
                for (int kb = 0; kb < KB; kb++) {
                    if (!mbar_wait(&bars.full[stage], phase, &bars.abort)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t a0 = smem_u32(smem + (size_t)stage * kStageBytes), b0 = a0 + kWBlock;
                    const int nkk = min(kSliceK / kUmmaK, (x.e - kb * kSliceK + kUmmaK - 1) / kUmmaK);
                    for (int kk = 0; kk < nkk; kk++) {
                        const uint32_t acc = (kb > 0 || kk > 0) ? 1u : 0u;
                        const uint64_t bl = sdesc64(b0 + kk * 32), bh = sdesc64(b0 + 4 * kLSlice + kk * 32);
#pragma unroll
                        for (int s = 0; s < kSlices; s++) {
                            // slice s against slices 0..7-s: the accumulators of g = s..7;
                            // s = 0 comes first and touches them all
                            const uint64_t a = sdesc64(a0 + s * kWSlice + kk * 32);
                            const int nn = kBN * (kSlices - s);
                            umma_bf16(tmem + s * kBN, a, bl, idesc_bf16(kBM, nn < 256 ? nn : 256), s ? 1u : acc);
                            if (nn > 256)
                                umma_bf16(tmem + s * kBN + 256, a, bh, idesc_bf16(kBM, nn - 256), s ? 1u : acc);
                        }
                    }
                    umma_commit(&bars.empty[stage]);
                    if (++stage == kStages) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
                if (ok) umma_commit(&bars.acc_full);
                accphase ^= 1u;
            }
            if (!ok) atomicExch(&bars.abort, 1);
        }
    } else {
        // ---------------- epilogue
        const int q = warp & 3;                        // TMEM lane quarter this warp may access
        const int cg = (warp - 2) >> 2;                // its 16 columns of the tile
        uint32_t accphase = 0;
        Tile x;
        for (int64_t k = 0; tile_at(wk, k, x); k++) {
            if (x.ti < 0) continue;
            const int64_t i = (int64_t)x.ti * kBM + q * 32 + lane, j0 = (int64_t)x.tj * kBN + cg * kCols;
            const int64_t m = x.m;
            const bool any = j0 < m && j0 <= (int64_t)x.ti * kBM + q * 32 + 31 && i - lane < m;  // warp-uniform
            const bool interior = (j0 + kCols - 1 <= (int64_t)x.ti * kBM + q * 32) && (i - lane + 31 < m);
            OutT *S = reinterpret_cast<OutT *>(x.S);
            OutT *ptr = S + (kPacked ? j0 * m - j0 * (j0 + 1) / 2 : j0 * x.lds) + i;
            int ei = kExpZero, ej = kExpZero;
            if (x.e > 0 && i < m) ei = x.sb.ew[i];
            if (x.e > 0 && lane < kCols && j0 + lane < m) ej = x.sb.el[j0 + lane];
            if (!mbar_wait(&bars.acc_full, accphase, &bars.abort)) {
                if (lane == 0) atomicExch(&bars.abort, 1);
                break;
            }
            accphase ^= 1u;
            tc_fence_after();
            // 2^(40 + f) is the weight of g = 0: as large as the 64 bits allow for e pivots
            const int f = x.e <= 16 ? 6 : (x.e <= 32 ? 5 : (x.e <= 64 ? 4 : (x.e <= 128 ? 3 : 2)));
            long long V[kCols];
            if (any && x.e > 0) {
                const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(cg * kCols);
                uint32_t r[16];
                float low[kCols];
                tmem_ld16_nowait(ta + 7 * kBN, r);
                tmem_wait_ld();
                const float w7 = __int_as_float((127 + f - 16) << 23), w6 = __int_as_float((127 + f - 8) << 23);
#pragma unroll
                for (int c = 0; c < kCols; c++) low[c] = __uint_as_float(r[c]) * w7;
                tmem_ld16_nowait(ta + 6 * kBN, r);
                tmem_wait_ld();
#pragma unroll
                for (int c = 0; c < kCols; c++) V[c] = __float2int_rn(fmaf(__uint_as_float(r[c]), w6, low[c]));
#pragma unroll
                for (int g = 5; g >= 0; g--) {
                    tmem_ld16_nowait(ta + g * kBN, r);
                    tmem_wait_ld();
#pragma unroll
                    for (int c = 0; c < kCols; c++) {
                        const int d = __float2int_rn(__uint_as_float(r[c]));
                        if (g > 1)
                            V[c] += (long long)d * (1 << ((40 - 8 * g + f) & 31));
                        else  // weights 2^(32 + f) and 2^(40 + f): the high word
                            V[c] += (long long)((unsigned long long)(unsigned)(d << (8 - 8 * g + f)) << 32);
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars.acc_empty);
            if (!any) continue;
            // marked rows and columns of this warp's block
            const bool wide_i = ei >= kExpWide / 2, wide_j = ej >= kExpWide / 2;
            const unsigned wides = __ballot_sync(0xffffffffu, wide_j);
            const bool any_wide = wides != 0u || __any_sync(0xffffffffu, wide_i);
#pragma unroll
            for (int h = 0; h < kCols; h += 8) {
                double pl[8];
                if (any_wide) {
                    if (i < m) plain_entries(x.L21, x.ldl, x.D, x.piv, x.e, i, j0 + h, pl);
                }
                // subtracting: eight old values loaded before any is stored
                double old[8];
                if (kSub) {
#pragma unroll
                    for (int c = 0; c < 8; c++) {
                        old[c] = 0.0;
                        if (interior || (i < m && j0 + h + c <= i)) old[c] = ptr[(int64_t)c * x.lds];
                    }
                }
#pragma unroll
                for (int c = 0; c < 8; c++) {
                    const int ex = ei + __shfl_sync(0xffffffffu, ej, h + c) - 52 - f;
                    double v = x.e > 0 ? to_fp64(V[h + c], ex) : 0.0;
                    if (any_wide && (wide_i || ((wides >> (h + c)) & 1u))) v = pl[c];
                    if (interior || (i < m && j0 + h + c <= i)) {
                        if (kSub)
                            *ptr = (OutT)(old[c] - v);
                        else
                            __stcs(ptr, (OutT)v);
                    }
                    ptr += kPacked ? m - 1 - (j0 + h + c) : x.lds;
                }
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && bars.abort) atomicCAS(info, kInfoOk, (int32_t)CTP_ETIMEOUT);
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// Slices of W21 = L21 D11 and L21 from a stored L21 (full-column pivoting writes no
// slices itself): a CTA per 32 rows.
constexpr int kSW = 8;
__global__ void __launch_bounds__(32 * kSW)
    k_slices_from_l(const double *__restrict__ A, int64_t lda, int p, int64_t m, const int32_t *__restrict__ piv,
                    const double *__restrict__ D, const double *__restrict__ Dinv, const int32_t *__restrict__ nelim,
                    SliceBuf sb) {
    extern __shared__ __align__(16) double xs[];  // [p][33]
    __shared__ short cexp[kMaxP];
    __shared__ int red[2 * kSW * 32], rexp[32];
    const int e = *nelim, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t row0 = (int64_t)blockIdx.x * 32;
    const int nrows = (int)min((int64_t)32, m - row0);
    for (int k = threadIdx.x; k < e; k += 32 * kSW) cexp[k] = (short)slice_col_exp(piv, Dinv, k);
    for (int k = w; k < e; k += kSW) xs[k * 33 + lane] = lane < nrows ? A[(int64_t)k * lda + p + row0 + lane] : 0.0;
    __syncthreads();
    write_slices<kLRows, kSW>(xs, e, row0, nrows, cexp, 1, sb.L, sb.el, sb.kb, red, rexp);
    __syncthreads();
    for (int k = w; k < e; k += kSW) {
        const int kd = piv[k];
        if (kd == CTP_PIVKIND_1X1) {
            xs[k * 33 + lane] *= D[2 * k];
        } else if (kd == CTP_PIVKIND_2X2_FIRST) {
            const double l0 = xs[k * 33 + lane], l1 = xs[(k + 1) * 33 + lane];
            xs[k * 33 + lane] = l0 * D[2 * k] + l1 * D[2 * k + 1];
            xs[(k + 1) * 33 + lane] = l0 * D[2 * k + 1] + l1 * D[2 * k + 2];
        }
    }
    __syncthreads();
    write_slices<kWRows, kSW>(xs, e, row0, nrows, cexp, -1, sb.W, sb.ew, sb.kb, red, rexp);
}

template <int kMode>
cudaError_t launch_mode(const Work &wk, int32_t *info, int num_sms, cudaStream_t st) {
    cudaError_t err = smem_at_least((const void *)k_form_fp64<kMode>, kSmem);
    if (err != cudaSuccess) return err;
    const unsigned grid = (unsigned)(wk.count < num_sms ? wk.count : num_sms);
    k_form_fp64<kMode><<<grid, kThreads, kSmem, st>>>(wk, info);
    return cudaGetLastError();
}

cudaError_t launch_any(const Work &wk, int smode, int32_t *info, int num_sms, cudaStream_t st) {
    switch (smode) {
    case CTP_S_FP64: return launch_mode<CTP_S_FP64>(wk, info, num_sms, st);
    case CTP_S_FP32: return launch_mode<CTP_S_FP32>(wk, info, num_sms, st);
    case CTP_S_FP64_SUB: return launch_mode<CTP_S_FP64_SUB>(wk, info, num_sms, st);
    case CTP_S_FP64_PACKED: return launch_mode<CTP_S_FP64_PACKED>(wk, info, num_sms, st);
    default: return launch_mode<CTP_S_FP32_PACKED>(wk, info, num_sms, st);
    }
}

}  // namespace

cudaError_t launch_form_fp64(const SliceBuf &sb, const double *L21, int64_t lda, const int32_t *piv,
                             const double *D, int64_t m, const int32_t *nelim, void *S, int64_t lds, int smode,
                             int32_t *info, int num_sms, cudaStream_t st) {
    if (m <= 0) return cudaSuccess;
    Work wk = {};
    wk.sb = sb;
    wk.L21 = L21;
    wk.ldl = lda;
    wk.piv = piv;
    wk.D = D;
    wk.m = m;
    wk.lds = lds;
    wk.nelim = nelim;
    wk.S = S;
    wk.count = walk_slots(m);
    return launch_any(wk, smode, info, num_sms, st);
}

cudaError_t launch_form_fp64_batch(const ctp_front *fronts, const BFront *tab, char *ws,
                                   const int *item_front, int64_t items, BatchOpts o, int32_t *info, int num_sms,
                                   cudaStream_t st, const int *item_tile) {
    if (items == 0) return cudaSuccess;
    Work wk = {};
    wk.fronts = fronts;
    wk.tab = tab;
    wk.ws = ws;
    wk.item_front = item_front;
    wk.item_tile = item_tile;
    wk.o = o;
    wk.count = items;
    return launch_any(wk, o.smode, info, num_sms, st);
}

cudaError_t launch_slices_from_l(const double *A, int64_t lda, int p, int64_t m, const int32_t *piv,
                                 const double *D, const double *Dinv, const int32_t *nelim, const SliceBuf &sb,
                                 cudaStream_t st) {
    if (m <= 0) return cudaSuccess;
    const size_t smem = sizeof(double) * (size_t)p * 33;
    cudaError_t err = smem_at_least((const void *)k_slices_from_l, smem);
    if (err != cudaSuccess) return err;
    k_slices_from_l<<<(unsigned)((m + 31) / 32), 32 * kSW, smem, st>>>(A, lda, p, m, piv, D, Dinv, nelim, sb);
    return cudaGetLastError();
}

// Tiles of a front's Form: row blocks of 128 by column blocks of 64 on or below the
// diagonal (the last row block may lack its last column block)
int64_t form_fp64_tiles(int64_t m) {
    const int64_t nM = (m + kBM - 1) / kBM, nN = (m + kBN - 1) / kBN;
    return nM * (nM + 1) - (2 * nM - nN);
}

}  // namespace ctp
