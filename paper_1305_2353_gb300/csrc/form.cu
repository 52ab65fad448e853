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
// The same kernel, kMode kUpdate, is the Solve's update of the later columns of A21
// with a block of 32 columns: A21(:, c0 + j) -= y L11(c0 + j, block)^T, all rows
// by all j, one K block.
// Bound: tensor pipe for e from about 100 on (n = 20000, p = e = 256: 2.26 ms, 1.6
// PFLOP/s of executed products, against 80.6 ms for FP64 multiply-adds at 0.99 of
// their pipe's rate); below, S traffic and the epilogue's instructions: the
// update of 224 columns of 200000 rows took 446 us with 144 instructions per entry,
// 210 with the test-free path, the 32-bit sums of neighbouring groups and the old
// values brought to L2 ahead (HBM's share: 121 us).
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
constexpr int kUpdate = 100;  // kMode of the Solve's update (the others are a ctp_smode)

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

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
    tmem_wait_ld();
}

struct Tile {
    int ti, tj, e, m, nc;  // m, nc: rows, columns (a Form: nc = m)
    int64_t lds, ldl;
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
    int c0;         // kUpdate: first column updated, 32 past the block's first
    int64_t nc;     // kUpdate, one supernode: columns updated
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
template <bool kUpd>
__device__ __forceinline__ bool tile_at(const Work &w, int64_t k, Tile &x) {
    const int64_t t = blockIdx.x + k * (int64_t)gridDim.x;
    if (t >= w.count) return false;
    if (kUpd) {
        // row block by row block, its column blocks one after another
        int64_t q = t;
        x.nc = (int)w.nc;
        x.sb = w.sb;
        x.m = (int)w.m;
        x.e = w.fronts != nullptr ? 0 : *w.nelim;
        x.L21 = w.L21;
        x.ldl = w.ldl;
        x.piv = w.piv;
        if (w.fronts != nullptr) {
            const int f = w.item_front[t];
            const BFront b = w.tab[f];
            const ctp_front &fr = w.fronts[f];
            q = w.item_tile[t];
            ctp_options oo;
            oo.pivot = w.o.pivot;
            oo.smode = w.o.smode;
            oo.prec = w.o.prec;
            x.sb = bsection_block(w.ws + b.ws, bsection(b.n, b.p, &oo));
            x.m = (int)b.m;
            x.nc = b.p - w.c0;
            x.e = *fr.nelim;
            x.L21 = fr.A + b.p;
            x.ldl = fr.lda;
            x.piv = fr.piv;
        }
        x.e = min(x.e - (w.c0 - kSliceK), kSliceK);
        x.S = const_cast<double *>(x.L21 + (int64_t)w.c0 * x.ldl);
        x.lds = x.ldl;
        const int nN = (x.nc + kBN - 1) / kBN;
        x.ti = x.e > 0 ? (int)(q / nN) : -1;  // nothing eliminated in the block: nothing to do
        x.tj = (int)(q % nN);
        return true;
    }
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
        x.m = x.nc = (int)b.m;
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
    x.m = x.nc = (int)w.m;
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

// V 2^ex rounded to nearest even in integer instructions, for results in the normal
// range of FP64 (the FP64 pipe takes 17 cycles per warp instruction and SM)
__device__ __forceinline__ double to_fp64(long long V, int ex) {
    const unsigned long long a = V < 0 ? 0ull - (unsigned long long)V : (unsigned long long)V;
    const int lz = __clzll((long long)a) & 63;
    const unsigned long long n = a << lz, t = n >> 11;
    const unsigned up = ((unsigned)n & 0x7FFu) + ((unsigned)t & 1u) > 0x400u ? 1u : 0u;
    // biased exponent - 1 (the hidden bit adds the 1) and sign in the high word
    const unsigned he = ((unsigned)(63 - lz + ex + 1022) << 20) | ((unsigned)(V >> 32) & 0x80000000u);
    const unsigned long long bits = ((unsigned long long)he << 32) + t + up;
    return V == 0 ? 0.0 : __longlong_as_double((long long)bits);
}
// any result
__device__ __noinline__ double to_fp64_any(long long V, int ex) {
    return ex > -900 && ex < 900 ? to_fp64(V, ex) : (V == 0 ? 0.0 : scalbn((double)V, ex));
}

// Entries (i, j..j+7) of the k-th tile's result by FP64 multiply-adds (i < m; columns
// past the result count as 0): the marked rows' path.  It looks its tile up again,
// so that the epilogue keeps no registers for it.
template <bool kUpd>
__device__ __noinline__ void plain_entries(const Work &wk, int64_t kt, int64_t i, int64_t j, double (&acc)[8]) {
    Tile x;
    tile_at<kUpd>(wk, kt, x);
#pragma unroll
    for (int c = 0; c < 8; c++) acc[c] = 0.0;
    const int first = kUpd ? wk.c0 - kSliceK : 0;
    for (int k = first; k < first + x.e; k++) {
        const int kd = x.piv[k];
        if (kd == CTP_PIVKIND_ZERO) continue;
        const double *col = x.L21 + (int64_t)k * x.ldl;
        double w = col[i];  // kUpd: y itself, in the block's columns of A21
        const double *l = col;
        if (kUpd) {
            l = col - (x.nc + wk.c0) + wk.c0;  // rows c0.. of L11's column
        } else {
            w *= x.D[2 * k];
            if (kd == CTP_PIVKIND_2X2_FIRST) w = fma(col[i + x.ldl], x.D[2 * k + 1], w);
            if (kd == CTP_PIVKIND_2X2_SECOND) w = fma(col[i - x.ldl], x.D[2 * k - 1], w);
        }
#pragma unroll
        for (int c = 0; c < 8; c++) {
            const bool d21 = kUpd && wk.c0 + j + c == k + 1 && kd == CTP_PIVKIND_2X2_FIRST;  // that slot holds D
            if (j + c <= (kUpd ? x.nc - 1 : i) && !d21) acc[c] = fma(w, l[j + c], acc[c]);
        }
    }
}

// The eight accumulators of 8 columns (group g at column g kBN) added up: V = sum_g
// T_g 2^(40 + f - 8 g), the last two groups rounded to whole units.  kSmall (K
// <= 32: every |T_g| <= 2^22): a float becomes an integer by adding 1.5 2^23 (its
// mantissa bits then hold the integer, offset by a constant that is taken off at
// the end), and two neighbouring groups fit one 32-bit integer; otherwise by the
// conversion instruction, a quarter as fast.
template <bool kSmall>
__device__ __forceinline__ void add_groups(uint32_t ta, int f, long long *V) {
    uint32_t r[8];
    float low[8];
    tmem_ld8(ta + 7 * kBN, r);
    const float w7 = __int_as_float((127 + f - 16) << 23), w6 = __int_as_float((127 + f - 8) << 23);
#pragma unroll
    for (int c = 0; c < 8; c++) low[c] = __uint_as_float(r[c]) * w7;
    tmem_ld8(ta + 6 * kBN, r);
    if (kSmall) {
        constexpr float kMagic = 12582912.0f;   // 1.5 2^23
        constexpr unsigned kOff = 0x4B400000u;  // its bits
        unsigned pr[8];
#pragma unroll
        for (int c = 0; c < 8; c++)  // |low| < 2^21: two groups of at most 2^22 by 2^(f - 8), f <= 6
            V[c] = (int)(__float_as_uint(fmaf(__uint_as_float(r[c]), w6, low[c]) + kMagic) - kOff);
#pragma unroll
        for (int g = 4; g >= 0; g -= 2) {
            tmem_ld8(ta + g * kBN, r);
#pragma unroll
            for (int c = 0; c < 8; c++) pr[c] = __float_as_uint(__uint_as_float(r[c]) + kMagic) * 256u - 257u * kOff;
            tmem_ld8(ta + (g + 1) * kBN, r);
#pragma unroll
            for (int c = 0; c < 8; c++) {
                const int two = (int)(pr[c] + __float_as_uint(__uint_as_float(r[c]) + kMagic));
                if (g > 0)  // groups 4, 5 weigh 2^f, groups 2, 3 2^(16 + f)
                    V[c] += (long long)two * (1 << (32 - 8 * g + f));
                else        // groups 0, 1 2^(32 + f): the high word
                    V[c] += (long long)((unsigned long long)(unsigned)(two << f) << 32);
            }
        }
    } else {
#pragma unroll
        for (int c = 0; c < 8; c++) V[c] = __float2int_rn(fmaf(__uint_as_float(r[c]), w6, low[c]));
#pragma unroll
        for (int g = 5; g >= 0; g--) {
            tmem_ld8(ta + g * kBN, r);
#pragma unroll
            for (int c = 0; c < 8; c++) {
                const int d = __float2int_rn(__uint_as_float(r[c]));
                if (g > 1)
                    V[c] += (long long)d * (1 << ((40 - 8 * g + f) & 31));
                else  // weights 2^(32 + f) and 2^(40 + f): the high word
                    V[c] += (long long)((unsigned long long)(unsigned)(d << (8 - 8 * g + f)) << 32);
            }
        }
    }
}

// kMode: ctp_smode of S, or kUpdate
template <int kMode>
__global__ void __launch_bounds__(kThreads, 1) k_form_fp64(const Work wk, int32_t *__restrict__ info) {
    using OutT = typename std::conditional<kMode == CTP_S_FP32 || kMode == CTP_S_FP32_PACKED, float, double>::type;
    constexpr bool kPacked = kMode == CTP_S_FP64_PACKED || kMode == CTP_S_FP32_PACKED;
    constexpr bool kUpd = kMode == kUpdate;
    constexpr bool kSub = kMode == CTP_S_FP64_SUB || kUpd;
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
            for (int64_t k = 0; ok && tile_at<kUpd>(wk, k, x); k++) {
                if (x.ti < 0) continue;
                // rows of the tile in use, in groups of 8
                const uint32_t rw = (uint32_t)(min(kBM, x.m - x.ti * kBM) + 7) & ~7u;
                const uint32_t rl = (uint32_t)(min(kBN, x.nc - x.tj * kBN) + 7) & ~7u;
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
            for (int64_t k = 0; ok && tile_at<kUpd>(wk, k, x); k++) {
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
        for (int64_t k = 0; tile_at<kUpd>(wk, k, x); k++) {
            if (x.ti < 0) continue;
            const int i = x.ti * kBM + q * 32 + lane, j0 = x.tj * kBN + cg * kCols, m = x.m;
            // entries (i, j) with i < m and j <= jmax belong to the result
            const int jmax = kUpd ? x.nc - 1 : i;
            const bool any = j0 <= (kUpd ? jmax : i - lane + 31) && j0 < x.nc && i - lane < m;  // warp-uniform
            const bool interior = j0 + kCols - 1 <= (kUpd ? jmax : i - lane) && i - lane + 31 < m;
            OutT *ptr = reinterpret_cast<OutT *>(x.S) +
                        (kPacked ? (int64_t)j0 * m - (int64_t)j0 * (j0 + 1) / 2 : j0 * x.lds) + i;
            int ei = kExpZero, ej = kExpZero;
            if (x.e > 0 && i < m) ei = x.sb.ew[i];
            if (x.e > 0 && lane < kCols && j0 + lane < x.nc) ej = x.sb.el[j0 + lane];
            // subtracting: the old values come to L2 while the products are computed
            if (kSub && any && i < m) {
#pragma unroll
                for (int c = 0; c < kCols; c++)
                    if (interior || j0 + c <= jmax)
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(ptr + (int64_t)c * x.lds));
            }
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
#pragma unroll
                for (int h = 0; h < kCols; h += 8)
                    if (kUpd || x.e <= 32)
                        add_groups<true>(ta + h, f, V + h);
                    else
                        add_groups<false>(ta + h, f, V + h);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars.acc_empty);
            if (!any) continue;
            // marked rows and columns of this warp's block
            const bool wide_i = ei >= kExpWide / 2, wide_j = ej >= kExpWide / 2;
            const unsigned wides = __ballot_sync(0xffffffffu, wide_j);
            const bool any_wide = wides != 0u || __any_sync(0xffffffffu, wide_i);
            // the plain case -- every entry of the warp's block belongs to the result, no
            // row is marked, exponents are moderate -- has no test in its loop
            const bool mild = abs(ei) < 400 && (lane >= kCols || abs(ej) < 400);
            if (interior && !any_wide && __all_sync(0xffffffffu, mild)) {
#pragma unroll
                for (int h = 0; h < kCols; h += 8) {
                    double old[8];  // eight old values loaded before any is stored
                    OutT *pl = ptr;
                    if (kSub) {
#pragma unroll
                        for (int c = 0; c < 8; c++) {
                            old[c] = *pl;
                            pl += x.lds;
                        }
                    }
#pragma unroll
                    for (int c = 0; c < 8; c++) {
                        const double v = to_fp64(V[h + c], ei + __shfl_sync(0xffffffffu, ej, h + c) - 52 - f);
                        if (kSub)
                            *ptr = (OutT)(old[c] - v);
                        else
                            __stcs(ptr, (OutT)v);
                        ptr += kPacked ? m - 1 - (j0 + h + c) : x.lds;
                    }
                }
                continue;
            }
#pragma unroll
            for (int h = 0; h < kCols; h += 8) {
                double pl[8], old[8];
                if (any_wide && i < m) plain_entries<kUpd>(wk, k, i, j0 + h, pl);
                if (kSub) {
#pragma unroll
                    for (int c = 0; c < 8; c++) old[c] = i < m && j0 + h + c <= jmax ? ptr[(int64_t)c * x.lds] : 0.0;
                }
#pragma unroll
                for (int c = 0; c < 8; c++) {
                    const int ex = ei + __shfl_sync(0xffffffffu, ej, h + c) - 52 - f;
                    if (i < m && j0 + h + c <= jmax) {
                        double v = x.e > 0 ? to_fp64_any(V[h + c], ex) : 0.0;
                        if (any_wide && (wide_i || ((wides >> (h + c)) & 1u))) v = pl[c];
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
    case kUpdate: return launch_mode<kUpdate>(wk, info, num_sms, st);
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

cudaError_t launch_update(const SliceBuf &u, double *A, int64_t lda, int p, int64_t m, int blk, const int32_t *piv,
                          const int32_t *nelim, int32_t *info, int num_sms, cudaStream_t st) {
    Work wk = {};
    wk.sb = u;
    wk.L21 = A + p;
    wk.ldl = lda;
    wk.piv = piv;
    wk.m = m;
    wk.nelim = nelim;
    wk.c0 = (blk + 1) * kSliceK;
    wk.nc = p - wk.c0;
    wk.count = (m + kBM - 1) / kBM * ((wk.nc + kBN - 1) / kBN);
    if (wk.count <= 0) return cudaSuccess;
    return launch_any(wk, kUpdate, info, num_sms, st);
}

int64_t update_tiles(int64_t m, int p) {
    return p > kSliceK ? (m + kBM - 1) / kBM * ((p - kSliceK + kBN - 1) / kBN) : 0;
}

cudaError_t launch_update_batch(const ctp_front *fronts, const BFront *tab, char *ws, const int *item_front,
                                const int *item_tile, int64_t items, BatchOpts o, int32_t *info, int num_sms,
                                cudaStream_t st) {
    if (items == 0) return cudaSuccess;
    Work wk = {};
    wk.fronts = fronts;
    wk.tab = tab;
    wk.ws = ws;
    wk.item_front = item_front;
    wk.item_tile = item_tile;
    wk.o = o;
    wk.c0 = kSliceK;
    wk.count = items;
    return launch_any(wk, kUpdate, info, num_sms, st);
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
