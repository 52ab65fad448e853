// form.cu -- K6 (FP64): the Form task S = L21 D11 L21^T = W21 L21^T (Section 1
// task list), lower triangle only, in FP64 on the tensor cores.
//
// GB300's FP64 pipe gives 1.26 TFLOP/s, its BF16 tensor cores about 1700, and a
// product of two FP64 matrices is 36 exact BF16 products: the operands come as
// eight digit slices each (slices.cuh), the products d_s d_t' of slices with
// g = s + t <= 7 are summed per g in FP32 without rounding, and the epilogue
// adds the eight sums, which are integers, in 64-bit integer arithmetic and
// rounds once to FP64.  slices.cuh says what this loses: less than FP64
// multiply-adds may, of every entry whose rows are large in common pivots.  The epilogue
// makes sure of that for every entry and takes the others by FP64 multiply-adds.
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
//   warp 18     scheduler: looks the tiles up (some 3000 clocks each: a walk over the
//               triangle or a chain of a batch's descriptors) and hands them to the others
//               through a ring of four.
//   warp 19     checker: tells for every 4 x 4 block of a tile's entries whether digits
//               serve it, from the groups' lower bounds (3 KB per K block): 512 sums of
//               e products, four rows and columns of them per lane.  The epilogue finds
//               a bit per block when the accumulators are full, and leaves entries of the
//               others out; they are computed after the CTA's last tile.
//   warps 2-17  epilogue: a thread holds 16 columns of one row of S as 64-bit
//               integers; the accumulators are handed back as soon as they have
//               been added up, and rounding and stores overlap the next tile.
// The same kernel, kMode kUpdate, is the Solve's update of the later columns of A21
// with a block of 32 columns: A21(:, c0 + j) -= y L11(c0 + j, block)^T, all rows
// by all j, one K block.
// Bound: tensor pipe for e from about 100 on (n = 20000, p = e = 256: 2.33 ms, 1.55
// PFLOP/s of executed products, against 80.6 ms for FP64 multiply-adds at 0.99 of
// their pipe's rate); below, S traffic and the epilogue's instructions: the
// update of 224 columns of 200000 rows took 446 us with 144 instructions per entry,
// 236 with the test-free path, the 32-bit sums of neighbouring groups and the old
// values brought to L2 ahead (HBM's share: 121 us).  The checker shares its issue slots with
// a quarter of the epilogue: without it the two take 2.26 ms and 196 us.  Where no two rows are
// large in a common pivot, nearly all entries go to FP64 multiply-adds (n = 20000, p = 256:
// 91 ms; 16 with 1% of such rows).
// Fronts of few rows have a kernel of their own, k_form_small.
// Every mbarrier wait is bounded; on timeout the kernel records CTP_ETIMEOUT,
// waits (bounded) for its copies in flight, frees its tensor memory and returns.
#include <cuda_fp16.h>

#include "slices.cuh"
#include "tc_common.cuh"

namespace ctp {

using namespace tc;

namespace {

constexpr int kBM = kWRows, kBN = kLRows;
constexpr int kEpiWarps = 16, kThreads = 32 * (4 + kEpiWarps);
constexpr int kCols = kBN / (kEpiWarps / 4);  // columns of S per epilogue thread
constexpr int kStages = 2;
constexpr uint32_t kStageBytes = kWBlock + kLBlock;
constexpr size_t kSmem = kStages * (size_t)kStageBytes + kWGroup + kLGroup + 1024;
constexpr int kPanel = 8;  // column blocks of a panel of the walk
constexpr int kUpdate = 100;  // kMode of the Solve's update (the others are a ctp_smode)

struct Tile {
    int64_t t;             // item or slot
    int ti, tj, e, m, nc;  // m, nc: rows, columns (a Form: nc = m); ti < 0: no tile
    int c0;                // kUpdate: first column updated, 32 past the block's first
    int64_t lds, ldl;
    SliceBuf sb;
    const double *L21, *D;
    const int32_t *piv;
    void *S;
};

constexpr int kRing = 4, kList = 256, kKept = 16;
struct Bars {
    unsigned long long full[kStages], empty[kStages], acc_full, acc_empty, grp_full, tile_full[kRing], tile_empty[kRing];
    Tile tile[kRing];
    int64_t list[kList];            // those tiles,
    Tile kept[kKept];               // the first of them as they were looked up,
    int64_t marked;                 // and the last that found no room there, -1: none
    int nlist, next;
    uint32_t unsure[2][kEpiWarps];  // by turns: blocks that digits may not serve,
    int linked[2];                  // the tile is in the list of those with entries left out
    int weak;                       // some entry was left out
    int nmarks;
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
    int64_t first, count;  // the launch's items, or slots of the walk: first .. count - 1
    TileMarks *marks;      // one for each of them
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

// Looks this CTA's tiles up, one after another.
template <bool kUpd>
struct Walk {
    const Work &w;
    int64_t t, panel = 0, before = 0, next;  // one supernode's Form: slots before this panel and the next
    int e = 0;
    __device__ __forceinline__ explicit Walk(const Work &w_) : w(w_), t(w_.first + blockIdx.x) {
        if (w.fronts == nullptr) e = *w.nelim;
        next = slots_before(1, (w.m + kBM - 1) / kBM);
    }
    // the next tile; ti < 0 past the end
    __device__ __forceinline__ void step(Tile &x) {
        for (x.ti = -1; t < w.count && x.ti < 0; t += gridDim.x) look(x);
    }
    // tile `to` is looked up next (any)
    __device__ __forceinline__ void seek(int64_t to) {
        t = to;
        panel = before = 0;
        next = slots_before(1, (w.m + kBM - 1) / kBM);
    }
    __device__ __forceinline__ void look(Tile &x) {
        int64_t q = x.t = t;
        x.sb = w.sb;
        x.m = x.nc = (int)w.m;
        x.e = e;
        x.L21 = w.L21;
        x.ldl = w.ldl;
        x.D = w.D;
        x.piv = w.piv;
        x.S = w.S;
        x.lds = w.lds;
        x.c0 = w.c0;
        if (kUpd) x.nc = (int)w.nc;
        if (w.fronts != nullptr) {
            const int f = w.item_front[t];
            const BFront b = w.tab[f];
            const ctp_front &fr = w.fronts[f];
            q = w.item_tile != nullptr ? (int64_t)w.item_tile[t] : t - b.f0;
            const BSection sec = bsection(b.n, b.p, w.o);
            x.sb = kUpd ? bsection_block(w.ws + b.ws, sec) : bsection_slices(w.ws + b.ws, sec, b.p);
            x.m = (int)b.m;
            x.nc = kUpd ? b.p - w.c0 : x.m;
            x.e = *fr.nelim;
            x.L21 = fr.A + b.p;
            x.ldl = fr.lda;
            x.D = fr.D;
            x.piv = fr.piv;
            x.S = fr.S;
            x.lds = fr.lds;
        }
        if (kUpd) {
            // row block by row block, its column blocks one after another
            x.e = min(x.e - (w.c0 - kSliceK), kSliceK);
            x.S = const_cast<double *>(x.L21 + (int64_t)w.c0 * x.ldl);
            x.lds = x.ldl;
            const int nN = (x.nc + kBN - 1) / kBN;
            const unsigned r = (unsigned)q / (unsigned)nN;  // (fewer than 2^31 tiles)
            x.ti = x.e > 0 ? (int)r : -1;  // nothing eliminated in the block: nothing to do
            x.tj = (int)((unsigned)q - r * (unsigned)nN);
        } else if (w.fronts != nullptr) {
            // row block i has 2 (i + 1) tiles, i (i + 1) precede it
            int64_t i = (int64_t)((sqrtf(4.0f * (float)q + 1.0f) - 1.0f) * 0.5f);
            while ((i + 1) * (i + 2) <= q) i++;
            while (i * (i + 1) > q) i--;
            x.ti = (int)i;
            x.tj = (int)(q - i * (i + 1));
        } else {
            const int64_t nM = (w.m + kBM - 1) / kBM;
            while (q >= next) {
                panel++;
                before = next;
                next = slots_before(panel + 1, nM);
            }
            const int64_t r = q - before, ti = panel * (kPanel / 2) + r / kPanel, tj = panel * kPanel + r % kPanel;
            x.tj = (int)tj;
            x.ti = (tj * kBN < w.m && tj <= 2 * ti + 1) ? (int)ti : -1;
        }
    }
};

// A role's way through the ring of tiles.
struct Ring {
    int slot = 0;
    uint32_t phase = 0;
    // the next tile is there; false on timeout
    __device__ __forceinline__ bool wait(Bars &b) { return mbar_wait(&b.tile_full[slot], phase, &b.abort); }
    // done with it (one lane of each role's warp)
    __device__ __forceinline__ void release(Bars &b) { mbar_arrive(&b.tile_empty[slot]); }
    __device__ __forceinline__ void step() {
        if (++slot == kRing) {
            slot = 0;
            phase ^= 1u;
        }
    }
};

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

// Which 4 x 4 blocks of a tile have pivots in which all their rows are large
// (slices.cuh): the dot products of four groups of rows (4 (lane / 4)..) by four of
// columns (4 (lane % 4)..) per lane, from the groups' bounds, a K block of them at a time
// (`fetch(kb)` brings it to shared memory; gw and gl groups per chunk of 8 pivots).  Bit 4 a + b: group a of the lane's rows by
// group b of its columns has not, and neither are they without a pivot in common
// (their results are then zero).  Rounded in FP16: a part in 2^11 per term of up to 128
// per sum.  From the last pivot on, where growth puts the large entries, and no
// further than needed: random data stop after the first block, which matters to the
// traffic from L2 (all blocks: 3% at e = 256).  From 24 pivots on, eight rows at a time are
// tried first, a quarter of the products: the checker shares its issue slots with a
// quarter of the epilogue.
constexpr float kSure = 0x1p-7f;
template <typename F>
__device__ __forceinline__ unsigned unsure_blocks(const uint8_t *grp, int e, int gw, int gl, bool in, F &&fetch) {
    const int lane = threadIdx.x & 31;
    const uint4 *pa = reinterpret_cast<const uint4 *>(grp) + 4 * (lane >> 2);
    const uint4 *pb = reinterpret_cast<const uint4 *>(grp + kWGroup) + 4 * (lane & 3);
    auto h2 = [](unsigned v) { return *reinterpret_cast<const __half2 *>(&v); };
    __half2 s[16];
#pragma unroll
    for (int j = 0; j < 16; j++) s[j] = __floats2half2_rn(0.0f, 0.0f);
    unsigned bad = 0xFFFFu;
    const int KB = (e + kSliceK - 1) / kSliceK;
    bool here = false;  // the last K block is in shared memory
    if (e >= 24) {
        const int kb = KB - 1, chunks = min(4, (e - kb * kSliceK + 7) / 8);
        fetch(kb);
        here = true;
        __half2 c[4];
#pragma unroll
        for (int j = 0; j < 4; j++) c[j] = __floats2half2_rn(0.0f, 0.0f);
#pragma unroll 1
        for (int k = 0; k < chunks; k++) {
            uint4 u[2], v[2];
            auto least = [](const uint4 &x, const uint4 &y) {  // FP16 pairs of magnitudes, -0 below them
                return make_uint4(__vminu2(x.x & 0x7FFF7FFFu, y.x & 0x7FFF7FFFu), __vminu2(x.y & 0x7FFF7FFFu, y.y & 0x7FFF7FFFu),
                                  __vminu2(x.z & 0x7FFF7FFFu, y.z & 0x7FFF7FFFu), __vminu2(x.w & 0x7FFF7FFFu, y.w & 0x7FFF7FFFu));
            };
#pragma unroll
            for (int i = 0; i < 2; i++) {
                u[i] = least(pa[k * gw + 2 * i], pa[k * gw + 2 * i + 1]);
                v[i] = least(pb[k * gl + 2 * i], pb[k * gl + 2 * i + 1]);
            }
#pragma unroll
            for (int i = 0; i < 2; i++)
#pragma unroll
                for (int j = 0; j < 2; j++) {
                    __half2 &t = c[2 * i + j];
                    t = __hfma2(h2(u[i].x), h2(v[j].x), t);
                    t = __hfma2(h2(u[i].y), h2(v[j].y), t);
                    t = __hfma2(h2(u[i].z), h2(v[j].z), t);
                    t = __hfma2(h2(u[i].w), h2(v[j].w), t);
                }
        }
        // (rows and columns past the result hold anything: their lanes decide nothing)
        bool all = true;
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const float2 t = __half22float2(c[j]);
            all = all && t.x + t.y >= kSure;
        }
        if (__all_sync(0xffffffffu, all || !in)) return 0u;
    }
#pragma unroll 1
    for (int kb = KB - 1; kb >= 0 && __any_sync(0xffffffffu, bad); kb--) {
        if (!here || kb < KB - 1) fetch(kb);
        const int chunks = min(4, (e - kb * kSliceK + 7) / 8);
#pragma unroll 1
        for (int c = 0; c < chunks; c++) {
            uint4 v[4];
#pragma unroll
            for (int j = 0; j < 4; j++) v[j] = pb[c * gl + j];
#pragma unroll
            for (int i = 0; i < 4; i++) {
                const uint4 u = pa[c * gw + i];
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    __half2 &t = s[4 * i + j];
                    t = __hfma2(h2(u.x), h2(v[j].x), t);
                    t = __hfma2(h2(u.y), h2(v[j].y), t);
                    t = __hfma2(h2(u.z), h2(v[j].z), t);
                    t = __hfma2(h2(u.w), h2(v[j].w), t);
                }
            }
        }
        bad = 0u;  // (two sums at a time; a NaN compares as false)
        const __half2 sure = __float2half2_rn(kSure);
#pragma unroll
        for (int j = 0; j < 16; j += 2)
            bad |= ~__hge2_mask(__hadd2(__lows2half2(s[j], s[j + 1]), __highs2half2(s[j], s[j + 1])), sure) &
                   (1u << j | 1u << (j + 1 + 15));
        bad = (bad & 0xFFFFu) | bad >> 15;
    }
    if (!__any_sync(0xffffffffu, bad)) return 0u;
    unsigned none[16];  // signs: no pivot in common
#pragma unroll
    for (int j = 0; j < 16; j++) none[j] = 0x80008000u;
#pragma unroll 1
    for (int kb = 0; kb < KB; kb++) {
        if (KB > 1) fetch(kb);
        const int chunks = min(4, (e - kb * kSliceK + 7) / 8);
#pragma unroll 1
        for (int c = 0; c < chunks; c++) {
            uint4 v[4];
#pragma unroll
            for (int j = 0; j < 4; j++) v[j] = pb[c * gl + j];
#pragma unroll
            for (int i = 0; i < 4; i++) {
                const uint4 u = pa[c * gw + i];
#pragma unroll
                for (int j = 0; j < 4; j++)
                    none[4 * i + j] &= (u.x | v[j].x) & (u.y | v[j].y) & (u.z | v[j].z) & (u.w | v[j].w);
            }
        }
    }
#pragma unroll
    for (int j = 0; j < 16; j++)
        if (none[j] == 0x80008000u) bad &= ~(1u << j);
    return bad;
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
struct FormOut {
    using T = typename std::conditional<kMode == CTP_S_FP32 || kMode == CTP_S_FP32_PACKED, float, double>::type;
    static constexpr bool kPacked = kMode == CTP_S_FP64_PACKED || kMode == CTP_S_FP32_PACKED;
    static constexpr bool kSub = kMode == CTP_S_FP64_SUB || kMode == kUpdate;
};
// 2^(40 + weight) is the weight of g = 0: as large as the 64 bits allow for e pivots
__device__ __forceinline__ int weight(int e) { return e <= 16 ? 6 : (e <= 32 ? 5 : (e <= 64 ? 4 : (e <= 128 ? 3 : 2))); }

// One pivot's entry of W21 (kUpd: of y) in row i, of kind kd, from L21 and D.
template <bool kUpd>
__device__ __forceinline__ double w21_entry(const Tile &x, int k, int kd, int i) {
    if (kd == CTP_PIVKIND_ZERO) return 0.0;
    const double *c = x.L21 + (int64_t)k * x.ldl + i;
    double w = *c;  // kUpd: y itself, in the block's columns of A21
    if (!kUpd) {
        w *= x.D[2 * k];
        if (kd == CTP_PIVKIND_2X2_FIRST) w = fma(c[x.ldl], x.D[2 * k + 1], w);
        if (kd == CTP_PIVKIND_2X2_SECOND) w = fma(c[-x.ldl], x.D[2 * k - 1], w);
    }
    return w;
}
// The same of L21 in row j (kUpd: of the rows c0.. of L11).
template <bool kUpd>
__device__ __forceinline__ double l21_entry(const Tile &x, int k, int kd, int64_t j) {
    const bool d21 = kUpd && x.c0 + j == k + 1 && kd == CTP_PIVKIND_2X2_FIRST;  // that slot holds D
    if (kd == CTP_PIVKIND_ZERO || d21 || j >= x.nc) return 0.0;
    return x.L21[(kUpd ? -(int64_t)x.nc : 0) + (int64_t)k * x.ldl + j];
}
template <int kMode>
__device__ __forceinline__ void put_entry(const Tile &x, int i, int64_t j, double v) {
    typedef typename FormOut<kMode>::T OutT;
    OutT *ptr = reinterpret_cast<OutT *>(x.S) +
                (FormOut<kMode>::kPacked ? j * x.m - j * (j + 1) / 2 : j * x.lds) + i;
    *ptr = FormOut<kMode>::kSub ? (OutT)(*ptr - v) : (OutT)v;
}

// The entries that digits do not serve, after the CTA's last tile, by FP64 multiply-adds in
// the order of the pivots.  Most tiles with any have a few (with two or three pivots
// one entry in 10^4 of random rows is one, and a tile has 8192): a warp takes such a
// tile, a lane an entry, and the CTA's warps hide each other's latency (4 us a tile).  A
// tile with many is taken by all threads, four columns of a row each, or up to four
// times that, 32 pivots of W21 and L21 at a time in shared memory; one with all of
// them left out takes what FP64's pipe takes for it.
constexpr int kFew = 32;  // entries of a tile that a warp takes
template <int kMode>
__device__ __forceinline__ void fix_few(const Work &wk, Bars &bars, uint8_t *smem) {
    constexpr bool kUpd = kMode == kUpdate;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n = bars.nlist;
    uint16_t *ids = reinterpret_cast<uint16_t *>(smem) + warp * kFew;
    Tile &x = reinterpret_cast<Tile *>(smem + kThreads / 32 * kFew * sizeof(uint16_t))[warp];
    for (;;) {
        int at = 0;
        if (lane == 0) at = atomicAdd(&bars.next, 1);
        at = __shfl_sync(0xffffffffu, at, 0);
        if (at >= n) break;
        const int64_t t = bars.list[at];
        unsigned mask[kEpiWarps];
        int cnt = 0;
#pragma unroll
        for (int b = 0; b < kEpiWarps; b++) mask[b] = wk.marks[t - wk.first].out[b][lane];
#pragma unroll
        for (int b = 0; b < kEpiWarps; b++) cnt += __popc(mask[b]);
        int pos = cnt;  // inclusive prefix sum
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, pos, o);
            if (lane >= o) pos += v;
        }
        const int total = __shfl_sync(0xffffffffu, pos, 31);
        if (total > kFew) continue;  // left in the list
        if (lane == 0) bars.list[at] = -1;
        if (total == 0) continue;
        pos -= cnt;
#pragma unroll
        for (int b = 0; b < kEpiWarps; b++)
            for (unsigned w = mask[b]; w; w &= w - 1)
                ids[pos++] = (uint16_t)(((b >> 2) * 32 + lane) * kBN + (b & 3) * kCols + __ffs(w) - 1);
        if (lane == 0 && at < kKept) x = bars.kept[at];
        if (lane == 0 && at >= kKept) {
            Walk<kUpd> walk(wk);
            Tile y;
            walk.seek(t);
            walk.look(y);
            x = y;
        }
        __syncwarp();
        const int first = kUpd ? x.c0 - kSliceK : 0, e = x.e;
        for (int q0 = lane; q0 < total; q0 += 32) {
            const int i = x.ti * kBM + ids[q0] / kBN;
            const int64_t j = x.tj * kBN + ids[q0] % kBN;
            double acc = 0.0;
            for (int k0 = 0; k0 < e; k0 += 8) {
                double w[8], l[8];
#pragma unroll
                for (int q = 0; q < 8; q++) {
                    const int kd = k0 + q < e ? x.piv[first + k0 + q] : CTP_PIVKIND_ZERO;
                    w[q] = w21_entry<kUpd>(x, first + k0 + q, kd, i);
                    l[q] = l21_entry<kUpd>(x, first + k0 + q, kd, j);
                }
#pragma unroll
                for (int q = 0; q < 8; q++) acc = fma(w[q], l[q], acc);
            }
            put_entry<kMode>(x, i, j, acc);
        }
        __syncwarp();
    }
}

constexpr int kFixW = kBM + 1, kFixL = kBN + 1;  // padded rows of the slabs
template <int kMode>
__device__ __forceinline__ void fix_tile(const Work &wk, Bars &bars, uint8_t *smem, int64_t t) {
    constexpr bool kUpd = kMode == kUpdate;
    constexpr int kItems = (kBM * kBN / 4 + kThreads - 1) / kThreads;
    double *ws = reinterpret_cast<double *>(smem), *ls = ws + kSliceK * kFixW;
    uint16_t *ids = reinterpret_cast<uint16_t *>(ls + kSliceK * kFixL);
    const Tile &x = bars.tile[0];
    const int lane = threadIdx.x & 31;
    // a thread holds a row's sixteen columns
    const unsigned mask = threadIdx.x < kBM * kBN / kCols ? wk.marks[t - wk.first].out[threadIdx.x >> 5][lane] : 0u;
    if (!__syncthreads_or(mask != 0u)) return;  // its own results served after all
    if (threadIdx.x == 0) {
        Walk<kUpd> walk(wk);
        Tile y;
        walk.seek(t);
        walk.look(y);
        bars.tile[0] = y;
        bars.nmarks = 0;
    }
    __syncthreads();
    if (threadIdx.x < kBM * kBN / kCols) {  // which fours of columns have any
#pragma unroll
        for (int c = 0; c < 4; c++) {
            const unsigned has = __ballot_sync(0xffffffffu, (mask >> (4 * c)) & 0xFu);
            int at = 0;
            if (lane == 0) at = atomicAdd(&bars.nmarks, __popc(has));
            at = __shfl_sync(0xffffffffu, at, 0) + __popc(has & ((1u << lane) - 1u));
            if ((has >> lane) & 1u) ids[at] = (uint16_t)(threadIdx.x * 4 + c);
        }
    }
    __syncthreads();
    const int n = bars.nmarks;
    double acc[kItems][4] = {};
    int row[kItems], col[kItems];
#pragma unroll
    for (int it = 0; it < kItems; it++) {
        const int q = threadIdx.x + it * kThreads, id = q < n ? ids[q] : 0;  // warp's block, lane, four
        row[it] = (id >> 9) * 32 + ((id >> 2) & 31);
        col[it] = ((id >> 7) & 3) * kCols + (id & 3) * 4;
    }
    const int i0 = x.ti * kBM, j0 = x.tj * kBN, first = kUpd ? x.c0 - kSliceK : 0;
    for (int k0 = 0; k0 < x.e; k0 += kSliceK) {
        const int cnt = min(kSliceK, x.e - k0);
        for (int idx = threadIdx.x; idx < cnt * kBM; idx += kThreads) {
            const int k = first + k0 + idx / kBM, r = idx % kBM, kd = x.piv[k];
            ws[idx / kBM * kFixW + r] = i0 + r < x.m ? w21_entry<kUpd>(x, k, kd, i0 + r) : 0.0;
        }
        for (int idx = threadIdx.x; idx < cnt * kBN; idx += kThreads) {
            const int k = first + k0 + idx / kBN, c = idx % kBN, kd = x.piv[k];
            ls[idx / kBN * kFixL + c] = l21_entry<kUpd>(x, k, kd, j0 + c);
        }
        __syncthreads();
#pragma unroll
        for (int it = 0; it < kItems; it++) {
            if (threadIdx.x + it * kThreads >= n) break;
            for (int k = 0; k < cnt; k++) {
                const double w = ws[k * kFixW + row[it]];
#pragma unroll
                for (int c = 0; c < 4; c++) acc[it][c] = fma(w, ls[k * kFixL + col[it] + c], acc[it][c]);
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int it = 0; it < kItems; it++) {
        if (threadIdx.x + it * kThreads >= n) break;
        const int i = i0 + row[it];
        const unsigned mask =
            wk.marks[t - wk.first].out[row[it] / 32 * 4 + col[it] / kCols][row[it] % 32] >> (col[it] % kCols);
#pragma unroll
        for (int c = 0; c < 4; c++) {
            const int64_t j = j0 + col[it] + c;
            if (!((mask >> c) & 1u)) continue;
            put_entry<kMode>(x, i, j, acc[it][c]);
        }
    }
}

template <int kMode>
__device__ __noinline__ void fix_tiles(const Work &wk, Bars &bars, uint8_t *smem) {
    fix_few<kMode>(wk, bars, smem);
    __syncthreads();
    for (int q = 0; q < bars.nlist; q++)
        if (bars.list[q] >= 0) fix_tile<kMode>(wk, bars, smem, bars.list[q]);
    for (int64_t t = bars.marked; t >= 0; t = wk.marks[t - wk.first].prev) fix_tile<kMode>(wk, bars, smem, t);
}

template <int kMode>
__global__ void __launch_bounds__(kThreads, 1) k_form_fp64(const __grid_constant__ Work wk, int32_t *__restrict__ info) {
    typedef typename FormOut<kMode>::T OutT;
    constexpr bool kPacked = FormOut<kMode>::kPacked, kUpd = kMode == kUpdate, kSub = FormOut<kMode>::kSub;
    extern __shared__ unsigned char smraw[];
    __shared__ Bars bars;
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; s++) {
            mbar_init(&bars.full[s], 1);
            mbar_init(&bars.empty[s], 1);
        }
        mbar_init(&bars.acc_full, 2);  // the MMAs and the checker
        mbar_init(&bars.acc_empty, kEpiWarps);
        mbar_init(&bars.grp_full, 1);
        for (int s = 0; s < kRing; s++) {
            mbar_init(&bars.tile_full[s], 1);
            mbar_init(&bars.tile_empty[s], 3 + kEpiWarps);
        }
        bars.abort = 0;
        bars.weak = bars.next = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc(&bars.tmem_base, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = bars.tmem_base;
    uint8_t *grp = smem + kStages * (size_t)kStageBytes;

    Ring ring;
    if (warp == 2 + kEpiWarps) {
        // ---------------- scheduler
        if (lane == 0) {
            Walk<kUpd> walk(wk);
            Tile x;
            bool ok = true;
            do {
                walk.step(x);
                ok = mbar_wait(&bars.tile_empty[ring.slot], ring.phase ^ 1u, &bars.abort);
                if (!ok) break;
                bars.tile[ring.slot] = x;
                mbar_arrive(&bars.tile_full[ring.slot]);
                ring.step();
            } while (x.ti >= 0);
            if (!ok) atomicExch(&bars.abort, 1);
        }
    } else if (warp == 3 + kEpiWarps) {
        // ---------------- checker
        uint32_t accphase = 0, grpphase = 0;
        bool ok, first = true;
        int64_t marked = -1;
        int nlist = 0;
        while ((ok = ring.wait(bars))) {
            const Tile &x = bars.tile[ring.slot];
            if (x.ti < 0) break;
            unsigned bits = 0u;
            bool linked = false;
            if (x.e > 0) {
                // groups of the tile's blocks of rows
                const int gw = min(kBM, (int)slice_rows(x.m - x.ti * kBM)) / kGroup;
                const int gl = min(kBN, (int)slice_rows(x.nc - x.tj * kBN)) / kGroup;
                // rows that hold an Inf or NaN
                const int r0 = x.ti * kBM + 4 * lane, c0 = x.tj * kBN + 2 * lane;
                int4 er = make_int4(0, 0, 0, 0);
                int2 ec = make_int2(0, 0);
                if (r0 < x.m) er = *reinterpret_cast<const int4 *>(x.sb.ew + r0);
                if (c0 < x.nc) ec = *reinterpret_cast<const int2 *>(x.sb.el + c0);
                auto fetch = [&](int kb) {
                    __syncwarp();
                    if (lane == 0) {
                        const uint32_t chunks = min(4u, (uint32_t)(x.e - kb * kSliceK + 7) / 8);
                        const uint32_t bw = chunks * gw * 16, bl = chunks * gl * 16;
                        mbar_expect_tx(&bars.grp_full, bw + bl);
                        bulk_load(grp, x.sb.gw + (size_t)x.ti * x.sb.kb * (kWGroup / 2) + (size_t)kb * gw * 32, bw,
                                  &bars.grp_full);
                        bulk_load(grp + kWGroup, x.sb.gl + (size_t)x.tj * x.sb.kb * (kLGroup / 2) + (size_t)kb * gl * 32,
                                  bl, &bars.grp_full);
                    }
                    int never = 0;  // no CTA leaves with copies in flight
                    ok = mbar_wait(&bars.grp_full, grpphase, &never) && ok;
                    grpphase ^= 1u;
                };
                // (a lane whose 16 rows or columns are not all there takes no part in the first test)
                const bool in = x.ti * kBM + 16 * (lane >> 2) < x.m && x.tj * kBN + 16 * (lane & 3) < x.nc;
                bits = unsure_blocks(grp, x.e, gw, gl, in, fetch);
                if (!__all_sync(0xffffffffu, ok)) {
                    ok = false;
                    break;
                }
                const bool nonfinite =
                    __any_sync(0xffffffffu, er.x >= kExpNonfinite || (r0 + 1 < x.m && er.y >= kExpNonfinite) ||
                                                (r0 + 2 < x.m && er.z >= kExpNonfinite) ||
                                                (r0 + 3 < x.m && er.w >= kExpNonfinite) || ec.x >= kExpNonfinite ||
                                                (c0 + 1 < x.nc && ec.y >= kExpNonfinite));
                if (__any_sync(0xffffffffu, bits)) {
#pragma unroll
                    for (int j = 0; j < 4; j++) {  // rows and columns past the result
                        if (x.ti * kBM + 16 * (lane >> 2) + 4 * j >= x.m) bits &= ~(0xFu << (4 * j));
                        if (x.tj * kBN + 16 * (lane & 3) + 4 * j >= x.nc) bits &= ~(0x1111u << j);
                    }
                    // a warp of the epilogue: rows of two of these lanes, bit 4 (row group) + column group
                    bits <<= 16 * ((lane >> 2) & 1);
                    bits |= __shfl_xor_sync(0xffffffffu, bits, 4);
                }
                linked = __any_sync(0xffffffffu, bits) || nonfinite;
                if (linked && nlist < kList) {
                    if (lane == 0) bars.list[nlist] = x.t;
                    if (lane == 0 && nlist < kKept) bars.kept[nlist] = x;
                    nlist++;
                } else if (linked) {
                    if (lane == 0) wk.marks[x.t - wk.first].prev = marked;
                    marked = x.t;
                }
            }
            __syncwarp();
            if (lane == 0) ring.release(bars);
            ring.step();
            // the bits of the tile before last have been read once the last one's accumulators are full
            if (!first) {
                ok = mbar_wait(&bars.acc_full, accphase, &bars.abort);
                if (!ok) break;
                accphase ^= 1u;
            }
            first = false;
            if (!((lane >> 2) & 1)) bars.unsure[accphase][(lane >> 3) * 4 + (lane & 3)] = bits;
            if (lane == 0) bars.linked[accphase] = linked;
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars.acc_full);
        }
        if (lane == 0) {
            bars.marked = marked;
            bars.nlist = nlist;
            if (!ok) atomicExch(&bars.abort, 1);
        }
    } else if (warp == 0) {
        // ---------------- producer of the slices
        if (lane == 0) {
            int stage = 0, issued = 0;
            uint32_t phase = 0;
            bool ok = true;
            while (ok && (ok = ring.wait(bars))) {
                const Tile x = bars.tile[ring.slot];
                ring.release(bars);
                ring.step();
                if (x.ti < 0) break;
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
                    const unsigned char *kW = srcW + (size_t)kb * kSlices * 64 * rw, *kL = srcL + (size_t)kb * kSlices * 64 * rl;
                    if (rw == kBM)
                        bulk_load(dW, kW, kWBlock, &bars.full[stage]);
                    else
                        for (int s = 0; s < kSlices; s++)
                            bulk_load(dW + s * kWSlice, kW + s * 64 * rw, rw * 64, &bars.full[stage]);
                    if (rl == kBN)
                        bulk_load(dL, kL, kLBlock, &bars.full[stage]);
                    else
                        for (int s = 0; s < kSlices; s++)
                            bulk_load(dL + s * kLSlice, kL + s * 64 * rl, rl * 64, &bars.full[stage]);
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
            bool ok = true;
            while (ok && (ok = ring.wait(bars))) {
                const Tile &slot = bars.tile[ring.slot];
                const struct { int ti, e; } x = {slot.ti, slot.e};
                ring.release(bars);
                ring.step();
                if (x.ti < 0) break;
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
        for (;; ring.step()) {
            if (!ring.wait(bars)) {
                if (lane == 0) atomicExch(&bars.abort, 1);
                break;
            }
            const Tile &x = bars.tile[ring.slot];
            if (x.ti < 0) break;
            const int i = x.ti * kBM + q * 32 + lane, j0 = x.tj * kBN + cg * kCols, m = x.m, e = x.e;
            const int64_t lds = x.lds;
            // entries (i, j) with i < m and j <= jmax belong to the result
            const int jmax = kUpd ? x.nc - 1 : i;
            const bool any = j0 <= (kUpd ? jmax : i - lane + 31) && j0 < x.nc && i - lane < m;  // warp-uniform
            const bool interior = j0 + kCols - 1 <= (kUpd ? jmax : i - lane) && i - lane + 31 < m;
            OutT *ptr = reinterpret_cast<OutT *>(x.S) +
                        (kPacked ? (int64_t)j0 * m - (int64_t)j0 * (j0 + 1) / 2 : j0 * lds) + i;
            int ei = kExpZero, ej = kExpZero;
            if (e > 0 && i < m) ei = x.sb.ew[i];
            if (e > 0 && lane < kCols && j0 + lane < x.nc) ej = x.sb.el[j0 + lane];
            // subtracting: the old values come to L2 while the products are computed
            if (kSub && any && i < m) {
#pragma unroll
                for (int c = 0; c < kCols; c++)
                    if (interior || j0 + c <= jmax)
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(ptr + (int64_t)c * lds));
            }
            if (!mbar_wait(&bars.acc_full, accphase, &bars.abort)) {
                if (lane == 0) atomicExch(&bars.abort, 1);
                break;
            }
            const unsigned unsure = *(volatile uint32_t *)&bars.unsure[accphase][q * 4 + cg];
            const bool linked = *(volatile int *)&bars.linked[accphase] != 0;
            accphase ^= 1u;
            tc_fence_after();
            const int f = weight(e);
            long long V[kCols];
            if (any && e > 0) {
                const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(cg * kCols);
#pragma unroll
                for (int h = 0; h < kCols; h += 8)
                    if (kUpd || e <= 32)
                        add_groups<true>(ta + h, f, V + h);
                    else
                        add_groups<false>(ta + h, f, V + h);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars.acc_empty);
            // this row's entries left out: of a block that digits may not serve, they do serve
            // those of which they make 2^-7 of the scales (a lower bound of P)
            unsigned weak = 0u;
            const bool nonfinite = ei >= kExpNonfinite || ej >= kExpNonfinite;
            if (linked && any && (unsure || __any_sync(0xffffffffu, nonfinite))) {
#pragma unroll
                for (int c = 0; c < kCols; c++) {
                    const int ejc = __shfl_sync(0xffffffffu, ej, c);
                    const unsigned long long a = V[c] < 0 ? 0ull - (unsigned long long)V[c] : (unsigned long long)V[c];
                    const bool low = ((unsure >> ((lane & ~3) | (c >> 2))) & 1u) && a >> (45 + f) == 0ull &&
                                     ei != kExpZero && ejc != kExpZero;
                    if (i < m && j0 + c <= jmax && (low || ei >= kExpNonfinite || ejc >= kExpNonfinite)) weak |= 1u << c;
                }
            }
            // the plain case -- every entry of the warp's block belongs to the result, its
            // digits serve all of them, exponents are moderate -- has no test in its loop
            const bool mild = weak == 0u && abs(ei) < 400 && (lane >= kCols || abs(ej) < 400);
            if (!any) {
            } else if (interior && __all_sync(0xffffffffu, mild)) {
#pragma unroll
                for (int h = 0; h < kCols; h += 8) {
                    double old[8];  // eight old values loaded before any is stored
                    OutT *pl = ptr;
                    if (kSub) {
#pragma unroll
                        for (int c = 0; c < 8; c++) {
                            old[c] = *pl;
                            pl += lds;
                        }
                    }
#pragma unroll
                    for (int c = 0; c < 8; c++) {
                        const double v = to_fp64(V[h + c], ei + __shfl_sync(0xffffffffu, ej, h + c) - 52 - f);
                        if (kSub)
                            *ptr = (OutT)(old[c] - v);
                        else
                            __stcs(ptr, (OutT)v);
                        ptr += kPacked ? m - 1 - (j0 + h + c) : lds;
                    }
                }
            } else {
#pragma unroll
                for (int h = 0; h < kCols; h += 8) {
                    double old[8];
                    if (kSub) {
#pragma unroll
                        for (int c = 0; c < 8; c++) old[c] = i < m && j0 + h + c <= jmax ? ptr[(int64_t)c * lds] : 0.0;
                    }
#pragma unroll
                    for (int c = 0; c < 8; c++) {
                        const int ex = ei + __shfl_sync(0xffffffffu, ej, h + c) - 52 - f;
                        if (i < m && j0 + h + c <= jmax && !((weak >> (h + c)) & 1u)) {
                            const double v = e > 0 ? to_fp64_any(V[h + c], ex) : 0.0;
                            if (kSub)
                                *ptr = (OutT)(old[c] - v);
                            else
                                __stcs(ptr, (OutT)v);
                        }
                        ptr += kPacked ? m - 1 - (j0 + h + c) : lds;
                    }
                }
            }
            if (linked) {
                wk.marks[x.t - wk.first].out[q * 4 + cg][lane] = (uint16_t)weak;
                if (weak) bars.weak = 1;
            }
            __syncwarp();
            if (lane == 0) ring.release(bars);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && bars.abort) atomicCAS(info, kInfoOk, (int32_t)CTP_ETIMEOUT);
    if (bars.weak && !bars.abort) fix_tiles<kMode>(wk, bars, smem);
    __syncwarp();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// Few rows (kFormSmall at most): S by FP64 multiply-adds in the order of the pivots, a CTA
// per front, 32 pivots of W21 and L21 at a time in shared memory, a thread an entry or
// up to five.  A latency of a few microseconds per front, sixteen fronts per SM at a
// time; a tile of slices takes 5 us of its SM whatever its rows.
constexpr int kSmallT = 128, kSmallE = (kFormSmall * (kFormSmall + 1) / 2 + kSmallT - 1) / kSmallT;
template <int kMode>
__global__ void __launch_bounds__(kSmallT) k_form_small(const __grid_constant__ Work wk, const double *W21) {
    typedef typename FormOut<kMode>::T OutT;
    constexpr bool kPacked = FormOut<kMode>::kPacked, kSub = FormOut<kMode>::kSub;
    __shared__ double ws[kSliceK][kFormSmall + 1], ls[kSliceK][kFormSmall + 1];
    const double *L21 = wk.L21, *D = wk.D;
    const int32_t *piv = wk.piv, *nelim = wk.nelim;
    int64_t ldl = wk.ldl, lds = wk.lds;
    int m = (int)wk.m;
    OutT *S = reinterpret_cast<OutT *>(wk.S);
    if (wk.fronts != nullptr) {
        const int f = wk.item_front[blockIdx.x];
        const BFront b = wk.tab[f];
        const ctp_front fr = wk.fronts[f];
        m = (int)b.m;
        L21 = fr.A + b.p;
        ldl = fr.lda;
        lds = fr.lds;
        S = reinterpret_cast<OutT *>(fr.S);
        nelim = fr.nelim;
        W21 = reinterpret_cast<const double *>(wk.ws + b.ws + bsection(b.n, b.p, wk.o).W21);
    }
    const int e = *nelim, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // entries of the lower triangle, column by column
    const int total = m * (m + 1) / 2;
    int row[kSmallE], col[kSmallE];
    double acc[kSmallE] = {};
#pragma unroll
    for (int q = 0; q < kSmallE; q++) {
        const int t = min((int)threadIdx.x + q * kSmallT, total - 1);
        int j = (int)((2 * m + 1 - sqrtf((float)((2 * m + 1) * (2 * m + 1) - 8 * t))) * 0.5f);
        while (j > 0 && j * m - j * (j - 1) / 2 > t) j--;
        while ((j + 1) * m - (j + 1) * j / 2 <= t) j++;
        col[q] = j;
        row[q] = t - (j * m - j * (j - 1) / 2) + j;
    }
    for (int k0 = 0; k0 < e; k0 += kSliceK) {
        const int cnt = min(kSliceK, e - k0);
        for (int k = warp; k < cnt; k += kSmallT / 32) {
            if (lane >= m) continue;
            const int kk = k0 + k;
            const double *c = L21 + (int64_t)kk * ldl + lane;
            const double l = *c;
            double w;
            if (W21 != nullptr) {
                w = W21[(int64_t)kk * m + lane];
            } else {  // W21 = L21 D11
                const int kd = piv[kk];
                w = kd == CTP_PIVKIND_ZERO ? 0.0 : l * D[2 * kk];
                if (kd == CTP_PIVKIND_2X2_FIRST) w = fma(c[ldl], D[2 * kk + 1], w);
                if (kd == CTP_PIVKIND_2X2_SECOND) w = fma(c[-ldl], D[2 * kk - 1], w);
            }
            ws[k][lane] = w;
            ls[k][lane] = l;
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kSmallE; q++) {
            if ((int)threadIdx.x + q * kSmallT >= total) break;
#pragma unroll 4
            for (int k = 0; k < cnt; k++) acc[q] = fma(ws[k][row[q]], ls[k][col[q]], acc[q]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int q = 0; q < kSmallE; q++) {
        const int t = threadIdx.x + q * kSmallT;
        if (t >= total) break;
        OutT *ptr = S + (kPacked ? (int64_t)t : (int64_t)col[q] * lds + row[q]);
        *ptr = kSub ? (OutT)(*ptr - acc[q]) : (OutT)acc[q];
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
    __shared__ int red[kSW * 32], rexp[32];
    const int e = *nelim, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t row0 = (int64_t)blockIdx.x * 32;
    const int nrows = (int)min((int64_t)32, m - row0);
    for (int k = threadIdx.x; k < e; k += 32 * kSW) cexp[k] = (short)slice_col_exp(piv, Dinv, k);
    for (int k = w; k < e; k += kSW) xs[k * 33 + lane] = lane < nrows ? A[(int64_t)k * lda + p + row0 + lane] : 0.0;
    __syncthreads();
    write_slices<kLRows, kSW>(xs, e, row0, nrows, cexp, 1, sb.L, sb.el, sb.gl, sb.kb, m, red, rexp);
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
    write_slices<kWRows, kSW>(xs, e, row0, nrows, cexp, -1, sb.W, sb.ew, sb.gw, sb.kb, m, red, rexp);
}

template <int kMode>
cudaError_t launch_mode(const Work &wk, int32_t *info, int num_sms, cudaStream_t st) {
    cudaError_t err = smem_at_least((const void *)k_form_fp64<kMode>, kSmem);
    if (err != cudaSuccess) return err;
    const int64_t items = wk.count - wk.first;
    const unsigned grid = (unsigned)(items < num_sms ? items : num_sms);
    k_form_fp64<kMode><<<grid, kThreads, kSmem, st>>>(wk, info);
    return cudaGetLastError();
}

template <int kMode>
cudaError_t launch_small_mode(const Work &wk, const double *W21, cudaStream_t st) {
    k_form_small<kMode><<<(unsigned)wk.count, kSmallT, 0, st>>>(wk, W21);
    return cudaGetLastError();
}

cudaError_t launch_small(const Work &wk, const double *W21, int smode, cudaStream_t st) {
    switch (smode) {
    case CTP_S_FP64: return launch_small_mode<CTP_S_FP64>(wk, W21, st);
    case CTP_S_FP32: return launch_small_mode<CTP_S_FP32>(wk, W21, st);
    case CTP_S_FP64_SUB: return launch_small_mode<CTP_S_FP64_SUB>(wk, W21, st);
    case CTP_S_FP64_PACKED: return launch_small_mode<CTP_S_FP64_PACKED>(wk, W21, st);
    default: return launch_small_mode<CTP_S_FP32_PACKED>(wk, W21, st);
    }
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

// Slots of the walk that one launch takes.  Their marks are 1/64 of S (2.5 GB at n =
// 200000, p = 256), so larger Forms go in several launches that use the same ones, 273 MB
// at most (there: ten launches, 233.5 ms; all tiles in one 233.7).
constexpr int64_t kLaunchSlots = 262144;

cudaError_t launch_form_fp64(const SliceBuf &sb, const double *L21, int64_t lda, const int32_t *piv,
                             const double *D, int64_t m, const int32_t *nelim, void *S, int64_t lds, int smode,
                             TileMarks *marks, int32_t *info, int num_sms, cudaStream_t st) {
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
    wk.marks = marks;
    const int64_t slots = walk_slots(m), launches = (slots + kLaunchSlots - 1) / kLaunchSlots;
    cudaError_t err = cudaSuccess;
    for (int64_t r = 0; r < launches && err == cudaSuccess; r++) {
        wk.first = slots * r / launches;
        wk.count = slots * (r + 1) / launches;
        err = launch_any(wk, smode, info, num_sms, st);
    }
    return err;
}

cudaError_t launch_form_small(const double *L21, int64_t lda, const double *W21, const int32_t *piv, const double *D,
                              int64_t m, const int32_t *nelim, void *S, int64_t lds, int smode, cudaStream_t st) {
    if (m <= 0) return cudaSuccess;
    Work wk = {};
    wk.L21 = L21;
    wk.ldl = lda;
    wk.piv = piv;
    wk.D = D;
    wk.m = m;
    wk.lds = lds;
    wk.nelim = nelim;
    wk.S = S;
    wk.count = 1;
    return launch_small(wk, W21, smode, st);
}

cudaError_t launch_form_small_batch(const ctp_front *fronts, const BFront *tab, char *ws, const int *list, int64_t count,
                                    BatchOpts o, cudaStream_t st) {
    if (count == 0) return cudaSuccess;
    Work wk = {};
    wk.fronts = fronts;
    wk.tab = tab;
    wk.ws = ws;
    wk.item_front = list;
    wk.o = o;
    wk.count = count;
    return launch_small(wk, nullptr, o.smode, st);
}

cudaError_t launch_form_fp64_batch(const ctp_front *fronts, const BFront *tab, char *ws,
                                   const int *item_front, int64_t items, BatchOpts o, TileMarks *marks, int32_t *info,
                                   int num_sms, cudaStream_t st, const int *item_tile) {
    if (items == 0) return cudaSuccess;
    Work wk = {};
    wk.fronts = fronts;
    wk.tab = tab;
    wk.ws = ws;
    wk.item_front = item_front;
    wk.item_tile = item_tile;
    wk.o = o;
    wk.count = items;
    wk.marks = marks;
    return launch_any(wk, o.smode, info, num_sms, st);
}

cudaError_t launch_update(const SliceBuf &u, double *A, int64_t lda, int p, int64_t m, int blk, const int32_t *piv,
                          const int32_t *nelim, TileMarks *marks, int32_t *info, int num_sms, cudaStream_t st) {
    Work wk = {};
    wk.sb = u;
    wk.marks = marks;
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

int64_t form_fp64_marks(int64_t m) {
    const int64_t slots = m > 0 ? walk_slots(m) : 0;
    return slots < kLaunchSlots ? slots : kLaunchSlots;
}

int64_t update_tiles(int64_t m, int p) {
    return p > kSliceK ? (m + kBM - 1) / kBM * ((p - kSliceK + kBN - 1) / kBN) : 0;
}

cudaError_t launch_update_batch(const ctp_front *fronts, const BFront *tab, char *ws, const int *item_front,
                                const int *item_tile, int64_t items, BatchOpts o, TileMarks *marks, int32_t *info,
                                int num_sms, cudaStream_t st) {
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
    wk.marks = marks;
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
    if (form_small(m)) return 0;  // not of slices
    const int64_t nM = (m + kBM - 1) / kBM, nN = (m + kBN - 1) / kBN;
    return nM * (nM + 1) - (2 * nM - nN);
}

}  // namespace ctp
