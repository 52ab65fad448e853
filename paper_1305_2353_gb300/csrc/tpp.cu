// tpp.cu -- K4: threshold partial pivoting on the whole supernode (Listing 1,
// Section 2), i.e. without compression: every test takes its column maxima over
// all n rows, which must be up to date.  This is the comparator of the
// compressed path, and the pivoting of a chain's or a root's last resort.
//
// GB300 design.  One cooperative, persistent launch (one CTA of 16 warps per SM
// at most, all co-resident).  The rows of A21 are dealt out in contiguous runs,
// one per CTA, held in shared memory when they fit (n p up to about 3.6 million
// entries on 152 SMs) and streamed from memory otherwise; the elements of W11's
// lower triangle are dealt out one by one, each owned by one thread, which
// keeps it in a register and writes it and its mirror to the current of two W11 buffers
// in L2.  Every CTA takes every decision itself, from the same numbers and so with the
// same outcome: nothing has to be sent back.  Per accepted pivot:
//   look ahead  warp 0 forms the next candidate's column of W11, its partner's
//               and their maxima on A11, applying the pivot at hand to the old
//               columns just as their owners do, while the others
//   update      apply the pivot to W11 and to the CTA's rows of A21;
//   exchange    all that is missing for the next decision are the two columns'
//               maxima over A21: each CTA publishes its two (16 bytes) and
//               reads all CTAs', one L2 write and read instead of a barrier and
//               two dependent reads; it also tells that all of W11 is written.
// After a search with rejections, or when the candidate looked ahead fails, all
// column maxima are merged in L2 behind a grid barrier (its spin bounded) and a window
// of up to 16 candidates (one warp each) is tested per step; rejected candidates change
// nothing, so the window's size does not matter to the outcome.
// What bounds a pivot at moderate n is latency: the exchange (3200 to 6000 clocks with 35
// to 152 CTAs), the decision and its broadcast (2500), the look-ahead beside
// the updates (4500, sharing the FP64 pipe); at large n the pass over the trailing
// A21, the traffic that the paper's compressed pivoting avoids (Section 6).
// Measured per pivot, with a grid barrier and the tests behind it -> looking ahead: 8.9
// -> 6.1 us at n = 1999, p = 256; 9.2 -> 5.2 at 1000, 256; 11.2 -> 8.4 at 20011, 127
// (FP64 work 3); 42.5 -> 39.7 at 60000, 256 (streamed).  How many CTAs share the
// rows hardly matters (24 to 152 CTAs: within 15%).
// At the end the A21 columns are scaled and permuted into pivot order and
// L11 / D / the delayed block are written from W11, in the same layout as the
// compressed path.  A barrier that gives up sets the abort flag and
// CTP_ETIMEOUT in the info word, and every CTA leaves the main loop.
#include "ctp_internal.cuh"
#include "pivot_tests.cuh"

namespace ctp {

namespace {

constexpr int kT = 512;
constexpr int kNW = kT / 32;
constexpr int kOwners = kT - 32;      // threads that own elements of W11 (warp 0 looks ahead)
constexpr long kBarSpin = 1L << 22;  // default polls (an L2 round trip each): about two seconds
constexpr size_t kTileBytes = 200 * 1024;  // shared memory for a CTA's rows of A21
constexpr int kMaxCtas = 256;              // records of the exchange

struct Ctl {
    unsigned bar_count;
    int abort;
};

struct TppArgs {
    double *A;
    int64_t lda, n;
    int p;
    double u, small;
    double *W11;                 // three p x p: two buffers by turns, then the pivots' frozen columns
    unsigned long long *M21;     // [3][p] column-maximum keys of the trailing A21
    ulonglong2 *rec;             // [2][CTAs] the exchanged maxima of two columns
    Ctl *ctl;
    int32_t *perm, *piv, *nelim;
    double *D, *Dinv;
    int32_t *info;
    long spin;                   // polls a grid barrier waits before it gives up
    int64_t rows;                // A21 rows per CTA
};

struct Shared {
    Decision res[kNW];
    double sD[2 * kMaxP + 2], sInv[2 * kMaxP + 2];
    double b0[kMaxP], b1[kMaxP], s0[kMaxP], s1[kMaxP];  // pivot column(s) on the A11 rows; times D^-1
    double cc[kMaxP], ct[kMaxP];      // the next candidate's and its partner's columns, looked ahead
    unsigned long long lmax[kMaxP];   // column maxima of this CTA's rows
    int order[kMaxP], kind[kMaxP], pos_of[kMaxP];
    unsigned char live[kMaxP];
    unsigned short lcol[kMaxP];  // the live columns after the pivot at hand
    int nlive, ok, job, lost;         // lost: warp 0 gave up
    int next, partner;                // the candidate looked ahead and its partner, -1: none
    double att, atm, amm;             // their entries
    unsigned long long vt, vm;        // their maxima on the other rows of A11
};

__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

// Software grid barrier for a cooperative launch (arrivals are counted up, never
// reset: the epoch's target is epoch * CTAs); false on timeout (more than
// `spin` polls) or when another CTA gave up.
__device__ __forceinline__ bool grid_sync(Ctl *ctl, unsigned target, int *s_ok, long spin) {
    __syncthreads();
    if (threadIdx.x == 0) {
        fence_gpu();
        unsigned seen = atomicAdd(&ctl->bar_count, 1u) + 1u;
        int ok = 1;
        for (long it = 0; (int)(seen - target) < 0; it++) {
            if (it >= spin) {
                ok = 0;
                atomicExch(&ctl->abort, 1);
                break;
            }
            seen = *(volatile unsigned *)&ctl->bar_count;
        }
        fence_gpu();
        *s_ok = ok && (*(volatile int *)&ctl->abort == 0);
    }
    __syncthreads();
    return *s_ok != 0;
}

// Every CTA's maxima of the two columns looked ahead, exchanged without a barrier: a
// CTA stores its two keys (their free sign bit is the tag: it flips each time
// the slot is used), and warps 0 and 1 read all CTAs' until every tag is there.
// Warp 1 publishes; its fence between the CTA's writes of W11 and the record was
// issued behind them, long before.  Records are double-buffered: a CTA
// publishes exchange g+2 after it has read all of g+1, whose writers have read g.
__device__ __forceinline__ unsigned long long record_tag(unsigned g) {
    return (unsigned long long)(((g >> 1) & 1) ^ 1) << 63;
}

__device__ __forceinline__ void publish(const TppArgs &a, unsigned g, unsigned long long kc, unsigned long long kt) {
    const unsigned long long tag = record_tag(g);
    asm volatile("st.volatile.global.v2.u64 [%0], {%1, %2};" ::"l"(a.rec + (g & 1) * kMaxCtas + blockIdx.x),
                 "l"(kc | tag), "l"(kt | tag)
                 : "memory");
}

// Waits for all records of exchange g (one warp; kB records per lane and pass): this lane's
// maxima.  False on timeout or abort.
template <int kB>
__device__ __forceinline__ bool gather(const TppArgs &a, unsigned g, unsigned long long &mc, unsigned long long &mt) {
    const int lane = threadIdx.x & 31, G = (int)gridDim.x;
    const ulonglong2 *buf = a.rec + (g & 1) * kMaxCtas;
    const unsigned long long tag = record_tag(g), mask = ~(1ull << 63);
    for (long it = 0;; it++) {
        unsigned long long miss = 0;
        mc = mt = 0;
        for (int i0 = lane; i0 - lane < G; i0 += 32 * kB) {
            unsigned long long x[kB], y[kB];
#pragma unroll
            for (int j = 0; j < kB; j++) {
                const int i = min(i0 + 32 * j, G - 1);  // the last record again instead of a branch
                asm volatile("ld.volatile.global.v2.u64 {%0, %1}, [%2];"
                             : "=l"(x[j]), "=l"(y[j])
                             : "l"(buf + i)
                             : "memory");
            }
#pragma unroll
            for (int j = 0; j < kB; j++) {
                miss |= (x[j] ^ tag) | (y[j] ^ tag);
                x[j] &= mask;
                y[j] &= mask;
                mc = x[j] > mc ? x[j] : mc;
                mt = y[j] > mt ? y[j] : mt;
            }
        }
        if (__all_sync(0xffffffffu, !(miss >> 63))) return true;
        if (it >= a.spin || ((it & 63) == 63 && *(volatile int *)&a.ctl->abort)) {
            if (lane == 0) atomicExch(&a.ctl->abort, 1);
            return false;
        }
    }
}

__device__ __forceinline__ bool gather(const TppArgs &a, unsigned g, unsigned long long &mc, unsigned long long &mt) {
    return gridDim.x <= 32   ? gather<1>(a, g, mc, mt)
           : gridDim.x <= 64 ? gather<2>(a, g, mc, mt)
                             : gather<5>(a, g, mc, mt);
}

// Listing 1's decision on candidate c with partner t (-1: none) from the entries and the
// maxima vt, vm of the two columns outside them; the 1x1 outcome leaves i0 to the caller.
__device__ __forceinline__ Decision tpp_decide(int c, int t, double att, double atm, double amm,
                                               unsigned long long vt, unsigned long long vm, double u,
                                               double rcp_u, unsigned long long small_k) {
    Decision d;
    d.kind = DEC_REJECT;
    d.t = -1;
    d.m = c;
    d.pad = 0;
    d.d0 = d.d1 = d.d2 = d.i0 = d.i1 = d.i2 = 0.0;
    const unsigned long long kmm = akey(amm), ktm = t >= 0 ? akey(atm) : 0ull;
    unsigned long long vall = vm > kmm ? vm : kmm;
    vall = ktm > vall ? ktm : vall;
    if (vall < small_k) {
        d.kind = DEC_ZERO;
        return d;
    }
    unsigned long long maxm1 = vm;
    if (t >= 0) {
        if (test_2x2(att, atm, amm, vt, vm, rcp_u, small_k, d)) {
            d.kind = DEC_2X2;
            d.t = t;
            return d;
        }
        maxm1 = ktm > vm ? ktm : vm;
    }
    if (kmm >= akey(__dmul_rn(u, key_val(maxm1)))) {
        d.kind = DEC_1X1;
        d.d0 = amm;
    }
    return d;
}

// Partner of candidate c: the live j < c with the largest |a(c, j)|, lowest j on ties; -1: none.
template <int NE>
__device__ __forceinline__ int partner(int c, const unsigned long long (&km)[NE], const bool (&lv)[NE]) {
    const int lane = threadIdx.x & 31;
    unsigned long long bv = 0;
    int bi = -1;
#pragma unroll
    for (int q = 0; q < NE; q++) {
        const int i = lane + 32 * q;
        if (lv[q] && i < c && (bi < 0 || km[q] > bv)) {
            bv = km[q];
            bi = i;
        }
    }
    const unsigned bh = bi >= 0 ? (unsigned)(bv >> 32) : 0u, bl = bi >= 0 ? (unsigned)bv : 0u;
    const unsigned BH = __reduce_max_sync(0xffffffffu, bh);
    const unsigned BL = __reduce_max_sync(0xffffffffu, bh == BH ? bl : 0u);
    const int t0 = __reduce_min_sync(0xffffffffu, (bi >= 0 && bh == BH && bl == BL) ? bi : 0x7fffffff);
    return t0 == 0x7fffffff ? -1 : t0;
}

// Largest key of the live entries but c's and t's.
template <int NE>
__device__ __forceinline__ unsigned long long rest_max(int c, int t, const unsigned long long (&km)[NE],
                                                       const bool (&lv)[NE]) {
    const int lane = threadIdx.x & 31;
    unsigned long long v = 0;
#pragma unroll
    for (int q = 0; q < NE; q++) {
        const int i = lane + 32 * q;
        if (lv[q] && i != t && i != c) v = km[q] > v ? km[q] : v;
    }
    return warp_max_key(v);
}

// Tests of Listing 1 for candidate c (one warp, p <= 256: eight entries of a column
// per lane, loaded together): the A11 part of every column maximum comes from
// W11, the A21 part is the key M[c].
__device__ __forceinline__ Decision tpp_test(int c, const double *W, const unsigned long long *M,
                                             const unsigned char *live, int p, double u, double rcp_u,
                                             unsigned long long small_k) {
    constexpr int NE = kMaxP / 32;
    const int lane = threadIdx.x & 31;
    const double *cm = W + (size_t)c * p;
    unsigned long long km[NE], vt = 0;
    bool lv[NE];
#pragma unroll
    for (int q = 0; q < NE; q++) {
        const int i = lane + 32 * q;
        lv[q] = i < p && live[i];
        km[q] = i < p ? akey(__ldcg(cm + i)) : 0ull;
    }
    const double amm = __ldcg(cm + c);
    const unsigned long long mc = __ldcg(M + c);
    const int t = partner(c, km, lv);
    double att = 0.0, atm = 0.0;
    if (t >= 0) {
        const double *ct = W + (size_t)t * p;
        unsigned long long kt[NE];
#pragma unroll
        for (int q = 0; q < NE; q++) {
            const int i = lane + 32 * q;
            kt[q] = i < p ? akey(__ldcg(ct + i)) : 0ull;
        }
        att = __ldcg(ct + t);
        atm = __ldcg(cm + t);
        const unsigned long long mt = __ldcg(M + t);
        vt = rest_max(c, t, kt, lv);
        vt = vt > mt ? vt : mt;
    }
    unsigned long long vm = rest_max(c, t, km, lv);
    vm = vm > mc ? vm : mc;
    Decision d = tpp_decide(c, t, att, atm, amm, vt, vm, u, rcp_u, small_k);
    if (d.kind == DEC_1X1) d.i0 = __drcp_rn(amm);
    return d;
}

// A pivot's update of this CTA's rows of A21 in memory: column k of the live list,
// entry r: a(r,k) - x0(r) s0(k) - x1(r) s1(k), one fused multiply-add per term, with x
// the pivot column(s) and s = D^-1 times the pivot row(s); the new maximum of the
// column goes to lmax[k].  A warp takes a column at a time, whichever is next (the first
// warp joins late), four loads per lane in flight.
template <bool k2x2>
__device__ __forceinline__ void update_rows(double *T, int64_t ldt, int64_t rows, int q0, int q1, Shared &sh) {
    const int lane = threadIdx.x & 31;
    const double *x0 = T + q0 * ldt, *x1 = k2x2 ? T + q1 * ldt : x0;
    for (;;) {
        int ci = 0;
        if (lane == 0) ci = atomicAdd(&sh.job, 1);
        ci = __shfl_sync(0xffffffffu, ci, 0);
        if (ci >= sh.nlive) break;
        const int k = sh.lcol[ci];
        const double s0 = sh.s0[k], s1 = k2x2 ? sh.s1[k] : 0.0;
        double *col = T + k * ldt;
        unsigned long long mx = 0;
        constexpr int U = 4;
        for (int64_t r0 = lane; r0 < rows; r0 += 32 * U) {
            double v[U], a[U], b[U];
#pragma unroll
            for (int q = 0; q < U; q++) {
                const bool in = r0 + 32 * q < rows;
                v[q] = in ? col[r0 + 32 * q] : 0.0;
                a[q] = in ? x0[r0 + 32 * q] : 0.0;
                b[q] = (k2x2 && in) ? x1[r0 + 32 * q] : 0.0;
            }
#pragma unroll
            for (int q = 0; q < U; q++) {
                if (r0 + 32 * q >= rows) break;
                double w = fma(-a[q], s0, v[q]);
                if (k2x2) w = fma(-b[q], s1, w);
                col[r0 + 32 * q] = w;
                const unsigned long long kk = akey(w);
                mx = kk > mx ? kk : mx;
            }
        }
        mx = warp_max_key(mx);
        if (lane == 0) sh.lmax[k] = mx;
    }
}

// The same in shared memory, a column per lane (rows in slices over the warps), so
// that every lane of a multiply-add has work however few rows a CTA holds, and
// nothing is reduced: maxima are taken from the tile where they are needed.
template <bool k2x2>
__device__ __forceinline__ void update_cols(double *T, int64_t ldt, int rows, int q0, int q1, const Shared &sh, int w,
                                            int nw) {
    constexpr int U = 8;
    const int lane = threadIdx.x & 31, nlive = sh.nlive;
    const double *x0 = T + q0 * ldt, *x1 = k2x2 ? T + q1 * ldt : x0;
    const int groups = (nlive + 31) / 32;
    int slices = groups > 0 ? nw / groups : 1;
    if (slices < 1) slices = 1;
    const int per = (rows + slices - 1) / slices;
    for (int job = w; job < groups * slices; job += nw) {
        const int g = job % groups, s = job / groups, r1 = min(rows, (s + 1) * per);
        const int ci = g * 32 + lane;
        const bool in = ci < nlive;
        const int k = in ? sh.lcol[ci] : q0;
        const double s0 = sh.s0[k], s1 = k2x2 ? sh.s1[k] : 0.0;
        double *col = T + k * ldt;
        int r = s * per;
        for (; r + U <= r1; r += U) {
            double v[U];
#pragma unroll
            for (int q = 0; q < U; q++) v[q] = col[r + q];
#pragma unroll
            for (int q = 0; q < U; q++) {
                v[q] = fma(-x0[r + q], s0, v[q]);
                if (k2x2) v[q] = fma(-x1[r + q], s1, v[q]);
            }
            if (in) {
#pragma unroll
                for (int q = 0; q < U; q++) col[r + q] = v[q];
            }
        }
#pragma unroll 1
        for (; r < r1; r++) {
            double v = fma(-x0[r], s0, col[r]);
            if (k2x2) v = fma(-x1[r], s1, v);
            if (in) col[r] = v;
        }
    }
}

// Largest key of a column of the tile (one warp).
__device__ __forceinline__ unsigned long long tile_max(const double *col, int64_t rows) {
    unsigned long long mx = 0;
    for (int64_t r = threadIdx.x & 31; r < rows; r += 32) {
        const unsigned long long k = akey(col[r]);
        mx = k > mx ? k : mx;
    }
    return warp_max_key(mx);
}

// kOwn: elements of W11's lower triangle a thread owns.
template <bool kSmem, int kOwn>
__global__ void __launch_bounds__(kT, 1) k_tpp(TppArgs a) {
    extern __shared__ __align__(16) double dsm[];  // kSmem: the CTA's rows [p][rows]; else staging [p][33]
    __shared__ Shared sh;
    const int p = a.p;
    const int64_t n = a.n, m = n - p, lda = a.lda;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    Ctl *ctl = a.ctl;
    const int64_t row0 = min((int64_t)blockIdx.x * a.rows, m), rows = min(a.rows, m - row0);
    double *T = kSmem ? dsm : a.A + p + row0;
    const int64_t ldt = kSmem ? (a.rows | 1) : lda;
    const int pp = p * p;
    double *fin = a.W11 + 2 * (size_t)pp;

    // ---- this thread's elements of W11's lower triangle (columns k and p-1-k share a
    // row of p+1 elements), this CTA's rows of A21 and their column maxima
    const int half = (p + 1) / 2;
    double own[kOwn];
    int oki[kOwn];  // column << 16 | row; -1: none
#pragma unroll
    for (int j = 0; j < kOwn; j++) {
        const int idx = tid < 32 ? half * (p + 1) : ((int)blockIdx.x + j * (int)gridDim.x) * kOwners + tid - 32;
        const int h = idx / (p + 1), o = idx - h * (p + 1);
        const bool low = o < p - h;
        const int k = low ? h : p - 1 - h, i = low ? h + o : k + o - (p - h);
        own[j] = 0.0;
        oki[j] = -1;
        if (h < half && (low || k != h)) {
            oki[j] = k << 16 | i;
            own[j] = a.A[(int64_t)k * lda + i];
            a.W11[k * p + i] = a.W11[i * p + k] = own[j];
        }
    }
    bool nonfinite = false;
    for (int k = warp; k < p; k += kNW) {
        const double *src = a.A + (int64_t)k * lda + p + row0;
        unsigned long long mx = 0;
        for (int64_t r0 = lane; r0 < rows; r0 += 128) {
            double v[4];
#pragma unroll
            for (int q = 0; q < 4; q++) v[q] = r0 + 32 * q < rows ? src[r0 + 32 * q] : 0.0;
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const unsigned long long kk = akey(v[q]);
                nonfinite |= kk >= 0x7FF0000000000000ull;
                mx = kk > mx ? kk : mx;
                if (kSmem && r0 + 32 * q < rows) T[k * ldt + r0 + 32 * q] = v[q];
            }
        }
        mx = warp_max_key(mx);
        if (!kSmem && lane == 0) sh.lmax[k] = mx;
    }
    if (nonfinite) atomicCAS(a.info, kInfoOk, (int32_t)CTP_ENONFINITE);
    for (int i = tid; i < p; i += kT) sh.live[i] = 1;
    if (tid == 0) sh.next = -1, sh.lost = 0;
    __syncthreads();

    const double u = a.u, rcp_u = __drcp_rn(a.u);
    const unsigned long long small_k = akey(a.small);
    int nelim = 0, c0 = p >= 2 ? 1 : 0, accepted = 0, win = 1, from = c0;
    unsigned round = 0, exchanges = 0, barriers = 0;
    bool ok = true;
    constexpr int NE = kMaxP / 32;
    double cv[NE];  // warp 0: the column of the next candidate
    int next = -1;
    for (;;) {
        const double *W = a.W11 + (size_t)(round & 1) * pp;
        double *Wn = a.W11 + (size_t)((round & 1) ^ 1) * pp;
        bool stop = false, ahead = false;
        int gap = 0;  // candidates rejected before the pivot
        Decision dv;
        // ---------------- decide on the candidate looked ahead: two maxima are all
        // that is not known here yet
        if (sh.next >= 0) {
            const int c = sh.next;
            if (warp == 1) {
                const int t = sh.partner;
                unsigned long long kc, kt;
                if (kSmem) {
                    kc = kt = 0;
                    const double *colc = T + c * ldt, *colt = T + (t < 0 ? c : t) * ldt;
                    for (int r = lane; r < (int)rows; r += 32) {
                        const unsigned long long x = akey(colc[r]), z = akey(colt[r]);
                        kc = x > kc ? x : kc;
                        kt = z > kt ? z : kt;
                    }
                    kc = warp_max_key(kc);
                    kt = t < 0 ? 0ull : warp_max_key(kt);
                } else {
                    kc = sh.lmax[c];
                    kt = t < 0 ? 0ull : sh.lmax[t];
                }
                if (lane == 0) publish(a, exchanges, kc, kt);
                // while the records travel
                const double att = sh.att, atm = sh.atm, amm = sh.amm, rcp = __drcp_rn(amm);
                const unsigned long long vt = sh.vt, vm = sh.vm;
                const bool got = gather(a, exchanges, kc, kt);
                kc = warp_max_key(kc);
                kt = warp_max_key(kt);
                Decision d = tpp_decide(c, t, att, atm, amm, kt > vt ? kt : vt, kc > vm ? kc : vm, u, rcp_u, small_k);
                if (d.kind == DEC_1X1) d.i0 = rcp;
                if (lane == 0) {
                    sh.res[0] = d;
                    sh.ok = got;
                }
            } else if (warp == 0) {
                // the column of the candidate after c, should c be accepted
                next = -1;
                for (int j0 = (c + 1) & ~31; j0 < p && next < 0; j0 += 32) {
                    const int j = j0 + lane;
                    const unsigned bal = __ballot_sync(0xffffffffu, j > c && j < p && sh.live[j]);
                    if (bal) next = j0 + __ffs(bal) - 1;
                }
                unsigned long long kc, kt;
                if (next >= 0) {
                    if (!gather(a, exchanges, kc, kt) && lane == 0) sh.lost = 1;
                    fence_gpu();
#pragma unroll
                    for (int q = 0; q < NE; q++) {
                        const int i = lane + 32 * q;
                        cv[q] = i < p ? __ldcg(W + (size_t)next * p + i) : 0.0;
                    }
                }
            }
            __syncthreads();
            exchanges++;
            if (!(ok = sh.ok && !sh.lost)) break;
            dv = sh.res[0];
            ahead = dv.kind == DEC_1X1 || dv.kind == DEC_2X2;
            from = c;
            c0 = c + 1;
            win = 4;
            if (dv.kind == DEC_ZERO) {
                if (tid == 0) {
                    sh.live[c] = 0;
                    sh.order[nelim] = c;
                    sh.kind[nelim] = CTP_PIVKIND_ZERO;
                    sh.sD[2 * nelim] = sh.sD[2 * nelim + 1] = 0.0;
                    sh.sInv[2 * nelim] = sh.sInv[2 * nelim + 1] = 0.0;
                }
                nelim++;
                from = c0;
                win = 1;
            }
        }
        const unsigned long long *M = a.M21 + (barriers % 3) * p;
        if (!ahead) {  // all maxima: a grid barrier
            for (int k = warp; k < p; k += kNW)
                if (sh.live[k]) {
                    const unsigned long long mx = kSmem ? tile_max(T + k * ldt, rows) : sh.lmax[k];
                    if (lane == 0 && mx) atomicMax(a.M21 + (barriers % 3) * p + k, mx);
                }
            ok = grid_sync(ctl, (barriers + 1) * gridDim.x, &sh.ok, a.spin);
            if (!ok) break;
            if (blockIdx.x == 0)  // read last in the decision before this barrier
                for (int k = tid; k < p; k += kT) a.M21[((barriers + 2) % 3) * p + k] = 0;
            barriers++;
        }
        // ---------------- decide: the same steps and outcome in every CTA
        while (!ahead) {
            if (nelim >= p) {
                stop = true;
                break;
            }
            while (c0 < p && !sh.live[c0]) c0++;
            if (c0 >= p) {
                if (!accepted) {  // a whole sweep without a pivot
                    stop = true;
                    break;
                }
                accepted = 0;
                c0 = from = 0;
                continue;
            }
            const int hi = min(p, c0 + win);
            {
                const int c = c0 + warp;
                int kind = DEC_REJECT;
                if (c < hi && sh.live[c]) {
                    const Decision d = tpp_test(c, W, M, sh.live, p, u, rcp_u, small_k);
                    kind = d.kind;
                    if (lane == 0) sh.res[warp] = d;
                }
                if (lane == 0 && kind == DEC_REJECT) sh.res[warp].kind = DEC_REJECT;
            }
            __syncthreads();
            int w = 0;
            while (w < hi - c0 && sh.res[w].kind == DEC_REJECT) w++;
            if (w >= hi - c0) {
                c0 = hi;
                win = win * 4 < kNW ? win * 4 : kNW;
                __syncthreads();
                continue;
            }
            dv = sh.res[w];
            // the next window: twice the distance that this search covered
            gap = dv.m - from;
            win = 1;
            while (win < 2 * gap && win < kNW) win *= 2;
            c0 = from = dv.m + 1;
            accepted = 1;
            __syncthreads();
            if (dv.kind != DEC_ZERO) break;
            if (tid == 0) {
                sh.live[dv.m] = 0;
                sh.order[nelim] = dv.m;
                sh.kind[nelim] = CTP_PIVKIND_ZERO;
                sh.sD[2 * nelim] = sh.sD[2 * nelim + 1] = 0.0;
                sh.sInv[2 * nelim] = sh.sInv[2 * nelim + 1] = 0.0;
            }
            nelim++;
            __syncthreads();
        }
        if (stop) break;
        // ---------------- the pivot's records, its column(s) and the live list
        const bool two = dv.kind == DEC_2X2;
        const int q0 = two ? dv.t : dv.m, q1 = two ? dv.m : -1;
        if (tid == 0) {
            sh.order[nelim] = q0;
            sh.kind[nelim] = two ? CTP_PIVKIND_2X2_FIRST : CTP_PIVKIND_1X1;
            sh.sD[2 * nelim] = dv.d0;
            sh.sD[2 * nelim + 1] = two ? dv.d1 : 0.0;
            sh.sInv[2 * nelim] = dv.i0;
            sh.sInv[2 * nelim + 1] = two ? dv.i1 : 0.0;
            if (two) {
                sh.order[nelim + 1] = q1;
                sh.kind[nelim + 1] = CTP_PIVKIND_2X2_SECOND;
                sh.sD[2 * nelim + 2] = dv.d2;
                sh.sD[2 * nelim + 3] = 0.0;
                sh.sInv[2 * nelim + 2] = dv.i2;
                sh.sInv[2 * nelim + 3] = 0.0;
            }
        }
        // the next candidate, looked ahead unless this search had rejections
        if (warp == 0) {
            const bool look = gap == 0 && nelim + (two ? 2 : 1) < p;
            if (!ahead) {
                next = -1;
                for (int j0 = (dv.m + 1) & ~31; look && j0 < p && next < 0; j0 += 32) {
                    const int j = j0 + lane;
                    const unsigned bal = __ballot_sync(0xffffffffu, j > dv.m && j < p && sh.live[j]);
                    if (bal) next = j0 + __ffs(bal) - 1;
                }
#pragma unroll
                for (int q = 0; q < NE; q++) {
                    const int i = lane + 32 * q;
                    cv[q] = next >= 0 && i < p ? __ldcg(W + (size_t)next * p + i) : 0.0;
                }
            }
            if (lane == 0) sh.next = look ? next : -1;
        } else if (warp == 1) {
            int r = 0;
            for (int j0 = 0; j0 < p; j0 += 32) {
                const int j = j0 + lane;
                const bool l = j < p && sh.live[j] && j != q0 && j != q1;
                const unsigned bal = __ballot_sync(0xffffffffu, l);
                if (l) sh.lcol[r + __popc(bal & ((1u << lane) - 1u))] = (unsigned short)j;
                r += __popc(bal);
            }
            if (lane == 0) {
                sh.nlive = r;
                sh.job = 0;
                sh.live[q0] = 0;
                if (two) sh.live[q1] = 0;
            }
        } else {
            for (int k = tid - 64; k < p; k += kT - 64) {
                const double x = ahead ? (two ? sh.ct[k] : sh.cc[k]) : __ldcg(W + (size_t)q0 * p + k);
                sh.b0[k] = x;
                if (!two) {
                    sh.s0[k] = x * dv.i0;
                } else {
                    const double y = ahead ? sh.cc[k] : __ldcg(W + (size_t)q1 * p + k);
                    sh.b1[k] = y;
                    sh.s0[k] = dv.i0 * x + dv.i1 * y;
                    sh.s1[k] = dv.i1 * x + dv.i2 * y;
                }
            }
        }
        __syncthreads();
        // ---------------- update: the own elements of W11 and their mirrors (the pivot
        // columns are frozen), then the own rows of A21
        if (warp > 0) {
#pragma unroll
            for (int j = 0; j < kOwn; j++)
                if (oki[j] >= 0) {
                    const int k = oki[j] >> 16, i = oki[j] & 0xffff;
                    if (sh.live[k] && sh.live[i]) {
                        own[j] = fma(-sh.b0[i], sh.s0[k], own[j]);
                        if (two) own[j] = fma(-sh.b1[i], sh.s1[k], own[j]);
                        Wn[k * p + i] = Wn[i * p + k] = own[j];
                    } else {
                        if (k == q0 || k == q1) fin[k * p + i] = own[j];
                        if (i == q0 || i == q1) fin[i * p + k] = own[j];
                    }
                }
            // warp 1's fence for the record that it will publish
            __syncwarp();
            asm volatile("bar.sync 1, %0;" ::"n"(kOwners) : "memory");
            if (warp == 1) fence_gpu();
        }
        if (warp == 0) {
            // the candidate's column, its partner's and their maxima on A11 after this pivot,
            // by the very operations of their owners
            const int c = sh.next;
            if (c >= 0) {
                unsigned long long km[NE];
                bool lv[NE];
                auto after = [&](int k, double x, int i) {
                    const int r = i > k ? i : k, s = i > k ? k : i;
                    x = fma(-sh.b0[r], sh.s0[s], x);
                    return two ? fma(-sh.b1[r], sh.s1[s], x) : x;
                };
#pragma unroll
                for (int q = 0; q < NE; q++) {
                    const int i = lane + 32 * q;
                    lv[q] = i < p && sh.live[i];
                    km[q] = 0;
                    if (__any_sync(0xffffffffu, lv[q])) {
                        const double x = after(c, cv[q], lv[q] ? i : c);
                        if (lv[q]) sh.cc[i] = x;
                        km[q] = akey(x);
                    }
                }
                const int t = partner(c, km, lv);
                double tv[NE];
#pragma unroll
                for (int q = 0; q < NE; q++) tv[q] = t >= 0 && lv[q] ? __ldcg(W + (size_t)t * p + lane + 32 * q) : 0.0;
                const unsigned long long vm = rest_max(c, t, km, lv);
                unsigned long long vt = 0;
                if (t >= 0) {
#pragma unroll
                    for (int q = 0; q < NE; q++) {
                        const int i = lane + 32 * q;
                        if (lv[q]) sh.ct[i] = tv[q] = after(t, tv[q], i);
                        km[q] = akey(tv[q]);
                    }
                    vt = rest_max(c, t, km, lv);
                }
                __syncwarp();
                if (lane == 0) {
                    sh.partner = t;
                    sh.amm = sh.cc[c];
                    sh.atm = t >= 0 ? sh.cc[t] : 0.0;
                    sh.att = t >= 0 ? sh.ct[t] : 0.0;
                    sh.vm = vm;
                    sh.vt = vt;
                }
            }
        } else if (kSmem) {
            if (two)
                update_cols<true>(T, ldt, (int)rows, q0, q1, sh, warp - 1, kNW - 1);
            else
                update_cols<false>(T, ldt, (int)rows, q0, q0, sh, warp - 1, kNW - 1);
        }
        if (!kSmem) {
            if (two)
                update_rows<true>(T, ldt, rows, q0, q1, sh);
            else
                update_rows<false>(T, ldt, rows, q0, q0, sh);
        }
        nelim += two ? 2 : 1;
        round++;
        // the next decision
        c0 = from = dv.m + 1;
        accepted = 1;
        if (ahead) win = 1;
        __syncthreads();
    }
    if (!ok) {
        if (blockIdx.x == 0 && tid == 0) atomicCAS(a.info, kInfoOk, (int32_t)CTP_ETIMEOUT);
        return;
    }

    // ---- the final order: accepted pivots, then the delayed columns in original order
    if (tid == 0) {
        int k = nelim;
        for (int c = 0; c < p; c++)
            if (sh.live[c]) {
                sh.order[k] = c;
                sh.kind[k] = CTP_PIVKIND_DELAYED;
                sh.sD[2 * k] = sh.sD[2 * k + 1] = 0.0;
                sh.sInv[2 * k] = sh.sInv[2 * k + 1] = 0.0;
                k++;
            }
    }
    __syncthreads();
    for (int k = tid; k < p; k += kT) sh.pos_of[sh.order[k]] = k;
    if (blockIdx.x == 0) {
        for (int k = tid; k < p; k += kT) {
            a.perm[k] = sh.order[k];
            a.piv[k] = sh.kind[k];
            a.D[2 * k] = sh.sD[2 * k];
            a.D[2 * k + 1] = sh.sD[2 * k + 1];
            a.Dinv[2 * k] = sh.sInv[2 * k];
            a.Dinv[2 * k + 1] = sh.sInv[2 * k + 1];
        }
        if (tid == 0) *a.nelim = nelim;
    }
    __syncthreads();

    // ---- output: A21 in pivot order, the pivots' columns times D^-1 (zero
    // pivots give zero columns)
    auto l21_entry = [&](const double *t, int64_t ld, int pos, int64_t r) -> double {
        const int kd = sh.kind[pos];
        const double x = t[sh.order[pos] * ld + r];
        if (kd == CTP_PIVKIND_1X1) return x * sh.sInv[2 * pos];
        if (kd == CTP_PIVKIND_2X2_FIRST)
            return x * sh.sInv[2 * pos] + t[sh.order[pos + 1] * ld + r] * sh.sInv[2 * pos + 1];
        if (kd == CTP_PIVKIND_2X2_SECOND)
            return t[sh.order[pos - 1] * ld + r] * sh.sInv[2 * pos - 1] + x * sh.sInv[2 * pos];
        return kd == CTP_PIVKIND_ZERO ? 0.0 : x;
    };
    if (kSmem) {
        for (int pos = warp; pos < p; pos += kNW)
            for (int64_t r = lane; r < rows; r += 32)
                a.A[(int64_t)pos * lda + p + row0 + r] = l21_entry(T, ldt, pos, r);
    } else {
        for (int64_t t0 = 0; t0 < rows; t0 += 32) {
            const int64_t r = t0 + lane;
            for (int k = warp; k < p; k += kNW) dsm[k * 33 + lane] = r < rows ? T[k * lda + r] : 0.0;
            __syncthreads();
            if (r < rows)
                for (int pos = warp; pos < p; pos += kNW) T[pos * lda + r] = l21_entry(dsm, 33, pos, lane);
            __syncthreads();
        }
    }
    // the A11 block from W11: frozen pivot columns, delayed Schur block
    const double *Wd = a.W11 + (size_t)(round & 1) * pp;
    for (int c = blockIdx.x; c < p; c += gridDim.x) {
        const int pos = sh.pos_of[c], kd = sh.kind[pos];
        double *out = a.A + (int64_t)pos * lda;
        for (int i = tid; i < p; i += kT) {
            const int pi = sh.pos_of[i];
            if (kd == CTP_PIVKIND_DELAYED) {
                if (pi >= pos) out[pi] = __ldcg(Wd + (size_t)c * p + i);
            } else if (kd == CTP_PIVKIND_ZERO) {
                if (pi >= pos) out[pi] = 0.0;
            } else {
                const bool first = kd == CTP_PIVKIND_2X2_FIRST;
                if (pi > (first ? pos + 1 : pos)) out[pi] = l21_entry(fin, p, pos, i);
                if (pi == pos) out[pi] = sh.sD[2 * pos];
                if (first && pi == pos + 1) out[pi] = sh.sD[2 * pos + 1];
            }
        }
    }
}

}  // namespace

// workspace: control word and exchange records, the maxima (both cleared per launch), W11
constexpr size_t kRecOff = 256, kMaxOff = kRecOff + 2 * kMaxCtas * sizeof(ulonglong2);

static size_t w11_off(int p) { return kMaxOff + align256(3 * sizeof(unsigned long long) * (size_t)p); }

size_t tpp_ws_bytes(int p) { return w11_off(p) + align256(3 * sizeof(double) * (size_t)p * p); }

cudaError_t launch_tpp(double *A, int64_t n, int p, int64_t lda, double u, double small, void *ws,
                       int32_t *perm, int32_t *piv, double *D, double *Dinv, int32_t *nelim,
                       int32_t *info, int num_sms, int spin, cudaStream_t st) {
    char *w = static_cast<char *>(ws);
    TppArgs a;
    a.spin = spin > 0 ? (long)spin : kBarSpin;
    a.A = A;
    a.lda = lda;
    a.n = n;
    a.p = p;
    a.u = u;
    a.small = small;
    a.ctl = reinterpret_cast<Ctl *>(w);
    a.rec = reinterpret_cast<ulonglong2 *>(w + kRecOff);
    a.M21 = reinterpret_cast<unsigned long long *>(w + kMaxOff);
    a.W11 = reinterpret_cast<double *>(w + w11_off(p));
    a.perm = perm;
    a.piv = piv;
    a.nelim = nelim;
    a.D = D;
    a.Dinv = Dinv;
    a.info = info;
    cudaError_t err = cudaMemsetAsync(w, 0, w11_off(p), st);
    if (err != cudaSuccess) return err;
    // CTAs: 32 rows of A21 each (a warp's width) until the SMs run out -- fewer
    // CTAs make the exchange cheaper -- and no more than two elements of W11 per thread
    const int64_t m = n - p, tri = (int64_t)((p + 1) / 2) * (p + 1);
    int64_t G = (m + 31) / 32;
    const int64_t gw = (tri + 2 * kOwners - 1) / (2 * kOwners);
    if (G < gw) G = gw;
    if (G > num_sms) G = num_sms;
    if (G > kMaxCtas) G = kMaxCtas;
    const int64_t own = (tri + G * kOwners - 1) / (G * kOwners);
    if (own > 8) return cudaErrorLaunchOutOfResources;  // fewer than nine SMs
    a.rows = (m + G - 1) / G;
    const size_t tile = sizeof(double) * (size_t)p * (size_t)(a.rows | 1);
    const bool in_smem = tile <= kTileBytes;
    const size_t smem = in_smem ? tile : sizeof(double) * (size_t)p * 33;
    const int o = own <= 1 ? 0 : own <= 2 ? 1 : 2;
    static const void *const fns[2][3] = {
        {(const void *)k_tpp<false, 1>, (const void *)k_tpp<false, 2>, (const void *)k_tpp<false, 8>},
        {(const void *)k_tpp<true, 1>, (const void *)k_tpp<true, 2>, (const void *)k_tpp<true, 8>}};
    const void *fn = fns[in_smem][o];
    err = smem_at_least(fn, smem);
    if (err != cudaSuccess) return err;
    void *args[] = {&a};
    return cudaLaunchCooperativeKernel(fn, dim3((unsigned)G), dim3(kT), args, smem, st);
}

}  // namespace ctp
