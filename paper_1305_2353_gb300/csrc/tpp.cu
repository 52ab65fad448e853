// tpp.cu -- K4: threshold partial pivoting on the whole supernode (Listing 1,
// Section 2), i.e. without compression: every test takes its column maxima over
// all n rows, which must be up to date.  This is the comparator of the
// compressed path, and the pivoting of a chain's or a root's last resort.
//
// GB300 design.  One cooperative, persistent launch (one CTA of 16 warps per SM
// at most, all co-resident).  The rows of A21 are dealt out in contiguous runs,
// one per CTA, held in shared memory when they fit (n p up to about 3.6 million
// entries on 152 SMs) and streamed from memory otherwise; the elements of W11,
// a full symmetric copy of A11, are dealt out one by one, each owned by one
// thread, which keeps it in a register.  Per accepted pivot:
//   barrier  one software grid barrier, its spin bounded;
//   decide   every CTA runs the tests of Listing 1 itself, on W11 and the
//            column maxima of the trailing A21 (integer keys of |a|) in L2:
//            the inputs are the same, so is the outcome, and nothing has to be
//            sent back (a decision by one CTA costs a second barrier per
//            pivot).  Rejected candidates change nothing, so a window of up to
//            16 candidates (one warp each) is tested per step; the window is one
//            candidate after an acceptance and grows fourfold while all fail;
//   update   every CTA applies the pivot to its rows of A21 (a warp per column,
//            which leaves the column's new maximum in the warp: one atomicMax
//            per column and CTA) and to its elements of W11, written to the other
//            of two W11 buffers, since slower CTAs may still be reading this
//            one; maxima are triple-buffered for the same reason.
// What bounds a pivot at moderate n is latency: the barrier (an atomic and a poll
// in L2), two dependent L2 reads of the tests and their FP64 chain; at large n
// the pass over the trailing A21, the traffic that the paper's compressed
// pivoting avoids (Section 6).  The column loop keeps four loads per lane in
// flight.  Measured: 11.3 us per pivot at n = 20011, p = 127 (FP64 work 2 us) and
// 9.1 us in the 256-wide panels of a dense system of order 1999; with one CTA
// deciding, and a warp per 128 rows going through the columns one load at a
// time, it was 62 and 105 us.
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
constexpr int kOwn = 8;              // elements of W11 a thread owns at most
constexpr long kBarSpin = 1L << 22;  // default polls (an L2 round trip each): about two seconds
constexpr size_t kTileBytes = 200 * 1024;  // shared memory for a CTA's rows of A21

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
    int order[kMaxP], kind[kMaxP], pos_of[kMaxP];
    unsigned char live[kMaxP];
    unsigned short lcol[kMaxP];  // the live columns after the pivot at hand
    int nlive, ok;
};

// Software grid barrier for a cooperative launch (arrivals are counted up, never
// reset: the epoch's target is epoch * CTAs); false on timeout (more than
// `spin` polls) or when another CTA gave up.
__device__ __forceinline__ bool grid_sync(Ctl *ctl, unsigned target, int *s_ok, long spin) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
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
        __threadfence();
        *s_ok = ok && (*(volatile int *)&ctl->abort == 0);
    }
    __syncthreads();
    return *s_ok != 0;
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
    Decision d;
    d.kind = DEC_REJECT;
    d.t = -1;
    d.m = c;
    d.pad = 0;
    d.d0 = d.d1 = d.d2 = d.i0 = d.i1 = d.i2 = 0.0;
    unsigned long long km[NE];
    bool lv[NE];
#pragma unroll
    for (int q = 0; q < NE; q++) {
        const int i = lane + 32 * q;
        lv[q] = i < p && live[i];
        km[q] = i < p ? akey(__ldcg(cm + i)) : 0ull;
    }
    const double amm = __ldcg(cm + c);
    const unsigned long long mc = __ldcg(M + c);
    // partner t: largest |a(c, j)| over live j < c, lowest j on ties
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
    const int t = t0 == 0x7fffffff ? -1 : t0;
    unsigned long long vt = 0, ktm = 0;
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
#pragma unroll
        for (int q = 0; q < NE; q++) {
            const int i = lane + 32 * q;
            if (lv[q] && i != t && i != c) vt = kt[q] > vt ? kt[q] : vt;
        }
        vt = warp_max_key(vt);
        vt = vt > mt ? vt : mt;
        ktm = akey(atm);
    }
    unsigned long long vm = 0;
#pragma unroll
    for (int q = 0; q < NE; q++) {
        const int i = lane + 32 * q;
        if (lv[q] && i != t && i != c) vm = km[q] > vm ? km[q] : vm;
    }
    vm = warp_max_key(vm);
    vm = vm > mc ? vm : mc;
    const unsigned long long kmm = akey(amm);
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
    const int f1 = test_1x1_f32(kmm, maxm1, u);
    if (f1 == 1 || (f1 < 0 && kmm >= akey(__dmul_rn(u, key_val(maxm1))))) {
        d.kind = DEC_1X1;
        d.d0 = amm;
        d.i0 = __drcp_rn(amm);
    }
    return d;
}

// A pivot's update of this CTA's rows of A21: column k of the live list, entry
// r: a(r,k) - x0(r) s0(k) - x1(r) s1(k), one fused multiply-add per term, with
// x the pivot column(s) and s = D^-1 times the pivot row(s); the new maximum of
// the column goes to Mn[k].
template <bool k2x2>
__device__ __forceinline__ void update_rows(double *T, int64_t ldt, int64_t rows, int q0, int q1, const Shared &sh,
                                            unsigned long long *Mn) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const double *x0 = T + q0 * ldt, *x1 = k2x2 ? T + q1 * ldt : x0;
    for (int ci = warp; ci < sh.nlive; ci += kNW) {
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
        if (lane == 0 && mx) atomicMax(Mn + k, mx);
    }
}

template <bool kSmem>
__global__ void __launch_bounds__(kT, 1) k_tpp(TppArgs a) {
    extern __shared__ __align__(16) double dsm[];  // kSmem: the CTA's rows [p][rows]; else staging [p][33]
    __shared__ Shared sh;
    const int p = a.p;
    const int64_t n = a.n, m = n - p, lda = a.lda;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    Ctl *ctl = a.ctl;
    const int64_t row0 = min((int64_t)blockIdx.x * a.rows, m), rows = min(a.rows, m - row0);
    double *T = kSmem ? dsm : a.A + p + row0;
    const int64_t ldt = kSmem ? a.rows : lda;
    const int pp = p * p;
    double *fin = a.W11 + 2 * (size_t)pp;

    // ---- this thread's elements of W11 (full symmetric), this CTA's rows of A21
    // and their initial column maxima
    const int e0 = (int)blockIdx.x * kT + tid, estep = (int)gridDim.x * kT;
    double own[kOwn];
#pragma unroll
    for (int j = 0; j < kOwn; j++) {
        const int idx = e0 + j * estep;
        own[j] = 0.0;
        if (idx < pp) {
            const int k = idx / p, i = idx - k * p;
            own[j] = i >= k ? a.A[(int64_t)k * lda + i] : a.A[(int64_t)i * lda + k];
            a.W11[idx] = own[j];
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
        if (lane == 0 && mx) atomicMax(a.M21 + k, mx);
    }
    if (nonfinite) atomicCAS(a.info, kInfoOk, (int32_t)CTP_ENONFINITE);
    for (int i = tid; i < p; i += kT) sh.live[i] = 1;

    const double u = a.u, rcp_u = __drcp_rn(a.u);
    const unsigned long long small_k = akey(a.small);
    int nelim = 0, c0 = p >= 2 ? 1 : 0, accepted = 0, win = 1, from = c0;
    unsigned round = 0;
    bool ok;
    while ((ok = grid_sync(ctl, (round + 1) * gridDim.x, &sh.ok, a.spin))) {
        const double *W = a.W11 + (size_t)(round & 1) * pp;
        double *Wn = a.W11 + (size_t)((round & 1) ^ 1) * pp;
        const unsigned long long *M = a.M21 + (round % 3) * p;
        unsigned long long *Mn = a.M21 + ((round + 1) % 3) * p;
        // ---------------- decide: the same steps and outcome in every CTA
        bool stop = false;
        Decision dv;
        for (;;) {
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
            const int gap = dv.m - from;
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
        if (warp == 0) {
            int r = 0;
            for (int j0 = 0; j0 < p; j0 += 32) {
                const int j = j0 + lane;
                const bool l = j < p && sh.live[j] && j != q0 && j != q1;
                const unsigned bal = __ballot_sync(0xffffffffu, l);
                if (l) sh.lcol[r + __popc(bal & ((1u << lane) - 1u))] = (unsigned short)j;
                if (j < p) sh.live[j] = l;
                r += __popc(bal);
            }
            if (lane == 0) sh.nlive = r;
        } else {
            for (int k = tid - 32; k < p; k += kT - 32) {
                const double x = __ldcg(W + (size_t)q0 * p + k);
                sh.b0[k] = x;
                if (!two) {
                    sh.s0[k] = x * dv.i0;
                } else {
                    const double y = __ldcg(W + (size_t)q1 * p + k);
                    sh.b1[k] = y;
                    sh.s0[k] = dv.i0 * x + dv.i1 * y;
                    sh.s1[k] = dv.i1 * x + dv.i2 * y;
                }
            }
        }
        if (blockIdx.x == 0)  // read last in the decision before this one
            for (int k = tid; k < p; k += kT) a.M21[((round + 2) % 3) * p + k] = 0;
        __syncthreads();
        // ---------------- update: the own elements of W11 (an entry above the
        // diagonal takes its mirror's operands, so W11 stays exactly symmetric;
        // the pivot columns are frozen), then the own rows of A21
#pragma unroll
        for (int j = 0; j < kOwn; j++) {
            const int idx = e0 + j * estep;
            if (idx < pp) {
                const int k = idx / p, i = idx - k * p;
                if (k == q0 || k == q1) {
                    fin[idx] = own[j];
                } else if (sh.live[k] && sh.live[i]) {
                    const int r = i > k ? i : k, c = i > k ? k : i;
                    own[j] = fma(-sh.b0[r], sh.s0[c], own[j]);
                    if (two) own[j] = fma(-sh.b1[r], sh.s1[c], own[j]);
                    Wn[idx] = own[j];
                }
            }
        }
        if (two)
            update_rows<true>(T, ldt, rows, q0, q1, sh, Mn);
        else
            update_rows<false>(T, ldt, rows, q0, q0, sh, Mn);
        nelim += two ? 2 : 1;
        round++;
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

size_t tpp_ws_bytes(int p) {
    return 256 + align256(3 * sizeof(double) * (size_t)p * p) + align256(3 * sizeof(unsigned long long) * (size_t)p);
}

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
    a.W11 = reinterpret_cast<double *>(w + 256);
    a.M21 = reinterpret_cast<unsigned long long *>(w + 256 + align256(3 * sizeof(double) * (size_t)p * p));
    a.perm = perm;
    a.piv = piv;
    a.nelim = nelim;
    a.D = D;
    a.Dinv = Dinv;
    a.info = info;
    cudaError_t err = cudaMemsetAsync(w, 0, 256, st);
    if (err != cudaSuccess) return err;
    err = cudaMemsetAsync(a.M21, 0, 3 * sizeof(unsigned long long) * (size_t)p, st);
    if (err != cudaSuccess) return err;
    // CTAs: 32 rows of A21 each (a warp's width) until the SMs run out -- fewer
    // CTAs make the barrier cheaper -- and no more than four elements of W11 per thread
    const int64_t m = n - p;
    int64_t G = (m + 31) / 32;
    const int64_t gw = ((int64_t)p * p + 4 * kT - 1) / (4 * kT);
    if (G < gw) G = gw;
    if (G > num_sms) G = num_sms;
    if (G * kT * kOwn < (int64_t)p * p) return cudaErrorLaunchOutOfResources;  // fewer than 16 SMs
    a.rows = (m + G - 1) / G;
    const size_t tile = sizeof(double) * (size_t)p * (size_t)a.rows;
    const bool in_smem = tile <= kTileBytes;
    const size_t smem = in_smem ? (tile > 0 ? tile : 16) : sizeof(double) * (size_t)p * 33;
    const void *fn = in_smem ? (const void *)k_tpp<true> : (const void *)k_tpp<false>;
    err = smem_at_least(fn, smem);
    if (err != cudaSuccess) return err;
    void *args[] = {&a};
    return cudaLaunchCooperativeKernel(fn, dim3((unsigned)G), dim3(kT), args, smem, st);
}

}  // namespace ctp
