// solve_plan.cu -- the solve with a multifrontal factorization and the residual
// helpers of iterative refinement (declared in solve_plan.cuh).
//
// The solve is the front-by-front substitution of system.cu (eq. (1.2) applied
// front by front), on groups of at most 64 consecutive pivots of a front: with
// group rows [L11; L21],
//   forward   y = L11^{-1} b,  b_rest -= L21 y;
//   diagonal  z = D^{-1} y, all pivots at once;
//   backward  x = L11^{-T} (z - L21^T x_rest).
// Groups of a level are independent; a level is one launch per sweep over items
// (group, up to four chunks of 32 rows below its pivots; fewer chunks where a level
// would leave SMs idle) by right-hand sides (as many per item as fill the
// chip: 16 share an item's triangular solve where items abound, down to 4):
//   forward   every item solves the group's small triangular system itself
//             (nothing is exchanged between CTAs) and subtracts its rows' share
//             with atomics; the group's first item stores y;
//   backward  every item subtracts its rows' L21^T x_rest from z with atomics;
//             the group's last item to finish (a fenced counter, no waiting)
//             solves with L11^T.
// What bounds a level is latency: consecutive groups of a front depend on each
// other, and the large fronts' groups are the whole level.  So an item's factor
// entries (two contiguous blocks) are copied to shared memory before the kernel
// waits for the level before it (programmatic dependent launch), the
// triangular solves keep a right-hand side in a warp's registers (a shuffle and a
// multiply-add per pivot, no shared-memory round trip), and the right-hand sides
// are held row by row in elimination order, so that gathers and atomics touch
// runs of memory.  One solve on a
// 64^3 grid with 16 right-hand sides: FP64 19 ms, FP32 3.4 ms (40 and 20 ms with a
// launch per panel, 973 of them instead of about 300, and the triangular solves
// in shared memory); on 48^3 with one right-hand side 2.0 ms (5.7).
// The sweeps compute in FP64, or in FP32 (the packed factors and z in FP32, the
// right-hand sides accumulated in FP64): the
// correction solves of a refinement whose residuals are FP64 (Section 7) need
// only to contract the error, and GB300's FP32 pipe is many times its FP64 one.
#include <algorithm>

#include "solve_plan.cuh"

namespace ctp {

namespace {

constexpr int kLT = 256;        // threads per item
constexpr int kRC = 32;         // rows of a chunk
constexpr int kMC = 4;          // chunks per item at most
constexpr int kLE = 64;         // pivots per group at most
constexpr int kLC = kRC + 1;    // padded length of a column of a chunk
constexpr int kWide = 76;       // items a level wants (half the SMs)

// A group.  Packed blocks: L11 column by column, le = e | 1 apart (zero on and
// above the diagonal and in the D slots of 2x2 pivots); L21 in chunks, each e
// columns of kLC.  Every block starts at a multiple of 4 elements.
struct Grp {
    int64_t l11, l21;  // element offsets in the pack
    int64_t voff;      // vars: e pivot positions, then the nr rows below (elimination order)
    int64_t zoff;      // first pivot
    int64_t nr;
    int32_t e, items;  // items: how many share it
    int32_t k0, k1;    // its panels
    int64_t c0;        // first pivot, counted within the front
};
__host__ __device__ inline int64_t up4(int64_t x) { return (x + 3) & ~int64_t(3); }
__host__ __device__ inline int64_t l11_elems(int e) { return up4((int64_t)e * (e | 1)); }
__host__ __device__ inline int64_t chunk_elems(int e) { return up4((int64_t)e * kLC); }

// A panel, for packing.
struct Pnl {
    ctp_sfront f;
    int64_t E;     // pivots of the front before it
    int64_t ioff;  // its inverse permutation in the scratch array
    int64_t zoff;  // its first pivot
    int32_t e, pad;
};
// The part of a panel that belongs to one group: columns q0..q1-1.
struct Seg {
    int32_t panel, q0, q1, grp;
};

// Position in the front of the variable in row r of panel k's factor, after panel k1:
// every later panel permutes its own fully-summed rows, while the rows of
// L21 stay where they are.
__device__ __forceinline__ int64_t front_row(const Pnl *P, const int32_t *invp, int k, int64_t r, int k1) {
    while (r >= P[k].e && k < k1) {
        r -= P[k].e;
        k++;
        if (r < P[k].f.p) r = invp[P[k].ioff + r];
    }
    return P[k].E + r;
}

// inverse permutations of the panels, and their pivot kinds and D in pivot order
__global__ void k_lv_panels(const Pnl *__restrict__ P, int32_t *invp, int32_t *kind, double *D) {
    const Pnl x = P[blockIdx.x];
    for (int q = threadIdx.x; q < x.f.p; q += blockDim.x) invp[x.ioff + x.f.perm[q]] = q;
    for (int q = threadIdx.x; q < x.e; q += blockDim.x) {
        kind[x.zoff + q] = x.f.piv[q];
        D[2 * (x.zoff + q)] = x.f.D[2 * q];
        D[2 * (x.zoff + q) + 1] = x.f.D[2 * q + 1];
    }
}

// positions (in elimination order) of a group's pivots and rows below
__global__ void k_lv_vars(const Pnl *__restrict__ P, const Grp *__restrict__ G, const int32_t *__restrict__ inv,
                          int32_t *vars) {
    const Grp g = G[blockIdx.x];
    const int64_t total = g.e + g.nr;
    for (int64_t i = threadIdx.x + (int64_t)blockIdx.y * blockDim.x; i < total; i += (int64_t)gridDim.y * blockDim.x) {
        const int64_t c = g.c0 + i;
        int k = g.k1;
        if (i < g.e)
            for (k = g.k0; c >= P[k].E + P[k].e;) k++;
        const ctp_sfront &f = P[k].f;
        const int64_t r = c - P[k].E;
        vars[g.voff + i] = inv[r < f.p ? f.rows[f.perm[r]] : f.rows[r]];
    }
}

// copy one segment's columns, 256 rows per CTA, into its group's blocks
template <typename T>
__global__ void __launch_bounds__(256) k_lv_pack(const Pnl *__restrict__ P, const Grp *__restrict__ G,
                                                 const Seg *__restrict__ S, const int2 *__restrict__ items,
                                                 const int32_t *__restrict__ invp, T *__restrict__ pack) {
    const int2 it = items[blockIdx.x];
    const Seg s = S[it.x];
    const Grp g = G[s.grp];
    const Pnl &x = P[s.panel];
    const int64_t r = (int64_t)it.y * 256 + threadIdx.x;
    if (r >= x.f.n || r <= s.q0) return;
    const int64_t row = front_row(P, invp, s.panel, r, g.k1) - g.c0;  // within the group's rows
    const int64_t i = row - g.e;                                      // row below the pivots
    const int le = g.e | 1;
    T *dst = i < 0 ? pack + g.l11 + row : pack + g.l21 + (i / kRC) * chunk_elems(g.e) + i % kRC;
    const int64_t ld = i < 0 ? le : kLC;
    const int c = (int)(x.E - g.c0);  // group column of the panel's column 0
    for (int q = s.q0; q < s.q1; q++) {
        if (r <= q || (r == q + 1 && x.f.piv[q] == CTP_PIVKIND_2X2_FIRST)) continue;
        dst[(int64_t)(c + q) * ld] = (T)x.f.L[(int64_t)q * x.f.ldl + r];
    }
}

// X in elimination order, row by row: Xp[i][r] = X(perm[i], r), and back
template <bool kBack>
__global__ void __launch_bounds__(kLT) k_lv_reorder(int64_t N, int nrhs, const int32_t *__restrict__ perm,
                                                    double *X, int64_t ldx, double *Xp) {
    for (int64_t i = (int64_t)blockIdx.x * kLT + threadIdx.x; i < N; i += (int64_t)gridDim.x * kLT) {
        const int64_t v = perm[i];
        for (int r = 0; r < nrhs; r++) {
            if (kBack)
                X[r * ldx + v] = Xp[i * nrhs + r];
            else
                Xp[i * nrhs + r] = X[r * ldx + v];
        }
    }
}

// z = D^{-1} y in place: 1x1, 2x2 (by its first pivot), zero pivot -> 0
template <typename T>
__global__ void __launch_bounds__(kLT) k_lv_dsolve(int64_t npiv, int nrhs, const int32_t *__restrict__ kind,
                                                   const double *__restrict__ D, T *Z) {
    const int64_t n = npiv * nrhs;
    for (int64_t x = (int64_t)blockIdx.x * kLT + threadIdx.x; x < n; x += (int64_t)gridDim.x * kLT) {
        const int64_t q = x / nrhs;
        const int k = kind[q];
        if (k == CTP_PIVKIND_1X1) {
            Z[x] = Z[x] / (T)D[2 * q];
        } else if (k == CTP_PIVKIND_2X2_FIRST) {
            const T d11 = (T)D[2 * q], d21 = (T)D[2 * q + 1], d22 = (T)D[2 * q + 2];
            const T det = d11 * d22 - d21 * d21, y0 = Z[x], y1 = Z[x + nrhs];
            Z[x] = (d22 * y0 - d21 * y1) / det;
            Z[x + nrhs] = (d11 * y1 - d21 * y0) / det;
        } else if (k == CTP_PIVKIND_ZERO) {
            Z[x] = T(0);
        }
    }
}

// Programmatic dependent launch: a level's kernel loads what no earlier kernel of
// the sweeps writes (descriptors, factor blocks) while the previous level runs,
// then waits for it before touching Xp and Z.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// n elements (a multiple of 4) from global to shared memory, asynchronously
template <typename T>
__device__ __forceinline__ void copy_async(T *dst, const T *src, int n) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    const int n16 = n * (int)sizeof(T) / 16;
    for (int i = threadIdx.x; i < n16; i += kLT)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + 16 * i), "l"((const char *)src + 16 * i)
                     : "memory");
}
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <typename T, int RG>
struct LvShape {
    static constexpr int RPW = RG >= 8 ? RG / 8 : 1;  // right-hand sides per warp of the triangular solves
    static constexpr int RS = RG >= 2 ? 2 : 1;        // forward: two thread groups share the right-hand sides
                                                      // of a row (the others its columns)
    static constexpr int BS = RG >= 4 ? 4 : RG;       // backward: quarters share the right-hand sides,
    static constexpr int BC = 4 / BS;                 //   and the rows
    // elements: L11, chunks, then b / z [kLE][RG], x of the chunks [kMC kRC][RG] (backward), sums
    static __host__ __device__ int64_t vec() { return kLE * RG + kMC * kRC * RG + kLT / RS * RG; }
    static size_t smem(int emax) { return sizeof(T) * (size_t)(l11_elems(emax) + kMC * chunk_elems(emax) + vec()); }
};

// An item's chunks of its group: first chunk and their number.
__device__ __forceinline__ int item_chunk(const int2 &it) { return it.y >> 3; }
__device__ __forceinline__ int item_count(const int2 &it) { return it.y & 7; }

// y <- L11^{-1} y for the right-hand sides of ys ([e][RG]): warp w takes RPW of them,
// lane i holds rows i and i + 32
template <typename T, int RG>
__device__ __forceinline__ void tri_forward(const T *Ls, T *ys, int e) {
    constexpr int RPW = LvShape<T, RG>::RPW;
    const int r0 = (threadIdx.x >> 5) * RPW, lane = threadIdx.x & 31, le = e | 1;
    if (r0 >= RG) return;
    T y0[RPW], y1[RPW];
#pragma unroll
    for (int t = 0; t < RPW; t++) {
        y0[t] = lane < e ? ys[lane * RG + r0 + t] : T(0);
        y1[t] = lane + 32 < e ? ys[(lane + 32) * RG + r0 + t] : T(0);
    }
    const int ea = e < 32 ? e : 32;
#pragma unroll 4
    for (int j = 0; j < ea; j++) {
        const T l0 = (lane > j && lane < e) ? Ls[j * le + lane] : T(0);
        const T l1 = lane + 32 < e ? Ls[j * le + lane + 32] : T(0);
#pragma unroll
        for (int t = 0; t < RPW; t++) {
            const T yj = __shfl_sync(0xffffffffu, y0[t], j);
            if (lane > j) y0[t] -= l0 * yj;
            if (e > 32) y1[t] -= l1 * yj;
        }
    }
#pragma unroll 4
    for (int j = 32; j < e; j++) {
        const T l1 = (lane + 32 > j && lane + 32 < e) ? Ls[j * le + lane + 32] : T(0);
#pragma unroll
        for (int t = 0; t < RPW; t++) {
            const T yj = __shfl_sync(0xffffffffu, y1[t], j - 32);
            if (lane + 32 > j) y1[t] -= l1 * yj;
        }
    }
#pragma unroll
    for (int t = 0; t < RPW; t++) {
        if (lane < e) ys[lane * RG + r0 + t] = y0[t];
        if (lane + 32 < e) ys[(lane + 32) * RG + r0 + t] = y1[t];
    }
}

// x <- L11^{-T} x, likewise
template <typename T, int RG>
__device__ __forceinline__ void tri_backward(const T *Ls, T *xs, int e) {
    constexpr int RPW = LvShape<T, RG>::RPW;
    const int r0 = (threadIdx.x >> 5) * RPW, lane = threadIdx.x & 31, le = e | 1;
    if (r0 >= RG) return;
    T x0[RPW], x1[RPW];
#pragma unroll
    for (int t = 0; t < RPW; t++) {
        x0[t] = lane < e ? xs[lane * RG + r0 + t] : T(0);
        x1[t] = lane + 32 < e ? xs[(lane + 32) * RG + r0 + t] : T(0);
    }
#pragma unroll 4
    for (int i = e - 1; i >= 32; i--) {
        const T l0 = Ls[lane * le + i], l1 = lane + 32 < i ? Ls[(lane + 32) * le + i] : T(0);
#pragma unroll
        for (int t = 0; t < RPW; t++) {
            const T xi = __shfl_sync(0xffffffffu, x1[t], i - 32);
            x0[t] -= l0 * xi;
            if (lane + 32 < i) x1[t] -= l1 * xi;
        }
    }
#pragma unroll 4
    for (int i = (e < 32 ? e : 32) - 1; i > 0; i--) {
        const T l0 = lane < i ? Ls[lane * le + i] : T(0);
#pragma unroll
        for (int t = 0; t < RPW; t++) {
            const T xi = __shfl_sync(0xffffffffu, x0[t], i);
            if (lane < i) x0[t] -= l0 * xi;
        }
    }
#pragma unroll
    for (int t = 0; t < RPW; t++) {
        if (lane < e) xs[lane * RG + r0 + t] = x0[t];
        if (lane + 32 < e) xs[(lane + 32) * RG + r0 + t] = x1[t];
    }
}

// Right-hand sides g0 .. g0 + RG - 1 with g0 = RG blockIdx.y.
template <typename T, int RG>
__global__ void __launch_bounds__(kLT, 2) k_lv_forward(const Grp *__restrict__ G, const int2 *__restrict__ items,
                                                       const T *__restrict__ pack, const int32_t *__restrict__ vars,
                                                       int emax, double *Xp, int nrhs, T *__restrict__ Z) {
    using S = LvShape<T, RG>;
    extern __shared__ __align__(16) unsigned char lv_smem[];
    __shared__ int32_t spv[kLE], srv[kMC * kRC];
    T *Ls = reinterpret_cast<T *>(lv_smem), *Lc = Ls + l11_elems(emax), *ys = Lc + kMC * chunk_elems(emax);
    T *red = ys + kLE * RG;
    const int2 it = items[blockIdx.x];
    const Grp g = G[it.x];
    const int e = g.e, t = threadIdx.x, c0 = item_chunk(it), nc = item_count(it);
    const int ce = (int)chunk_elems(e), R = nc * kRC;
    const int nr = (int)min((int64_t)R, g.nr - (int64_t)c0 * kRC);
    copy_async(Ls, pack + g.l11, (int)l11_elems(e));
    copy_async(Lc, pack + g.l21 + (int64_t)c0 * ce, nc * ce);
    if (t < e) spv[t] = vars[g.voff + t];
    if (t < nr) srv[t] = vars[g.voff + e + (int64_t)c0 * kRC + t];
    pdl_trigger();
    copy_wait();
    __syncthreads();
    pdl_wait();
    const int g0 = blockIdx.y * RG, ng = min(RG, nrhs - g0);
    for (int idx = t; idx < e * RG; idx += kLT) {
        const int q = idx / RG, r = idx % RG;
        ys[idx] = r < ng ? (T)Xp[(int64_t)spv[q] * nrhs + g0 + r] : T(0);
    }
    __syncthreads();
    tri_forward<T, RG>(Ls, ys, e);
    __syncthreads();
    if (c0 == 0)
        for (int idx = t; idx < e * RG; idx += kLT) {
            const int q = idx / RG, r = idx % RG;
            if (r < ng) Z[(g.zoff + q) * nrhs + g0 + r] = ys[idx];
        }
    if (nr <= 0) return;
    // b_rest -= L21 y: thread (row, slice); a slice takes RT of the right-hand sides and
    // every CS-th column
    constexpr int RT = RG / S::RS;
    const int slices = kLT / R, CS = slices / S::RS, row = t % R, sl = t / R;
    const int hr = sl % S::RS, hc = sl / S::RS;
    T acc[RT];
#pragma unroll
    for (int r = 0; r < RT; r++) acc[r] = T(0);
    if (sl < slices) {
        const T *y = ys + hr * RT, *l = Lc + (row / kRC) * ce + row % kRC;
#pragma unroll 4
        for (int j = hc; j < e; j += CS) {
            const T lj = l[j * kLC];
#pragma unroll
            for (int r = 0; r < RT; r++) acc[r] += lj * y[j * RG + r];
        }
#pragma unroll
        for (int r = 0; r < RT; r++) red[(hc * R + row) * RG + hr * RT + r] = acc[r];
    }
    __syncthreads();
    for (int idx = t; idx < nr * RG; idx += kLT) {
        const int q = idx / RG, r = idx % RG;
        if (r >= ng) continue;
        T v = red[idx];
        for (int c = 1; c < CS; c++) v += red[c * R * RG + idx];
        atomicAdd(Xp + (int64_t)srv[q] * nrhs + g0 + r, -(double)v);
    }
}

template <typename T, int RG>
__global__ void __launch_bounds__(kLT, 2) k_lv_backward(const Grp *__restrict__ G, const int2 *__restrict__ items,
                                                        const T *__restrict__ pack, const int32_t *__restrict__ vars,
                                                        int emax, double *Xp, int nrhs, T *Z, int *cnt) {
    using S = LvShape<T, RG>;
    extern __shared__ __align__(16) unsigned char lv_smem[];
    __shared__ int32_t spv[kLE], srv[kMC * kRC];
    __shared__ int last;
    T *Ls = reinterpret_cast<T *>(lv_smem), *Lc = Ls + l11_elems(emax), *zs = Lc + kMC * chunk_elems(emax);
    T *xs = zs + kLE * RG, *red = xs + kMC * kRC * RG;
    const int2 it = items[blockIdx.x];
    const Grp g = G[it.x];
    const int e = g.e, t = threadIdx.x, c0 = item_chunk(it), nc = item_count(it);
    const int ce = (int)chunk_elems(e), R = nc * kRC;
    const int nr = (int)min((int64_t)R, g.nr - (int64_t)c0 * kRC);
    copy_async(Ls, pack + g.l11, (int)l11_elems(e));
    copy_async(Lc, pack + g.l21 + (int64_t)c0 * ce, nc * ce);
    if (t < e) spv[t] = vars[g.voff + t];
    if (t < nr) srv[t] = vars[g.voff + e + (int64_t)c0 * kRC + t];
    pdl_trigger();
    copy_wait();
    __syncthreads();
    pdl_wait();
    const int g0 = blockIdx.y * RG, ng = min(RG, nrhs - g0);
    const bool shared_z = g.items > 1;  // several items add into the group's z
    if (nr > 0) {
        for (int idx = t; idx < R * RG; idx += kLT) {
            const int q = idx / RG, r = idx % RG;
            xs[idx] = (q < nr && r < ng) ? (T)Xp[(int64_t)srv[q] * nrhs + g0 + r] : T(0);
        }
        __syncthreads();
        // z -= L21^T x_rest: thread (pivot, quarter); a quarter takes RT of the right-hand
        // sides and its share of the chunks' rows
        constexpr int RT = RG / S::BS;
        const int j = t & (kLE - 1), s = t / kLE, sr = s % S::BS, sc = s / S::BS;
        T acc[RT];
#pragma unroll
        for (int r = 0; r < RT; r++) acc[r] = T(0);
        if (j < e) {
            for (int c = 0; c < nc; c++) {
                const T *l = Lc + c * ce + j * kLC, *x = xs + c * kRC * RG + sr * RT;
#pragma unroll 8
                for (int q = sc * (kRC / S::BC); q < (sc + 1) * (kRC / S::BC); q++) {
                    const T lq = l[q];
#pragma unroll
                    for (int r = 0; r < RT; r++) acc[r] += lq * x[q * RG + r];
                }
            }
        }
#pragma unroll
        for (int r = 0; r < RT; r++) red[(sc * kLE + j) * RG + sr * RT + r] = acc[r];
        __syncthreads();
    }
    for (int idx = t; idx < e * RG; idx += kLT) {
        const int q = idx / RG, r = idx % RG;
        T v = T(0);
        if (nr > 0) {
#pragma unroll
            for (int c = 0; c < S::BC; c++) v += red[c * kLE * RG + idx];
        }
        T *z = Z + (g.zoff + q) * nrhs + g0 + r;
        if (!shared_z)
            zs[idx] = r < ng ? *z - v : T(0);
        else if (r < ng)
            atomicAdd(z, -v);
    }
    if (shared_z) {
        // the last item of the group to get here solves with L11^T
        __threadfence();
        __syncthreads();
        if (t == 0) last = atomicAdd(cnt + (int64_t)it.x * nrhs + blockIdx.y, 1) == g.items - 1;
        __syncthreads();
        if (!last) return;
        __threadfence();
        for (int idx = t; idx < e * RG; idx += kLT) {
            const int q = idx / RG, r = idx % RG;
            zs[idx] = r < ng ? __ldcg(Z + (g.zoff + q) * nrhs + g0 + r) : T(0);
        }
    }
    __syncthreads();
    tri_backward<T, RG>(Ls, zs, e);
    __syncthreads();
    for (int idx = t; idx < e * RG; idx += kLT) {
        const int q = idx / RG, r = idx % RG;
        if (r < ng) Xp[(int64_t)spv[q] * nrhs + g0 + r] = (double)zs[idx];
    }
}

struct Sweep {
    const Grp *G;
    const int2 *items;
    int64_t nitems;
    const int32_t *vars;
    int emax, nrhs;
    double *Xp;
    int *cnt;
};

template <typename T, int RG>
cudaError_t launch_level(bool forward, const Sweep &w, const T *pack, T *Z, cudaStream_t st) {
    if (w.nitems == 0) return cudaSuccess;
    const size_t smem = LvShape<T, RG>::smem(w.emax);
    const void *fn = forward ? (const void *)k_lv_forward<T, RG> : (const void *)k_lv_backward<T, RG>;
    cudaError_t e = smem_at_least(fn, smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)w.nitems, (unsigned)((w.nrhs + RG - 1) / RG));
    cfg.blockDim = dim3(kLT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr_pdl[1];
    attr_pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr_pdl[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr_pdl;
    cfg.numAttrs = 1;
    if (forward)
        return cudaLaunchKernelEx(&cfg, k_lv_forward<T, RG>, w.G, w.items, pack, w.vars, w.emax, w.Xp, w.nrhs, Z);
    return cudaLaunchKernelEx(&cfg, k_lv_backward<T, RG>, w.G, w.items, pack, w.vars, w.emax, w.Xp, w.nrhs, Z, w.cnt);
}

template <typename T>
cudaError_t launch_level_rg(bool forward, const Sweep &w, const T *pack, T *Z, cudaStream_t st) {
    if (w.nrhs <= 1) return launch_level<T, 1>(forward, w, pack, Z, st);
    if (w.nrhs <= 2) return launch_level<T, 2>(forward, w, pack, Z, st);
    // at least four to an item; more where that still leaves an item for every SM
    const int64_t want = 2 * kWide;
    if (w.nrhs <= 4 || w.nitems * ((w.nrhs + 7) / 8) < want) return launch_level<T, 4>(forward, w, pack, Z, st);
    if (w.nrhs <= 8 || w.nitems * ((w.nrhs + 15) / 16) < want) return launch_level<T, 8>(forward, w, pack, Z, st);
    return launch_level<T, 16>(forward, w, pack, Z, st);
}

}  // namespace

bool DevBuf::need(size_t bytes) {
    if (bytes <= cap) return true;
    release();
    if (cudaMalloc(&p, bytes) != cudaSuccess) {
        p = nullptr;
        return false;
    }
    cap = bytes;
    return true;
}
void DevBuf::release() {
    if (p) cudaFree(p);
    p = nullptr;
    cap = 0;
}

SolvePlan::~SolvePlan() {
    for (DevBuf *b : {&grp, &items, &vars, &perm, &pack64, &pack32, &kind, &D}) b->release();
}

ctp_status SolvePlan::build(const std::vector<ctp_sfront> &panels, const std::vector<int32_t> &nelim,
                            const std::vector<SolveChain> &fronts, const std::vector<int32_t> &perm_host,
                            const std::vector<int32_t> &inv_host, bool fp32, cudaStream_t st) {
    clear();
    N = (int64_t)perm_host.size();
    std::vector<Pnl> pn(panels.size());
    std::vector<Grp> gr;
    std::vector<Seg> seg;
    std::vector<int2> sitem;
    std::vector<int> glev, first(fronts.size(), 0);  // first: level of a front's first group
    int64_t z = 0, io = 0, vo = 0, po = 0, maxtotal = 1;
    for (size_t f = 0; f < fronts.size(); f++) {
        const SolveChain &c = fronts[f];
        int64_t E = 0;
        for (int64_t k = c.pa; k < c.pb; k++) {
            const ctp_sfront &s = panels[k];
            if (nelim[k] < 0 || nelim[k] > s.p || s.p > kMaxP || s.n < s.p) return CTP_EINVAL;
            pn[k] = {s, E, io, z + E, nelim[k], 0};
            io += s.p;
            E += nelim[k];
        }
        const int64_t nf = c.pb > c.pa ? panels[c.pa].n : 0;
        int lv = first[f];
        int64_t k = c.pa;
        for (int64_t c0 = 0; c0 < E; c0 += kLE) {
            const int64_t c1 = std::min<int64_t>(c0 + kLE, E);
            Grp g = {};
            g.e = (int32_t)(c1 - c0);
            g.nr = nf - c1;
            const int64_t nch = (g.nr + kRC - 1) / kRC;
            if (nch > (1 << 27)) return CTP_EINVAL;
            g.c0 = c0;
            g.zoff = z + c0;
            g.voff = vo;
            vo += g.e + g.nr;
            g.l11 = po;
            g.l21 = po + l11_elems(g.e);
            po = g.l21 + nch * chunk_elems(g.e);
            maxtotal = std::max(maxtotal, g.e + g.nr);
            while (pn[k].E + pn[k].e <= c0) k++;
            g.k0 = g.k1 = (int32_t)k;
            for (int64_t q = k; q < c.pb && pn[q].E < c1; q++) {
                const int a = (int)std::max<int64_t>(0, c0 - pn[q].E), b = (int)std::min<int64_t>(pn[q].e, c1 - pn[q].E);
                if (b <= a) continue;
                g.k1 = (int32_t)q;
                seg.push_back({(int32_t)q, a, b, (int32_t)gr.size()});
                for (int64_t r = a / 256; r * 256 < panels[q].n; r++)
                    sitem.push_back(make_int2((int)seg.size() - 1, (int)r));
            }
            gr.push_back(g);
            glev.push_back(lv++);
        }
        if (c.parent >= 0) first[c.parent] = std::max(first[c.parent], lv);
        z += E;
    }
    npiv = z;
    const int ng = (int)gr.size();
    int levels = 0;
    for (int l : glev) levels = std::max(levels, l + 1);
    std::vector<int2> it;
    item_ptr.assign(1, 0);
    level_e.assign(levels, 1);
    {
        std::vector<std::vector<int>> by(levels);
        for (int g = 0; g < ng; g++) by[glev[g]].push_back(g);
        for (int l = 0; l < levels; l++) {
            auto count = [&](int per) {
                int64_t n = 0;
                for (int g : by[l]) n += std::max<int64_t>(1, ((gr[g].nr + kRC - 1) / kRC + per - 1) / per);
                return n;
            };
            int per = kMC;
            while (per > 1 && count(per) < kWide) per >>= 1;
            for (int g : by[l]) {
                level_e[l] = std::max(level_e[l], gr[g].e);
                const int nch = (int)((gr[g].nr + kRC - 1) / kRC);
                gr[g].items = std::max(1, (nch + per - 1) / per);
                for (int c = 0; c == 0 || c < nch; c += per)
                    it.push_back(make_int2(g, c * 8 + std::min(per, nch - c)));
            }
            item_ptr.push_back((int64_t)it.size());
        }
    }
    if (ng == 0) return CTP_OK;
    DevBuf d_pn, d_seg, d_sitem, d_invp, d_inv;
    const bool mem = grp.need(sizeof(Grp) * ng) && items.need(sizeof(int2) * it.size()) &&
                     vars.need(sizeof(int32_t) * (size_t)vo) && perm.need(sizeof(int32_t) * (size_t)N) &&
                     pack64.need(sizeof(double) * (size_t)po) && (!fp32 || pack32.need(sizeof(float) * (size_t)po)) &&
                     kind.need(sizeof(int32_t) * (size_t)npiv) && D.need(sizeof(double) * 2 * (size_t)npiv) &&
                     d_pn.need(sizeof(Pnl) * pn.size()) && d_seg.need(sizeof(Seg) * seg.size()) &&
                     d_sitem.need(sizeof(int2) * sitem.size()) && d_invp.need(sizeof(int32_t) * (size_t)io) &&
                     d_inv.need(sizeof(int32_t) * (size_t)N);
    bool ok = mem;
    auto up = [&](DevBuf &b, const void *src, size_t bytes) {
        ok = ok && cudaMemcpyAsync(b.p, src, bytes, cudaMemcpyHostToDevice, st) == cudaSuccess;
    };
    if (ok) {
        up(grp, gr.data(), sizeof(Grp) * ng);
        up(items, it.data(), sizeof(int2) * it.size());
        up(perm, perm_host.data(), sizeof(int32_t) * (size_t)N);
        up(d_inv, inv_host.data(), sizeof(int32_t) * (size_t)N);
        up(d_pn, pn.data(), sizeof(Pnl) * pn.size());
        up(d_seg, seg.data(), sizeof(Seg) * seg.size());
        up(d_sitem, sitem.data(), sizeof(int2) * sitem.size());
        ok = ok && cudaMemsetAsync(pack64.p, 0, sizeof(double) * (size_t)po, st) == cudaSuccess &&
             (!fp32 || cudaMemsetAsync(pack32.p, 0, sizeof(float) * (size_t)po, st) == cudaSuccess);
    }
    if (ok) {
        k_lv_panels<<<(unsigned)pn.size(), 128, 0, st>>>(d_pn.as<Pnl>(), d_invp.as<int32_t>(), kind.as<int32_t>(),
                                                        D.as<double>());
        const unsigned gy = (unsigned)std::min<int64_t>((maxtotal + 255) / 256, 16);
        k_lv_vars<<<dim3((unsigned)ng, gy), 256, 0, st>>>(d_pn.as<Pnl>(), grp.as<Grp>(), d_inv.as<int32_t>(),
                                                          vars.as<int32_t>());
        k_lv_pack<double><<<(unsigned)sitem.size(), 256, 0, st>>>(d_pn.as<Pnl>(), grp.as<Grp>(), d_seg.as<Seg>(),
                                                                 d_sitem.as<int2>(), d_invp.as<int32_t>(),
                                                                 pack64.as<double>());
        if (fp32)
            k_lv_pack<float><<<(unsigned)sitem.size(), 256, 0, st>>>(d_pn.as<Pnl>(), grp.as<Grp>(), d_seg.as<Seg>(),
                                                                    d_sitem.as<int2>(), d_invp.as<int32_t>(),
                                                                    pack32.as<float>());
        ok = cudaGetLastError() == cudaSuccess;
    }
    ok = cudaStreamSynchronize(st) == cudaSuccess && ok;
    for (DevBuf *b : {&d_pn, &d_seg, &d_sitem, &d_invp, &d_inv}) b->release();
    if (!ok) return mem ? CTP_ECUDA : CTP_ENOMEM;
    ngrp = ng;
    nlev = levels;
    return CTP_OK;
}

// workspace: the right-hand sides in elimination order, z, the groups' counters
size_t SolvePlan::ws_bytes(int nrhs) const {
    return align256(sizeof(double) * (size_t)(N > 0 ? N : 1) * nrhs) +
           align256(sizeof(double) * (size_t)(npiv > 0 ? npiv : 1) * nrhs) + align256(sizeof(int) * (size_t)(ngrp + 1) * nrhs);
}

template <typename T>
static cudaError_t plan_sweeps(ctp_ctx *ctx, const SolvePlan &pl, const T *pack, double *X, int64_t ldx, int nrhs,
                               void *ws, cudaStream_t st) {
    char *w = (char *)ws;
    Sweep s;
    s.G = pl.grp.as<Grp>();
    s.vars = pl.vars.as<int32_t>();
    s.nrhs = nrhs;
    s.Xp = (double *)w;
    w += align256(sizeof(double) * (size_t)pl.N * nrhs);
    T *Z = (T *)w;
    s.cnt = (int *)(w + align256(sizeof(double) * (size_t)pl.npiv * nrhs));
    cudaError_t e = cudaMemsetAsync(s.cnt, 0, sizeof(int) * (size_t)pl.ngrp * nrhs, st);
    if (e != cudaSuccess) return e;
    const unsigned gb = (unsigned)std::min<int64_t>((pl.N + kLT - 1) / kLT, 4096);
    e = timed(ctx, K_SYS_FWD, st, [&] {
        k_lv_reorder<false><<<gb, kLT, 0, st>>>(pl.N, nrhs, pl.perm.as<int32_t>(), X, ldx, s.Xp);
        return cudaGetLastError();
    });
    if (e != cudaSuccess) return e;
    auto level = [&](bool forward, int l) {
        s.items = pl.items.as<int2>() + pl.item_ptr[l];
        s.nitems = pl.item_ptr[l + 1] - pl.item_ptr[l];
        s.emax = pl.level_e[l];
        return timed(ctx, forward ? K_SYS_FWD : K_SYS_BWD, st, [&] { return launch_level_rg<T>(forward, s, pack, Z, st); });
    };
    for (int l = 0; l < pl.nlev; l++)
        if ((e = level(true, l)) != cudaSuccess) return e;
    e = timed(ctx, K_SYS_FWD, st, [&] {
        const unsigned g = (unsigned)std::min<int64_t>((pl.npiv * nrhs + kLT - 1) / kLT, 4096);
        k_lv_dsolve<T><<<g, kLT, 0, st>>>(pl.npiv, nrhs, pl.kind.as<int32_t>(), pl.D.as<double>(), Z);
        return cudaGetLastError();
    });
    if (e != cudaSuccess) return e;
    for (int l = pl.nlev - 1; l >= 0; l--)
        if ((e = level(false, l)) != cudaSuccess) return e;
    return timed(ctx, K_SYS_BWD, st, [&] {
        k_lv_reorder<true><<<gb, kLT, 0, st>>>(pl.N, nrhs, pl.perm.as<int32_t>(), X, ldx, s.Xp);
        return cudaGetLastError();
    });
}

cudaError_t SolvePlan::solve(ctp_ctx *ctx, double *X, int64_t ldx, int nrhs, void *ws, cudaStream_t st,
                             bool fp32) const {
    return fp32 ? plan_sweeps<float>(ctx, *this, pack32.as<float>(), X, ldx, nrhs, ws, st)
                : plan_sweeps<double>(ctx, *this, pack64.as<double>(), X, ldx, nrhs, ws, st);
}

RefineLayout refine_layout(int64_t N, size_t solve_ws, int nrhs) {
    RefineLayout L;
    size_t off = 0;
    L.solve = off;
    off += align256(solve_ws);
    L.R = off;
    off += align256(sizeof(double) * (size_t)N * nrhs);
    L.rowsum = off;
    off += align256(sizeof(double) * (size_t)N);
    L.mx = off;
    off += align256(sizeof(double) * (3 * (size_t)nrhs + 1));
    L.berr = off;
    off += align256(sizeof(double) * (size_t)nrhs);
    L.total = off;
    return L;
}

static cudaError_t mat_residual(ctp_ctx *ctx, const MatOp &A, int64_t N, int nrhs, const double *X,
                                int64_t ldx, double *R, cudaStream_t st) {
    if (A.sparse())
        return timed(ctx, K_SPMV, st, [&] {
            return launch_spmv_csc_residual(N, A.colptr, A.rowind, A.val, nrhs, X, ldx, R, N, st);
        });
    return timed(ctx, K_SYMV, st, [&] { return launch_symv_residual(N, A.M, A.ldm, nrhs, X, ldx, R, N, st); });
}

cudaError_t mat_abs_rowsum(ctp_ctx *ctx, const MatOp &A, int64_t N, double *rowsum, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(rowsum, 0, sizeof(double) * N, st);
    if (e != cudaSuccess) return e;
    if (A.sparse())
        return timed(ctx, K_SPMV, st, [&] {
            return launch_spmv_csc_abs_rowsum(N, A.colptr, A.rowind, A.val, rowsum, st);
        });
    return timed(ctx, K_SYMV, st, [&] { return launch_abs_rowsum(N, A.M, A.ldm, rowsum, st); });
}

cudaError_t residual_berr(ctp_ctx *ctx, const MatOp &A, int64_t N, int nrhs, const double *B, int64_t ldb,
                          const double *X, int64_t ldx, double *R, const double *rowsum, double *mx,
                          double *berr, cudaStream_t st) {
    cudaError_t e = cudaMemcpy2DAsync(R, sizeof(double) * N, B, sizeof(double) * ldb, sizeof(double) * N, nrhs,
                                      cudaMemcpyDeviceToDevice, st);
    if (e != cudaSuccess) return e;
    e = mat_residual(ctx, A, N, nrhs, X, ldx, R, st);
    if (e != cudaSuccess) return e;
    return timed(ctx, K_BERR, st, [&] {
        return launch_backward_error(N, nrhs, R, N, X, ldx, B, ldb, rowsum, mx, berr, st);
    });
}

}  // namespace ctp
