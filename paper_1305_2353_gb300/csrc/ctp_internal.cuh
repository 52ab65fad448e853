// ctp_internal.cuh -- internal declarations shared by the libctp translation units.
// Product code only: nothing here is used by, or uses, the CPU oracle.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/ctp.h"

namespace ctp {

// Largest supernode width handled on chip by the pivot search (kernel K3).
constexpr int kMaxP = 256;

// Device info word codes (first int32 of the workspace).
constexpr int kInfoOk = 0;

// Digit slices of the FP64 Form's operands (slices.cuh).
constexpr int kSlices = 8;
constexpr int kSliceK = 32;                       // pivots per K block
constexpr int kWRows = 128, kLRows = 64;          // rows per block
constexpr uint32_t kWSlice = kWRows * 64, kLSlice = kLRows * 64;  // bytes of one slice of one K block
constexpr uint32_t kWBlock = kSlices * kWSlice, kLBlock = kSlices * kLSlice;
constexpr int kExpZero = -100000, kExpNonfinite = 1 << 20;
constexpr int kGroup = 4;  // rows that share a lower bound of their entries
constexpr uint32_t kWGroup = kWRows / kGroup * kSliceK * 2, kLGroup = kLRows / kGroup * kSliceK * 2;  // a block's bytes

// Fronts of at most this many rows below the pivots form S by FP64 multiply-adds from W21 itself
// (form.cu): a tile of slices is 128 rows by 32 pivots, and they would take up to 40 times
// the room of W21.
constexpr int kFormSmall = 32;
__host__ __device__ inline bool form_small(int64_t m) { return m <= kFormSmall; }

// Where a supernode's slices live: blocks at (row block * kb + K block), the
// rows' exponents E, the groups' lower bounds (FP16) in blocks like the slices'; kb =
// ceil(p / 32).
struct SliceBuf {
    unsigned char *W, *L;
    int32_t *ew, *el;
    uint16_t *gw, *gl;
    int kb;
};
__host__ __device__ inline int slice_kb(int p) { return (p + kSliceK - 1) / kSliceK; }
// Rows are rounded up to 8 (what the MMA's layout and a bulk copy want), also in the last
// block: a front with few rows takes room for those only.
__host__ __device__ inline int64_t slice_rows(int64_t m) { return (m + 7) & ~int64_t(7); }
__host__ __device__ inline size_t slice_bytes(int64_t m, int p) {
    return (size_t)slice_rows(m) * slice_kb(p) * (kSlices * 64);
}
__host__ __device__ inline size_t slice_g_bytes(int64_t m, int p) {
    return (size_t)(slice_rows(m) / kGroup) * slice_kb(p) * (kSliceK * 2);
}

// Which entries of a tile of the FP64 Form (or of the Solve's update) digits do not serve,
// for the kernel's own use: a bit per column for every row of a warp's block, and
// the CTA's tile before it that has any.
struct TileMarks {
    uint16_t out[kWRows * kLRows / 512][32];
    int64_t prev, pad;
};

// Workspace layout (all offsets 256-byte aligned):
//   [0, 256)            info word + scratch counters
//   C                   p*p doubles, row-major compressed matrix (strict: as uint64 keys)
//   Dinv                2p doubles: inverse pivot blocks, same slots as D
//   W21                 m*p doubles (Y = L21 D11) when the FP64 Form of few rows runs
//   Ws, Ls, ew, el,     digit slices of Y = L21 D11 and L21, their row exponents and
//     gw, gl            lower bounds (slices.cuh) when the FP64 Form step runs
//   Yb, Lx, ey, ex,     the same of one block's y and of L11 for the blocked FP64 Solve
//     gy, gx
//   marks               a TileMarks per tile of a launch of the FP64 Form or of the Solve's updates
//   Wb, Lb              m*Kp BF16 copies of Y and L21 for the tensor-core Form
//   aux                 method-specific scratch (relaxed candidate lists)
struct WsLayout {
    size_t info, C, Dinv, W21, Ws, Ls, ew, el, gw, gl, Yb, Lx, ey, ex, gy, gx, marks, Wb, Lb, aux, Xs, flags, total;
};

inline size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

// Make sure `func` may launch with `bytes` of dynamic shared memory on the
// current device: raises cudaFuncAttributeMaxDynamicSharedMemorySize when it is
// below `bytes` and never lowers it.  The attribute belongs to the function,
// not to one launch: a CUDA graph node captured with more shared memory than a
// later, lower setting allows fails when the graph is replayed, so no launcher
// may lower it.  (A device reset restores the default; the current value is
// queried each time, so the next launch raises it again.)
cudaError_t smem_at_least(const void *func, size_t bytes);

WsLayout ws_layout(int64_t n, int p, const ctp_options *opt, int num_sms);
int ctx_batch_smem_kb(const ctp_ctx *ctx);  // CTP_TUNE_BATCH_SMEM_KB of a context
// BF16 pieces per operand of the tensor-core Form for a precision (0: FP64 Form)
inline int prec_pieces(int prec) {
    return prec == CTP_BF16 ? 1 : (prec == CTP_BF16X3 ? 2 : (prec == CTP_BF16X6 ? 3 : 0));
}
size_t factor_batch_max_dynamic_smem();     // dynamic shared memory the batched pivot search can take
size_t factor_smem_bytes(int p, int R, int G);  // dynamic shared memory of a pivot-search CTA
size_t factor_warp_smem_bytes(int pcap, int ldcap);  // of a CTA of the warp-per-front kernel
// kinds of batched pivot-search launch: a warp per front (p <= 32, at most 64
// rows of [A11; C]), a CTA per front, a cluster of G CTAs per front
constexpr int kFactorWarp = 0, kFactorCta = 1, kFactorCluster = 2;

// ---------------------------------------------------------------------------
// kernel launchers (each returns cudaError_t of the launch)
// rowbits (optional, ceil(p/32) words cleared by the caller): bit j set for
// every row j of C that receives an A21 row (the rows the pivot search must keep)
cudaError_t launch_compress_strict(const double *A21, int64_t m, int p, int64_t lda,
                                   unsigned long long *Ckeys, int32_t *J, uint32_t *rowbits, int32_t *info,
                                   int num_sms, cudaStream_t st);
// single-row compression: ckey[k] (p keys, zeroed by the caller) = max_i |a21(i,k)|
cudaError_t launch_compress_single_row(const double *A21, int64_t m, int p, int64_t lda,
                                       unsigned long long *ckey, int32_t *info, int num_sms, cudaStream_t st);
int relaxed_block_lg(int64_t m, int p);
size_t relaxed_aux_bytes(int64_t m, int p, int num_sms);
cudaError_t launch_compress_relaxed(const double *A21, int64_t m, int p, int64_t lda, double *C,
                                    int32_t *rows, void *aux, int32_t *info, int num_sms,
                                    cudaStream_t st);
cudaError_t launch_keys_to_rowmajor(const unsigned long long *Ckeys, double *C, int p,
                                    cudaStream_t st);

struct FactorArgs {
    double *A;          // n x p supernode (in/out)
    int64_t lda;
    int p;
    int R;              // outer rows held on chip: p (compressed) or 0 (restricted)
    int abs_update;     // 1: strict worst-case update of the outer rows
    const double *C;    // R x p row-major outer rows (doubles), or nullptr
    const uint32_t *rowbits;  // R bits: set for rows of C that may be nonzero (nullptr: scan C)
    double u, small;
    int32_t *perm, *piv, *nelim;
    double *D, *Dinv;
    int32_t *info;
};
cudaError_t launch_factor_cluster(const FactorArgs &a, int G /* 0: by p */, cudaStream_t st);

// ---------------------------------------------------------------------------
// batched path: per-front table (built on the host by the plan, uploaded into
// the workspace) and the per-front workspace sections
struct BFront {
    int64_t n, m;
    int32_t p, nM;       // nM: 128-row blocks of S (tensor-core Form)
    int64_t ws;          // byte offset of this front's workspace section
    int64_t row0;        // first row of this front in the stacked BF16 operand buffers
    int64_t c0, s0, f0;  // first compression / solve / form work item of this front
    // tensor-core Solve: first 128 x 64 tile of x_e and of Z^T, first GEMM item,
    // K blocks and output windows at most (from p)
    int64_t xt0, zt0, q0, r0;  // r0: first prep item (8 identity rows each)
    int32_t kbx, nwz;
};
struct BatchOpts {
    double u, small;
    int pivot;  // ctp_pivot
    int smode, prec;
    int64_t lo_off;  // elements between the BF16 pieces of the operand copies
    int pieces;      // BF16 pieces per operand (1: plain; 2, 3: split)
    int stc;         // the Solve runs on the tensor cores
    int64_t xoff, zoff;  // elements between the pieces of the x_e / Z^T tile arrays
};

// Whether a front of a batch may solve for its rows in blocks (solve.cu): one block of 32
// columns, the tensor cores' update of the others and the rest.  Measured, all Solves of
// batches of equal fronts, one pass / in blocks, m x p.  Strict pivoting, a dozen
// accepted: 60 x 96 430 / 518 us, 200 x 96 504 / 424, 60 x 128 512 / 618, 200 x 128 589 / 439,
// 60 x 200 553 / 635, 60 x 256 612 / 600, 800 x 256 565 / 324; 200 x 64 475 / 563, 800 x 64
// 485 / 440, 2400 x 64 385 / 393.  All accepted: 60 x 64 1396 / 1316, 60 x 96 1989 / 1612,
// 800 x 200 3767 / 3187; 200 x 48 1143 / 1230, 800 x 48 1020 / 983.
__host__ __device__ inline bool front_blocked(int64_t m, int p, const BatchOpts &o) {
    const int64_t right = m * (p - kSliceK);  // entries that the update touches
    return o.pivot == CTP_PIV_STRICT ? p > 56 && right >= 12000 : p > 48 && right >= 1900;
}

// offsets inside a front's section: info word, compressed matrix (strict),
// Dinv, and when an FP64 Form follows W21 = L21 D11 (few rows) or the digit slices of
// W21 and L21
struct BSection {
    size_t info, C, Dinv, W21, Ws, Ls, ew, el, gw, gl, Yb, Lx, ey, ex, gy, gx, nz, total;
};
__host__ __device__ inline size_t align256hd(size_t x) { return (x + 255) & ~size_t(255); }
__host__ __device__ inline BSection bsection(int64_t n, int p, const BatchOpts &o) {
    BSection s;
    size_t off = 0;
    s.info = off;
    off += 256;
    s.C = off;
    off += align256hd(o.pivot == CTP_PIV_STRICT ? sizeof(double) * (size_t)p * p : 0);
    s.Dinv = off;
    off += align256hd(sizeof(double) * (2 * (size_t)p + 2));
    s.nz = off;  // strict: which rows of C receive an A21 row (one bit per row)
    off += align256hd(o.pivot == CTP_PIV_STRICT ? sizeof(int32_t) * (size_t)p : 0);
    const int64_t mf = o.smode != CTP_S_NONE && o.prec == CTP_FP64 ? n - p : 0;
    const int64_t ms = form_small(mf) ? 0 : mf;
    s.W21 = off;
    off += align256hd(sizeof(double) * (size_t)(mf - ms) * p);
    s.Ws = off;
    off += align256hd(slice_bytes(ms, p));
    s.Ls = off;
    off += align256hd(slice_bytes(ms, p));
    s.ew = off;
    off += align256hd(sizeof(int32_t) * (size_t)ms);
    s.el = off;
    off += align256hd(sizeof(int32_t) * (size_t)ms);
    s.gw = off;
    off += align256hd(slice_g_bytes(ms, p));
    s.gl = off;
    off += align256hd(slice_g_bytes(ms, p));
    // the blocked Solve's first block: slices of y (where those of W21 come later, if there
    // are any) and of L11's rows below it
    const bool blk = !o.stc && front_blocked(n - p, p, o);
    const int64_t mb = blk && ms == 0 ? n - p : 0;
    const int pb = blk ? p - kSliceK : 0;
    s.Yb = blk && ms > 0 ? s.Ws : off;
    off += align256hd(slice_bytes(mb, kSliceK));
    s.ey = blk && ms > 0 ? s.ew : off;
    off += align256hd(sizeof(int32_t) * (size_t)mb);
    s.gy = blk && ms > 0 ? s.gw : off;
    off += align256hd(slice_g_bytes(mb, kSliceK));
    s.Lx = off;
    off += align256hd(slice_bytes(pb, kSliceK));
    s.ex = off;
    off += align256hd(sizeof(int32_t) * (size_t)pb);
    s.gx = off;
    off += align256hd(slice_g_bytes(pb, kSliceK));
    s.total = off;
    return s;
}

__host__ __device__ inline SliceBuf bsection_slices(char *base, const BSection &s, int p) {
    SliceBuf b;
    b.W = reinterpret_cast<unsigned char *>(base + s.Ws);
    b.L = reinterpret_cast<unsigned char *>(base + s.Ls);
    b.ew = reinterpret_cast<int32_t *>(base + s.ew);
    b.el = reinterpret_cast<int32_t *>(base + s.el);
    b.gw = reinterpret_cast<uint16_t *>(base + s.gw);
    b.gl = reinterpret_cast<uint16_t *>(base + s.gl);
    b.kb = slice_kb(p);
    return b;
}

__host__ __device__ inline SliceBuf bsection_block(char *base, const BSection &s) {
    SliceBuf b;
    b.W = reinterpret_cast<unsigned char *>(base + s.Yb);
    b.L = reinterpret_cast<unsigned char *>(base + s.Lx);
    b.ew = reinterpret_cast<int32_t *>(base + s.ey);
    b.el = reinterpret_cast<int32_t *>(base + s.ex);
    b.gw = reinterpret_cast<uint16_t *>(base + s.gy);
    b.gl = reinterpret_cast<uint16_t *>(base + s.gx);
    b.kb = 1;
    return b;
}

// pivot search of the fronts list[0..count) of one class: kind (kFactor*), the
// cluster width G, the dynamic shared memory per CTA, and for the warp kernel
// the largest p and p + R of the class (its per-warp slice)
cudaError_t launch_factor_batch(const ctp_front *fronts, const BFront *tab, char *ws, const int *list,
                                int count, int kind, int G, size_t smem, int pcap, int ldcap, BatchOpts o,
                                cudaStream_t st);
// bucket[b] .. bucket[b+1]: the items (32-row tiles) of the fronts with p <= 32 << b
cudaError_t launch_compress_strict_batch(const ctp_front *fronts, const BFront *tab, char *ws,
                                         const int *item_front, const int64_t (&bucket)[5], BatchOpts o,
                                         cudaStream_t st);
// items: (front, tile) pairs; plain: no slices are written
cudaError_t launch_solve_batch(const ctp_front *fronts, const BFront *tab, char *ws,
                               const int *item_front, int64_t items, int rows, bool plain, BatchOpts o, void *Wb, void *Lb,
                               int pmax, cudaStream_t st, const int *item_tile);
// rows per tile (32, 16 or 8) of a Solve with this many 32-row tiles
int solve_rows(int64_t tiles, bool blocked, int num_sms);
// item_tile (optional, both batched Forms): each item's tile of its front;
// without it the items of a front are consecutive, from tab[front].f0 on
cudaError_t launch_form_fp64_batch(const ctp_front *fronts, const BFront *tab, char *ws,
                                   const int *item_front, int64_t items, BatchOpts o, TileMarks *marks, int32_t *info,
                                   int num_sms, cudaStream_t st, const int *item_tile = nullptr);
// the fronts of few rows, by number (W21 from their sections)
cudaError_t launch_form_small_batch(const ctp_front *fronts, const BFront *tab, char *ws, const int *list, int64_t count,
                                    BatchOpts o, cudaStream_t st);
cudaError_t launch_form_tc_batch(const ctp_front *fronts, const BFront *tab, const int *item_front,
                                 int64_t items, int64_t total_rows, const void *Wb, const void *Lb,
                                 int pieces, int layout /* 2 tiled, 3 subtract */, int32_t *info, int num_sms,
                                 cudaStream_t st, const int *item_tile = nullptr);
constexpr int kBatchKp = 256;  // K stride of the stacked BF16 operand buffers

// the batched launch sequence (batch.cu); the plan type is declared in ctp.h
int batch_num_classes(const ctp_plan *P);
int batch_class_kind(const ctp_plan *P, int c);  // kFactor*
int batch_class_G(const ctp_plan *P, int c);
size_t batch_total(const ctp_plan *P);
size_t batch_blob_bytes(const ctp_plan *P);
const void *batch_blob(const ctp_plan *P);
cudaError_t batch_upload(const ctp_plan *P, const void *blob, char *w, cudaStream_t st);
cudaError_t batch_flags(const ctp_plan *P, char *w, int32_t *flags_host, cudaStream_t st);
// ctp_factor_batch with one of the context's two sets of side streams; the stream
// from which a second batch in flight runs (ordered behind st; false: none)
ctp_status factor_batch_on(ctp_ctx *ctx, const ctp_plan *plan, const ctp_front *fronts, void *workspace,
                           size_t ws_bytes, cudaStream_t st, int set);
bool second_stream(ctp_ctx *ctx, cudaStream_t st, cudaStream_t *out);
cudaError_t batch_prepare(const ctp_plan *P, char *w, cudaStream_t st);
cudaError_t batch_compress(const ctp_plan *P, const ctp_front *fr, char *w, int num_sms, cudaStream_t st);
cudaError_t batch_factor_class(const ctp_plan *P, int ci, const ctp_front *fr, char *w, cudaStream_t st);
cudaError_t batch_solve(const ctp_plan *P, const ctp_front *fr, char *w, int num_sms, cudaStream_t st);
bool batch_solve_per_class(const ctp_plan *P);
cudaError_t batch_solve_class(const ctp_plan *P, int ci, const ctp_front *fr, char *w, int num_sms, cudaStream_t st);
cudaError_t batch_form_class(const ctp_plan *P, int ci, const ctp_front *fr, char *w, int num_sms, cudaStream_t st);
cudaError_t batch_form(const ctp_plan *P, const ctp_front *fr, char *w, int num_sms, cudaStream_t st);

// Tensor-core Solve (solve_tc.cu): BF16 pieces of its operands, its scratch
// bytes, and the launch sequence (prep of Z^T, gather of x_e, the GEMM with its
// epilogue).  Its outputs are stored factors, so it always takes three pieces
// (products close to FP32, whatever the Form's pieces): with two, a chain of
// fronts whose every Solve and Form was split in two stopped refining at 2e-13.
inline int solve_tc_pieces(int) { return 3; }
// the tensor-core Solve runs when asked for and the Form runs on the tensor cores
inline bool solve_on_tc(const ctp_options *o) {
    return o->solve == CTP_SOLVE_TC && o->prec != CTP_FP64 && o->smode != CTP_S_NONE && o->pivot != CTP_PIV_TPP;
}
size_t solve_tc_ws_bytes(int64_t m, int p, int spieces);
cudaError_t launch_solve_tc(double *A, int64_t n, int p, int64_t lda, const int32_t *perm, const int32_t *piv,
                            const double *Dinv, const int32_t *nelim, void *ws, int spieces, void *Wb, void *Lb,
                            int64_t foff, int fpieces, int32_t *info, int num_sms, cudaStream_t st);

// Batched tensor-core Solve: x_e and Z^T of every front in 128 x 64 BF16 tiles
// (three pieces each), GEMM items (front, 128-row block, output window).
size_t solve_tc_tile_elems();  // elements of one tile
int solve_tc_windows(int p);   // output windows of a front of width p, at most
cudaError_t launch_solve_tc_batch(const ctp_front *fronts, const BFront *tab, char *ws, const int *sitem,
                                  int64_t s_items, const int *qitem, int64_t q_items, const int *ritem,
                                  int64_t r_items, BatchOpts o,
                                  void *Xt, void *Zt, int64_t nxt, int64_t nzt, void *Wb, void *Lb,
                                  int32_t *ginfo, int num_sms, cudaStream_t st);

cudaError_t launch_solve_fp64(double *A, int64_t n, int p, int64_t lda, const int32_t *perm,
                              const int32_t *piv, const double *Dinv, const int32_t *nelim,
                              double *W21, const SliceBuf &sb, const SliceBuf &blk, int blocks, void *Wb, void *Lb, int Kp,
                              int64_t lo_off, int pieces, TileMarks *marks, int32_t *info, int num_sms, cudaStream_t st);
int solve_blocks(int64_t m, int p, int pivot);  // 0: a whole pass
// A21(:, 32 (blk+1)..p-1) -= y_blk L11(32 (blk+1).., block blk)^T from the slices (form.cu)
cudaError_t launch_update(const SliceBuf &u, double *A, int64_t lda, int p, int64_t m, int blk, const int32_t *piv,
                          const int32_t *nelim, TileMarks *marks, int32_t *info, int num_sms, cudaStream_t st);
// the same for block 0 of a batch's fronts, by (front, tile) items
cudaError_t launch_update_batch(const ctp_front *fronts, const BFront *tab, char *ws, const int *item_front,
                                const int *item_tile, int64_t items, BatchOpts o, TileMarks *marks, int32_t *info,
                                int num_sms, cudaStream_t st);
int64_t update_tiles(int64_t m, int p);  // of a front, for block 0
int64_t form_fp64_marks(int64_t m);      // TileMarks that a single supernode's Form needs
// a batch class's Solve in one block of 32 columns, its update and the tail
cudaError_t launch_solve_batch_blocked(const ctp_front *fronts, const BFront *tab, char *ws, const int *list,
                                       int count, const int *item_front, const int *item_tile, int64_t items,
                                       int rows, const int *uitem, const int *utile, int64_t uitems, BatchOpts o, void *Wb,
                                       void *Lb, int pmax, TileMarks *marks, int32_t *info, int num_sms, cudaStream_t st);

// Threshold partial pivoting on all n rows (the comparator of the compressed path).
size_t tpp_ws_bytes(int p);
// spin: polls a grid barrier waits before it reports CTP_ETIMEOUT (0: the default)
cudaError_t launch_tpp(double *A, int64_t n, int p, int64_t lda, double u, double small, void *ws,
                       int32_t *perm, int32_t *piv, double *D, double *Dinv, int32_t *nelim,
                       int32_t *info, int num_sms, int spin, cudaStream_t st);

// K-padding of the BF16 operand copies used by the tensor-core Form.
int form_tc_kpad(int p);
// pieces: BF16 pieces per operand (1 plain, 2 or 3 split), piece_off elements apart.
cudaError_t launch_form_tc(const void *Wb, const void *Lb, int64_t piece_off, int pieces, int64_t m, int Kp,
                           const int32_t *nelim, float *S, int64_t lds,
                           int layout /* 0 full, 1 packed, 2 tiled, 3 subtract from FP64 */,
                           int32_t *info, int num_sms, int walk /* ctp_walk */, cudaStream_t st);

// S = W21 L21^T in FP64 from the operands' slices (form.cu)
// (L21, D and the pivot kinds serve the rows that the slices do not represent)
cudaError_t launch_form_fp64(const SliceBuf &sb, const double *L21, int64_t lda, const int32_t *piv,
                             const double *D, int64_t m, const int32_t *nelim, void *S, int64_t lds, int smode,
                             TileMarks *marks, int32_t *info, int num_sms, cudaStream_t st);
// the same for few rows (W21 null: from L21 and D)
cudaError_t launch_form_small(const double *L21, int64_t lda, const double *W21, const int32_t *piv, const double *D,
                              int64_t m, const int32_t *nelim, void *S, int64_t lds, int smode, cudaStream_t st);
// the slices from a stored L21 and its D, D^-1 (full-column pivoting)
cudaError_t launch_slices_from_l(const double *A, int64_t lda, int p, int64_t m, const int32_t *piv,
                                 const double *D, const double *Dinv, const int32_t *nelim, const SliceBuf &sb,
                                 cudaStream_t st);

// Complete systems: front-list solve, residual, backward error (system.cu).
size_t sys_solve_ws_bytes(int64_t nmax, int nrhs);
cudaError_t launch_sys_forward(const ctp_sfront &f, double *X, int64_t ldx, int nrhs, void *ws,
                               cudaStream_t st);
cudaError_t launch_sys_backward(const ctp_sfront &f, double *X, int64_t ldx, int nrhs, void *ws,
                                cudaStream_t st);
cudaError_t launch_symv_residual(int64_t N, const double *M, int64_t ldm, int nrhs, const double *X,
                                 int64_t ldx, double *R, int64_t ldr, cudaStream_t st);
cudaError_t launch_abs_rowsum(int64_t N, const double *M, int64_t ldm, double *rowsum,
                              cudaStream_t st);
cudaError_t launch_backward_error(int64_t N, int nrhs, const double *R, int64_t ldr, const double *X,
                                  int64_t ldx, const double *B, int64_t ldb, const double *rowsum,
                                  double *mx, double *berr, cudaStream_t st);
cudaError_t launch_axpy(int64_t N, int nrhs, double *X, int64_t ldx, const double *Dx, int64_t ldd,
                        cudaStream_t st);
cudaError_t launch_sym_grad_dense(int64_t N, int nrhs, const double *G, int64_t ldg, const double *X,
                                  int64_t ldx, double *out, int64_t ldo, cudaStream_t st);
cudaError_t launch_sym_grad_pattern(int64_t nnz, const int32_t *row, const int32_t *col, int nrhs,
                                    const double *G, int64_t ldg, const double *X, int64_t ldx,
                                    double *out, cudaStream_t st);
cudaError_t launch_spmv_csc_residual(int64_t N, const int64_t *colptr, const int32_t *rowind,
                                     const double *val, int nrhs, const double *X, int64_t ldx, double *R,
                                     int64_t ldr, cudaStream_t st);
cudaError_t launch_spmv_csc_abs_rowsum(int64_t N, const int64_t *colptr, const int32_t *rowind,
                                       const double *val, double *rowsum, cudaStream_t st);

}  // namespace ctp
