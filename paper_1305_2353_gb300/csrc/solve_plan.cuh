// solve_plan.cuh -- the solve with a multifrontal factorization, planned by levels of
// groups of pivots (groups of a level are independent: one launch per level and
// sweep), and FP64 iterative refinement (Section 7) around any solve: the
// helpers shared by the ABI's complete-system entry points.
#pragma once

#include <vector>

#include "ctx.cuh"

namespace ctp {

// A device buffer that only grows.
struct DevBuf {
    void *p = nullptr;
    size_t cap = 0;
    bool need(size_t bytes);
    void release();
    template <typename T>
    T *as() const { return static_cast<T *>(p); }
};

// A front's panels, in order: panels [pa, pb) of the list, and its parent front
// (-1: a root; children come before parents).
struct SolveChain {
    int64_t pa, pb;
    int parent;
};

// The factors repacked for solving.  The pivots of a front's panels, in
// elimination order, are cut into groups of at most 64; a group's L11 and its
// rows below (L21, in chunks of rows) are copied into contiguous blocks, with
// the rows in the order they have after the group's last panel, so that a
// sweep needs one launch per level of groups instead of one per panel
// (strict pivoting makes panels of about 15 pivots), and an item's factor entries
// are one contiguous copy.
struct SolvePlan {
    int ngrp = 0, nlev = 0;
    int64_t N = 0, npiv = 0;
    std::vector<int64_t> item_ptr;  // items (group, chunk) of level l: [item_ptr[l], item_ptr[l+1])
    std::vector<int> level_e;       // largest group of each level
    DevBuf grp, items, vars, perm, pack64, pack32, kind, D;
    SolvePlan() = default;
    SolvePlan(const SolvePlan &) = delete;
    SolvePlan &operator=(const SolvePlan &) = delete;
    ~SolvePlan();
    void clear() { ngrp = nlev = 0; }  // forgets the plan, keeps its memory for the next one
    // panels of all fronts; perm_host: the elimination order (variable of position i),
    // inv_host its inverse; fp32: also pack for FP32 sweeps.  Reads the panels'
    // device arrays on `st` (synchronised before returning).
    ctp_status build(const std::vector<ctp_sfront> &panels, const std::vector<int32_t> &nelim,
                     const std::vector<SolveChain> &fronts, const std::vector<int32_t> &perm_host,
                     const std::vector<int32_t> &inv_host, bool fp32, cudaStream_t st);
    size_t ws_bytes(int nrhs) const;
    // X <- M^{-1} X; fp32: the sweeps' arithmetic in FP32 (X read and written in FP64)
    cudaError_t solve(ctp_ctx *ctx, double *X, int64_t ldx, int nrhs, void *ws, cudaStream_t st,
                      bool fp32 = false) const;
};

// The system matrix of a residual: dense (lower triangle, column-major) or
// sparse (lower triangle in compressed columns), symmetric either way.
struct MatOp {
    const double *M = nullptr;
    int64_t ldm = 0;
    const int64_t *colptr = nullptr;
    const int32_t *rowind = nullptr;
    const double *val = nullptr;
    bool sparse() const { return colptr != nullptr; }
};

struct RefineLayout {
    size_t solve, R, rowsum, mx, berr, total;
};
RefineLayout refine_layout(int64_t N, size_t solve_ws, int nrhs);

// Residual R = B - A X and the Section 7 backward errors into berr (device).
cudaError_t residual_berr(ctp_ctx *ctx, const MatOp &A, int64_t N, int nrhs, const double *B, int64_t ldb,
                          const double *X, int64_t ldx, double *R, const double *rowsum, double *mx,
                          double *berr, cudaStream_t st);
cudaError_t mat_abs_rowsum(ctp_ctx *ctx, const MatOp &A, int64_t N, double *rowsum, cudaStream_t st);

// X = solve(B); while the worst backward error exceeds tol and fewer than
// max_steps corrections were made: X += solve(B - A X).  `solve(Y, ldy, ws)`
// overwrites the N x nrhs array Y with the solution (cudaError_t).
template <typename Solve>
ctp_status refine_core(ctp_ctx *ctx, Solve &&solve, size_t solve_ws, int64_t N, const MatOp &A, int32_t nrhs,
                       const double *B, int64_t ldb, double *X, int64_t ldx, int32_t max_steps, double tol,
                       double *berr_host, int32_t *steps_host, void *workspace, size_t ws_bytes,
                       cudaStream_t st) {
    RefineLayout L = refine_layout(N, solve_ws, nrhs);
    if (ws_bytes < L.total) return CTP_ENOMEM;
    char *w = (char *)workspace;
    void *sws = w + L.solve;
    double *R = (double *)(w + L.R), *rowsum = (double *)(w + L.rowsum);
    double *mx = (double *)(w + L.mx), *berr = (double *)(w + L.berr);
    *steps_host = 0;
    CTP_CUDA(mat_abs_rowsum(ctx, A, N, rowsum, st));
    CTP_CUDA(cudaMemcpy2DAsync(X, sizeof(double) * ldx, B, sizeof(double) * ldb, sizeof(double) * N, nrhs,
                               cudaMemcpyDeviceToDevice, st));
    CTP_CUDA(solve(X, ldx, sws));
    for (int32_t k = 0;; k++) {
        CTP_CUDA(residual_berr(ctx, A, N, nrhs, B, ldb, X, ldx, R, rowsum, mx, berr, st));
        double *bh = berr_host + (size_t)k * nrhs;
        CTP_CUDA(cudaMemcpyAsync(bh, berr, sizeof(double) * nrhs, cudaMemcpyDeviceToHost, st));
        CTP_CUDA(cudaStreamSynchronize(st));
        double worst = 0.0;
        for (int r = 0; r < nrhs; r++) worst = bh[r] > worst || bh[r] != bh[r] ? bh[r] : worst;
        if (!(worst > tol) || k == max_steps) break;
        CTP_CUDA(solve(R, N, sws));
        CTP_CUDA(timed(ctx, K_AXPY, st, [&] { return launch_axpy(N, nrhs, X, ldx, R, N, st); }));
        *steps_host = k + 1;
    }
    return CTP_OK;
}

}  // namespace ctp
