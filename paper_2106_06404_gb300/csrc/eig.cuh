// Batched block subspace iteration with Rayleigh-Ritz for the local GEVPs
//   abar(w, v) = lambda b(w, v)                     (Eq. theGEVP)
// through the spectral transformation with the shifted matrix
// K = Abar + sigma B (mu = 1 / (lambda + sigma), largest mu wanted; cf. the
// shift-invert use of Section 4.2/4.3 and the transformation in the proof of
// the non-defectiveness lemma of Section 3.3).
//
// One iteration for every unconverged problem i (X B-orthonormal Ritz vectors
// with Ritz values theta, AX = Abar X, BX = B X, S = K^{-1} B):
//   W = BX - (AX + sigma BX) diag(mu),      mu_k = 1 / (theta_k + sigma)
//   W <- K^{-1} W        (tile LDL^T solve, FP64 or FP32 factors), so that S X = X diag(mu) + W
//   Y = the Chebyshev step of S X, X and Q (the block before X in the basis of
//       X) that damps [0, c], c = 0.95 times the smallest Ritz value of S in
//       the block; the first iteration, and blocks that span more than the
//       range of B, Y = S X
//   AY, BY; H = Y^T AY, M = Y^T BY (FP64); Rayleigh-Ritz H c = theta M c
//   Q = X C, X = Y C, AX = AY C, BX = BY C (with a cheap operator X and Q only, AX
//       and BX afresh); residuals |AX_k - theta_k BX_k| / ((theta_k + sigma) |BX_k|).
// The residual form lets an inexact (lower precision) K^{-1} still converge
// to the FP64 eigenpairs: its fixed point does not depend on the solve.
#pragma once
#include "common.cuh"
#include "tile_ldlt.cuh"

namespace msdd {

struct GevpBatch {
    int P = 0;
    int ldx = PMAX;                   // columns stored per row
    std::vector<int> p;               // block size per problem (<= PMAX)
    DevBuf<int> d_p;
    TileBatch K;                      // factor of Abar + sigma B (rows = problem size)
    DevBuf<double> X, AX, BX, Y, AY, BY, W;        // (total_rows x ldx); W with FP64 factors only
    // right-hand sides and solutions beside FP32 factors (total_rows x ldw,
    // ldw = the largest p rounded up to 4): the solves round them to FP32
    // either way, so FP32 storage halves their traffic at the same results
    DevBuf<float> W32;
    int ldw = PMAX;
    DevBuf<int> sdone, sstop, smax;   // FP32 start phase: ended, its iterations; per group the largest of them
    DevBuf<unsigned> ticket;          // per problem: row ranges of the FP32 Gram that are done
    // the block before X in its basis (Chebyshev recurrence); where AX and BX are only needed by the first iteration
    // (`fused` of alloc: the operator is applied afresh), a view of AX
    DevBuf<double> Q;
    // per problem: end of the damped interval of S = K^{-1} B; 0: plain step next; negative: the step before was plain
    DevBuf<double> cheb;
    DevBuf<double> H, M, C, theta, res;            // per problem PMAX^2 / PMAX
    int gsplit = 1;                                // row splits of the Gram products
    DevBuf<double> Hp, Mp;                         // per (problem, split) PMAX^2 partial Grams
    DevBuf<double> partial;                        // per (problem, row block) sums
    DevBuf<int> done, m, rank, iters;   // done: 0 running, 1 converged, 2 maxit, 3 at noise floor
    DevBuf<double> best;                 // best worst-selected residual so far
    DevBuf<int> best_it;
    DevBuf<int> n_active;
    int nblk_max = 0;
    bool knorm = false;           // residual measured in the K^+-norm (coarse levels)
    void alloc(cudaStream_t s, bool fused = false);
    // Non-owning view of problems [p0, p0 + np) with its own active counter
    // (group < 2): per-problem arrays offset, block vectors shared (they are
    // addressed by absolute row offsets).
    GevpBatch slice(int p0, int np, int group) const;
};

struct EigParams {
    double sigma = 1e-2;
    double tol = 1e-6;
    double eta = 0.3;
    int nev_max = 8;
    int maxit = 100;
    unsigned long long seed = 12345;
};

// Fill X with counter-based random numbers (rows < n_i, columns < p_i) and
// zero the rest; reset per-problem state.
void eig_init(GevpBatch& g, unsigned long long seed, cudaStream_t s);
// X[:, c] <- Wst rows (woff[i] + r), columns c < min(wc, p_i), for rows r < n_i
// (caller-provided start vectors; the remaining columns keep eig_init's).
void eig_load_start(GevpBatch& g, const double* Wst, int wc, const long long* d_woff, cudaStream_t s);
// W = BX - (AX + sigma BX) diag(mu) (first == true: W = BX).
void eig_form_rhs(GevpBatch& g, double sigma, bool first, cudaStream_t s);
// The next block from X, W = S X - X diag(mu) (S = K^{-1} B) and Q, the block
// before X: FORM_FIRST Y = W (which then is S X), FORM_CHEB1 the first and
// FORM_CHEB every further step of the Chebyshev recurrence that damps
// [0, cheb[i]] (plain S X where cheb[i] is 0).
enum EigForm { FORM_FIRST = 0, FORM_CHEB1 = 1, FORM_CHEB = 2 };
void eig_form_y(GevpBatch& g, double sigma, EigForm mode, cudaStream_t s);
// FP32 start phase: W <- X in FP32; V = S X (FORM_FIRST: V is SX and the
// damped interval is set) or the Chebyshev step of SX, X and Q (V written),
// and C (FP32, in the buffer of g.C) with V C an orthonormal basis of span(V)
// by Euclidean CholQR; X <- W C of the problems that end after `steps`
// iterations (last: or later).  The first START_SETTLE iterations are power
// steps and every eighth after them; with `early`, after the settling part sstop
// holds each problem's number of iterations, one of the stops of start_stop.
constexpr int START_SETTLE = 6;
constexpr int START_ITERS = 20;   // the default number of iterations, under which a problem may end earlier
__host__ __device__ inline int start_stop(int steps) {
    return steps <= 10 ? 10 : steps <= 13 ? 13 : 1 << 20;
}
void eig_start32(GevpBatch& g, float* W, cudaStream_t s);
void eig_cholqr32(GevpBatch& g, const EigParams& ep, int it, EigForm mode, bool early, const float* SX,
                  const float* X, const float* Q, float* V, cudaStream_t s);
void eig_update32(GevpBatch& g, const float* W, int steps, bool last, cudaStream_t s);
// The same with the K^+-norm residual partial sums of X.
void eig_form_y_knorm(GevpBatch& g, double sigma, EigForm mode, cudaStream_t s);
// Convergence test on the K^+-norm residuals (regularised coarse pencils).
void eig_check_knorm(GevpBatch& g, const EigParams& ep, int it, cudaStream_t s);
// H = Y^T AY, M = Y^T BY.
void eig_gram(GevpBatch& g, cudaStream_t s);
// Rayleigh-Ritz: theta ascending, C with C^T M C = I; the next damped interval.
void eig_rayleigh_ritz(GevpBatch& g, double sigma, cudaStream_t s);
// X = Y C, AX = AY C, BX = BY C, residual partial sums; want_q: Q = (old X) C.
void eig_update(GevpBatch& g, bool want_q, cudaStream_t s);
// X = Y C only: with a cheap operator (stored stencils) AX and BX are applied
// afresh, together with the next right-hand side (apply_local_rhs).
void eig_update_x(GevpBatch& g, bool want_q, cudaStream_t s);
// Selection count m = min(nev_max, #{theta < eta}) of the running problems.
void eig_select(GevpBatch& g, const EigParams& ep, cudaStream_t s);
// Residuals, selection count m, convergence flags.
void eig_check(GevpBatch& g, const EigParams& ep, int it, cudaStream_t s);

// Dense operators for the coarse levels: Abar dense (problem i at aoff[i],
// leading dimension n_i); own generators are rows < nown[i] and B = X Abar X
// with X the indicator of the own rows (chi_{l,i} of Section 4.2).
void apply_dense_pencil(const double* Abar, const long long* d_aoff, const int* d_n, const int* d_nown,
                        const TileBatch& layout, const double* X, double* AX, double* BX, int ldx, int ncols,
                        const int* skip, int P, int nmax, cudaStream_t s);

}  // namespace msdd
