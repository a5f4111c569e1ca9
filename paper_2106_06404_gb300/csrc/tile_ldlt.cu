// Batched tile-band LDL^T factorisation and triangular solves (one CTA per
// local matrix).  See tile_ldlt.cuh for the storage format.
#include "tile_ldlt.cuh"

#include <cuda.h>
#include <cstring>
#include <mutex>
#include <type_traits>

namespace msdd {

namespace {

constexpr int TPB = 256;     // threads per CTA; each owns 4 entries of a 32 x 32 tile
constexpr int LDS = NB + 1;  // padded shared-memory row stride

template <typename T>
__device__ __forceinline__ void load_tile(T (*dst)[LDS], const T* __restrict__ src) {
    for (int e = threadIdx.x; e < NB2; e += TPB) dst[e / NB][e % NB] = src[e];
}

template <typename T>
__device__ __forceinline__ void store_tile(T* __restrict__ dst, T (*src)[LDS]) {
    for (int e = threadIdx.x; e < NB2; e += TPB) dst[e] = src[e / NB][e % NB];
}

// ------------------------------------------------------------------ factor
// Dense LDL^T of the diagonal tile R held in W (lower triangle; rows >=
// rows_valid are padding): pivots d with d <= reg_tol * od (the original
// diagonal) are null pivots (D^{-1} = 0, counted in s_nreg), other
// non-positive pivots set s_status to the first failing row + 1.  T_R =
// L_RR^{-1} (unit lower) is built in Sa and stored to Tdst, D^{-1} to ddst.
template <typename T>
__device__ void factor_diag_tile(T (*W)[LDS], T (*Sa)[LDS], T* sd, const T* od, T& piv_inv, int rows_valid,
                                 double reg_tol, int R, int& s_status, int& s_nreg, T* __restrict__ Tdst,
                                 T* __restrict__ ddst) {
    const int t = threadIdx.x;
    for (int k = 0; k < NB; ++k) {
        if (t == 0) {
            T d = W[k][k];
            T dinv_k;
            if (k >= rows_valid) {
                dinv_k = T(1);
            } else if (reg_tol > 0.0 && !(d > T(reg_tol) * od[k])) {
                dinv_k = T(0);
                ++s_nreg;
            } else if (!(d > T(0))) {
                dinv_k = T(0);
                if (s_status == 0) s_status = R * NB + k + 1;
            } else {
                dinv_k = T(1) / d;
            }
            piv_inv = dinv_k;
            sd[k] = dinv_k;
        }
        __syncthreads();
        const T pinv = piv_inv;
        // trailing update W[a][b] -= W[a][k] W[b][k] / d for k < b <= a
        for (int e = t; e < NB2; e += TPB) {
            int a = e / NB, b = e % NB;
            if (b > k && a >= b) W[a][b] -= W[a][k] * W[b][k] * pinv;
        }
        __syncthreads();
        if (t > k && t < NB) W[t][k] = (k >= rows_valid || t >= rows_valid) ? T(0) : W[t][k] * pinv;
        __syncthreads();
    }
    for (int e = t; e < NB2; e += TPB) Sa[e / NB][e % NB] = (e / NB == e % NB) ? T(1) : T(0);
    __syncthreads();
    for (int k = 0; k < NB - 1; ++k) {
        for (int e = t; e < NB2; e += TPB) {
            int a = e / NB, b = e % NB;
            if (a > k && b <= k) Sa[a][b] -= W[a][k] * Sa[k][b];
        }
        __syncthreads();
    }
    store_tile(Tdst, Sa);
    if (t < NB) ddst[t] = sd[t];
}

template <typename T>
__global__ void __launch_bounds__(TPB) k_tile_factor(
    T* __restrict__ tiles, T* __restrict__ dinv, const int* __restrict__ n_, const int* __restrict__ kb_,
    const int* __restrict__ K_, const long long* __restrict__ toff_, const long long* __restrict__ roff_,
    int* __restrict__ status, int* __restrict__ nreg, double reg_tol)
{
    __shared__ T W[NB][LDS];
    __shared__ T Sa[NB][LDS];
    __shared__ T Sb[NB][LDS];
    __shared__ T sd[NB];
    __shared__ T od[NB];
    __shared__ T piv_inv;
    __shared__ int s_status, s_nreg;

    const int i = blockIdx.x;
    const int n = n_[i], kb = kb_[i], K = K_[i];
    const long long toff = toff_[i], roff = roff_[i];
    const int t = threadIdx.x;
    const int r = t >> 3, c0 = t & 7;
    if (t == 0) { s_status = 0; s_nreg = 0; }

    for (int R = 0; R < K; ++R) {
        const int Cmin = R - kb > 0 ? R - kb : 0;
        for (int C = Cmin; C <= R; ++C) {
            __syncthreads();
            load_tile(W, tiles + tile_index(toff, kb, R, C));
            __syncthreads();
            if (C == R && t < NB) od[t] = W[t][t];
            // W -= sum_J L_RJ D_J L_CJ^T
            const int Jmin = (C - kb > Cmin) ? C - kb : Cmin;
            T acc[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[q] = W[r][c0 + 8 * q];
            for (int J = Jmin; J < C; ++J) {
                __syncthreads();
                load_tile(Sa, tiles + tile_index(toff, kb, R, J));
                load_tile(Sb, tiles + tile_index(toff, kb, C, J));
                if (t < NB) {
                    T di = dinv[roff + (long long)J * NB + t];
                    sd[t] = di != T(0) ? T(1) / di : T(0);
                }
                __syncthreads();
#pragma unroll 8
                for (int k = 0; k < NB; ++k) {
                    T a = Sa[r][k] * sd[k];
#pragma unroll
                    for (int q = 0; q < 4; ++q) acc[q] -= a * Sb[c0 + 8 * q][k];
                }
            }
            __syncthreads();
#pragma unroll
            for (int q = 0; q < 4; ++q) W[r][c0 + 8 * q] = acc[q];
            __syncthreads();
            if (C < R) {
                // L_RC = W T_C^T D_C^{-1}
                load_tile(Sb, tiles + tile_index(toff, kb, C, C));
                if (t < NB) sd[t] = dinv[roff + (long long)C * NB + t];
                __syncthreads();
                T out[4] = {0, 0, 0, 0};
#pragma unroll 8
                for (int k = 0; k < NB; ++k) {
                    T w = W[r][k];
#pragma unroll
                    for (int q = 0; q < 4; ++q) out[q] += w * Sb[c0 + 8 * q][k];
                }
                T* dst = tiles + tile_index(toff, kb, R, C);
#pragma unroll
                for (int q = 0; q < 4; ++q) dst[r * NB + c0 + 8 * q] = out[q] * sd[c0 + 8 * q];
            } else {
                factor_diag_tile<T>(W, Sa, sd, od, piv_inv, n - R * NB, reg_tol, R, s_status, s_nreg,
                                    tiles + tile_index(toff, kb, R, R), dinv + roff + (long long)R * NB);
            }
        }
    }
    __syncthreads();
    if (t == 0) { status[i] = s_status; nreg[i] = s_nreg; }
}

// ------------------------------------------------------------------ solve
// acc[r][c] for the 4 (row, column) pairs owned by a thread: row r = t>>3,
// columns c0 + 8q.
template <typename T, typename XT>
__global__ void __launch_bounds__(TPB) k_tile_solve(
    const T* __restrict__ tiles, const T* __restrict__ dinv, const int* __restrict__ n_,
    const int* __restrict__ kb_, const int* __restrict__ K_, const long long* __restrict__ toff_,
    const long long* __restrict__ roff_, XT* __restrict__ X, int ldx, int ncols,
    const int* __restrict__ skip, const int* __restrict__ gdone)
{
    __shared__ T Sa[NB][LDS];
    __shared__ T Sx[NB][LDS];   // operand block of X (rows x columns)
    __shared__ T Acc[NB][LDS];

    const int i = blockIdx.x;
    if (skip && skip[i]) return;
    if (gdone && *gdone) return;
    const int kb = kb_[i], K = K_[i];
    const long long toff = toff_[i], roff = roff_[i];
    const int t = threadIdx.x;
    const int r = t >> 3, c0 = t & 7;
    (void)n_;
    // this CTA handles the columns [32 * blockIdx.y, 32 * blockIdx.y + 32)
    const int c_lo = blockIdx.y * NB;
    X += c_lo;
    ncols = min(NB, ncols - c_lo);
    if (ncols <= 0) return;

    // forward: z_R = T_R (x_R - sum_J L_RJ z_J)
    for (int R = 0; R < K; ++R) {
        T acc[4];
        XT* xr = X + (roff + (long long)R * NB) * ldx;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            int c = c0 + 8 * q;
            acc[q] = c < ncols ? T(xr[(long long)r * ldx + c]) : T(0);
        }
        const int Jmin = R - kb > 0 ? R - kb : 0;
        for (int J = Jmin; J < R; ++J) {
            __syncthreads();
            load_tile(Sa, tiles + tile_index(toff, kb, R, J));
            const XT* xj = X + (roff + (long long)J * NB) * ldx;
            for (int e = t; e < NB * NB; e += TPB) {
                int a = e / NB, c = e % NB;
                Sx[a][c] = c < ncols ? T(xj[(long long)a * ldx + c]) : T(0);
            }
            __syncthreads();
#pragma unroll 8
            for (int k = 0; k < NB; ++k) {
                T l = Sa[r][k];
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[q] -= l * Sx[k][c0 + 8 * q];
            }
        }
        __syncthreads();
        load_tile(Sa, tiles + tile_index(toff, kb, R, R));
#pragma unroll
        for (int q = 0; q < 4; ++q) Acc[r][c0 + 8 * q] = acc[q];
        __syncthreads();
        T out[4] = {0, 0, 0, 0};
        for (int k = 0; k <= r; ++k) {
            T l = Sa[r][k];
#pragma unroll
            for (int q = 0; q < 4; ++q) out[q] += l * Acc[k][c0 + 8 * q];
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            int c = c0 + 8 * q;
            if (c < ncols) xr[(long long)r * ldx + c] = XT(out[q]);
        }
    }
    // backward: x_R = T_R^T (D_R^{-1} z_R - sum_I L_IR^T x_I)
    for (int R = K - 1; R >= 0; --R) {
        __syncthreads();
        T acc[4];
        XT* xr = X + (roff + (long long)R * NB) * ldx;
        const T dr = dinv[roff + (long long)R * NB + r];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            int c = c0 + 8 * q;
            acc[q] = c < ncols ? dr * T(xr[(long long)r * ldx + c]) : T(0);
        }
        const int Imax = R + kb < K - 1 ? R + kb : K - 1;
        for (int I = R + 1; I <= Imax; ++I) {
            __syncthreads();
            load_tile(Sa, tiles + tile_index(toff, kb, I, R));
            const XT* xi = X + (roff + (long long)I * NB) * ldx;
            for (int e = t; e < NB * NB; e += TPB) {
                int a = e / NB, c = e % NB;
                Sx[a][c] = c < ncols ? T(xi[(long long)a * ldx + c]) : T(0);
            }
            __syncthreads();
#pragma unroll 8
            for (int k = 0; k < NB; ++k) {
                T l = Sa[k][r];
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[q] -= l * Sx[k][c0 + 8 * q];
            }
        }
        __syncthreads();
        load_tile(Sa, tiles + tile_index(toff, kb, R, R));
#pragma unroll
        for (int q = 0; q < 4; ++q) Acc[r][c0 + 8 * q] = acc[q];
        __syncthreads();
        T out[4] = {0, 0, 0, 0};
        for (int k = r; k < NB; ++k) {
            T l = Sa[k][r];
#pragma unroll
            for (int q = 0; q < 4; ++q) out[q] += l * Acc[k][c0 + 8 * q];
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            int c = c0 + 8 * q;
            if (c < ncols) xr[(long long)r * ldx + c] = XT(out[q]);
        }
    }
}


// ------------------------------------------------------------------ factor, right-looking
// Dense batches (coarse-level matrices) and FP64 bands are factored one tile
// column k per launch triple, so that many CTAs share each step instead of
// one CTA per matrix: the diagonal tile (one CTA per problem), the panel
// L_ik = A_ik T_k^T D_k^{-1} (one CTA per tile), and the trailing update
// A_ij -= L_ik D_k L_jk^T for k < j <= i <= k + kb (one CTA per tile).  In
// FP64 the pipe bounds the panel and the update, so both skip the zeros: T_k
// is lower triangular, and columns below 32 (i - k) - b of tile (i, k) lie
// outside the band.  k_save_diag first parks the original diagonal (the
// null-pivot reference) in dinv and clears the status.
// Measured (GB300, Dirichlet and Neumann batches side by side): 27 FP64
// matrices of n = 1452..1872, b = 133..157 17.1 -> 4.5 ms a factorisation
// against one CTA per matrix, 144 of n ~ 1300, b = 36 6.0 -> 3.7 ms.
template <typename T>
__global__ void __launch_bounds__(TPB) k_save_diag(const T* __restrict__ tiles, T* __restrict__ dinv,
                                                   const int* __restrict__ kb_, const int* __restrict__ K_,
                                                   const long long* __restrict__ toff_,
                                                   const long long* __restrict__ roff_, int* __restrict__ status,
                                                   int* __restrict__ nreg) {
    const int i = blockIdx.x;
    const int kb = kb_[i], K = K_[i];
    const long long toff = toff_[i], roff = roff_[i];
    for (int e = threadIdx.x; e < K * NB; e += TPB) {
        const int R = e / NB, r = e % NB;
        dinv[roff + e] = tiles[tile_index(toff, kb, R, R) + r * NB + r];
    }
    if (threadIdx.x == 0) { status[i] = 0; nreg[i] = 0; }
}

// LDL^T of the diagonal tile and T = L^{-1} in one elimination of [A | I]:
// lane = row, warp w holds columns w + 4 j of both in registers.  Step k: the
// warp that owns column k publishes it and the reciprocal pivot (shared
// memory, one barrier); with m_a = A_ak / d_k, entry (a, b) of A takes off
// A_ak m_b (columns b > k, m_b by shuffle from lane b) and of T m_a T_kb
// (columns b <= k, T_kb by shuffle from lane k).  The 32 pivots are the chain (a division, a barrier and
// about eight FP64 operations of every warp each), so one barrier a pivot
// instead of three, and the inverse in the same pass instead of a second one.
template <typename T>
__global__ void __launch_bounds__(128) k_rl_diag(T* __restrict__ tiles, T* __restrict__ dinv,
                                                 const int* __restrict__ n_, const int* __restrict__ kb_,
                                                 const int* __restrict__ K_, const long long* __restrict__ toff_,
                                                 const long long* __restrict__ roff_, int* __restrict__ status,
                                                 int* __restrict__ nreg, double reg_tol, int k0) {
    __shared__ T S[NB][LDS];
    __shared__ T col[2][NB], piv[2], sd[NB], od[NB];
    __shared__ int s_status, s_nreg;
    const int i = blockIdx.x;
    if (k0 >= K_[i]) return;
    const int kb = kb_[i], t = threadIdx.x, a = t & 31, w = t >> 5;
    T* tile = tiles + tile_index(toff_[i], kb, k0, k0);
    T* dv = dinv + roff_[i] + (long long)k0 * NB;
    const int valid = n_[i] - k0 * NB;                 // rows from here on are padding
    if (t == 0) { s_status = status[i]; s_nreg = nreg[i]; }
    for (int e = t; e < NB2; e += 128) S[e / NB][e % NB] = tile[e];
    if (t < NB) od[t] = dv[t];
    __syncthreads();
    T A[NB / 4], L[NB / 4];
#pragma unroll
    for (int j = 0; j < NB / 4; ++j) {
        const int b = w + 4 * j;
        A[j] = S[a][b];
        L[j] = a == b ? T(1) : T(0);
    }
#pragma unroll
    for (int k = 0; k < NB; ++k) {
        const int buf = k & 1;
        if (w == (k & 3)) {
            const T v = A[k >> 2];
            col[buf][a] = v;
            if (a == k) {
                T r;
                if (k >= valid) r = T(1);
                else if (reg_tol > 0.0 && !(v > T(reg_tol) * od[k])) { r = T(0); ++s_nreg; }
                else if (!(v > T(0))) { r = T(0); if (s_status == 0) s_status = k0 * NB + k + 1; }
                else r = T(1) / v;
                piv[buf] = r;
                sd[k] = r;
            }
        }
        __syncthreads();
        const T m = a > k && a < valid && k < valid ? col[buf][a] * piv[buf] : T(0);
#pragma unroll
        for (int j = 0; j < NB / 4; ++j) {
            const int b = w + 4 * j;                   // (the same side of k for the whole warp)
            if (4 * j + 3 > k && b > k) A[j] -= col[buf][a] * __shfl_sync(0xffffffffu, m, b);
            if (4 * j <= k && b <= k) L[j] -= m * __shfl_sync(0xffffffffu, L[j], k);
        }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < NB / 4; ++j) S[a][w + 4 * j] = L[j];
    __syncthreads();
    for (int e = t; e < NB2; e += 128) tile[e] = S[e / NB][e % NB];
    if (t < NB) dv[t] = sd[t];
    if (t == 0) { status[i] = s_status; nreg[i] = s_nreg; }
}

// grid.y: tile row k + 1 + blockIdx.y
template <typename T>
__global__ void __launch_bounds__(TPB) k_rl_panel(T* __restrict__ tiles, const T* __restrict__ dinv,
                                                  const int* __restrict__ kb_, const int* __restrict__ K_,
                                                  const int* __restrict__ b_, const long long* __restrict__ toff_,
                                                  const long long* __restrict__ roff_, int k) {
    __shared__ T W[NB][LDS];
    __shared__ T Sb[NB][LDS];
    __shared__ T sd[NB];
    const int i = blockIdx.x, d = 1 + blockIdx.y, R = k + d;
    const int kb = kb_[i];
    if (R >= K_[i] || d > kb) return;
    const int t = threadIdx.x, r = t >> 3, c0 = t & 7;
    const long long toff = toff_[i], roff = roff_[i];
    T* dst = tiles + tile_index(toff, kb, R, k);
    load_tile(W, dst);
    load_tile(Sb, tiles + tile_index(toff, kb, k, k));
    if (t < NB) sd[t] = dinv[roff + (long long)k * NB + t];
    __syncthreads();
    const int kk0 = max(0, NB * d - b_[i]) & ~7;       // columns of A_Rk before it are zero
    T out[4] = {0, 0, 0, 0};
#pragma unroll
    for (int g = 0; g < 4; ++g) {                      // columns 8 g .. 8 g + 7 of A reach the rows >= 8 g of T
        if (8 * g < kk0) continue;
#pragma unroll
        for (int kk = 8 * g; kk < 8 * g + 8; ++kk) {
            const T w = W[r][kk];
#pragma unroll
            for (int q = g; q < 4; ++q) out[q] += w * Sb[c0 + 8 * q][kk];
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) dst[r * NB + c0 + 8 * q] = out[q] * sd[c0 + 8 * q];
}

// grid.y, continued in grid.z beyond its 65535 blocks (kb > 361), enumerates
// the tiles (R, C), k < C <= R <= k + kb, row by row
template <typename T>
__global__ void __launch_bounds__(TPB) k_rl_update(T* __restrict__ tiles, const T* __restrict__ dinv,
                                                   const int* __restrict__ kb_, const int* __restrict__ K_,
                                                   const int* __restrict__ b_, const long long* __restrict__ toff_,
                                                   const long long* __restrict__ roff_, int k) {
    __shared__ T Sa[NB][LDS];
    __shared__ T Sb[NB][LDS];
    __shared__ T sd[NB];
    const int i = blockIdx.x;
    const int K = K_[i], kb = kb_[i];
    int e = blockIdx.y + blockIdx.z * gridDim.y, R = k + 1;
    while (R < K && e >= R - k) { e -= R - k; ++R; }
    if (R >= K || R - k > kb) return;
    const int C = k + 1 + e;
    const int t = threadIdx.x, r = t >> 3, c0 = t & 7;
    const long long toff = toff_[i], roff = roff_[i];
    T* dst = tiles + tile_index(toff, kb, R, C);
    T acc[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[q] = dst[r * NB + c0 + 8 * q];
    if (t < NB) {
        T di = dinv[roff + (long long)k * NB + t];
        sd[t] = di != T(0) ? T(1) / di : T(0);
    }
    load_tile(Sa, tiles + tile_index(toff, kb, R, k));
    const T* lb = tiles + tile_index(toff, kb, C, k);
    __syncthreads();
    for (int x = t; x < NB2; x += TPB) Sb[x / NB][x % NB] = lb[x] * sd[x % NB];   // L_Ck D_k
    __syncthreads();
    const int kk0 = max(0, NB * (R - k) - b_[i]);      // columns of L_Rk before it are zero
    // a warp has rows r .. r + 3; of a diagonal tile the column groups beyond them are not stored
    const int nq = R == C ? (4 * (t >> 5) + 3) / 8 + 1 : 4;
    if (nq == 4) {
#pragma unroll 4
        for (int kk = kk0; kk < NB; ++kk) {
            const T a = Sa[r][kk];
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[q] -= a * Sb[c0 + 8 * q][kk];
        }
    } else {
        for (int kk = kk0; kk < NB; ++kk) {
            const T a = Sa[r][kk];
            acc[0] -= a * Sb[c0][kk];
            if (nq > 1) acc[1] -= a * Sb[c0 + 8][kk];
            if (nq > 2) acc[2] -= a * Sb[c0 + 16][kk];
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) dst[r * NB + c0 + 8 * q] = acc[q];
}

// ------------------------------------------------------------------ factor, FP32, half-bandwidth <= 2 tiles
// The steps and the arithmetic of k_tile_factor<float> (same expressions in
// the same order), arranged for latency: the tiles of the last three tile
// rows (L, T and the pivots) stay in shared memory, so nothing the CTA
// produced is read back from global memory; the original tiles of row R + 1
// are copied with cp.async while row R is factored; the diagonal tiles are
// factored and inverted by one warp holding a row per lane in registers
// (shuffles instead of block barriers).
constexpr int FB_T = 256, FB_LD = NB + 1, FB_ROWS = 3;
constexpr size_t factor_band32_smem() {
    return sizeof(float) * ((size_t)2 * FB_ROWS * NB2 + (size_t)FB_ROWS * FB_ROWS * NB * FB_LD + (size_t)NB * FB_LD +
                            (size_t)2 * FB_ROWS * NB + NB) + 16;
}

__global__ void __launch_bounds__(FB_T) k_tile_factor_band32(
    float* __restrict__ tiles, float* __restrict__ dinv, const int* __restrict__ n_, const int* __restrict__ kb_,
    const int* __restrict__ K_, const long long* __restrict__ toff_, const long long* __restrict__ roff_,
    int* __restrict__ status, int* __restrict__ nreg, double reg_tol)
{
    extern __shared__ __align__(16) float fb_sm[];
    float* stg = fb_sm;                                                          // [2][3][32*32] original tiles
    float (*cache)[NB][FB_LD] = reinterpret_cast<float (*)[NB][FB_LD]>(stg + 2 * FB_ROWS * NB2);  // [row%3 * 3 + d]
    float (*Wsm)[FB_LD] = reinterpret_cast<float (*)[FB_LD]>(&cache[FB_ROWS * FB_ROWS][0][0]);
    float* cpiv = &Wsm[NB][0];                                                   // [3][32] D = 1 / D^{-1}
    float* cdinv = cpiv + FB_ROWS * NB;                                          // [3][32] D^{-1}
    float* od = cdinv + FB_ROWS * NB;                                            // original diagonal
    __shared__ int s_status, s_nreg;

    const int i = blockIdx.x;
    const int n = n_[i], kb = kb_[i], K = K_[i];
    const long long toff = toff_[i], roff = roff_[i];
    const int t = threadIdx.x;
    const int r = t >> 3, c0 = t & 7;
    if (t == 0) { s_status = 0; s_nreg = 0; }
    auto issue_row = [&](int R) {
        if (R < K) {
            const int Cmin = R - kb > 0 ? R - kb : 0;
            for (int C = Cmin; C <= R; ++C) {
                const float* src = tiles + tile_index(toff, kb, R, C);
                float* dst = stg + ((R & 1) * FB_ROWS + (R - C)) * NB2;
                for (int ch = t; ch < NB2 / 4; ch += FB_T) cp_async16(dst + ch * 4, src + ch * 4);
            }
        }
        cp_async_commit();
    };
    issue_row(0);
    for (int R = 0; R < K; ++R) {
        issue_row(R + 1);
        cp_async_wait_n<1>();                       // row R landed (row R + 1 may be in flight)
        __syncthreads();
        const int Cmin = R - kb > 0 ? R - kb : 0;
        const int rs = R % FB_ROWS;
        for (int C = Cmin; C <= R; ++C) {
            __syncthreads();                        // the previous step's cache and Wsm accesses are done
            const float* A = stg + ((R & 1) * FB_ROWS + (R - C)) * NB2;
            if (C == R && t < NB) od[t] = A[t * NB + t];
            float acc[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[q] = A[r * NB + c0 + 8 * q];
            // W -= sum_J L_RJ D_J L_CJ^T
            for (int J = Cmin; J < C; ++J) {
                const float (*LR)[FB_LD] = cache[rs * FB_ROWS + (R - J)];
                const float (*LC)[FB_LD] = cache[(C % FB_ROWS) * FB_ROWS + (C - J)];
                const float* Dj = cpiv + (J % FB_ROWS) * NB;
#pragma unroll 8
                for (int k = 0; k < NB; ++k) {
                    const float a = LR[r][k] * Dj[k];
#pragma unroll
                    for (int q = 0; q < 4; ++q) acc[q] -= a * LC[c0 + 8 * q][k];
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) Wsm[r][c0 + 8 * q] = acc[q];
            __syncthreads();
            if (C < R) {
                // L_RC = W T_C^T D_C^{-1}
                const float (*TC)[FB_LD] = cache[(C % FB_ROWS) * FB_ROWS];
                const float* dC = cdinv + (C % FB_ROWS) * NB;
                float out[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
                for (int k = 0; k < NB; ++k) {
                    const float w = Wsm[r][k];
#pragma unroll
                    for (int q = 0; q < 4; ++q) out[q] += w * TC[c0 + 8 * q][k];
                }
                float* dst = tiles + tile_index(toff, kb, R, C);
                float (*Lc)[FB_LD] = cache[rs * FB_ROWS + (R - C)];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float v = out[q] * dC[c0 + 8 * q];
                    Lc[r][c0 + 8 * q] = v;
                    dst[r * NB + c0 + 8 * q] = v;
                }
            } else if (t < 32) {
                // dense LDL^T of the diagonal tile by warp 0, lane a holding
                // row a of W in registers (W[b][k] by shuffle from lane b);
                // then T_R = L_RR^{-1}, lane a building row a of T
                const int lane = t;
                const int rows_valid = n - R * NB;
                float row[NB];
#pragma unroll
                for (int b = 0; b < NB; ++b) row[b] = Wsm[lane][b];
                float dl = 0.f;                     // D^{-1} of this lane's row
                int nr = 0, st = 0;
#pragma unroll
                for (int k = 0; k < NB; ++k) {
                    const float d = __shfl_sync(0xffffffffu, row[k], k);
                    float dinv_k;
                    if (k >= rows_valid) {
                        dinv_k = 1.f;
                    } else if (reg_tol > 0.0 && !(d > (float)reg_tol * od[k])) {
                        dinv_k = 0.f;
                        ++nr;
                    } else if (!(d > 0.f)) {
                        dinv_k = 0.f;
                        if (st == 0) st = R * NB + k + 1;
                    } else {
                        dinv_k = 1.f / d;
                    }
                    if (lane == k) dl = dinv_k;
                    const float pinv = dinv_k;
                    const float wak = row[k];
                    // W[a][b] -= W[a][k] W[b][k] / d for k < b <= a
#pragma unroll
                    for (int b = 0; b < NB; ++b) {
                        if (b > k) {
                            const float wbk = __shfl_sync(0xffffffffu, wak, b);
                            if (lane >= b) row[b] -= wak * wbk * pinv;
                        }
                    }
                    if (lane > k) row[k] = (k >= rows_valid || lane >= rows_valid) ? 0.f : wak * pinv;
                }
                float tr[NB];
#pragma unroll
                for (int b = 0; b < NB; ++b) tr[b] = (b == lane) ? 1.f : 0.f;
#pragma unroll
                for (int k = 0; k < NB - 1; ++k) {
                    const float lak = row[k];
#pragma unroll
                    for (int b = 0; b < NB; ++b) {
                        if (b <= k) {
                            const float tkb = __shfl_sync(0xffffffffu, tr[b], k);
                            if (lane > k) tr[b] -= lak * tkb;
                        }
                    }
                }
                float* dst = tiles + tile_index(toff, kb, R, R);
                float (*Tc)[FB_LD] = cache[rs * FB_ROWS];
#pragma unroll
                for (int b = 0; b < NB; ++b) {
                    Tc[lane][b] = tr[b];
                    dst[lane * NB + b] = tr[b];
                }
                cdinv[rs * NB + lane] = dl;
                cpiv[rs * NB + lane] = dl != 0.f ? 1.f / dl : 0.f;
                dinv[roff + (long long)R * NB + lane] = dl;
                if (lane == 0) { s_nreg += nr; if (s_status == 0 && st != 0) s_status = st; }
            }
        }
        __syncthreads();                            // row R complete before its stage is refilled
    }
    cp_async_wait_n<0>();
    __syncthreads();
    if (t == 0) { status[i] = s_status; nreg[i] = s_nreg; }
}

constexpr int S1T = 128;

// One right-hand side where the streamed kernels below do not fit (very wide
// bands, dense matrices) or keep too few CTAs on an SM (large batches of wide FP64
// bands): tiles are read as needed without prefetch.
template <typename T>
__global__ void __launch_bounds__(S1T) k_tile_solve1_dense(
    const T* __restrict__ tiles, const T* __restrict__ dinv, const int* __restrict__ kb_, const int* __restrict__ K_,
    const long long* __restrict__ toff_, const long long* __restrict__ roff_, double* __restrict__ X,
    const int* __restrict__ gdone)
{
    extern __shared__ double zs[];
    __shared__ double accs[NB];
    __shared__ double part[S1T / 32][NB + 1];
    if (gdone && *gdone) return;
    const int i = blockIdx.x;
    const int kb = kb_[i], K = K_[i];
    const long long toff = toff_[i], roff = roff_[i];
    const int t = threadIdx.x;
    for (int e = t; e < K * NB; e += S1T) zs[e] = X[roff + e];
    __syncthreads();
    {
        const int r = t >> 2, c0 = (t & 3) * 8;
        for (int R = 0; R < K; ++R) {
            double acc = 0.0;
            for (int J = (R - kb > 0 ? R - kb : 0); J < R; ++J) {
                const T* src = tiles + tile_index(toff, kb, R, J) + r * NB + c0;
                const double* zj = zs + J * NB + c0;
#pragma unroll
                for (int q = 0; q < 8; ++q) acc += (double)src[q] * zj[q];
            }
            acc += __shfl_xor_sync(0xffffffffu, acc, 1);
            acc += __shfl_xor_sync(0xffffffffu, acc, 2);
            if ((t & 3) == 0) accs[r] = zs[R * NB + r] - acc;
            __syncthreads();
            const T* tr = tiles + tile_index(toff, kb, R, R) + r * NB + c0;
            double s = 0.0;
#pragma unroll
            for (int q = 0; q < 8; ++q) s += (double)tr[q] * accs[c0 + q];
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            s += __shfl_xor_sync(0xffffffffu, s, 2);
            if ((t & 3) == 0) zs[R * NB + r] = s;
            __syncthreads();
        }
    }
    for (int e = t; e < K * NB; e += S1T) zs[e] *= (double)dinv[roff + e];
    __syncthreads();
    {
        const int lane = t & 31, warp = t >> 5, k0 = warp * 8;
        for (int R = K - 1; R >= 0; --R) {
            double s = 0.0;
            const int Imax = R + kb < K - 1 ? R + kb : K - 1;
            for (int I = R + 1; I <= Imax; ++I) {
                const T* src = tiles + tile_index(toff, kb, I, R);
                const double* xi = zs + I * NB + k0;
#pragma unroll
                for (int q = 0; q < 8; ++q) s += (double)src[(k0 + q) * NB + lane] * xi[q];
            }
            part[warp][lane] = s;
            __syncthreads();
            if (warp == 0) {
                double v = 0.0;
#pragma unroll
                for (int w = 0; w < S1T / 32; ++w) v += part[w][lane];
                accs[lane] = zs[R * NB + lane] - v;
            }
            __syncthreads();
            const T* tr = tiles + tile_index(toff, kb, R, R);
            double s2 = 0.0;
#pragma unroll
            for (int q = 0; q < 8; ++q) s2 += (double)tr[(k0 + q) * NB + lane] * accs[k0 + q];
            part[warp][lane] = s2;
            __syncthreads();
            if (warp == 0) {
                double v = 0.0;
#pragma unroll
                for (int w = 0; w < S1T / 32; ++w) v += part[w][lane];
                zs[R * NB + lane] = v;
            }
            __syncthreads();
        }
    }
    for (int e = t; e < K * NB; e += S1T) X[roff + e] = zs[e];
}


// ---- TMA / mbarrier helpers of the FP32 band solve.  Every mbarrier wait is
// bounded; a kernel whose wait runs out records it in g_wait_timeouts.
__device__ int g_wait_timeouts;

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
constexpr long long kWaitTries = 1LL << 22;
__device__ __forceinline__ bool mbar_wait_bounded(unsigned long long* bar, unsigned parity) {
    for (long long k = 0; k < kWaitTries; ++k)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}
__device__ __forceinline__ void tma_load_tile(void* dst, const CUtensorMap* map, int row, unsigned long long* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n" ::"r"(
            smem_u32(dst)),
        "l"(map), "r"(0), "r"(row), "r"(smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ void bulk_load(void* dst, const void* src, unsigned bytes, unsigned long long* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory"); }

// ---- FP32 band LDL^T with the panel updates on the tensor cores (3 <= kb <= 12)
// Left-looking by tile column C, one CTA (one warpgroup) per matrix.  The
// update of column C,
//   U_R = sum_{J} L_RJ D_J L_CJ^T,  R = C .. min(C + kb, K - 1),
//   J = max(C - kb, R - kb) .. C - 1,
// is a product D = A B^T with A = [L_RJ] (tile rows R stacked, 128-row
// blocks of four tile rows, tiles outside the band zero) and
// B = [L_CJ D_J] (32 x 32 per J), done by tcgen05.mma kind::tf32 into a
// TMEM accumulator (four 128 x 32 FP32 blocks).  FP32 accuracy from TF32
// operands by the three-product split x = hi + lo, hi = x with the low 13
// mantissa bits cleared: A_hi B_hi + A_hi B_lo + A_lo B_hi (the lo * lo
// term is below FP32 rounding).  The tensor cores of this GPU take a
// kind::tf32 operand as its top 19 bits (truncation, measured), so the FP32
// L tiles themselves serve as hi parts, and lo = x - hi of each L tile is
// written once, when the tile is computed, to a scratch array.  The A
// operands (hi from the tiles, lo from the scratch) are streamed by TMA
// (3-stage ring, one pair (block, J) per stage, tiles outside the band read
// as zeros from out-of-range coordinates); the B operands are scaled by D_J
// and split in shared memory.  Then, as in
// k_tile_factor: W_RC = A_RC - U_R, the diagonal tile is factored and
// inverted by warp 0 in registers (null pivots as there), and
// L_RC = W_RC T_C^T D_C^{-1}.  Operands are K-major with the 128-byte
// swizzle (row r of a tile at 128 r bytes, 16-byte chunk g at g ^ (r & 7)),
// descriptors: start >> 4, stride between 8-row groups 1024 B, the K step
// of 8 elements advances the start by 32 B.
constexpr int TF_NT = 128, TF_KBM = 12, TF_NS = 3;
constexpr int TF_MAXPAIRS = TF_KBM * ((TF_KBM + 1 + 3) / 4);
constexpr size_t tf_smem_bytes() {
    return 1024 + (size_t)TF_NS * 8 * NB2 * 4            // A stages: 4 hi + 4 lo tiles
           + (size_t)TF_KBM * 2 * NB2 * 4                // B_J hi and lo
           + (size_t)NB2 * 4 + NB * 4                    // T_C, D_C^{-1}
           + (size_t)TF_KBM * NB * 4                     // D_J of the B operands
           + 64 * (TF_NS * 2 + 3) + TF_MAXPAIRS * 4 + 64;
}

__device__ __forceinline__ float tf32_hi(float x) { return __uint_as_float(__float_as_uint(x) & 0xffffe000u); }

__device__ __forceinline__ uint64_t umma_desc_sw128(unsigned saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);          // start address
    d |= (uint64_t)1 << 16;                             // leading byte offset (unused: K-major, 128 B rows)
    d |= (uint64_t)(1024 >> 4) << 32;                   // stride byte offset: 8 rows x 128 B
    d |= (uint64_t)1 << 46;                             // descriptor version
    d |= (uint64_t)2 << 61;                             // 128-byte swizzle
    return d;
}
__device__ __forceinline__ void umma_tf32(unsigned tmem, uint64_t a, uint64_t b, unsigned idesc, unsigned acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}
__device__ __forceinline__ void umma_commit(unsigned long long* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void tmem_ld32(unsigned taddr, float (&v)[32]) {
    unsigned r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,"
        "%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int k = 0; k < 32; ++k) v[k] = __uint_as_float(r[k]);
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async_global() { asm volatile("fence.proxy.async.global;\n" ::: "memory"); }

// lo: E floats (E = total tile elements), lo parts of the L tiles in the tile layout;
// tm_hi / tm_lo: [E / 32][32] tensor maps of the tiles and of lo
__global__ void __launch_bounds__(TF_NT) k_tile_factor_tc(
    const __grid_constant__ CUtensorMap tm_hi, const __grid_constant__ CUtensorMap tm_lo, float* __restrict__ tiles,
    float* __restrict__ lo, long long total_elems, float* __restrict__ dinv, const int* __restrict__ n_, const int* __restrict__ kb_,
    const int* __restrict__ K_, const long long* __restrict__ toff_, const long long* __restrict__ roff_,
    int* __restrict__ status, int* __restrict__ nreg, double reg_tol)
{
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    float* Ast = reinterpret_cast<float*>(base);                                   // [NS][8][1024]
    float* Bst = Ast + (size_t)TF_NS * 8 * NB2;                                     // [KBM][2][1024]
    float* Tc = Bst + (size_t)TF_KBM * 2 * NB2;                                     // [32][32]
    float* Dc = Tc + NB2;                                                           // [32]
    float* Dj = Dc + NB;                                                            // [KBM][32]
    unsigned long long* bars = reinterpret_cast<unsigned long long*>(Dj + TF_KBM * NB);  // full[NS], empty[NS], acc, b
    unsigned long long* full = bars;
    unsigned long long* empty = bars + TF_NS;
    unsigned long long* accb = bars + 2 * TF_NS;
    unsigned long long* bfull = bars + 2 * TF_NS + 1;
    int* pairs = reinterpret_cast<int*>(bars + 2 * TF_NS + 3);                     // (J << 8) | mb
    __shared__ unsigned s_tmem;
    __shared__ int s_status, s_nreg, s_abort, s_npairs, s_used;

    const int i = blockIdx.x;
    const int n = n_[i], kb = kb_[i], K = K_[i];
    const long long toff = toff_[i], roff = roff_[i];
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    if (kb > TF_KBM) {                                  // never launched so (host dispatch)
        if (t == 0) status[i] = -1;
        return;
    }
    const int oob_row = (int)(total_elems / NB);        // first row beyond both tensors: zero fill
    if (t == 0) {
        s_status = 0; s_nreg = 0; s_abort = 0;
        for (int s = 0; s < TF_NS; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        mbar_init(accb, 1);
        mbar_init(bfull, 1);
        fence_mbar_init();
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 128;\n" ::"r"(smem_u32(&s_tmem)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem = s_tmem;
    // D f32, A and B tf32, both K-major, N = 32, M = 128
    const unsigned idesc = (1u << 4) | (2u << 7) | (2u << 10) | ((32u >> 3) << 17) | ((128u >> 4) << 24);
    // parity bits: ph_full (product thread), ph_empty and par_issued (copy
    // thread), ph_acc (all threads); pair_base counts the ring's pairs so far
    unsigned ph_full = 0, ph_empty = 0, ph_acc = 0, par_issued = 0, ph_b = 0;
    int pair_base = 0;

    auto issue_pair = [&](int C, int Rend, int pr, int stage) {
        // A operand tiles of pair (J, mb): hi into slots 0..3, lo into 4..7
        const int J = pr >> 8, mb = pr & 0xff;
        float* dst = Ast + (size_t)stage * 8 * NB2;
        mbar_expect_tx(&full[stage], 8 * NB2 * 4);
        for (int q = 0; q < 4; ++q) {
            const int R = C + 4 * mb + q;
            const bool valid = R <= Rend && R - J <= kb;
            const long long ti = valid ? tile_index(toff, kb, R, J) : 0;
            const int row = valid ? (int)(ti / NB) : oob_row;
            tma_load_tile(dst + (size_t)q * NB2, &tm_hi, row, &full[stage]);
            tma_load_tile(dst + (size_t)(4 + q) * NB2, &tm_lo, row, &full[stage]);
        }
    };

    for (int C = 0; C < K && !s_abort; ++C) {
        const int Rend = min(C + kb, K - 1);
        const int J0 = max(0, C - kb);
        const int nJ = C - J0;
        const int nmb = (Rend - C + 1 + 3) / 4;
        // ---- pair list and B operands: B_J[n][j] = L_CJ[n][j] * D_J[j], split
        if (t == 0) {
            int np = 0, used = 0;
            for (int J = J0; J < C; ++J)
                for (int mb = 0; mb < nmb; ++mb) {
                    const int R0 = C + 4 * mb;
                    if (R0 <= Rend && R0 - J <= kb) {       // the block's first row has the most J's
                        pairs[np++] = (J << 8) | mb;
                        used |= 1 << mb;
                    }
                }
            s_npairs = np;
            s_used = used;
        }
        // raw tiles L_CJ by TMA into the lo slots, D_J into shared memory
        if (t == 32 && nJ > 0) {
            mbar_expect_tx(bfull, nJ * NB2 * 4);
            for (int jj = 0; jj < nJ; ++jj)
                tma_load_tile(Bst + (size_t)(2 * jj + 1) * NB2, &tm_hi,
                              (int)(tile_index(toff, kb, C, J0 + jj) / NB), bfull);
        }
        for (int e = t; e < nJ * NB; e += TF_NT) {
            const float di = dinv[roff + (long long)J0 * NB + e];
            Dj[e] = di != 0.f ? 1.f / di : 0.f;
        }
        __syncthreads();
        if (nJ > 0) {
            if (!mbar_wait_bounded(bfull, ph_b & 1u)) {
                if (atomicExch(&s_abort, 1) == 0) atomicAdd(&g_wait_timeouts, 1);
            } else {
                ph_b ^= 1u;
            }
        }
        for (int e = t; e < nJ * NB2; e += TF_NT) {
            // element (r, c) of tile jj; the same swizzled position in both slots
            const int jj = e / NB2, w = e % NB2, r = w / NB, c = w % NB;
            const int sidx = r * NB + ((((c >> 2) ^ (r & 7))) << 2) + (c & 3);
            float* lo_slot = Bst + (size_t)(2 * jj + 1) * NB2;
            const float b = lo_slot[sidx] * Dj[jj * NB + c];
            const float hi = tf32_hi(b);
            Bst[(size_t)(2 * jj) * NB2 + sidx] = hi;
            lo_slot[sidx] = b - hi;
        }
        fence_proxy_async_smem();
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        const int np = s_npairs, used = s_used;
        // ---- tensor-core update: lane 0 of warp 1 streams the A operands into the
        // ring, lane 0 of warp 0 issues the products (each side waits only for
        // the other: "full" when a stage's copies landed, "empty" when the
        // products that read a stage are done)
        if (t == 32 && np > 0) {
            for (int p = 0; p < np; ++p) {
                const int g = pair_base + p, st = g % TF_NS;
                if (g >= TF_NS) {
                    if (!mbar_wait_bounded(&empty[st], (ph_empty >> st) & 1u)) {
                        if (atomicExch(&s_abort, 1) == 0) atomicAdd(&g_wait_timeouts, 1);
                        break;
                    }
                    ph_empty ^= 1u << st;
                }
                if (*(volatile int*)&s_abort) break;
                issue_pair(C, Rend, pairs[p], st);
                par_issued = (par_issued & ~(1u << st)) | ((unsigned)((g / TF_NS) & 1) << st);
            }
        }
        if (t == 0 && np > 0) {
            unsigned started = 0;                       // M-blocks whose accumulator has been started
            for (int p = 0; p < np; ++p) {
                const int g = pair_base + p, st = g % TF_NS;
                if (!mbar_wait_bounded(&full[st], (ph_full >> st) & 1u)) {
                    if (atomicExch(&s_abort, 1) == 0) atomicAdd(&g_wait_timeouts, 1);
                    break;
                }
                ph_full ^= 1u << st;
                tc_fence_after();
                const int J = pairs[p] >> 8, mb = pairs[p] & 0xff, jj = J - J0;
                const unsigned a_hi = smem_u32(Ast + (size_t)st * 8 * NB2), a_lo = a_hi + 4 * NB2 * 4;
                const unsigned b_hi = smem_u32(Bst + (size_t)(2 * jj) * NB2), b_lo = b_hi + NB2 * 4;
                const unsigned d = tmem + 32u * mb;
                for (int k = 0; k < 4; ++k) {
                    const unsigned ko = 32u * k;
                    const unsigned acc = (started >> mb) & 1u;
                    umma_tf32(d, umma_desc_sw128(a_hi + ko), umma_desc_sw128(b_hi + ko), idesc, acc);
                    started |= 1u << mb;
                    umma_tf32(d, umma_desc_sw128(a_hi + ko), umma_desc_sw128(b_lo + ko), idesc, 1u);
                    umma_tf32(d, umma_desc_sw128(a_lo + ko), umma_desc_sw128(b_hi + ko), idesc, 1u);
                }
                umma_commit(&empty[st]);                // the stage is free once these products are done
            }
            umma_commit(accb);
        }
        pair_base += np;
        __syncthreads();
        if (s_abort) break;
        // ---- W_RC = A_RC - U_R for the rows of this thread: tile row C + 4 mb + warp, row lane
        if (np > 0) {
            if (!mbar_wait_bounded(accb, ph_acc & 1u)) {
                if (atomicExch(&s_abort, 1) == 0) atomicAdd(&g_wait_timeouts, 1);
            } else {
                ph_acc ^= 1u;                           // (on a timeout the phase stays pending)
            }
        }
        tc_fence_after();
        __syncthreads();
        if (s_abort) break;
        float w[4][NB];
#pragma unroll
        for (int mb = 0; mb < 4; ++mb) {
            const int R = C + 4 * mb + warp;
            if (mb < nmb && ((used >> mb) & 1)) {
                float u[NB];
                tmem_ld32(tmem + ((unsigned)(32 * warp) << 16) + 32u * mb, u);
                if (R <= Rend) {
                    const float* a = tiles + tile_index(toff, kb, R, C) + lane * NB;
#pragma unroll
                    for (int c = 0; c < NB; ++c) w[mb][c] = a[c] - u[c];
                }
            } else if (mb < nmb && R <= Rend) {
                const float* a = tiles + tile_index(toff, kb, R, C) + lane * NB;
#pragma unroll
                for (int c = 0; c < NB; ++c) w[mb][c] = a[c];
            }
        }
        tc_fence_before();
        // ---- diagonal tile (warp 0, mb 0: R = C): L D L^T in registers, T_C = L_CC^{-1}
        if (warp == 0) {
            const int rows_valid = n - C * NB;
            // original diagonal entry of this row (null-pivot reference)
            const float od_l = tiles[tile_index(toff, kb, C, C) + lane * NB + lane];
            float row[NB];
#pragma unroll
            for (int b = 0; b < NB; ++b) row[b] = w[0][b];
            float dl = 0.f;
            int nr = 0, stc = 0;
#pragma unroll
            for (int k = 0; k < NB; ++k) {
                const float d = __shfl_sync(0xffffffffu, row[k], k);
                const float odk = __shfl_sync(0xffffffffu, od_l, k);
                float dinv_k;
                if (k >= rows_valid) {
                    dinv_k = 1.f;
                } else if (reg_tol > 0.0 && !(d > (float)reg_tol * odk)) {
                    dinv_k = 0.f;
                    ++nr;
                } else if (!(d > 0.f)) {
                    dinv_k = 0.f;
                    if (stc == 0) stc = C * NB + k + 1;
                } else {
                    dinv_k = 1.f / d;
                }
                if (lane == k) dl = dinv_k;
                const float wak = row[k];
#pragma unroll
                for (int b = 0; b < NB; ++b) {
                    if (b > k) {
                        const float wbk = __shfl_sync(0xffffffffu, wak, b);
                        if (lane >= b) row[b] -= wak * wbk * dinv_k;
                    }
                }
                if (lane > k) row[k] = (k >= rows_valid || lane >= rows_valid) ? 0.f : wak * dinv_k;
            }
            float tr[NB];
#pragma unroll
            for (int b = 0; b < NB; ++b) tr[b] = (b == lane) ? 1.f : 0.f;
#pragma unroll
            for (int k = 0; k < NB - 1; ++k) {
                const float lak = row[k];
#pragma unroll
                for (int b = 0; b < NB; ++b) {
                    if (b <= k) {
                        const float tkb = __shfl_sync(0xffffffffu, tr[b], k);
                        if (lane > k) tr[b] -= lak * tkb;
                    }
                }
            }
            float* dst = tiles + tile_index(toff, kb, C, C) + lane * NB;
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                Tc[lane * NB + b] = tr[b];
                dst[b] = tr[b];
            }
            Dc[lane] = dl;
            dinv[roff + (long long)C * NB + lane] = dl;
            if (lane == 0) {
                s_nreg += nr;
                if (s_status == 0 && stc != 0) s_status = stc;
            }
        }
        __syncthreads();
        // ---- panel: L_RC = W_RC T_C^T D_C^{-1}, stored with its hi / lo parts for later columns
#pragma unroll
        for (int mb = 0; mb < 4; ++mb) {
            const int R = C + 4 * mb + warp;
            if (mb >= nmb || R <= C || R > Rend) continue;
            float out[NB];
#pragma unroll
            for (int c = 0; c < NB; ++c) {
                float s = 0.f;
#pragma unroll
                for (int g = 0; g < NB / 4; ++g) {
                    const float4 tv = *reinterpret_cast<const float4*>(Tc + c * NB + 4 * g);
                    s += w[mb][4 * g] * tv.x;
                    s += w[mb][4 * g + 1] * tv.y;
                    s += w[mb][4 * g + 2] * tv.z;
                    s += w[mb][4 * g + 3] * tv.w;
                }
                out[c] = s * Dc[c];
            }
            const long long ti = tile_index(toff, kb, R, C) + lane * NB;
#pragma unroll
            for (int c = 0; c < NB; ++c) {
                tiles[ti + c] = out[c];
                lo[ti + c] = out[c] - tf32_hi(out[c]);
            }
        }
        fence_proxy_async_global();                     // the next columns read these by TMA
        __syncthreads();
    }
    // ---- end: wait (bounded) for copies and products still in flight, free TMEM
    if (s_abort) {
        // copies still in flight land, and the products issued complete, before the CTA exits
        if (t == 32)
            for (int s = 0; s < TF_NS && s < pair_base; ++s) mbar_wait_bounded(&full[s], (par_issued >> s) & 1u);
        if (t == 0) mbar_wait_bounded(accb, ph_acc & 1u);  // a column's products, if their wait gave up
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 128;\n" ::"r"(tmem));
    if (t == 0) { status[i] = s_status; nreg[i] = s_nreg; }
}

template <int C>
__device__ __forceinline__ void ws_ld(const float* p, float (&v)[C]) {
    if constexpr (C == 4) {
        const float4 x = *reinterpret_cast<const float4*>(p);
        v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
    } else if constexpr (C == 2) {
        const float2 x = *reinterpret_cast<const float2*>(p);
        v[0] = x.x; v[1] = x.y;
    } else {
        v[0] = *p;
    }
}
template <int C>
__device__ __forceinline__ void ws_st(float* p, const float (&v)[C]) {
    if constexpr (C == 4) *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    else if constexpr (C == 2) *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
    else *p = v[0];
}
// element (row, col) of a 128-byte-swizzled 32 x 32 FP32 tile
__device__ __forceinline__ int swz(int row, int col) { return row * NB + ((((col >> 2) ^ (row & 7))) << 2) + (col & 3); }

// acc[c] += SIGN * sum_{K0 <= k < K1} tile[lane][k] V[k][c]  (row access of a
// swizzled tile; V: [32][C] floats, read by broadcast).  Fully unrolled so
// that all loads issue ahead of the products.
template <int C, int K0, int K1, int SIGN>
__device__ __forceinline__ void ws_row_product(const float* tile, const float* V, int lane, float (&acc)[C]) {
    float l[K1 - K0];
#pragma unroll
    for (int g = K0 / 4; g < K1 / 4; ++g) {
        const float4 x = *reinterpret_cast<const float4*>(tile + lane * NB + ((g ^ (lane & 7)) << 2));
        l[4 * g - K0] = x.x; l[4 * g - K0 + 1] = x.y; l[4 * g - K0 + 2] = x.z; l[4 * g - K0 + 3] = x.w;
    }
#pragma unroll
    for (int k = K0; k < K1; ++k) {
        float v[C];
        ws_ld<C>(V + k * C, v);
#pragma unroll
        for (int c = 0; c < C; ++c) {
            if (SIGN > 0) acc[c] += l[k - K0] * v[c];
            else acc[c] -= l[k - K0] * v[c];
        }
    }
}
// acc[c] += SIGN * sum_{0 <= k < K1} tile[k][lane] V[k][c]  (column access)
template <int C, int K1, int SIGN>
__device__ __forceinline__ void ws_col_product(const float* tile, const float* V, int lane, float (&acc)[C]) {
    float l[K1];
#pragma unroll
    for (int k = 0; k < K1; ++k) l[k] = tile[swz(k, lane)];
#pragma unroll
    for (int k = 0; k < K1; ++k) {
        float v[C];
        ws_ld<C>(V + k * C, v);
#pragma unroll
        for (int c = 0; c < C; ++c) {
            if (SIGN > 0) acc[c] += l[k] * v[c];
            else acc[c] -= l[k] * v[c];
        }
    }
}

// Wide-band forms of the two products: the loads are volatile shared
// loads issued eight k at a time ahead of their products (the compiler keeps
// their order), with two partial sums per column.  With 13 tiles a step the
// products dominate and this ordering is 2-12% faster; with 3 tiles the
// plain forms above are.
__device__ __forceinline__ float4 lds4_ordered(const float* p) {
    float4 r;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];\n"
                 : "=f"(r.x), "=f"(r.y), "=f"(r.z), "=f"(r.w)
                 : "r"(smem_u32(p)));
    return r;
}
__device__ __forceinline__ float lds1_ordered(const float* p) {
    float r;
    asm volatile("ld.shared.f32 %0, [%1];\n" : "=f"(r) : "r"(smem_u32(p)));
    return r;
}
__device__ __forceinline__ float2 lds2_ordered(const float* p) {
    float2 r;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];\n" : "=f"(r.x), "=f"(r.y) : "r"(smem_u32(p)));
    return r;
}
template <int C>
__device__ __forceinline__ void ws_ld_ordered(const float* p, float (&v)[C]) {
    if constexpr (C == 4) {
        const float4 x = lds4_ordered(p);
        v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
    } else if constexpr (C == 2) {
        const float2 x = lds2_ordered(p);
        v[0] = x.x; v[1] = x.y;
    } else {
        ws_ld<C>(p, v);
    }
}
template <int C, int K0, int K1, int SIGN>
__device__ __forceinline__ void ws_row_product_wide(const float* tile, const float* V, int lane, float (&acc)[C]) {
    constexpr int NK = K1 - K0;
    static_assert(NK % 8 == 0, "k range in multiples of 8");
    float l[NK];
#pragma unroll
    for (int g = K0 / 4; g < K1 / 4; ++g) {
        const float4 x = lds4_ordered(tile + lane * NB + ((g ^ (lane & 7)) << 2));
        l[4 * g - K0] = x.x; l[4 * g - K0 + 1] = x.y; l[4 * g - K0 + 2] = x.z; l[4 * g - K0 + 3] = x.w;
    }
    float a0[C], a1[C];
#pragma unroll
    for (int c = 0; c < C; ++c) { a0[c] = acc[c]; a1[c] = 0.f; }
#pragma unroll
    for (int k8 = 0; k8 < NK; k8 += 8) {
        float v[8][C];
#pragma unroll
        for (int k = 0; k < 8; ++k) ws_ld_ordered<C>(V + (K0 + k8 + k) * C, v[k]);
#pragma unroll
        for (int k = 0; k < 8; k += 2)
#pragma unroll
            for (int c = 0; c < C; ++c) {
                if (SIGN > 0) { a0[c] += l[k8 + k] * v[k][c]; a1[c] += l[k8 + k + 1] * v[k + 1][c]; }
                else { a0[c] -= l[k8 + k] * v[k][c]; a1[c] -= l[k8 + k + 1] * v[k + 1][c]; }
            }
    }
#pragma unroll
    for (int c = 0; c < C; ++c) acc[c] = a0[c] + a1[c];
}
template <int C, int K1, int SIGN>
__device__ __forceinline__ void ws_col_product_wide(const float* tile, const float* V, int lane, float (&acc)[C]) {
    static_assert(K1 % 8 == 0, "k range in multiples of 8");
    float l[K1];
#pragma unroll
    for (int k = 0; k < K1; ++k) l[k] = lds1_ordered(tile + swz(k, lane));
    float a0[C], a1[C];
#pragma unroll
    for (int c = 0; c < C; ++c) { a0[c] = acc[c]; a1[c] = 0.f; }
#pragma unroll
    for (int k8 = 0; k8 < K1; k8 += 8) {
        float v[8][C];
#pragma unroll
        for (int k = 0; k < 8; ++k) ws_ld_ordered<C>(V + (k8 + k) * C, v[k]);
#pragma unroll
        for (int k = 0; k < 8; k += 2)
#pragma unroll
            for (int c = 0; c < C; ++c) {
                if (SIGN > 0) { a0[c] += l[k8 + k] * v[k][c]; a1[c] += l[k8 + k + 1] * v[k + 1][c]; }
                else { a0[c] -= l[k8 + k] * v[k][c]; a1[c] -= l[k8 + k + 1] * v[k + 1][c]; }
            }
    }
#pragma unroll
    for (int c = 0; c < C; ++c) acc[c] = a0[c] + a1[c];
}
// the form a configuration uses: ordered for wide bands (more than 2 tiles)
// with 2 or 4 columns a warp (the configurations that were measured)
template <bool WIDE, int C, int K0, int K1, int SIGN>
__device__ __forceinline__ void ws_rowp(const float* tile, const float* V, int lane, float (&acc)[C]) {
    if constexpr (WIDE) ws_row_product_wide<C, K0, K1, SIGN>(tile, V, lane, acc);
    else ws_row_product<C, K0, K1, SIGN>(tile, V, lane, acc);
}
template <bool WIDE, int C, int K1, int SIGN>
__device__ __forceinline__ void ws_colp(const float* tile, const float* V, int lane, float (&acc)[C]) {
    if constexpr (WIDE) ws_col_product_wide<C, K1, SIGN>(tile, V, lane, acc);
    else ws_col_product<C, K1, SIGN>(tile, V, lane, acc);
}

__device__ __forceinline__ void mbar_arrive(unsigned long long* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}

// ---- the FP32 band solve of several right-hand sides (kb <= 12), TMA tile
// loads, k split over warps.  Forward z_R = T_R (x_R - sum_J L_RJ z_J),
// backward x_R = T_R^T (D_R^{-1} z_R - sum_I L_IR^T x_I); all sums in FP32.
//
// A solve is a chain of 2 K dependent steps of one CTA; a step's products
// are (kb + 1) tiles of 32 x 32 by 4 J columns.  Letting every warp run over
// all tiles for columns of its own (k_tile_solve_band_ws below) makes each tile
// element travel from shared memory once per warp.  Here the NW consumer warps
// split the k index instead, so that every tile element is read once: a warp
// takes groups of four k and accumulates all 32 rows x 4 J columns in registers
// (lane = 8 row groups x 4 column groups, 4 rows x J columns each: 4 + J wide
// loads per 16 J FMA).  The partial sums are exchanged through shared memory:
// warp w sums and finishes the 32 / NW rows of its slice, which are exactly the
// rows it then multiplies as its k-slice of T_R, and of the next step's nearest
// tile.  The exchange costs two barriers of the consumer warps a step, which
// pays where a step has many tiles or columns (solve_band_f32 has the line): of
// 128 problems of n = 1500, b = 380, 20 columns, FP32 X 400 -> 324 us a launch;
// of 128 with b = 38, 16 columns 107 -> 121.  Still bound by shared memory: 4 + J
// 16-byte loads, four LSU cycles each, feed 16 J FMA.
//
// A producer warp streams the tiles of each step by TMA (128-byte swizzle,
// ring of nst stages of S = maxkb + 1 tiles, "full" mbarriers by byte count,
// "empty" ones released by each consumer warp after its last read).  Column
// blocks of a tile that lie outside the band (element (r, k) of L_{R,R-d} is
// zero unless 32 d + r - k <= b) are skipped in groups of four k.  Every wait
// is bounded; after a timeout (recorded in g_wait_timeouts) the producer
// waits (bounded) for its copies in flight and the consumers leave together
// at the end of the step.
__device__ __forceinline__ float as_f32(double x) { return f64_to_f32(x); }
__device__ __forceinline__ float as_f32(float x) { return x; }
constexpr int KS_LD = 40;        // column stride of the exchange blocks: 16-byte reads of 4 columns or 8 row groups are conflict-free

constexpr size_t band_ks_smem(int NW, int J, int S, int nst) {
    return 1024 + (size_t)nst * S * NB2 * 4 + 16 * (size_t)nst + sizeof(float) * (size_t)(2 * NW + S + 1) * 4 * J * KS_LD;
}

template <int NW, int J, typename XT>
__global__ void __launch_bounds__(32 * (NW + 1)) k_tile_solve_band_ks(
    const __grid_constant__ CUtensorMap tmt, const float* __restrict__ dinv, const int* __restrict__ kb_,
    const int* __restrict__ K_, const int* __restrict__ b_, const long long* __restrict__ toff_,
    const long long* __restrict__ roff_, XT* Xall, int ldx, int ncols_all, const int* __restrict__ skip,
    const int* __restrict__ gdone, int S, int nst)
{
    constexpr int COLS = 4 * J, RS = NB / NW, QS = RS / 4;   // columns, rows and k-groups of a warp's slice
    constexpr int UNITS = COLS * QS, UN = (UNITS + 31) / 32;  // (column, four rows) units of a slice per lane
    constexpr int BLK = COLS * KS_LD;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    float* St = reinterpret_cast<float*>(base);                        // [nst][S][32*32]
    unsigned long long* full = reinterpret_cast<unsigned long long*>(St + (size_t)nst * S * NB2);
    unsigned long long* empty = full + nst;
    float* P1 = reinterpret_cast<float*>(empty + nst);                 // [NW][COLS][KS_LD] partial sums
    float* P2 = P1 + NW * BLK;
    float* Zr = P2 + NW * BLK;                                         // [S][COLS][KS_LD] solutions
    float* Ac = Zr + S * BLK;                                          // [COLS][KS_LD]
    __shared__ int s_abort, s_stop;

    const int i = blockIdx.x;
    if (skip && skip[i]) return;
    if (gdone && *gdone) return;
    const int kb = kb_[i], K = K_[i], bw = b_[i];
    if (kb >= S || K == 0) return;                   // never launched so (host dispatch)
    const long long toff = toff_[i], roff = roff_[i];
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    if (t == 0) {
        s_abort = 0;
        s_stop = 0;
        for (int s = 0; s < nst; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], NW);
        }
        fence_mbar_init();
    }
    __syncthreads();
    auto give_up = [&]() {
        if (atomicExch(&s_abort, 1) == 0) atomicAdd(&g_wait_timeouts, 1);
    };
    const int total = 2 * K;                         // steps of both sweeps

    if (warp == NW) {
        // ---------------- producer: one lane issues every copy
        if (lane == 0) {
            unsigned pending = 0, par = 0, ph = 0;   // stages with copies in flight, their parity; use parity of each stage
            int st = 0;
            for (int it = 0; it < total; ++it) {
                if (it >= nst) {
                    if (!mbar_wait_bounded(&empty[st], ((ph >> st) & 1u) ^ 1u)) { give_up(); break; }
                    pending &= ~(1u << st);
                }
                if (*(volatile int*)&s_abort) break;
                const bool fwd = it < K;
                const int R = fwd ? it : total - 1 - it;
                const int nd = min(kb, fwd ? R : K - 1 - R);
                float* dst = St + (size_t)st * S * NB2;
                mbar_expect_tx(&full[st], (nd + 1) * NB2 * 4);
                for (int d = nd; d >= 0; --d) {
                    const long long ti = fwd ? tile_index(toff, kb, R, R - d) : tile_index(toff, kb, R + d, R);
                    tma_load_tile(dst + (size_t)d * NB2, &tmt, (int)(ti / NB), &full[st]);
                }
                pending |= 1u << st;
                par = (par & ~(1u << st)) | (((ph >> st) & 1u) << st);
                ph ^= 1u << st;
                st = st + 1 == nst ? 0 : st + 1;
            }
            // after an abort, copies still in flight must land before the CTA exits
            if (*(volatile int*)&s_abort)
                for (int s = 0; s < nst; ++s)
                    if (pending & (1u << s)) mbar_wait_bounded(&full[s], (par >> s) & 1u);
        }
        return;
    }

    // ---------------- consumer warps
    auto consumers_sync = [&]() { asm volatile("bar.sync 1, %0;\n" ::"r"(32 * NW) : "memory"); };
    const int rg = lane & 7, cg = lane >> 3;
    const int cbase = blockIdx.y * COLS;
    // this lane's units of the warp's slice: column uc[u], rows ur[u] .. ur[u] + 3
    int uc[UN], ur[UN];
    bool uon[UN], uok[UN];
#pragma unroll
    for (int u = 0; u < UN; ++u) {
        const int e = lane + 32 * u;
        uc[u] = e / QS;
        ur[u] = RS * warp + 4 * (e % QS);
        uon[u] = e < UNITS;
        uok[u] = uon[u] && cbase + uc[u] < ncols_all;
    }
    XT xn[UN][4];                                    // next right-hand side rows, as loaded (converted when used)
    float dn[UN][4], zl[UN][4];                      // next D^{-1}, last solution rows
    auto load_rhs = [&](int it) {
        const bool fwd = it < K;
        const int R = fwd ? it : total - 1 - it;
#pragma unroll
        for (int u = 0; u < UN; ++u) {
            const long long row = roff + (long long)R * NB + ur[u];
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                xn[u][a] = uok[u] ? Xall[(row + a) * ldx + cbase + uc[u]] : XT(0);
                dn[u][a] = 1.f;
            }
            if (!fwd && uok[u]) {
                const float4 d4 = *reinterpret_cast<const float4*>(dinv + row);
                dn[u][0] = d4.x; dn[u][1] = d4.y; dn[u][2] = d4.z; dn[u][3] = d4.w;
            }
        }
    };
    float acc[4][J];
    auto clear = [&]() {
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int j = 0; j < J; ++j) acc[a][j] = 0.f;
    };
    // acc += (32 x 4 columns 4 q .. of the tile, or of its transpose) V[:, 4 q ..]; forward rows rg + 8 a, backward 4 rg + a
    auto product = [&](const float* T, const float* V, int q, bool fwd) {
        float4 v[J];
#pragma unroll
        for (int j = 0; j < J; ++j) v[j] = *reinterpret_cast<const float4*>(V + (cg + 4 * j) * KS_LD + 4 * q);
        if (fwd) {
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const float4 l = *reinterpret_cast<const float4*>(T + (rg + 8 * a) * NB + ((q ^ rg) << 2));
#pragma unroll
                for (int j = 0; j < J; ++j) {
                    acc[a][j] = fmaf(l.x, v[j].x, acc[a][j]);
                    acc[a][j] = fmaf(l.y, v[j].y, acc[a][j]);
                    acc[a][j] = fmaf(l.z, v[j].z, acc[a][j]);
                    acc[a][j] = fmaf(l.w, v[j].w, acc[a][j]);
                }
            }
        } else {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                const int k = 4 * q + kk;
                const float4 l = *reinterpret_cast<const float4*>(T + k * NB + ((rg ^ (k & 7)) << 2));
#pragma unroll
                for (int j = 0; j < J; ++j) {
                    const float x = kk == 0 ? v[j].x : kk == 1 ? v[j].y : kk == 2 ? v[j].z : v[j].w;
                    acc[0][j] = fmaf(l.x, x, acc[0][j]);
                    acc[1][j] = fmaf(l.y, x, acc[1][j]);
                    acc[2][j] = fmaf(l.z, x, acc[2][j]);
                    acc[3][j] = fmaf(l.w, x, acc[3][j]);
                }
            }
        }
    };
    auto store_partial = [&](float* P, bool fwd) {
        float* dst = P + warp * BLK;
#pragma unroll
        for (int j = 0; j < J; ++j) {
            if (fwd) {
#pragma unroll
                for (int a = 0; a < 4; ++a) dst[(cg + 4 * j) * KS_LD + rg + 8 * a] = acc[a][j];
            } else {
                *reinterpret_cast<float4*>(dst + (cg + 4 * j) * KS_LD + 4 * rg) =
                    make_float4(acc[0][j], acc[1][j], acc[2][j], acc[3][j]);
            }
        }
    };
    // four-k groups of the outermost tile that hold nonzeros (the last ones forward, the first ones backward)
    const int nql = kb > 0 ? min(8, 8 - (NB * kb - bw) / 4) : 0;
    load_rhs(0);
    int st = 0;
    unsigned ph = 0;                                 // parity of each stage's next use
    int zs = 0;                                      // ring slot of this step's solution
    for (int it = 0; it < total; ++it) {
        const bool fwd = it < K;
        const int R = fwd ? it : total - 1 - it;
        const int nd = min(kb, fwd ? R : K - 1 - R);
        if (it == K) zs = (K - 1) % S;               // the backward sweep overwrites z_R by x_R in its slot
        float x[UN][4];
#pragma unroll
        for (int u = 0; u < UN; ++u)
#pragma unroll
            for (int a = 0; a < 4; ++a) x[u][a] = as_f32(xn[u][a]) * dn[u][a];
        if (it == K) {                               // the last forward step's rows are still in registers
#pragma unroll
            for (int u = 0; u < UN; ++u)
                if (uok[u]) {
                    const float4 d4 = *reinterpret_cast<const float4*>(dinv + roff + (long long)R * NB + ur[u]);
                    x[u][0] = zl[u][0] * d4.x; x[u][1] = zl[u][1] * d4.y;
                    x[u][2] = zl[u][2] * d4.z; x[u][3] = zl[u][3] * d4.w;
                }
        }
        if (it + 1 < total && it + 1 != K) load_rhs(it + 1);
        const float* tiles = St + (size_t)st * S * NB2;
        const bool ok = mbar_wait_bounded(&full[st], (ph >> st) & 1u);
        if (!ok) give_up();
        clear();
        if (ok && nd > 0) {
            // tiles d >= 2: all k groups, spread over the warps
            const int nfar = nd < 2 ? 0 : 8 * (nd - 2) + (nd == kb ? nql : 8);
            for (int f = warp; f < nfar; f += NW) {
                const int d = 2 + (f >> 3);
                const int q = (f & 7) + (fwd && d == kb ? 8 - nql : 0);
                int slot = fwd ? zs - d : zs + d;
                slot += slot < 0 ? S : 0;
                slot -= slot >= S ? S : 0;
                product(tiles + (size_t)d * NB2, Zr + slot * BLK, q, fwd);
            }
            // the nearest tile: this warp's slice of z_{R-1} (x_{R+1})
            int slot = fwd ? zs - 1 : zs + 1;
            slot += slot < 0 ? S : 0;
            slot -= slot >= S ? S : 0;
#pragma unroll
            for (int m = 0; m < QS; ++m) {
                const int q = QS * warp + m;
                if (kb > 1 || (fwd ? q >= 8 - nql : q < nql)) product(tiles + NB2, Zr + slot * BLK, q, fwd);
            }
        }
        store_partial(P1, fwd);
        consumers_sync();                            // every partial sum is in P1
#pragma unroll
        for (int u = 0; u < UN; ++u)
            if (uon[u]) {
                float4 y = make_float4(x[u][0], x[u][1], x[u][2], x[u][3]);
#pragma unroll
                for (int w = 0; w < NW; ++w) {
                    const float4 p = *reinterpret_cast<const float4*>(P1 + w * BLK + uc[u] * KS_LD + ur[u]);
                    y.x -= p.x; y.y -= p.y; y.z -= p.z; y.w -= p.w;
                }
                *reinterpret_cast<float4*>(Ac + uc[u] * KS_LD + ur[u]) = y;
            }
        __syncwarp();
        clear();
        if (ok) {
#pragma unroll
            for (int m = 0; m < QS; ++m) product(tiles, Ac, QS * warp + m, fwd);
        }
        store_partial(P2, fwd);
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[st]);
        if (t == 0) *(volatile int*)&s_stop = *(volatile int*)&s_abort;
        consumers_sync();                            // every partial of the solution is in P2
        if (*(volatile int*)&s_stop) break;          // sampled once: every warp leaves after this step
#pragma unroll
        for (int u = 0; u < UN; ++u)
            if (uon[u]) {
                float4 z = *reinterpret_cast<const float4*>(P2 + uc[u] * KS_LD + ur[u]);
#pragma unroll
                for (int w = 1; w < NW; ++w) {
                    const float4 p = *reinterpret_cast<const float4*>(P2 + w * BLK + uc[u] * KS_LD + ur[u]);
                    z.x += p.x; z.y += p.y; z.z += p.z; z.w += p.w;
                }
                *reinterpret_cast<float4*>(Zr + zs * BLK + uc[u] * KS_LD + ur[u]) = z;
                zl[u][0] = z.x; zl[u][1] = z.y; zl[u][2] = z.z; zl[u][3] = z.w;
                if (uok[u]) {
                    XT* xw = Xall + (roff + (long long)R * NB + ur[u]) * ldx + cbase + uc[u];
#pragma unroll
                    for (int a = 0; a < 4; ++a) {
                        if constexpr (sizeof(XT) == 8) xw[(long long)a * ldx] = f32_to_f64(zl[u][a]);
                        else xw[(long long)a * ldx] = zl[u][a];
                    }
                }
            }
        __syncwarp();
        ph ^= 1u << st;
        st = st + 1 == nst ? 0 : st + 1;
        if (fwd) zs = zs + 1 == S ? 0 : zs + 1;
        else zs = zs == 0 ? S - 1 : zs - 1;
    }
}

// ---- the FP32 band solve of several right-hand sides (kb <= 12), a warp per
// few columns.  No block barrier sits on the sweeps' chain: each of W consumer
// warps owns C right-hand-side columns and all 32 rows of a tile row (lane =
// row), so a step's data exchange is warp-internal (__syncwarp).  Producer
// warp, bounded waits and time-outs as in k_tile_solve_band_ks.  Each lane
// prefetches its own row of the right-hand sides with cp.async, XD steps ahead
// (X rows start on 16 bytes: host dispatch).  Column k of tile L_{R,R-d} can be
// nonzero only where 32 d + r - k <= b (the band), so the forward products
// start at k = 32 d - b and the backward ones stop at k = b - 32 d + 31.
template <int KBP, int W, int C, int NST, int XD, typename XT>
struct BandWs {
    // The backward sweep's first right-hand side read from X (block K-1-S,
    // written by forward step K-1-S) is issued XD - 1 steps ahead, at step
    // K - XD + 1: it must come after that write, so XD <= S + 1 = KBP + 2.
    static_assert(XD <= KBP + 2, "X prefetch deeper than the solution ring allows");
    static constexpr int SLOTS = KBP + 1;            // tiles per step; also the solution ring per warp
    static constexpr int NT = 32 * (W + 1);
    static constexpr int COLS = W * C;
    static constexpr size_t stage_bytes = (size_t)SLOTS * NB2 * sizeof(float);
    static constexpr size_t warp_bytes =
        sizeof(float) * ((size_t)SLOTS * NB * C + (size_t)NB * C) + sizeof(XT) * (size_t)XD * NB * C;
    static constexpr size_t smem_bytes =
        1024 + (size_t)NST * stage_bytes + (size_t)NST * NB * sizeof(float) + 16 * (size_t)NST + (size_t)W * warp_bytes;
};

// Half-bandwidth b at most KBP tiles (kb <= KBP); a step needs the diagonal
// tile and kb off-diagonal tiles, and z_{R-1} .. z_{R-kb} (forward) or
// x_{R+1} .. x_{R+kb} (backward) from the warp's ring of KBP + 1 solution
// blocks.  When the backward sweep starts, the ring still holds z_R for the
// last KBP + 1 rows, so only the rows before those are read back from X.
template <int KBP, int W, int C, int NST, int XD, typename XT>
__global__ void __launch_bounds__(32 * (W + 1)) k_tile_solve_band_ws(
    const __grid_constant__ CUtensorMap tmt, const float* __restrict__ dinv, const int* __restrict__ kb_,
    const int* __restrict__ K_, const int* __restrict__ b_, const long long* __restrict__ toff_,
    const long long* __restrict__ roff_, XT* Xall, int ldx, int ncols_all,
    const int* __restrict__ skip, const int* __restrict__ gdone)
{
    using Cfg = BandWs<KBP, W, C, NST, XD, XT>;
    constexpr int S = Cfg::SLOTS;
    static_assert(C == 2 || C == 4, "2 or 4 columns per warp");
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    float* St = reinterpret_cast<float*>(base);                                        // [NST][S][32*32]
    float* Sd = St + (size_t)NST * S * NB2;                                            // [NST][32]
    unsigned long long* full = reinterpret_cast<unsigned long long*>(Sd + (size_t)NST * NB);
    unsigned long long* empty = full + NST;
    unsigned char* wbase = reinterpret_cast<unsigned char*>(empty + NST);
    __shared__ int s_abort;

    const int i = blockIdx.x;
    if (skip && skip[i]) return;
    if (gdone && *gdone) return;
    const int kb = kb_[i], K = K_[i], bw = b_[i];
    if (kb > KBP) return;                            // never launched so (host dispatch)
    const long long toff = toff_[i], roff = roff_[i];
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    if (t == 0) {
        s_abort = 0;
        for (int s = 0; s < NST; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], W);
        }
        fence_mbar_init();
    }
    __syncthreads();
    auto stile = [&](int st, int slot) { return St + (size_t)(st * S + slot) * NB2; };
    auto give_up = [&]() {
        if (atomicExch(&s_abort, 1) == 0) atomicAdd(&g_wait_timeouts, 1);
    };
    const int total = 2 * K;                         // steps of both sweeps

    if (warp == W) {
        // ---------------- producer: one lane issues every copy
        if (lane == 0) {
            unsigned pending = 0, par = 0;           // stages with copies in flight, their phase parity
            for (int it = 0; it < total; ++it) {
                const int st = it % NST;
                if (it >= NST) {
                    if (!mbar_wait_bounded(&empty[st], ((it / NST) - 1) & 1u)) { give_up(); break; }
                    pending &= ~(1u << st);
                }
                if (*(volatile int*)&s_abort) break;
                const bool fwd = it < K;
                const int R = fwd ? it : total - 1 - it;
                int nt = 1;
                for (int d = 1; d <= kb; ++d) {
                    const int o = fwd ? R - d : R + d;
                    if (o >= 0 && o < K) ++nt;
                }
                mbar_expect_tx(&full[st], nt * NB2 * 4 + (fwd ? 0 : NB * 4));
                tma_load_tile(stile(st, 0), &tmt, (int)(tile_index(toff, kb, R, R) / NB), &full[st]);
                for (int d = 1; d <= kb; ++d) {
                    const int o = fwd ? R - d : R + d;
                    if (o < 0 || o >= K) continue;
                    const long long ti = fwd ? tile_index(toff, kb, R, o) : tile_index(toff, kb, o, R);
                    tma_load_tile(stile(st, d), &tmt, (int)(ti / NB), &full[st]);
                }
                if (!fwd) bulk_load(Sd + st * NB, dinv + roff + (long long)R * NB, NB * 4, &full[st]);
                pending |= 1u << st;
                par = (par & ~(1u << st)) | (((unsigned)(it / NST) & 1u) << st);
            }
            // after an abort, copies still in flight must land before the CTA exits
            if (*(volatile int*)&s_abort)
                for (int s = 0; s < NST; ++s)
                    if (pending & (1u << s)) mbar_wait_bounded(&full[s], (par >> s) & 1u);
        }
        return;
    }

    // ---------------- consumer warp: columns [c_lo, c_lo + nc)
    const int c_lo = blockIdx.y * Cfg::COLS + warp * C;
    const int nc = max(0, min(C, ncols_all - c_lo));
    float* Zr = reinterpret_cast<float*>(wbase + (size_t)warp * Cfg::warp_bytes);     // [S][32][C]
    float* Acc = Zr + (size_t)S * NB * C;                                               // [32][C]
    XT* Xs = reinterpret_cast<XT*>(Acc + (size_t)NB * C);                      // [XD][32][C]
    XT* X = Xall + c_lo;
    // loads of this lane's row: index q < K: forward step q (row q); q >= K:
    // backward row K - 1 - S - (q - K) (backward steps s >= S)
    const int nload = K + max(0, K - S);
    auto issue_load = [&](int q) {
        if (q < nload && nc > 0) {
            if (q >= K) __threadfence_block();       // rows written by this lane in the forward sweep
            const int R = q < K ? q : K - 1 - S - (q - K);
            const XT* src = X + (roff + (long long)R * NB + lane) * ldx;
            XT* dst = Xs + ((size_t)(q % XD) * NB + lane) * C;
            if constexpr (C * sizeof(XT) == 8) {
                asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(smem_u32(dst)), "l"(src));
            } else {
                cp_async16(dst, src);
                if (C * sizeof(XT) == 32 && nc > 2) cp_async16(dst + 2, src + 2);
            }
        }
        cp_async_commit();
    };
    for (int q = 0; q < XD - 1; ++q) issue_load(q);
    int q_next = XD - 1, q_use = 0;
    for (int it = 0; it < total; ++it) {
        const int st = it % NST;
        const bool fwd = it < K;
        const int R = fwd ? it : total - 1 - it;
        float acc[C];
        // right-hand side of this step (own row)
        if (fwd || (it - K) >= S) {
            issue_load(q_next++);
            cp_async_wait_n<XD - 1>();
            const XT* xs = Xs + ((size_t)(q_use % XD) * NB + lane) * C;
#pragma unroll
            for (int c = 0; c < C; ++c) acc[c] = c < nc ? as_f32(xs[c]) : 0.f;
            ++q_use;
        } else {
            ws_ld<C>(Zr + ((size_t)(R % S) * NB + lane) * C, acc);
        }
        if (!mbar_wait_bounded(&full[st], (it / NST) & 1u)) { give_up(); break; }
        if (nc > 0) {
            if (!fwd) {
                const float dr = Sd[st * NB + lane];
#pragma unroll
                for (int c = 0; c < C; ++c) acc[c] *= dr;
            }
            for (int d = 1; d <= kb; ++d) {
                const int o = fwd ? R - d : R + d;
                if (o < 0 || o >= K) continue;
                const float* L = stile(st, d);
                const float* Z = Zr + (size_t)(o % S) * NB * C;
                if (fwd) {
                    // acc -= L_{R,o}[lane][k] z_o[k]; nonzero only for k >= 32 d - b
                    const int k0 = NB * d - bw;
                    if (k0 >= 24) ws_rowp<(KBP > 2 && C >= 2), C, 24, 32, -1>(L, Z, lane, acc);
                    else if (k0 >= 16) ws_rowp<(KBP > 2 && C >= 2), C, 16, 32, -1>(L, Z, lane, acc);
                    else ws_rowp<(KBP > 2 && C >= 2), C, 0, 32, -1>(L, Z, lane, acc);
                } else {
                    // acc -= L_{o,R}[k][lane] x_o[k]; nonzero only for k <= b - 32 d + 31
                    const int kend = bw - NB * d + NB;
                    if (kend <= 8) ws_colp<(KBP > 2 && C >= 2), C, 8, -1>(L, Z, lane, acc);
                    else if (kend <= 16) ws_colp<(KBP > 2 && C >= 2), C, 16, -1>(L, Z, lane, acc);
                    else ws_colp<(KBP > 2 && C >= 2), C, 32, -1>(L, Z, lane, acc);
                }
            }
            ws_st<C>(Acc + lane * C, acc);
            __syncwarp();
            const float* T = stile(st, 0);
            float out[C];
#pragma unroll
            for (int c = 0; c < C; ++c) out[c] = 0.f;
            if (fwd) ws_rowp<(KBP > 2 && C >= 2), C, 0, 32, 1>(T, Acc, lane, out);
            else ws_colp<(KBP > 2 && C >= 2), C, 32, 1>(T, Acc, lane, out);
            __syncwarp();                                   // Acc reads done before the next step's writes
            ws_st<C>(Zr + ((size_t)(R % S) * NB + lane) * C, out);
            XT* xw = X + (roff + (long long)R * NB + lane) * ldx;
#pragma unroll
            for (int c = 0; c < C; ++c)
                if (c < nc) {
                    if constexpr (sizeof(XT) == 8) xw[c] = f32_to_f64(out[c]);
                    else xw[c] = out[c];
                }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[st]);
    }
    cp_async_wait_n<0>();
}

// Launch of k_tile_solve_band_ws for one configuration.
template <int KBP, int W, int C, int NST, int XD, typename XT>
void launch_band_ws(const TileBatch& tb, const CUtensorMap& tm, XT* X, int ldx, int ncols, const int* skip,
                    cudaStream_t s, const int* gdone) {
    using Cfg = BandWs<KBP, W, C, NST, XD, XT>;
    static_assert(Cfg::smem_bytes <= 227 * 1024, "shared memory per CTA");
    auto kern = k_tile_solve_band_ws<KBP, W, C, NST, XD, XT>;
    raise_smem_limit(kern, Cfg::smem_bytes);
    kern<<<dim3(tb.P, (ncols + Cfg::COLS - 1) / Cfg::COLS), Cfg::NT, Cfg::smem_bytes, s>>>(
        tm, tb.dinv_f.p, tb.d_kb.p, tb.d_K.p, tb.d_b.p, tb.d_toff.p, tb.d_roff.p, X, ldx, ncols, skip, gdone);
    MSDD_LAUNCH_CHECK();
}

// stages of k_tile_solve_band_ks: up to four, with two CTAs an SM where that leaves at least two
int band_ks_stages(int NW, int J, int S) {
    const size_t half = 112 * 1024, full = 226 * 1024;
    const size_t limit = band_ks_smem(NW, J, S, 2) <= half ? half : full;
    int nst = 4;
    while (nst > 2 && band_ks_smem(NW, J, S, nst) > limit) --nst;
    return nst;
}

template <int NW, int J, typename XT>
void launch_band_ks(const TileBatch& tb, const CUtensorMap& tm, int maxkb, XT* X, int ldx, int ncols, int chunks,
                    const int* skip, cudaStream_t s, const int* gdone) {
    const int S = maxkb + 1, nst = band_ks_stages(NW, J, S);
    const size_t b = band_ks_smem(NW, J, S, nst);
    auto kern = k_tile_solve_band_ks<NW, J, XT>;
    raise_smem_limit(kern, b);
    kern<<<dim3(tb.P, chunks), 32 * (NW + 1), b, s>>>(tm, tb.dinv_f.p, tb.d_kb.p, tb.d_K.p, tb.d_b.p, tb.d_toff.p,
                                                      tb.d_roff.p, X, ldx, ncols, skip, gdone, S, nst);
    MSDD_LAUNCH_CHECK();
}

// FP32 factors, several columns, kb <= 12.
//
// k_tile_solve_band_ks takes column groups of 4 J <= 20 columns, as even as
// they come; fewer columns a CTA while that still leaves every CTA an SM of its
// own (the tiles are then read by several CTAs, but a step's products and loads
// are shared out).  Four consumer warps, eight where a step's tiles outweigh the
// exchange of the partial sums: wide bands with one group of columns or with
// five, and J >= 4 beside an FP64 X (whose conversions take four warps' registers).
// k_tile_solve_band_ws takes 16 (kb <= 2) or 20 columns a CTA, two and one CTA an SM.
//
// Which one: the kernel that takes fewer rounds of CTAs over the SMs; in a tie
// the column split for kb <= 2 (its step has no block barrier), but the k split
// at kb = 2 where its CTAs have an SM each and at most 8 columns; for kb >= 3 the
// k split from 11 (FP32 X) or 15 (FP64 X) columns on, where a warp's run over
// the step's tiles is longer than the exchange.  Measured, us a launch with cold
// L2, n = 1500, column split / k split, FP32 X unless said:
//   kb 1, 128 problems, 12 columns 70 / 103; 500, 8 columns 154 / 140;
//   kb 2, 128, 16: 107 / 121; 300, 20: 226 / 187; 8, 8: 101 / 97;
//   kb 3, 72, 8: 109 / 119; 72, 16: 138 / 121; 300, 8: 214 / 150;
//   kb 12, 48, 16: 341 / 279; 128, 16 with FP64 X 365 / 324; 128, 6 with FP64 X 287 / 343.
// Over 2320 such cells (b 5 to 380, 1 to 961 problems, 2 to 32 columns, both types)
// the choice takes 1.1% more than the faster kernel on average, 29% at most.  The k
// split alone, with eight warps from kb = 3, took 16% more, 85% at most, and was
// the slower one in 1301 of them (through the band API, b = 100, 8 problems of
// 5000, 8 columns: 0.54 -> 0.70 ms).
template <typename XT>
void solve_band_f32(const TileBatch& tb, const CUtensorMap& tm, int maxkb, XT* X, int ldx, int ncols, const int* skip,
                    cudaStream_t s, const int* gdone) {
    constexpr bool F64X = sizeof(XT) == 8;
    int chunks = (ncols + 19) / 20, J = (ncols + 4 * chunks - 1) / (4 * chunks);
    while (J > 1 && (long long)tb.P * ((ncols + 4 * (J - 1) - 1) / (4 * (J - 1))) <= NUM_SMS) --J;
    chunks = (ncols + 4 * J - 1) / (4 * J);
    const long long ctas = (long long)tb.P * chunks;
    const bool own_sm = ctas <= NUM_SMS;
    const int NW = maxkb <= 2 ? 4
                   : F64X && J >= 4 ? 8
                   : maxkb <= 6 ? (J == 5 && own_sm && maxkb > 4 ? 8 : 4)
                   : J == 1 || J == 5 ? 8 : 4;
    const size_t bytes = band_ks_smem(NW, J, maxkb + 1, band_ks_stages(NW, J, maxkb + 1));
    const long long ks_rounds = ceil_div(ctas, NUM_SMS * std::max<long long>(1, 227 * 1024 / (bytes + 1024)));
    const int ws_cols = maxkb <= 2 ? 16 : 20;
    const long long ws_rounds = ceil_div((long long)tb.P * ((ncols + ws_cols - 1) / ws_cols), maxkb <= 2 ? 2 * NUM_SMS : NUM_SMS);
    bool ks;
    if (maxkb <= 2)
        ks = ks_rounds != ws_rounds ? ks_rounds < ws_rounds : maxkb == 2 && ((own_sm && J <= 2) || (!F64X && ncols > 28));
    else if (F64X && J >= 4 && maxkb <= 6)
        ks = false;
    else
        ks = ks_rounds < ws_rounds || (ncols > (F64X ? 14 : 10) && (J < 5 || maxkb > 4));
    const bool aligned = ldx * sizeof(XT) % 16 == 0 && (uintptr_t)X % 16 == 0;
    if (!ks && aligned) {
        if (maxkb <= 2) launch_band_ws<2, 4, 4, 6, 4>(tb, tm, X, ldx, ncols, skip, s, gdone);
        else launch_band_ws<12, 10, 2, 2, 4>(tb, tm, X, ldx, ncols, skip, s, gdone);
        return;
    }
    auto go = [&](auto nw) {
        constexpr int W = decltype(nw)::value;
        switch (J) {
            case 1: launch_band_ks<W, 1>(tb, tm, maxkb, X, ldx, ncols, chunks, skip, s, gdone); break;
            case 2: launch_band_ks<W, 2>(tb, tm, maxkb, X, ldx, ncols, chunks, skip, s, gdone); break;
            case 3: launch_band_ks<W, 3>(tb, tm, maxkb, X, ldx, ncols, chunks, skip, s, gdone); break;
            case 4: launch_band_ks<W, 4>(tb, tm, maxkb, X, ldx, ncols, chunks, skip, s, gdone); break;
            default: launch_band_ks<W, 5>(tb, tm, maxkb, X, ldx, ncols, chunks, skip, s, gdone); break;
        }
    };
    if (NW == 4) go(std::integral_constant<int, 4>{});
    else go(std::integral_constant<int, 8>{});
}

// ---- one right-hand side, wide bands: the off-diagonal tiles of a step split
// over warps.  With one column a step is a chain of kb tile products and the
// T_R product in one warp; here WS consumer warps each take the tiles d = w + 1,
// w + 1 + WS, ... of the step and store their partial sums, and warp 0 forms
// the right-hand side minus those sums and applies T_R (T_R^T backward), writes
// the step's solution to the ring and to X, under two named barriers of the
// consumer warps.  The producer warp streams the tiles as in
// k_tile_solve_band_ks; warp 0 alone releases a stage, after the barrier that
// ends every warp's reads of it.
template <int KBP, int WS, int NST, int XD>
struct BandSplit {
    static_assert(XD <= KBP + 2, "X prefetch deeper than the solution ring allows");
    static constexpr int S = KBP + 1;
    static constexpr int NT = 32 * (WS + 1);
    static constexpr size_t smem_bytes = 1024 + (size_t)NST * S * NB2 * sizeof(float) + (size_t)NST * NB * 4 +
                                         16 * (size_t)NST + (size_t)(S + WS + 1) * NB * 4 + 16 + (size_t)XD * NB * 8;
};

template <int KBP, int WS, int NST, int XD>
__global__ void __launch_bounds__(32 * (WS + 1)) k_tile_solve_band_split(
    const __grid_constant__ CUtensorMap tmt, const float* __restrict__ dinv, const int* __restrict__ kb_,
    const int* __restrict__ K_, const int* __restrict__ b_, const long long* __restrict__ toff_,
    const long long* __restrict__ roff_, double* __restrict__ X, const int* __restrict__ gdone)
{
    using Cfg = BandSplit<KBP, WS, NST, XD>;
    constexpr int S = Cfg::S;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    float* St = reinterpret_cast<float*>(base);                                        // [NST][S][32*32]
    float* Sd = St + (size_t)NST * S * NB2;                                            // [NST][32]
    unsigned long long* full = reinterpret_cast<unsigned long long*>(Sd + (size_t)NST * NB);
    unsigned long long* empty = full + NST;
    float* Zr = reinterpret_cast<float*>(empty + NST);                                // [S][32] solutions
    float* Pp = Zr + (size_t)S * NB;                                                   // [WS][32] partial sums
    float* Acc = Pp + (size_t)WS * NB;                                                 // [32]
    double* Xs = reinterpret_cast<double*>(                                            // [XD][32]
        base + ((reinterpret_cast<unsigned char*>(Acc + NB) - base + 15) & ~(size_t)15));
    __shared__ int s_abort, s_stop;

    const int i = blockIdx.x;
    if (gdone && *gdone) return;
    const int kb = kb_[i], K = K_[i], bw = b_[i];
    if (kb > KBP) return;                            // never launched so (host dispatch)
    const long long toff = toff_[i], roff = roff_[i];
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    if (t == 0) {
        s_abort = 0;
        for (int s = 0; s < NST; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        fence_mbar_init();
    }
    __syncthreads();
    auto stile = [&](int st, int slot) { return St + (size_t)(st * S + slot) * NB2; };
    auto give_up = [&]() {
        if (atomicExch(&s_abort, 1) == 0) atomicAdd(&g_wait_timeouts, 1);
    };
    const int total = 2 * K;

    if (warp == WS) {
        // ---------------- producer (as in k_tile_solve_band_ks)
        if (lane == 0) {
            unsigned pending = 0, par = 0;
            for (int it = 0; it < total; ++it) {
                const int st = it % NST;
                if (it >= NST) {
                    if (!mbar_wait_bounded(&empty[st], ((it / NST) - 1) & 1u)) { give_up(); break; }
                    pending &= ~(1u << st);
                }
                if (*(volatile int*)&s_abort) break;
                const bool fwd = it < K;
                const int R = fwd ? it : total - 1 - it;
                int nt = 1;
                for (int d = 1; d <= kb; ++d) {
                    const int o = fwd ? R - d : R + d;
                    if (o >= 0 && o < K) ++nt;
                }
                mbar_expect_tx(&full[st], nt * NB2 * 4 + (fwd ? 0 : NB * 4));
                tma_load_tile(stile(st, 0), &tmt, (int)(tile_index(toff, kb, R, R) / NB), &full[st]);
                for (int d = 1; d <= kb; ++d) {
                    const int o = fwd ? R - d : R + d;
                    if (o < 0 || o >= K) continue;
                    const long long ti = fwd ? tile_index(toff, kb, R, o) : tile_index(toff, kb, o, R);
                    tma_load_tile(stile(st, d), &tmt, (int)(ti / NB), &full[st]);
                }
                if (!fwd) bulk_load(Sd + st * NB, dinv + roff + (long long)R * NB, NB * 4, &full[st]);
                pending |= 1u << st;
                par = (par & ~(1u << st)) | (((unsigned)(it / NST) & 1u) << st);
            }
            if (*(volatile int*)&s_abort)
                for (int s = 0; s < NST; ++s)
                    if (pending & (1u << s)) mbar_wait_bounded(&full[s], (par >> s) & 1u);
        }
        return;
    }

    auto consumers_sync = [&]() { asm volatile("bar.sync 1, %0;\n" ::"r"(32 * WS) : "memory"); };
    // X prefetch of warp 0 (lane = row): index u < K forward block u; u >= K
    // backward block K - 1 - S - (u - K) (backward steps s >= S)
    const int nload = K + max(0, K - S);
    auto issue_load = [&](int u) {
        if (u < nload) {
            if (u >= K) __threadfence_block();       // rows written by this lane in the forward sweep
            const int R = u < K ? u : K - 1 - S - (u - K);
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(smem_u32(Xs + (u % XD) * NB + lane)),
                         "l"(X + roff + (long long)R * NB + lane));
        }
        cp_async_commit();
    };
    if (warp == 0)
        for (int u = 0; u < XD - 1; ++u) issue_load(u);
    int u_next = XD - 1, u_use = 0;
    for (int it = 0; it < total; ++it) {
        const int st = it % NST;
        const bool fwd = it < K;
        const int R = fwd ? it : total - 1 - it;
        float rhs[1] = {0.f};
        if (warp == 0) {
            if (fwd || (it - K) >= S) {
                issue_load(u_next++);
                cp_async_wait_n<XD - 1>();
                rhs[0] = f64_to_f32(Xs[(u_use % XD) * NB + lane]);
                ++u_use;
            } else {
                rhs[0] = Zr[(R % S) * NB + lane];
            }
        }
        const bool ok = mbar_wait_bounded(&full[st], (it / NST) & 1u);
        if (!ok) give_up();
        float part[1] = {0.f};
        if (ok) {
            for (int d = warp + 1; d <= kb; d += WS) {
                const int o = fwd ? R - d : R + d;
                if (o < 0 || o >= K) continue;
                const float* L = stile(st, d);
                const float* Z = Zr + (size_t)(o % S) * NB;
                if (fwd) {
                    const int k0 = NB * d - bw;
                    if (k0 >= 24) ws_row_product<1, 24, 32, 1>(L, Z, lane, part);
                    else if (k0 >= 16) ws_row_product<1, 16, 32, 1>(L, Z, lane, part);
                    else ws_row_product<1, 0, 32, 1>(L, Z, lane, part);
                } else {
                    const int kend = bw - NB * d + NB;
                    if (kend <= 8) ws_col_product<1, 8, 1>(L, Z, lane, part);
                    else if (kend <= 16) ws_col_product<1, 16, 1>(L, Z, lane, part);
                    else ws_col_product<1, 32, 1>(L, Z, lane, part);
                }
            }
        }
        Pp[warp * NB + lane] = part[0];
        consumers_sync();                            // every partial is in Pp
        if (warp == 0) {
            if (ok) {
                float acc = fwd ? rhs[0] : rhs[0] * Sd[st * NB + lane];
                for (int w = 0; w < WS; ++w) acc -= Pp[w * NB + lane];
                Acc[lane] = acc;
                __syncwarp();
                float out[1] = {0.f};
                const float* T = stile(st, 0);
                if (fwd) ws_row_product<1, 0, 32, 1>(T, Acc, lane, out);
                else ws_col_product<1, 32, 1>(T, Acc, lane, out);
                Zr[(R % S) * NB + lane] = out[0];
                X[roff + (long long)R * NB + lane] = f32_to_f64(out[0]);
            }
            if (lane == 0) *(volatile int*)&s_stop = *(volatile int*)&s_abort;
        }
        consumers_sync();                            // the solution is in the ring; the stage and Pp are free
        if (warp == 0 && lane == 0) mbar_arrive(&empty[st]);
        if (*(volatile int*)&s_stop) break;          // sampled once by warp 0: every warp leaves after this step
    }
    if (warp == 0) cp_async_wait_n<0>();
}

template <int KBP, int WS, int NST, int XD>
void launch_band_split(const TileBatch& tb, const CUtensorMap& tm, double* X, cudaStream_t s, const int* gdone) {
    using Cfg = BandSplit<KBP, WS, NST, XD>;
    static_assert(Cfg::smem_bytes <= 227 * 1024, "shared memory per CTA");
    auto kern = k_tile_solve_band_split<KBP, WS, NST, XD>;
    raise_smem_limit(kern, Cfg::smem_bytes);
    kern<<<tb.P, Cfg::NT, Cfg::smem_bytes, s>>>(tm, tb.dinv_f.p, tb.d_kb.p, tb.d_K.p, tb.d_b.p, tb.d_toff.p,
                                                tb.d_roff.p, X, gdone);
    MSDD_LAUNCH_CHECK();
}

// ---- one right-hand side, kb <= 2, FP32 (the PCG local solves of 2D boxes)
// The solve is a chain of 2 K dependent steps, z_R = T_R (x_R - L_{R,R-1}
// z_{R-1} - L_{R,R-2} z_{R-2}) forward, and a step's 64 multiply-adds a row are
// a small part of it: with four warps sharing each step, the barriers, shuffle
// sums and copy instructions around them took 1400 cycles.  Here one warp does
// a step alone (lane = row, its rows of T and L_{R,R-1} in registers, the 32
// values of z_{R-1} and of the right-hand side broadcast through shared
// memory: 133 + 126 cycles), and four warps take turns: while one runs its
// step, the others wait for the tiles of their next ones, load their rows into
// registers (some 600 cycles, off the chain) and take the far tile's part off
// the right-hand side.  Warps hand over in pairs (named barriers: z_R is
// announced to the warps of the next two steps).  (One warp doing all of it was
// no faster than four sharing a step, a warp issues in order; a barrier of all
// four a step made each wait for the slowest load; a fifth warp issuing every
// copy took 830 cycles a step for it.)  Each warp streams the tiles of its own
// steps by TMA, D turns (4 D steps) ahead; of the far tile, whose columns
// before 64 - b are zero, only the 8-column boxes that hold nonzeros are copied
// (at b = 38 a step moves 9 of 12 KB).  Every wait is bounded; after a timeout
// (recorded in g_wait_timeouts) the chain runs to its end without waiting for
// tiles, and each warp waits (bounded) for its copies in flight.
// Measured: 256 problems of n = 1369, b = 38 with cold caches 60 -> 53 us (DRAM
// from there on), with the factors in L2 59 -> 32 us; 128 of them 57 -> 29 us.
constexpr int S1W_W = 4;
// the box of a tile map at (col, row)
__device__ __forceinline__ void tma_load_box(void* dst, const CUtensorMap* map, int col, int row,
                                               unsigned long long* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n" ::"r"(
            smem_u32(dst)),
        "l"(map), "r"(col), "r"(row), "r"(smem_u32(bar))
        : "memory");
}
// first 8-column group of the far tile (R, R - 2) that holds nonzeros
__host__ __device__ inline int s1w_group0(int b) { return b >= 64 ? 0 : (64 - b) >> 3; }

constexpr size_t s1w_bytes(int D, int nbox, int K) {
    return 1024 + sizeof(float) * ((size_t)D * S1W_W * (2 * NB2 + nbox * 8 * NB) + (size_t)S1W_W * nbox * 8 * NB + NB +
                                   (size_t)K * NB);
}

template <int D>
__global__ void __launch_bounds__(32 * S1W_W) k_tile_solve1_warp(
    const __grid_constant__ CUtensorMap tmt, const __grid_constant__ CUtensorMap tmc, const float* __restrict__ dinv,
    const int* __restrict__ kb_, const int* __restrict__ K_, const int* __restrict__ b_,
    const long long* __restrict__ toff_, const long long* __restrict__ roff_, double* __restrict__ X,
    const int* __restrict__ gdone, int nbox)
{
    constexpr int NTC = 32 * S1W_W, NST = D * S1W_W;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    const int stage_floats = 2 * NB2 + nbox * 8 * NB;      // T, near tile, far tile's boxes
    float* St = reinterpret_cast<float*>(base);
    float* Fr = St + (size_t)NST * stage_floats;         // [S1W_W][boxes] far boxes of the step each warp prepares
    float* Ac = Fr + (size_t)S1W_W * nbox * 8 * NB;          // [32]
    float* zs = Ac + NB;                                     // [K * 32]
    __shared__ unsigned long long full[NST];
    __shared__ int s_abort;
    if (gdone && *gdone) return;
    const int i = blockIdx.x;
    const int kb = kb_[i], K = K_[i], bw = b_[i];
    if (kb > 2 || K == 0) return;                            // never launched so (host dispatch)
    const long long toff = toff_[i], roff = roff_[i];
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int g0 = s1w_group0(bw), nb = kb == 2 ? min(nbox, 4 - g0) : 0;
    if (t == 0) {
        s_abort = 0;
        for (int s = 0; s < NST; ++s) mbar_init(&full[s], 1);
        fence_mbar_init();
    }
    for (int e = t; e < K * NB; e += NTC) zs[e] = f64_to_f32(X[roff + e]);
    __syncthreads();
    auto give_up = [&]() {
        if (atomicExch(&s_abort, 1) == 0) atomicAdd(&g_wait_timeouts, 1);
    };
    const int total = 2 * K;

    // turn u of a warp is step 4 u + warp, its tiles go to stage D warp + u % D
    auto stage = [&](int u) { return D * warp + u % D; };
    auto issue = [&](int u) {                                // one lane issues a step's copies
        const int it = S1W_W * u + warp;
        if (lane != 0 || it >= total) return;
        const bool fwd = it < K;
        const int R = fwd ? it : total - 1 - it, nd = min(kb, fwd ? R : K - 1 - R), st = stage(u);
        float* dst = St + (size_t)st * stage_floats;
        mbar_expect_tx(&full[st], (1 + (nd > 0)) * NB2 * 4 + (nd > 1 ? nb * 8 * NB * 4 : 0));
        tma_load_tile(dst, &tmt, (int)(tile_index(toff, kb, R, R) / NB), &full[st]);
        if (nd > 0) {
            const long long ti = fwd ? tile_index(toff, kb, R, R - 1) : tile_index(toff, kb, R + 1, R);
            tma_load_tile(dst + NB2, &tmt, (int)(ti / NB), &full[st]);
        }
        if (nd > 1) {
            const long long ti = fwd ? tile_index(toff, kb, R, R - 2) : tile_index(toff, kb, R + 2, R);
            for (int q = 0; q < nb; ++q)
                tma_load_box(dst + 2 * NB2 + q * 8 * NB, &tmc, 8 * (g0 + q), (int)(ti / NB), &full[st]);
        }
    };
    for (int u = 0; u < D; ++u) issue(u);

    // ---------------- the chain warps, lane = row (column in the backward sweep)
    auto announce = [&](int id) { asm volatile("bar.arrive %0, 64;\n" ::"r"(id) : "memory"); };
    auto await = [&](int id) { asm volatile("bar.sync %0, 64;\n" ::"r"(id) : "memory"); };
    float* far = Fr + (size_t)warp * nbox * 8 * NB;
    float l[NB], tr[NB], xfar = 0.f, dv = 1.f;               // near tile's and T's row, the far tile's part, D^{-1}
    // the rows of step `it` (turn u) into registers, its far boxes to this warp's copy, the next copies into its stage
    auto fetch = [&](int it, int u) -> bool {
        const int st = stage(u);
        const bool fwd = it < K;
        const int R = fwd ? it : total - 1 - it, nd = min(kb, fwd ? R : K - 1 - R);
        if (!fwd) dv = dinv[roff + (long long)R * NB + lane];
        if (*(volatile int*)&s_abort) return false;          // the chain ends without the tiles
        if (!mbar_wait_bounded(&full[st], (u / D) & 1u)) { give_up(); return false; }
        const float *T = St + (size_t)st * stage_floats, *L = T + NB2, *F = L + NB2;
        if (fwd) {
#pragma unroll
            for (int g = 0; g < 8; ++g) {
                const float4 a = *reinterpret_cast<const float4*>(T + lane * NB + ((g ^ (lane & 7)) << 2));
                tr[4 * g] = a.x; tr[4 * g + 1] = a.y; tr[4 * g + 2] = a.z; tr[4 * g + 3] = a.w;
                const float4 c = *reinterpret_cast<const float4*>(L + lane * NB + ((g ^ (lane & 7)) << 2));
                l[4 * g] = c.x; l[4 * g + 1] = c.y; l[4 * g + 2] = c.z; l[4 * g + 3] = c.w;
            }
        } else {
#pragma unroll
            for (int k = 0; k < NB; ++k) {
                tr[k] = T[swz(k, lane)];
                l[k] = L[swz(k, lane)];
            }
        }
        if (nd == 0)                                         // (no near tile: the stage holds an older one)
#pragma unroll
            for (int k = 0; k < NB; ++k) l[k] = 0.f;
        if (nd > 1)
            for (int e = lane; e < nb * 2 * NB; e += 32)
                *reinterpret_cast<float4*>(far + 4 * e) = *reinterpret_cast<const float4*>(F + 4 * e);
        __syncwarp();
        issue(u + D);
        return true;
    };
    // the far tile's product of step `it` (z of step it - 2 is there)
    auto far_part = [&](int it) {
        const bool fwd = it < K;
        const int R = fwd ? it : total - 1 - it, nd = min(kb, fwd ? R : K - 1 - R);
        xfar = 0.f;
        if (nd < 2) return;
        if (fwd) {
            for (int q = 0; q < nb; ++q) {
                const float4 a = *reinterpret_cast<const float4*>(far + q * 8 * NB + lane * 8);
                const float4 c = *reinterpret_cast<const float4*>(far + q * 8 * NB + lane * 8 + 4);
                const float4 u = *reinterpret_cast<const float4*>(zs + (R - 2) * NB + 8 * (g0 + q));
                const float4 v = *reinterpret_cast<const float4*>(zs + (R - 2) * NB + 8 * (g0 + q) + 4);
                xfar += (fmaf(a.x, u.x, fmaf(a.y, u.y, fmaf(a.z, u.z, a.w * u.w)))) +
                        (fmaf(c.x, v.x, fmaf(c.y, v.y, fmaf(c.z, v.z, c.w * v.w))));
            }
        } else if ((lane >> 3) >= g0 && (lane >> 3) - g0 < nb) {
            const float* f = far + ((lane >> 3) - g0) * 8 * NB + (lane & 7);
            const float* z = zs + (R + 2) * NB;
            const int kend = min(NB, bw - 31);               // rows of the far tile with nonzeros
            float s1 = 0.f;
            int k = 0;
            for (; k + 1 < kend; k += 2) {
                xfar = fmaf(f[k * 8], z[k], xfar);
                s1 = fmaf(f[k * 8 + 8], z[k + 1], s1);
            }
            if (k < kend) xfar = fmaf(f[k * 8], z[k], xfar);
            xfar += s1;
        }
    };
    auto dot = [&](const float (&a)[NB], const float* v) {   // sum_k a[k] v[k], v broadcast from shared memory
        float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll
        for (int g = 0; g < 8; ++g) {
            const float4 x = *reinterpret_cast<const float4*>(v + 4 * g);
            s0 = fmaf(a[4 * g], x.x, s0); s1 = fmaf(a[4 * g + 1], x.y, s1);
            s2 = fmaf(a[4 * g + 2], x.z, s2); s3 = fmaf(a[4 * g + 3], x.w, s3);
        }
        return (s0 + s1) + (s2 + s3);
    };
#pragma unroll
    for (int k = 0; k < NB; ++k) { l[k] = 0.f; tr[k] = 0.f; }
    int u = 0, landed = 0;                                   // turn; turns whose copies have been waited for
    for (int it = warp; it < total; it += S1W_W, ++u) {
        const bool fwd = it < K;
        const int R = fwd ? it : total - 1 - it, other = fwd ? max(R - 1, 0) : min(R + 1, K - 1);
        if (fetch(it, u)) landed = u + 1;
        if (it >= 2) await(1 + ((it - 2) & 3));              // z of step it - 2
        far_part(it);
        if (it >= 1) await(5 + ((it - 1) & 3));              // z of step it - 1
        const float x = fmaf(dv, zs[R * NB + lane], -xfar);  // (dv = 1 forward)
        Ac[lane] = x - dot(l, zs + other * NB);
        __syncwarp();
        const float z = dot(tr, Ac);
        zs[R * NB + lane] = z;
        __syncwarp();
        if (it + 1 < total) announce(5 + warp);
        if (it + 2 < total) announce(1 + warp);
    }
    for (int v = landed; v < landed + D && S1W_W * v + warp < total; ++v)     // after a timeout only
        mbar_wait_bounded(&full[stage(v)], (v / D) & 1u);
    asm volatile("bar.sync 9, %0;\n" ::"r"(NTC) : "memory");
    for (int e = t; e < K * NB; e += NTC) X[roff + e] = f32_to_f64(zs[e]);
}

// ---- one right-hand side, FP64 bands (the local solves of the plain form)
// A DFMA holds a scheduler's FP64 pipe for some 67 cycles whatever its active
// lanes, so a step's products are spread over four warps (four pipes) by k:
// warp w multiplies columns 8 w .. 8 w + 7 of every tile, lane = row, and the
// partial sums are exchanged through shared memory.  Warp w then sums and
// finishes exactly the rows 8 w .. 8 w + 7 that it multiplies next, as its
// k-slice of T_R and of the next step's nearest tile: two barriers and two
// two-level sums a step, where every lane group of a row summing its own part
// with each product took 3700 cycles a step at kb = 2.  The columns of the
// outermost tile that lie in the band are dealt out singly.  A fifth warp
// streams the tiles by TMA in halves of 16 columns (128-byte swizzle), of the
// outermost tile only the halves that hold nonzeros.  Waits and time-outs as in
// k_tile_solve_band_ks.  Ring and vector share 226 KB: at two stages of kb + 1
// tiles, n <= 24,400 at kb = 1, 12,100 at kb = 7, 8,000 at kb = 9, 3,900 at kb = 11,
// 1,900 at kb = 12; beyond, and for wide bands in large batches, k_tile_solve1_dense.
// Measured (warm L2): 144 problems of n = 1296, b = 37 147 -> 125 us, 27 of
// n = 1728, b = 157 331 -> 295 us.
constexpr int S1D_W = 4, S1D_HALF = NB * 16;           // doubles of a half tile
__host__ __device__ constexpr size_t s1d_bytes(int S, int nst, int K) {
    return 1024 + sizeof(double) * ((size_t)nst * S * NB2 + 2 * S1D_W * NB + NB + (size_t)K * NB);
}

__global__ void __launch_bounds__(32 * (S1D_W + 1)) k_tile_solve1_f64(
    const __grid_constant__ CUtensorMap tmt, const double* __restrict__ dinv, const int* __restrict__ kb_,
    const int* __restrict__ K_, const int* __restrict__ b_, const long long* __restrict__ toff_,
    const long long* __restrict__ roff_, double* __restrict__ X, const int* __restrict__ gdone, int S, int nst)
{
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    double* St = reinterpret_cast<double*>(base);            // [nst][S][2][32][16]
    double* P1 = St + (size_t)nst * S * NB2;                 // [4][32] partial sums
    double* P2 = P1 + S1D_W * NB;
    double* Ac = P2 + S1D_W * NB;                            // [32]
    double* zs = Ac + NB;                                    // [K * 32]
    __shared__ unsigned long long full[4], empty[4];
    __shared__ int s_abort, s_stop;
    if (gdone && *gdone) return;
    const int i = blockIdx.x;
    const int kb = kb_[i], K = K_[i], bw = b_[i];
    if (kb >= S || K == 0) return;                           // never launched so (host dispatch)
    const long long toff = toff_[i], roff = roff_[i];
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int k_out = max(0, NB * kb - bw);                  // columns of the outermost tile before it are zero
    const int h_out = k_out >> 4;                            // its first half with nonzeros
    if (t == 0) {
        s_abort = 0;
        s_stop = 0;
        for (int s = 0; s < nst; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], S1D_W);
        }
        fence_mbar_init();
    }
    for (int e = t; e < K * NB; e += 32 * (S1D_W + 1)) zs[e] = X[roff + e];
    __syncthreads();
    auto give_up = [&]() {
        if (atomicExch(&s_abort, 1) == 0) atomicAdd(&g_wait_timeouts, 1);
    };
    const int total = 2 * K;

    if (warp == S1D_W) {
        // ---------------- producer: one lane issues every copy
        if (lane == 0) {
            unsigned pending = 0, par = 0, ph = 0;
            int st = 0;
            for (int it = 0; it < total; ++it) {
                if (it >= nst) {
                    if (!mbar_wait_bounded(&empty[st], ((ph >> st) & 1u) ^ 1u)) { give_up(); break; }
                    pending &= ~(1u << st);
                }
                if (*(volatile int*)&s_abort) break;
                const bool fwd = it < K;
                const int R = fwd ? it : total - 1 - it, nd = min(kb, fwd ? R : K - 1 - R);
                const int skipped = nd == kb && kb > 0 ? h_out : 0;
                double* dst = St + (size_t)st * S * NB2;
                mbar_expect_tx(&full[st], (2 * (nd + 1) - skipped) * S1D_HALF * 8);
                for (int d = nd; d >= 0; --d) {
                    const long long ti = fwd ? tile_index(toff, kb, R, R - d) : tile_index(toff, kb, R + d, R);
                    for (int h = d == kb && kb > 0 ? h_out : 0; h < 2; ++h)
                        tma_load_box(dst + (size_t)d * NB2 + h * S1D_HALF, &tmt, 16 * h, (int)(ti / NB), &full[st]);
                }
                pending |= 1u << st;
                par = (par & ~(1u << st)) | (((ph >> st) & 1u) << st);
                ph ^= 1u << st;
                st = st + 1 == nst ? 0 : st + 1;
            }
            // after an abort, copies still in flight must land before the CTA exits
            if (*(volatile int*)&s_abort)
                for (int s = 0; s < nst; ++s)
                    if (pending & (1u << s)) mbar_wait_bounded(&full[s], (par >> s) & 1u);
        }
        return;
    }

    // ---------------- consumer warps
    auto consumers_sync = [&]() { asm volatile("bar.sync 1, %0;\n" ::"r"(32 * S1D_W) : "memory"); };
    // a0 += columns 8 w .. 8 w + 7 (rows, backward) of a tile times v[8 w ..]: lane = row (column).  One chain: a
    // dependent DFMA starts as soon as the pipe is free
    double a0;
    auto slice = [&](const double* T, const double* v, bool fwd) {
        const double2* vv = reinterpret_cast<const double2*>(v + 8 * warp);
        if (fwd) {
            const double* Tr = T + (warp >> 1) * S1D_HALF + lane * 16;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const double2 l = *reinterpret_cast<const double2*>(Tr + (((4 * (warp & 1) + c) ^ (lane & 7)) << 1));
                const double2 x = vv[c];
                a0 = fma(l.x, x.x, a0);
                a0 = fma(l.y, x.y, a0);
            }
        } else {
            const double* Tc = T + (lane >> 4) * S1D_HALF + (lane & 1);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int k = 8 * warp + 2 * c;
                const double2 x = vv[c];
                a0 = fma(Tc[k * 16 + ((((lane >> 1) & 7) ^ (k & 7)) << 1)], x.x, a0);
                a0 = fma(Tc[(k + 1) * 16 + ((((lane >> 1) & 7) ^ ((k + 1) & 7)) << 1)], x.y, a0);
            }
        }
    };
    const int row = 8 * warp + (lane >> 2), part = lane & 3;  // the slice's row that this lane helps to sum
    auto sum4 = [&](const double* P) {
        double v = P[part * NB + row];
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        v += __shfl_xor_sync(0xffffffffu, v, 2);
        return v;
    };
    int st = 0;
    unsigned ph = 0;
    for (int it = 0; it < total; ++it) {
        const bool fwd = it < K;
        const int R = fwd ? it : total - 1 - it, sg = fwd ? -1 : 1, nd = min(kb, fwd ? R : K - 1 - R);
        const double dv = fwd ? 1.0 : dinv[roff + (long long)R * NB + row];
        const double* tiles = St + (size_t)st * S * NB2;
        const bool ok = mbar_wait_bounded(&full[st], (ph >> st) & 1u);
        if (!ok) give_up();
        a0 = 0.0;
        if (ok) {
            for (int d = 2; d <= nd; ++d) {
                const double *T = tiles + (size_t)d * NB2, *z = zs + (R + sg * d) * NB;
                if (d < kb) {
                    slice(T, z, fwd);
                } else if (fwd) {                            // columns k_out .. 31, dealt out
                    for (int k = k_out + warp; k < NB; k += S1D_W)
                        a0 = fma(T[(k >> 4) * S1D_HALF + lane * 16 + ((((k >> 1) & 7) ^ (lane & 7)) << 1) + (k & 1)],
                                 z[k], a0);
                } else if (lane >> 4 >= h_out) {             // rows 0 .. 31 - k_out, dealt out
                    for (int k = warp; k < NB - k_out; k += S1D_W)
                        a0 = fma(T[(lane >> 4) * S1D_HALF + k * 16 + ((((lane >> 1) & 7) ^ (k & 7)) << 1) + (lane & 1)],
                                 z[k], a0);
                }
            }
            if (nd > 0) {
                // (kb = 1: the halves that were not copied hold zeros of the band)
                const double *T = tiles + NB2, *z = zs + (R + sg) * NB;
                if (kb > 1) slice(T, z, fwd);
                else if (fwd ? (warp >> 1) >= h_out : (lane >> 4) >= h_out) slice(T, z, fwd);
            }
        }
        P1[warp * NB + lane] = a0;
        consumers_sync();                                    // every partial sum is in P1
        const double y = fma(dv, zs[R * NB + row], -sum4(P1));
        if (part == 0) Ac[row] = y;
        __syncwarp();
        a0 = 0.0;
        if (ok) slice(tiles, Ac, fwd);
        P2[warp * NB + lane] = a0;
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[st]);
        if (t == 0) *(volatile int*)&s_stop = *(volatile int*)&s_abort;
        consumers_sync();                                    // every partial of the solution is in P2
        if (*(volatile int*)&s_stop) break;                  // sampled once: every warp leaves after this step
        const double z = sum4(P2);
        if (part == 0) zs[R * NB + row] = z;
        __syncwarp();
        ph ^= 1u << st;
        st = st + 1 == nst ? 0 : st + 1;
    }
    consumers_sync();
    for (int e = t; e < K * NB; e += 32 * S1D_W) X[roff + e] = zs[e];
}

using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_tiled() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    });
    return fn;
}

// [elems / 32][32] FP32 view of a tile array, 32 x 32 boxes, 128-byte swizzle.
bool encode_tile_map(const float* base, long long elems, CUtensorMap* m) {
    EncodeTiledFn enc = encode_tiled();
    if (!enc || !base || elems <= 0) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)NB, (cuuint64_t)(elems / NB)};
    const cuuint64_t strides[1] = {(cuuint64_t)NB * sizeof(float)};
    const cuuint32_t box[2] = {(cuuint32_t)NB, (cuuint32_t)NB};
    const cuuint32_t estr[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, (void*)base, dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// [elems / 32][32] view, boxes of `cols` columns x 32 rows.
bool encode_box_map(const void* base, CUtensorMapDataType type, size_t esize, long long elems, int cols,
                    CUtensorMapSwizzle swizzle, CUtensorMap* m) {
    EncodeTiledFn enc = encode_tiled();
    if (!enc || !base || elems <= 0) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)NB, (cuuint64_t)(elems / NB)};
    const cuuint64_t strides[1] = {(cuuint64_t)NB * esize};
    const cuuint32_t box[2] = {(cuuint32_t)cols, (cuuint32_t)NB};
    const cuuint32_t estr[2] = {1, 1};
    return enc(m, type, 2, (void*)base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
               CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The tile descriptor of an FP32 batch (built once per tiles_f allocation).
const CUtensorMap* tile_tensor_map(const TileBatch& tb) {
    if (!tb.prec || !tb.tiles_f.p || tb.total_tile_elems <= 0) return nullptr;
    if (tb.tmap_base == tb.tiles_f.p) return reinterpret_cast<const CUtensorMap*>(tb.tmap_tiles);
    CUtensorMap* m = reinterpret_cast<CUtensorMap*>(tb.tmap_tiles);
    if (!encode_tile_map(tb.tiles_f.p, tb.total_tile_elems, m)) return nullptr;
    tb.tmap_base = tb.tiles_f.p;
    return m;
}

// FP32 factors, any number of columns
template <typename XT>
void solve_f32(const TileBatch& tb, XT* X, int ldx, int ncols, const int* skip, cudaStream_t s, const int* gdone) {
    int maxkb = 0;
    for (int v : tb.kb) maxkb = std::max(maxkb, v);
    const CUtensorMap* tm = maxkb <= 12 ? tile_tensor_map(tb) : nullptr;
    if (tm) {
        solve_band_f32(tb, *tm, maxkb, X, ldx, ncols, skip, s, gdone);
        return;
    }
    k_tile_solve<float, XT><<<dim3(tb.P, (ncols + NB - 1) / NB), TPB, 0, s>>>(
        tb.tiles_f.p, tb.dinv_f.p, tb.d_n.p, tb.d_kb.p, tb.d_K.p, tb.d_toff.p, tb.d_roff.p, X, ldx, ncols, skip, gdone);
    MSDD_LAUNCH_CHECK();
}

__global__ void k_fill_identity(double* __restrict__ E, const int* __restrict__ n_, const int* __restrict__ K_,
                                const long long* __restrict__ roff_, int lde) {
    const int i = blockIdx.y;
    const int n = n_[i];
    const long long rows = (long long)K_[i] * NB;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < rows * lde;
         e += (long long)gridDim.x * blockDim.x) {
        long long r = e / lde, c = e % lde;
        E[(roff_[i] + r) * lde + c] = (r == c && r < n) ? 1.0 : 0.0;
    }
}

template <typename T>
__global__ void k_tile_from_dense(T* __restrict__ tiles, const int* __restrict__ n_, const int* __restrict__ kb_,
                                  const int* __restrict__ K_, const long long* __restrict__ toff_,
                                  const int* __restrict__ b_, const double* __restrict__ src,
                                  const long long* __restrict__ soff, const int* __restrict__ lds)
{
    const int i = blockIdx.y;
    const int n = n_[i], kb = kb_[i], K = K_[i], bw = b_[i];
    const long long ntile = (long long)K * (kb + 1) * NB2;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < ntile;
         e += (long long)gridDim.x * blockDim.x) {
        long long tileno = e / NB2;
        int within = (int)(e % NB2);
        int R = (int)(tileno / (kb + 1)), d = (int)(tileno % (kb + 1));
        int C = R - d;
        int rr = R * NB + within / NB, cc = C * NB + within % NB;
        T v = 0;
        if (C >= 0 && rr < n && cc < n && cc >= 0 && cc <= rr && rr - cc <= bw)
            v = (T)src[soff[i] + (long long)rr * lds[i] + cc];
        tiles[toff_[i] + e] = v;
    }
}

}  // namespace

TileBatch TileBatch::slice(int p0, int np) const {
    TileBatch v;
    v.P = np;
    v.prec = prec;
    auto sub = [&](const auto& vec) { return std::decay_t<decltype(vec)>(vec.begin() + p0, vec.begin() + p0 + np); };
    v.n = sub(n); v.kb = sub(kb); v.K = sub(K); v.b = sub(b); v.toff = sub(toff); v.roff = sub(roff);
    v.total_tile_elems = total_tile_elems;
    v.total_rows = total_rows;
    v.max_K = 0;
    for (int k : v.K) v.max_K = std::max(v.max_K, k);
    v.d_n = d_n.view(p0, np); v.d_kb = d_kb.view(p0, np); v.d_K = d_K.view(p0, np); v.d_b = d_b.view(p0, np);
    v.d_status = d_status.view(p0, np); v.d_nreg = d_nreg.view(p0, np);
    v.d_toff = d_toff.view(p0, np); v.d_roff = d_roff.view(p0, np);
    v.tiles_d = tiles_d.view(0, tiles_d.n); v.dinv_d = dinv_d.view(0, dinv_d.n);
    v.tiles_f = tiles_f.view(0, tiles_f.n); v.dinv_f = dinv_f.view(0, dinv_f.n);
    tile_tensor_map(*this);                     // build the shared descriptor once, then copy it
    memcpy(v.tmap_tiles, tmap_tiles, sizeof(tmap_tiles));
    v.tmap_base = tmap_base;
    return v;
}

void TileBatch::layout(const std::vector<int>& n_, const std::vector<int>& b_, int precision, cudaStream_t s) {
    P = (int)n_.size();
    prec = precision;
    tmap_base = nullptr;
    n = n_;
    kb.resize(P);
    K.resize(P);
    b.resize(P);
    toff.resize(P);
    roff.resize(P);
    total_tile_elems = 0;
    total_rows = 0;
    max_K = 0;
    for (int i = 0; i < P; ++i) {
        K[i] = n[i] > 0 ? (int)ceil_div(n[i], NB) : 0;
        int bi = b_[i] < n[i] - 1 ? b_[i] : n[i] - 1;
        if (bi < 0) bi = 0;
        b[i] = bi;
        kb[i] = (int)ceil_div(bi, NB);
        if (kb[i] > K[i] - 1) kb[i] = K[i] > 0 ? K[i] - 1 : 0;
        toff[i] = total_tile_elems;
        roff[i] = total_rows;
        total_tile_elems += (long long)K[i] * (kb[i] + 1) * NB2;
        total_rows += (long long)K[i] * NB;
        if (K[i] > max_K) max_K = K[i];
    }
    d_n.upload(n, s);
    d_kb.upload(kb, s);
    d_b.upload(b, s);
    d_K.upload(K, s);
    d_toff.upload(toff, s);
    d_roff.upload(roff, s);
    d_status.alloc(P);
    d_nreg.alloc(P);
    if (prec) {
        tiles_f.alloc(total_tile_elems);
        dinv_f.alloc(total_rows);
        tiles_d.release();
        dinv_d.release();
    } else {
        tiles_d.alloc(total_tile_elems);
        dinv_d.alloc(total_rows);
        tiles_f.release();
        dinv_f.release();
    }
}

void tile_zero(TileBatch& tb, cudaStream_t s) {
    if (tb.prec) tb.tiles_f.zero(s); else tb.tiles_d.zero(s);
}

void tile_from_dense(TileBatch& tb, const double* src, const long long* d_soff, const int* d_lds, cudaStream_t s) {
    if (tb.P == 0) return;
    long long maxt = 0;
    for (int i = 0; i < tb.P; ++i) maxt = std::max(maxt, (long long)tb.K[i] * (tb.kb[i] + 1) * NB2);
    dim3 grid(std::min<long long>(ceil_div(maxt, 256), 1024), tb.P);
    if (tb.prec)
        k_tile_from_dense<float><<<grid, 256, 0, s>>>(tb.tiles_f.p, tb.d_n.p, tb.d_kb.p, tb.d_K.p, tb.d_toff.p, tb.d_b.p, src, d_soff, d_lds);
    else
        k_tile_from_dense<double><<<grid, 256, 0, s>>>(tb.tiles_d.p, tb.d_n.p, tb.d_kb.p, tb.d_K.p, tb.d_toff.p, tb.d_b.p, src, d_soff, d_lds);
    MSDD_LAUNCH_CHECK();
}

void tile_identity(const TileBatch& tb, double* E, int lde, cudaStream_t s) {
    if (tb.P == 0) return;
    dim3 grid(64, tb.P);
    k_fill_identity<<<grid, 256, 0, s>>>(E, tb.d_n.p, tb.d_K.p, tb.d_roff.p, lde);
    MSDD_LAUNCH_CHECK();
}

void tile_factor(TileBatch& tb, double reg_tol, cudaStream_t s) {
    if (tb.P == 0) return;
    int maxkb = 0;
    for (int v : tb.kb) maxkb = std::max(maxkb, v);
    bool dense = tb.max_K >= 3;
    for (int i = 0; i < tb.P && dense; ++i) dense = tb.kb[i] >= tb.K[i] - 1;
    if (dense || !tb.prec) {
        auto run = [&](auto* tl, auto* dv) {
            using T = std::remove_pointer_t<decltype(tl)>;
            k_save_diag<T><<<tb.P, TPB, 0, s>>>(tl, dv, tb.d_kb.p, tb.d_K.p, tb.d_toff.p, tb.d_roff.p, tb.d_status.p,
                                               tb.d_nreg.p);
            MSDD_LAUNCH_CHECK();
            for (int k = 0; k < tb.max_K; ++k) {
                k_rl_diag<T><<<tb.P, 128, 0, s>>>(tl, dv, tb.d_n.p, tb.d_kb.p, tb.d_K.p, tb.d_toff.p, tb.d_roff.p,
                                                 tb.d_status.p, tb.d_nreg.p, reg_tol, k);
                MSDD_LAUNCH_CHECK();
                const int m = std::min(maxkb, tb.max_K - 1 - k);
                if (m == 0) continue;
                k_rl_panel<T><<<dim3(tb.P, m), TPB, 0, s>>>(tl, dv, tb.d_kb.p, tb.d_K.p, tb.d_b.p, tb.d_toff.p,
                                                           tb.d_roff.p, k);
                MSDD_LAUNCH_CHECK();
                const int nt = m * (m + 1) / 2, ny = std::min(nt, 65535);
                k_rl_update<T><<<dim3(tb.P, ny, (nt + ny - 1) / ny), TPB, 0, s>>>(
                    tl, dv, tb.d_kb.p, tb.d_K.p, tb.d_b.p, tb.d_toff.p, tb.d_roff.p, k);
                MSDD_LAUNCH_CHECK();
            }
        };
        if (tb.prec) run(tb.tiles_f.p, tb.dinv_f.p);
        else run(tb.tiles_d.p, tb.dinv_d.p);
        return;
    }
    if (tb.prec && maxkb <= 2) {
        const size_t b = factor_band32_smem();
        raise_smem_limit(k_tile_factor_band32, b);
        k_tile_factor_band32<<<tb.P, FB_T, b, s>>>(tb.tiles_f.p, tb.dinv_f.p, tb.d_n.p, tb.d_kb.p, tb.d_K.p,
                                                  tb.d_toff.p, tb.d_roff.p, tb.d_status.p, tb.d_nreg.p, reg_tol);
        MSDD_LAUNCH_CHECK();
        return;
    }
    if (tb.prec && maxkb <= TF_KBM) {
        // 3 <= kb <= 12: panel updates on the tensor cores (lo parts of the factor in scratch)
        const CUtensorMap* thi = tile_tensor_map(tb);
        DevBuf<float> lo(tb.total_tile_elems);
        alignas(64) CUtensorMap tlo;
        if (thi && encode_tile_map(lo.p, tb.total_tile_elems, &tlo)) {
            const size_t b = tf_smem_bytes();
            raise_smem_limit(k_tile_factor_tc, b);
            k_tile_factor_tc<<<tb.P, TF_NT, b, s>>>(*thi, tlo, tb.tiles_f.p, lo.p, tb.total_tile_elems, tb.dinv_f.p,
                                                   tb.d_n.p, tb.d_kb.p, tb.d_K.p, tb.d_toff.p, tb.d_roff.p,
                                                   tb.d_status.p, tb.d_nreg.p, reg_tol);
            MSDD_LAUNCH_CHECK();
            return;
        }
    }
    k_tile_factor<float><<<tb.P, TPB, 0, s>>>(tb.tiles_f.p, tb.dinv_f.p, tb.d_n.p, tb.d_kb.p, tb.d_K.p, tb.d_toff.p,
                                             tb.d_roff.p, tb.d_status.p, tb.d_nreg.p, reg_tol);
    MSDD_LAUNCH_CHECK();
}

void tile_check_waits() {
    int n = 0;
    MSDD_CUDA(cudaMemcpyFromSymbol(&n, g_wait_timeouts, sizeof(int)));
    if (n) {
        const int zero = 0;
        MSDD_CUDA(cudaMemcpyToSymbol(g_wait_timeouts, &zero, sizeof(int)));
        throw WaitTimeout("a band solve gave up waiting for its tile copies (" + std::to_string(n) + " CTAs)");
    }
}

void tile_solve(const TileBatch& tb, double* X, int ldx, int ncols, const int* skip, cudaStream_t s,
                const int* gdone) {
    if (tb.P == 0) return;
    if (ncols > ldx) throw std::runtime_error("tile_solve: more columns than the leading dimension");
    const size_t zbytes = (size_t)tb.max_K * NB * sizeof(double);   // upper bound for both precisions
    if (ncols == 1 && ldx == 1 && skip == nullptr) {
        int maxkb = 0;
        for (int v : tb.kb) maxkb = std::max(maxkb, v);
        if (tb.prec && maxkb <= 2) {
            const CUtensorMap* tm = tile_tensor_map(tb);
            alignas(64) CUtensorMap tc;
            int nbox = 0;
            for (int i = 0; i < tb.P; ++i)
                if (tb.kb[i] == 2) nbox = std::max(nbox, 4 - s1w_group0(tb.b[i]));
            // one turn ahead where two do not fit beside the vector (n = 38500, b = 38: 3.4 ms without the ring, 0.73 with
            // it), and where two leave one CTA an SM to more CTAs than SMs (n = 1369, b = 60, 256 problems: 126 -> 103 us)
            const size_t deep = s1w_bytes(2, nbox, tb.max_K);
            const int D = deep <= (tb.P > NUM_SMS ? 112 : 226) * 1024 ? 2 : 1;
            const size_t bytes = s1w_bytes(D, nbox, tb.max_K);
            if (tm && bytes <= 226 * 1024 &&
                encode_box_map(tb.tiles_f.p, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, tb.total_tile_elems, 8,
                               CU_TENSOR_MAP_SWIZZLE_NONE, &tc)) {
                auto kern = D == 2 ? k_tile_solve1_warp<2> : k_tile_solve1_warp<1>;
                raise_smem_limit(kern, bytes);
                kern<<<tb.P, 32 * S1W_W, bytes, s>>>(*tm, tc, tb.dinv_f.p, tb.d_kb.p, tb.d_K.p, tb.d_b.p,
                                                     tb.d_toff.p, tb.d_roff.p, X, gdone, nbox);
                MSDD_LAUNCH_CHECK();
                return;
            }
        }
        if (!tb.prec) {
            int nst = 4;
            while (nst > 2 && s1d_bytes(maxkb + 1, nst, tb.max_K) > 200 * 1024) --nst;
            const size_t bytes = s1d_bytes(maxkb + 1, nst, tb.max_K);
            // wide bands: while the ring's CTAs (one an SM mostly) take at most two rounds over the SMs; many small CTAs
            // without a ring hide the tiles' latency better in more (b = 157, n = 1369: 152 problems 526 -> 278 us, 300
            // 575 -> 504, but 700 894 -> 1181; b = 100, n = 441, 700 problems 254 -> 334)
            const bool ring = maxkb <= 2 || zbytes > 160 * 1024 ||
                              tb.P <= 2 * NUM_SMS * (int)std::max<size_t>(1, 227 * 1024 / (bytes + 1024));
            alignas(64) CUtensorMap tm;
            if (ring && bytes <= 226 * 1024 &&
                encode_box_map(tb.tiles_d.p, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 8, tb.total_tile_elems, 16,
                               CU_TENSOR_MAP_SWIZZLE_128B, &tm)) {
                raise_smem_limit(k_tile_solve1_f64, bytes);
                k_tile_solve1_f64<<<tb.P, 32 * (S1D_W + 1), bytes, s>>>(tm, tb.dinv_d.p, tb.d_kb.p, tb.d_K.p, tb.d_b.p,
                                                                       tb.d_toff.p, tb.d_roff.p, X, gdone, maxkb + 1,
                                                                       nst);
                MSDD_LAUNCH_CHECK();
                return;
            }
        }
        if (tb.prec && maxkb > 2 && maxkb <= 12) {
            // wide bands, one right-hand side (PCG local solves of 3D boxes):
            // the step's off-diagonal tiles split over 6 warps, two stages of 13 tiles
            const CUtensorMap* tm = tile_tensor_map(tb);
            if (tm) {
                launch_band_split<12, 6, 2, 4>(tb, *tm, X, s, gdone);
                return;
            }
        }
        if (zbytes <= 160 * 1024) {
            raise_smem_limit(k_tile_solve1_dense<float>, zbytes);
            raise_smem_limit(k_tile_solve1_dense<double>, zbytes);
            if (tb.prec) k_tile_solve1_dense<float><<<tb.P, S1T, zbytes, s>>>(tb.tiles_f.p, tb.dinv_f.p, tb.d_kb.p, tb.d_K.p, tb.d_toff.p, tb.d_roff.p, X, gdone);
            else k_tile_solve1_dense<double><<<tb.P, S1T, zbytes, s>>>(tb.tiles_d.p, tb.dinv_d.p, tb.d_kb.p, tb.d_K.p, tb.d_toff.p, tb.d_roff.p, X, gdone);
            MSDD_LAUNCH_CHECK();
            return;
        }
    }
    if (!tb.prec && tile_solve_f64(tb, X, ldx, ncols, skip, s, gdone)) return;
    if (tb.prec) {
        solve_f32(tb, X, ldx, ncols, skip, s, gdone);
        return;
    }
    const dim3 grid(tb.P, (ncols + NB - 1) / NB);
    k_tile_solve<double, double><<<grid, TPB, 0, s>>>(tb.tiles_d.p, tb.dinv_d.p, tb.d_n.p, tb.d_kb.p, tb.d_K.p,
                                                      tb.d_toff.p, tb.d_roff.p, X, ldx, ncols, skip, gdone);
    MSDD_LAUNCH_CHECK();
}

void tile_solve(const TileBatch& tb, float* X, int ldx, int ncols, const int* skip, cudaStream_t s) {
    if (tb.P == 0) return;
    if (!tb.prec || ncols > ldx) throw std::runtime_error("tile_solve: FP32 blocks need FP32 factors and ncols <= ldx");
    solve_f32(tb, X, ldx, ncols, skip, s, nullptr);
}

}  // namespace msdd
