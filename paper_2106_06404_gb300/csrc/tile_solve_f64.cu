// FP64 tile-band solves (the plain form's fine level, every dense coarse
// inverse).  See tile_ldlt.cuh for the storage format.
#include "tile_ldlt.cuh"

#include <algorithm>

namespace msdd {

namespace {

constexpr int F6_T = 128;       // 4 warps; warp w owns rows 8 w .. 8 w + 7 of a tile row
constexpr int F6_NST = 4;       // tiles in flight (8 KB each)

// z_R = T_R (x_R - sum_J L_RJ z_J) forward, x_R = T_R^T (D_R^{-1} z_R -
// sum_I L_IR^T x_I) backward, for C right-hand-side columns per CTA.
//
// The narrow FP64 pipe bounds this kernel (about 1.6 DFMA a clock on an SM),
// so everything is arranged around issuing few of them and on every SM:
//  - a thread owns one row and one column (lane = 8 rows x C columns x KS
//    parts of k), so a warp's k-range follows the zeros of its eight rows:
//    T_R is lower triangular, and element (r, k) of the tile d below the
//    diagonal is zero unless 32 d + r - k <= b.  Of the 3 x 1024 products a
//    column takes per step at b = 36, 1408 are left.
//  - the columns of a problem are spread over CTAs (C = 4, 2 or 1) until
//    there are enough of them for the chip; with C < 4 the k-range of a row
//    is split over KS = 4 / C lanes and summed by shuffles.  The tiles are
//    then read once per column group, from L2.
// Tiles come through a ring of F6_NST stages by cp.async, 16-byte chunk q of
// row r at position q ^ (r & 7): the eight rows of a warp (forward) and eight
// neighbouring columns of a row (backward) then fall in distinct banks.
//
// Measured (GB300): 14 columns of 27 problems of n = 1452..1872, b = 133..157
// 8.75 -> 0.75 ms a launch against one CTA of full tiles a problem; 16 columns
// of 72 problems of n ~ 1300, b = 36 1.28 -> 0.54 ms; dense inverses of 27
// matrices of order ~1000 and their copy about 20 ms less in the 96^3 set-up.
//
// INV: the right-hand sides are the identity columns c_lo .. c_lo + C - 1 (X is
// not read); z_R = 0 above the first of them, so the forward sweep starts there
// (three quarters of the products of n full solves).  The backward sweep runs over
// all rows: taking the upper triangle from the other columns, by symmetry, leaves
// columns whose errors belong to different solves, and K times such a column is off
// by the condition number: eigensolves of near-dependent generating systems then
// stalled at residuals around 1 where they reach 1e-4.
template <int C, bool INV>
__global__ void __launch_bounds__(F6_T) k_tile_solve_f64(
    const double* __restrict__ tiles, const double* __restrict__ dinv, const int* __restrict__ n_,
    const int* __restrict__ kb_, const int* __restrict__ K_, const int* __restrict__ b_,
    const long long* __restrict__ toff_, const long long* __restrict__ roff_, double* Xall, int ldx, int ncols,
    const int* __restrict__ skip, const int* __restrict__ gdone)
{
    constexpr int KS = 4 / C;
    extern __shared__ __align__(16) double f6_smem[];
    __shared__ double Acc[NB][C];
    const int i = blockIdx.x;
    if (skip && skip[i]) return;
    if (gdone && *gdone) return;
    const int n = n_[i], kb = kb_[i], K = K_[i], bw = b_[i];
    const int c_lo = blockIdx.y * C;
    if (INV && c_lo >= n) return;
    double* ring = f6_smem;                                    // [F6_NST][32 * 32]
    double* Zr = ring + F6_NST * NB2;                          // [kb + 1][32][C]
    const int S = kb + 1;
    const long long toff = toff_[i], roff = roff_[i];
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int r = 8 * warp + (lane >> 2), c = lane & (C - 1), part = (lane & 3) / C;
    const int wr0 = 8 * warp;                                   // first row of the warp
    const bool owner = part == 0 && c_lo + c < ncols;           // this lane reads and writes X
    double* X = Xall + c_lo + c;
    const int R0 = INV ? c_lo / NB : 0;

    // the tiles of a sweep, one after the other: (R, d) with d = dmax .. 1
    // (off-diagonal, far to near) and then 0 (T_R)
    auto issue = [&](int st, int R, int d, bool fwd) {
        if (R >= (fwd ? R0 : 0) && R < K) {
            const double* src = tiles + (fwd ? tile_index(toff, kb, R, R - d) : tile_index(toff, kb, R + d, R));
            double* dst = ring + st * NB2;
#pragma unroll
            for (int q = 0; q < NB2 / 2 / F6_T; ++q) {
                const int ch = t + q * F6_T, row = ch >> 4, g = ch & 15;
                cp_async16(dst + row * NB + ((g ^ (row & 7)) << 1), src + 2 * ch);
            }
        }
        cp_async_commit();
    };
    for (int sweep = 0; sweep < 2; ++sweep) {
        const bool fwd = sweep == 0;
        const int Rbeg = fwd ? R0 : K - 1, step = fwd ? 1 : -1;
        auto dmax = [&](int R) { return min(kb, fwd ? R - R0 : K - 1 - R); };
        int iR = Rbeg, id = dmax(Rbeg), ist = 0;                // next tile to issue
        auto issue_next = [&]() {
            issue(ist, iR, id, fwd);
            ist = ist + 1 == F6_NST ? 0 : ist + 1;
            if (id > 0) --id;
            else { iR += step; id = dmax(iR); }
        };
        for (int k = 0; k < F6_NST - 1; ++k) issue_next();
        auto load_x = [&](int R) -> double {
            if (R < R0 || R >= K) return 0.0;        // (backward, above R0: z_R = 0)
            const int row = R * NB + r;
            if (INV && fwd) return (row == c_lo + c && row < n) ? 1.0 : 0.0;
            return owner ? X[(roff + row) * ldx] : 0.0;
        };
        double xnext = load_x(Rbeg), dnext = fwd ? 0.0 : dinv[roff + Rbeg * NB + r];
        int st = 0;
        for (int R = Rbeg; R >= (fwd ? R0 : 0) && R < K; R += step) {
            const double xr = fwd ? xnext : dnext * xnext;
            xnext = load_x(R + step);                           // one step ahead
            if (!fwd && R > 0) dnext = dinv[roff + (R - 1) * NB + r];
            double a0 = 0.0, a1 = 0.0;
            for (int d = dmax(R); d >= 0; --d) {
                cp_async_wait_n<F6_NST - 2>();
                __syncthreads();
                issue_next();
                const double* T = ring + st * NB2;
                st = st + 1 == F6_NST ? 0 : st + 1;
                const double* V;
                int k0, k1;                                     // nonzero k of the warp's rows
                if (d > 0) {
                    V = Zr + (size_t)((fwd ? R - d : R + d) % S) * NB * C + c;
                    k0 = fwd ? max(0, NB * d + wr0 - bw) : 0;
                    k1 = fwd ? NB : min(NB, bw - NB * d + wr0 + 8);
                } else {
                    // sum over the parts, y = x - acc, then z = T y
                    double a = a0 + a1;
#pragma unroll
                    for (int o = C; o < 4; o <<= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
                    if (part == 0) Acc[r][c] = xr - a;
                    __syncthreads();
                    V = &Acc[0][c];
                    a0 = a1 = 0.0;
                    k0 = fwd ? 0 : wr0;
                    k1 = fwd ? wr0 + 8 : NB;
                }
                if (fwd) {
                    const double* Tr = T + r * NB;
                    for (int q = (k0 >> 1) + part; q < (k1 >> 1); q += KS) {
                        const double2 l = *reinterpret_cast<const double2*>(Tr + ((q ^ (r & 7)) << 1));
                        a0 = fma(l.x, V[2 * q * C], a0);
                        a1 = fma(l.y, V[(2 * q + 1) * C], a1);
                    }
                } else {
                    const int rc = r >> 1, ro = r & 1;
                    int k = k0 + part;
                    for (; k + KS < k1; k += 2 * KS) {
                        const double l0 = T[k * NB + ((rc ^ (k & 7)) << 1) + ro];
                        const double l1 = T[(k + KS) * NB + ((rc ^ ((k + KS) & 7)) << 1) + ro];
                        a0 = fma(l0, V[k * C], a0);
                        a1 = fma(l1, V[(k + KS) * C], a1);
                    }
                    if (k < k1) a0 = fma(T[k * NB + ((rc ^ (k & 7)) << 1) + ro], V[k * C], a0);
                }
            }
            double z = a0 + a1;
#pragma unroll
            for (int o = C; o < 4; o <<= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
            if (part == 0) Zr[(size_t)(R % S) * NB * C + r * C + c] = z;
            if (owner) X[(roff + R * NB + r) * ldx] = z;
        }
        cp_async_wait_n<0>();
        __syncthreads();
    }
}

__global__ void k_copy_squares(const double* __restrict__ E, int lde, const int* __restrict__ n_,
                               const long long* __restrict__ roff_, const long long* __restrict__ ooff,
                               const int* __restrict__ ldo, double* __restrict__ out) {
    const int i = blockIdx.x, n = n_[i], r1 = min(n, (int)(blockIdx.y + 1) * NB);
    const double* Ei = E + roff_[i] * lde;
    double* o = out + ooff[i];
    const int ld = ldo[i];
    for (int r = blockIdx.y * NB + (threadIdx.x >> 5); r < r1; r += 8)
        for (int c = threadIdx.x & 31; c < n; c += 32) o[(long long)r * ld + c] = Ei[(long long)r * lde + c];
}

size_t f6_bytes(int maxkb, int C) { return sizeof(double) * ((size_t)F6_NST * NB2 + (size_t)(maxkb + 1) * NB * C); }
constexpr size_t F6_MAX = 200 * 1024;

template <int C, bool INV>
void launch_f64(const TileBatch& tb, int maxkb, double* X, int ldx, int ncols, const int* skip, cudaStream_t s,
                const int* gdone) {
    const size_t b = f6_bytes(maxkb, C);
    raise_smem_limit(k_tile_solve_f64<C, INV>, b);
    k_tile_solve_f64<C, INV><<<dim3(tb.P, (ncols + C - 1) / C), F6_T, b, s>>>(
        tb.tiles_d.p, tb.dinv_d.p, tb.d_n.p, tb.d_kb.p, tb.d_K.p, tb.d_b.p, tb.d_toff.p, tb.d_roff.p, X, ldx, ncols,
        skip, gdone);
    MSDD_LAUNCH_CHECK();
}

// Columns per CTA: 4 while that gives 1.5 CTAs for each SM, else
// 2 or 1 (fewer columns cost shuffles and tile reads, idle SMs cost more).
// 0: the solution ring does not fit shared memory (dense problems beyond
// 21,000 rows).
int f64_columns(const TileBatch& tb, int maxkb, int ncols) {
    for (int c : {4, 2, 1})
        if ((c == 1 || (c <= ncols && (long long)tb.P * ((ncols + c - 1) / c) >= 3 * NUM_SMS / 2)) && f6_bytes(maxkb, c) <= F6_MAX)
            return c;
    return 0;
}

template <bool INV>
bool solve_f64(const TileBatch& tb, double* X, int ldx, int ncols, const int* skip, cudaStream_t s, const int* gdone) {
    int maxkb = 0;
    for (int v : tb.kb) maxkb = std::max(maxkb, v);
    switch (f64_columns(tb, maxkb, ncols)) {
        case 4: launch_f64<4, INV>(tb, maxkb, X, ldx, ncols, skip, s, gdone); return true;
        case 2: launch_f64<2, INV>(tb, maxkb, X, ldx, ncols, skip, s, gdone); return true;
        case 1: launch_f64<1, INV>(tb, maxkb, X, ldx, ncols, skip, s, gdone); return true;
        default: return false;
    }
}

}  // namespace

bool tile_solve_f64(const TileBatch& tb, double* X, int ldx, int ncols, const int* skip, cudaStream_t s,
                    const int* gdone) {
    return solve_f64<false>(tb, X, ldx, ncols, skip, s, gdone);
}

bool tile_inverse_f64(const TileBatch& tb, double* E, int lde, int ncols, cudaStream_t s) {
    return solve_f64<true>(tb, E, lde, ncols, nullptr, s, nullptr);
}

void copy_squares(const TileBatch& tb, const double* E, int lde, int maxn, const long long* d_ooff, const int* d_ld,
                  double* out, cudaStream_t s) {
    if (tb.P == 0 || maxn <= 0) return;
    k_copy_squares<<<dim3(tb.P, (maxn + NB - 1) / NB), 256, 0, s>>>(E, lde, tb.d_n.p, tb.d_roff.p, d_ooff, d_ld, out);
    MSDD_LAUNCH_CHECK();
}

}  // namespace msdd
