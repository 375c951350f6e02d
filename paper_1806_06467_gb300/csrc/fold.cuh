// fold.cuh -- matrix Fourier transforms on even / odd halves (real bases).
//
// A centred transform F[u'] = sum_j f[j'] exp(sigma 2 pi i c j' u') on symmetric grids (j' = j - n/2,
// u' = u - m/2) splits into the halves of f: with fe[k] = f[k] + f[-k], fo[k] = f[k] - f[-k]
// (fe[0] = f[0], fo[0] = 0; k = n/2 of an even n has no positive partner, which counts as 0),
//     F[+-u] = P[u] +- sigma i Q[u],  P = sum_k fe[k] cos(2 pi c k u),  Q = sum_k fo[k] sin(2 pi c k u).
// The two products have half the inner length and half the outputs, and their bases are real: a
// quarter of the multiply-adds of the complex product. In two dimensions the field becomes four
// parity classes T[py][px] on [k_y][k_x] half grids,
//     F[sv v, su u] = T00 + su sigma i T01 + sv sigma i T10 - su sv T11     (su, sv = +-1).
//
// A chain contracts the first index and appends the new one: Y[m][p][n] = sum_k X[p][k][m] W[p][k][n],
// p the parity of the contracted axis, W[0] = cos, W[1] = sin, m = (parity, index) of the other
// axis. The output has the input's form with the axes exchanged, so two of them transform a plane
// and bring its axes back in order, without a transpose.
//
// A plane masked symmetrically stays in its classes: the fold of the masked F is w_v w_u T (w_0 = 1,
// w_k = 2, the factor (sigma i)^(py + px) of the way out cancels against the way back), provided the
// mask is zero on the unpaired samples k = m/2 of an even m.
#pragma once
#include <cuda_runtime.h>

namespace coro {

// Samples of one half, the axis included: k = 0 ... n/2.
__host__ __device__ inline int fold_len(int n) { return n / 2 + 1; }

template <typename C> struct FoldReal;
template <> struct FoldReal<float2> { using type = float; };
template <> struct FoldReal<double2> { using type = double; };

enum FoldEpi : int {
    FOLD_PLAIN = 0,     // Y
    FOLD_MASK = 1,      // w_m w_n Y inside the disk m^2 + n^2 <= thr, else 0 (operand of the way back)
    FOLD_BABINET = 2    // a - w_m w_n scale Y inside the disk, else 0, a = base at (p, n, m)
};

// One contraction of `items` planes (grid z = item x parity).
//   X [item][2][K][M]  complex, M = 2 Hm: (parity, index) of the other axis; item stride sX
//   W [item][2][K][ldw] real, zero-filled beyond N up to ldw (a multiple of 32); item stride sW
//   Y [item][M][2][N]  complex; item stride sY (K splits: partial planes in `part`, then summed)
// base (FOLD_BABINET): class plane [2][base_h][2][base_h] read at (parity m, index m, p, n).
template <typename C>
struct FoldGemm {
    using R = typename FoldReal<C>::type;
    int M, N, K, items;
    const C* X;
    long long sX;
    const R* W;
    long long sW;
    int ldw;
    C* Y;
    long long sY;
    int epi;
    long long thr;
    R scale;
    const C* base;
    int base_h;
    long long thr_in = -1;   // X is zero where k^2 + (index of m)^2 > thr_in (< 0: no known zeros)
};

inline int fold_ldw(int n) { return (n + 31) / 32 * 32; }

// Fill bases and fold fields of up to `batch` items: W[b][2][K][ldw] (b-th constant c[b], K x N),
// F[b][2][hy][2][hx] from in[b][n][n] (hy, hx <= fold_len(n): what lies beyond is not read; samples
// with k_y^2 + k_x^2 > keep_r2 become 0, keep_r2 < 0: all kept). Either part may be left out (NULL).
template <typename C>
cudaError_t fold_prepare(const C* in, int n, int h, long long keep_r2, C* F, const double* c, int K, int N,
                         typename FoldReal<C>::type* W, int batch, cudaStream_t stream);

// Y = X W; FP32: 64 x 32 tiles in packed FP32x2 arithmetic, K split when the tiles leave the chip
// idle (then `part` of fold_part_elems() elements is needed); FP64: 32-row warp tiles.
size_t fold_part_elems(int M, int N, int K, int items);
cudaError_t fold_gemm(const FoldGemm<float2>& g, float2* part, cudaStream_t stream);
cudaError_t fold_gemm(const FoldGemm<double2>& g, double2* part, cudaStream_t stream);

// out[b][m][m] = scale[b] * (the four sign combinations of T[b][2][hm][2][hm]), sigma = sign.
template <typename C>
cudaError_t fold_expand(const C* T, int m, int sign, const double* scale, C* out, int batch, cudaStream_t stream);

}  // namespace coro
