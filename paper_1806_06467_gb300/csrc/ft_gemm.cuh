// ft_gemm.cuh -- folded matrix Fourier transforms on the 5th-generation tensor cores: the parity
// classes and real bases of fold.cuh, contracted by split-precision GEMMs.
//
// One contraction: Y[q][p][c][n][i] = sum_k X[p][q][c][i][k] W[p][n][k], p the parity of the
// contracted axis (W[0] = cos, W[1] = sin), q and i parity and index of the other axis, c = 0 real,
// 1 imaginary part (the bases are real, so the parts never mix). The result has the operand's form
// with the axes exchanged and its inner index contiguous, so GEMMs chain without transposes.
//
// Formats (FtFormat): an operand value is held as planes whose leading products are summed,
//   FT_TF32            hi + lo (22 bits); hi.hi + hi.lo + lo.hi
//   FT_BF16            hi + mid + lo (24 bits); the six products down to 2^-16. Folding gathers
//                      a symmetric pupil in one class of four times its amplitude, and two planes
//                      (16 bits) then leave 1.1e-9 in a dark hole where the complex GEMM left 6.5e-10
//   Both are drained from the tensor-core accumulator into FP32 registers every 32 of K.
//   FT_EXT             four BF16 slices in groups of 64 of K (tcx_gemm.cuh: exact level-0 sums, ten
//                      products, two-float accumulation)
// Storage of an X operand [item][p][plane pair][(q, c, i)][2 ld], of a basis [p][plane pair][n][2 ld]: two
// planes share a row in alternating blocks of 64 bytes (ft_ke elements), so that a K slice of
// both is one 128-byte row of a TMA box. The copy engine takes rows at a fixed rate, some 2.5 clocks
// each: with one plane per 64-byte row every contraction loaded some 25 bytes per SM and clock at
// most (168-item Lyot set, pupil to occulter: 0.73 ms, 0.67 with shared rows).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

#include "tc_gemm.cuh"

namespace coro {

enum FtFormat : int { FT_TF32 = 0, FT_BF16 = 1, FT_EXT = 2 };

enum FtEpi : int {
    FT_SPLIT = 0,      // w scale Y inside the disk i^2 + n^2 <= thr_out, else 0 -> operand planes (w: see weights)
    FT_BABINET = 1,    // base - w scale Y inside the disk, else 0 -> operand planes
    FT_FLOAT = 2,      // Y as float planes (FT_EXT: float2, two-float)
    FT_DIFF = 3,       // base / w - scale Y as float planes (base 0 beyond its extent)
    FT_SEED = 4        // w inv_peak scale Y on lo <= i^2 + n^2 <= thr_out -> operand planes; dark-hole sums
};

struct FtItem {
    int K, N, H;                 // inner length, columns (outputs), valid rows i of each (q, c)
    int w_idx;                   // basis
    int thr_in;                  // X is zero where i^2 + k^2 > thr_in (-1: no known zeros)
    int thr_out, lo_out;         // mask of the masking epilogues
    double scale, inv_peak;
};

struct FtArgs {
    const FtItem* items;
    int* err;
    int R;                       // rows of each (q, c) of X (pitch; valid rows: item.H)
    int weights;                 // w = w_i w_n (w_0 = 1, w_k = 2) instead of 1
    void* dst;                   // operand planes, or floats [item][q][p][c][dst_R][dst_ld]
    long long dst_bstride;       // elements of one item
    int dst_R, dst_ld;
    const void* base;            // FT_BABINET / FT_DIFF: operand planes like dst with base_R, base_ld
    long long base_bstride;
    int base_R, base_ld, base_H; // base_H: valid extent of both indices
    double* dh_acc;              // FT_SEED: dark-hole sums [item]
};

struct FtOperand {               // X operand or basis
    void* base = nullptr;
    int items = 0;               // items, or bases
    int R = 0, cols = 0, ld = 0; // rows of each (q, c) (a basis: rows), inner length, its pitch
    long long stride = 0;        // elements of one item
};

inline int ft_planes(int fmt) { return fmt + 2; }
inline size_t ft_elem(int fmt) { return fmt == FT_TF32 ? 4 : 2; }
// Elements of a 64-byte block.
inline int ft_ke(int fmt) { return fmt == FT_TF32 ? 16 : 32; }
// Pitches in whole blocks (FT_EXT: in its groups of 64, which stay inside one plane), of rows and of
// the (q, c) planes alike: every sector that an epilogue's warp writes is written whole.
inline int ft_pitch(int fmt, int n) {
    const int q = fmt == FT_EXT ? 64 : ft_ke(fmt);
    return (n + q - 1) / q * q;
}
inline int ft_pairs(int fmt) { return fmt == FT_TF32 ? 1 : 2; }
FtOperand ft_operand(int fmt, int items, int rows, int cols);          // shape only
FtOperand ft_basis_operand(int fmt, int bases, int rows, int cols);
inline size_t ft_bytes(int fmt, const FtOperand& o) { return (size_t)o.items * o.stride * ft_elem(fmt); }

// A prepared contraction: tensor maps, tile width, launch shape.
struct FtGemm {
    CUtensorMap mx, mw;
    int fmt, items, nt, tiles_n, tiles_m, stages;
};
// max_n: columns over all items; max_nt: widest tile (128, or less).
cudaError_t ft_make(int fmt, const FtOperand& x, const FtOperand& w, int items, int max_n, int max_nt, FtGemm* g);
cudaError_t ft_launch(const FtGemm& g, int epi, const FtArgs& a, cudaStream_t stream);
// Tensor work over host copies of the items: products of valid outputs inside the known support,
// and of every tile and K slice that runs (2 flops each, all split products). Added to the outputs.
void ft_count_flops(const FtGemm& g, int epi, const FtItem* items, int R, double* useful, double* issued);

// complex64 [items][n][n] (pitch ld, item stride) -> its parity classes as an X operand contracting x
// ([px][plane][(py, c, ky)][kx]), up to extent h; keep_r2 >= 0: samples beyond become 0.
cudaError_t ft_fold(int fmt, const float2* src, long long src_bstride, int src_ld, int n, int h, int keep_r2,
                    const FtOperand& dst, cudaStream_t stream);
// basis `index` of w: W[p][n][k] = cos / sin(2 pi c k n), n < N, k < K
cudaError_t ft_basis(int fmt, double c, int K, int N, const FtOperand& w, int index, cudaStream_t stream);
// All of w at once, c = items[index].scale (device). One launch: six of 221 x 58 one by one cost an MFT
// 114^2 -> 440^2 of six fields 12 of its 74 us.
cudaError_t ft_bases(int fmt, const FtItem* items, int K, int N, const FtOperand& w, cudaStream_t stream);

// Classes T [item][px][py][c][R][ld] (FT_FLOAT of two GEMMs; v rows, u columns) to the plane: field =
// scale F, intensity |scale F|^2 inv_peak, its sum over lo <= r^2 <= thr_out, its largest value.
struct FtPlane {
    const FtItem* items;         // scale, inv_peak, lo_out, thr_out of the last contraction
    const void* T;
    int ext, R, ld;
    long long bstride;           // of T, in values
    int m, sign;
    float* image;                // [item][m][m] or NULL
    float2* field;               // [item][m][m] or NULL
    double* dh;                  // dark-hole sums [item], or NULL
    double* dh_part;             // with dh: [item][ft_plane_parts(m)] work, and
    unsigned* dh_count;          //   [item] zeros (left as zeros)
    float* peak;                 // running maximum, or NULL
    double* peak64;
};
size_t ft_plane_parts(int m);
cudaError_t ft_plane(const FtPlane& p, int items, cudaStream_t stream);
// FT_DIFF classes [item][px][py][c][R][ld] -> dst[item][n][n] (pitch ld): the plane of all signs
cudaError_t ft_unfold(const float* T, int R, int ld, long long bstride, int n, int items, float2* dst, int dst_ld,
                      long long dst_bstride, cudaStream_t stream);

}  // namespace coro
