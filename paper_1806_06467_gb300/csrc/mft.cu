// mft.cu -- matrix Fourier transform (Sec. 1.1: the semi-analytic coronagraph method of
// Soummer et al. uses "discrete matrix Fourier transforms of modest sized arrays"; Sec. 2.3:
// the "sines and cosines ... needed in the matrix DFT").
//
//   out = s * A_y . in . A_x^T,   A[u][j] = exp(-+ 2 pi i X_j U_u)
//
// evaluated as two batched GEMMs over even / odd halves with real bases: on the CUDA cores
// (fold.cuh) or on the tensor cores (ft_gemm.cuh). The bases are generated on the device in FP64
// (the phase X_j U_u = j' u' du / npix is an exact integer times one FP64 constant, reduced to its
// fractional cycle before sincospi) and rounded.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "capi_common.h"
#include "fft_engine.cuh"
#include "fold.cuh"
#include "ft_gemm.cuh"

using namespace coro;

namespace {

coro_status check_mft_wf(const char* fn, const coro_wavefront* wf) {
    if (!wf || !wf->data) { coro::set_error("%s: wavefront or data is NULL", fn); return CORO_EINVAL; }
    if (wf->dtype != CORO_C64 && wf->dtype != CORO_C128) { coro::set_error("%s: bad dtype %d", fn, wf->dtype); return CORO_EINVAL; }
    if (wf->batch < 1 || wf->batch > 65535) { coro::set_error("%s: batch %d", fn, wf->batch); return CORO_ESIZE; }
    if (wf->n < 1 || wf->n > 8192) { coro::set_error("%s: size %d outside [1, 8192]", fn, wf->n); return CORO_ESIZE; }
    return CORO_OK;
}

// Items of a batch that one round takes: their workspace stays within 2 GiB, or is that of one item.
// (The classes of a plane are as large as the plane: a batch that fills most of the device would
// otherwise need as much again. Rounds of 2 GiB are far past what fills the chip.)
int round_items(int batch, size_t item_bytes, int most) {
    const size_t fit = ((size_t)2 << 30) / item_bytes;
    return (int)std::max<size_t>(1, std::min<size_t>({fit, (size_t)batch, (size_t)most}));
}

// Tensor-core MFT (3xTF32, 3xBF16, EXT) on even / odd halves (ft_gemm.cuh): fold, bases, two
// contractions to the parity classes of the result, and the plane of all signs.
coro_status mft_tensor_core(coro_ctx ctx, const coro_wavefront* in, int direction, int m, const std::vector<double>& c,
                            int fmt, coro_wavefront* out) {
    coro_status st = CORO_OK;
    const int n = in->n, hn = fold_len(n), hm = fold_len(m), ld_t = ft_pitch(FT_TF32, hm);
    const size_t t_item = (size_t)8 * hm * ld_t * (fmt == FT_EXT ? sizeof(float2) : sizeof(float));
    auto align = [](size_t v) { return (v + 1023) & ~(size_t)1023; };
    FtOperand X, W, Y;
    // T, written when X has been read, takes its place
    size_t xb, wb, yb;
    auto shape = [&](int items) {
        X = ft_operand(fmt, items, hn, hn);
        W = ft_basis_operand(fmt, items, hm, hn);
        Y = ft_operand(fmt, items, hm, hn);
        xb = align(std::max(ft_bytes(fmt, X), t_item * items));
        wb = align(ft_bytes(fmt, W));
        yb = align(ft_bytes(fmt, Y));
    };
    shape(1);
    const int round = round_items(in->batch, xb + wb + yb, in->batch);
    shape(round);
    unsigned char* work = (unsigned char*)coro::ctx_work(ctx, xb + wb + yb, &st);
    if (!work) return st;
    for (int b0 = 0; b0 < in->batch; b0 += round) {
        const int batch = std::min(round, in->batch - b0);
        shape(batch);
        X.base = work;
        W.base = work + xb;
        Y.base = work + xb + wb;
        void* T = work;
        std::vector<FtItem> items(batch);
        for (int b = 0; b < batch; ++b) items[b] = FtItem{hn, hm, 0, b, -1, 0x7fffffff, 0, 1.0, 1.0};
        std::vector<FtItem> both(items);
        both.insert(both.end(), items.begin(), items.end());
        for (int b = 0; b < batch; ++b) {
            both[b].H = hn;                              // rows: k of the other axis, then u
            both[batch + b].H = hm;
        }
        std::vector<FtItem> plane(items);
        for (int b = 0; b < batch; ++b) plane[b].scale = c[b0 + b];
        both.insert(both.end(), plane.begin(), plane.end());
        FtItem* it = (FtItem*)coro::upload_async(ctx, both.data(), both.size() * sizeof(FtItem), &st);
        if (!it) return st;
        FtGemm g1, g2;
        cudaError_t e = ft_fold(fmt, (const float2*)in->data + (size_t)b0 * n * n, (long long)n * n, n, n, hn, -1, X, ctx->stream);
        if (e == cudaSuccess) e = ft_bases(fmt, it + 2 * batch, hn, hm, W, ctx->stream);      // scale = c
        if (e == cudaSuccess) e = ft_make(fmt, X, W, batch, hm, 128, &g1);
        if (e == cudaSuccess) e = ft_make(fmt, Y, W, batch, hm, 128, &g2);
        if (e == cudaSuccess) {
            FtArgs a{};
            a.items = it;
            a.err = ctx->err;
            a.R = X.R;
            a.dst = Y.base;
            a.dst_bstride = Y.stride;
            a.dst_R = Y.R;
            a.dst_ld = Y.ld;
            e = ft_launch(g1, FT_SPLIT, a, ctx->stream);
        }
        if (e == cudaSuccess) {
            FtArgs a{};
            a.items = it + batch;
            a.err = ctx->err;
            a.R = Y.R;
            a.dst = T;
            a.dst_bstride = (long long)8 * hm * ld_t;
            a.dst_R = hm;
            a.dst_ld = ld_t;
            e = ft_launch(g2, FT_FLOAT, a, ctx->stream);
        }
        if (e == cudaSuccess) {
            FtPlane p{};
            p.items = it + 2 * batch;
            p.T = T;
            p.ext = fmt == FT_EXT;
            p.R = hm;
            p.ld = ld_t;
            p.bstride = (long long)8 * hm * ld_t;
            p.m = m;
            p.sign = direction < 0 ? -1 : 1;
            p.field = (float2*)out->data + (size_t)b0 * m * m;
            e = ft_plane(p, batch, ctx->stream);
        }
        coro::free_async(ctx, it);
        if (e == cudaErrorNotSupported) {
            coro::set_error("coro_propagate_mft: tensor maps unavailable (driver entry point missing)");
            return CORO_ENOTIMPL;
        }
        if (e != cudaSuccess) return coro::cuda_fail(e, "tensor-core MFT");
    }
    return CORO_OK;
}

// CUDA-core MFT: complex64 with FP32 arithmetic or complex128 with FP64 arithmetic, on even / odd
// halves (fold.cuh): fold and bases in one launch, two contractions, the expansion.
template <typename C>
coro_status mft_cuda_cores(coro_ctx ctx, const coro_wavefront* in, int direction, int m, const std::vector<double>& c,
                           coro_wavefront* out) {
    using R = typename real_of<C>::type;
    coro_status st = CORO_OK;
    const int batch = in->batch, n = in->n, hn = fold_len(n), hm = fold_len(m), ldw = fold_ldw(hm);
    auto align = [](size_t v) { return (v + 255) & ~(size_t)255; };
    // T, written when F has been read, takes its place
    auto f_bytes = [&](size_t k) { return align(k * 4 * std::max((size_t)hn * hn, (size_t)hm * hm) * sizeof(C)); };
    auto w_bytes = [&](size_t k) { return align(k * 2 * hn * ldw * sizeof(R)); };
    auto y_bytes = [&](size_t k) { return align(k * 4 * hn * hm * sizeof(C)); };
    // the contractions carry item x parity (x K split) in grid z: 4096 items at most
    const int round = round_items(batch, f_bytes(1) + w_bytes(1) + y_bytes(1), 4096);
    const int rest = batch % round ? batch % round : round;       // items of the last round: other K splits
    size_t part_elems = 0;
    if (std::is_same<C, float2>::value)
        for (int k : {round, rest})
            part_elems = std::max({part_elems, fold_part_elems(2 * hn, hm, hn, k), fold_part_elems(2 * hm, hm, hn, k)});
    unsigned char* work = (unsigned char*)coro::ctx_work(ctx, f_bytes(round) + w_bytes(round) + y_bytes(round) + part_elems * sizeof(C), &st);
    if (!work) return st;
    C *F = (C*)work, *T = F;
    R* W = (R*)(work + f_bytes(round));
    C* Y = (C*)(work + f_bytes(round) + w_bytes(round));
    C* part = part_elems ? (C*)(work + f_bytes(round) + w_bytes(round) + y_bytes(round)) : nullptr;
    cudaError_t e = cudaSuccess;
    for (int b0 = 0; b0 < batch && e == cudaSuccess; b0 += round) {
        const int nb = std::min(round, batch - b0);
        e = fold_prepare<C>((const C*)in->data + (size_t)b0 * n * n, n, hn, -1, F, c.data() + b0, hn, hm, W, nb, ctx->stream);
        FoldGemm<C> g{2 * hn, hm, hn, nb, F, (long long)4 * hn * hn, W, (long long)2 * hn * ldw, ldw, Y, (long long)4 * hn * hm,
                      FOLD_PLAIN, 0, (R)1, nullptr, 0};
        if (e == cudaSuccess) e = fold_gemm(g, part, ctx->stream);
        g.M = 2 * hm;
        g.X = Y;
        g.sX = (long long)4 * hn * hm;
        g.Y = T;
        g.sY = (long long)4 * hm * hm;
        if (e == cudaSuccess) e = fold_gemm(g, part, ctx->stream);
        if (e == cudaSuccess)
            e = fold_expand<C>(T, m, direction < 0 ? -1 : 1, c.data() + b0, (C*)out->data + (size_t)b0 * m * m, nb, ctx->stream);
    }
    return e == cudaSuccess ? CORO_OK : coro::cuda_fail(e, "mft (folded)");
}

}  // namespace

extern "C" coro_status coro_propagate_mft(coro_ctx ctx, const coro_wavefront* in, double npix, int direction,
                                          int m, const double* du, int precision, coro_wavefront* out) {
    coro::clear_error();
    if (!ctx) { coro::set_error("coro_propagate_mft: ctx is NULL"); return CORO_EINVAL; }
    coro_status st = check_mft_wf("coro_propagate_mft(in)", in);
    if (st != CORO_OK) return st;
    if ((st = check_mft_wf("coro_propagate_mft(out)", out)) != CORO_OK) return st;
    if (direction != -1 && direction != 1) { coro::set_error("coro_propagate_mft: direction must be -1 or +1"); return CORO_EINVAL; }
    if (!(npix > 0)) { coro::set_error("coro_propagate_mft: npix must be > 0"); return CORO_EINVAL; }
    if (!du) { coro::set_error("coro_propagate_mft: du is NULL"); return CORO_EINVAL; }
    if (out->batch != in->batch) { coro::set_error("coro_propagate_mft: batch mismatch"); return CORO_EINVAL; }
    if (out->n != m) { coro::set_error("coro_propagate_mft: out->n (%d) must equal m (%d)", out->n, m); return CORO_EINVAL; }
    if (in->dtype != out->dtype) { coro::set_error("coro_propagate_mft: in and out dtypes differ"); return CORO_EINVAL; }
    const bool dbl = in->dtype == CORO_C128;
    if (dbl ? precision != CORO_MFT_FP64
            : (precision != CORO_MFT_FP32 && precision != CORO_MFT_3XTF32 && precision != CORO_MFT_3XBF16 &&
                 precision != CORO_MFT_EXT)) {
        coro::set_error("coro_propagate_mft: precision %d does not apply to %s fields", precision,
                        dbl ? "complex128 (use CORO_MFT_FP64)" : "complex64");
        return CORO_EINVAL;
    }
    const int batch = in->batch;
    std::vector<double> c(batch);
    for (int b = 0; b < batch; ++b) {
        if (!(du[b] > 0) || !std::isfinite(du[b])) { coro::set_error("coro_propagate_mft: du[%d] must be > 0", b); return CORO_EINVAL; }
        c[b] = du[b] / npix;
    }
    coro::DeviceGuard g(ctx->device);
    if (precision == CORO_MFT_EXT) return mft_tensor_core(ctx, in, direction, m, c, FT_EXT, out);
    if (precision == CORO_MFT_3XTF32 || precision == CORO_MFT_3XBF16)
        return mft_tensor_core(ctx, in, direction, m, c, precision == CORO_MFT_3XBF16 ? FT_BF16 : FT_TF32, out);
    return dbl ? mft_cuda_cores<double2>(ctx, in, direction, m, c, out) : mft_cuda_cores<float2>(ctx, in, direction, m, c, out);
}

