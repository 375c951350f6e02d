// mft.cu -- matrix Fourier transform (Sec. 1.1: the semi-analytic coronagraph method of
// Soummer et al. uses "discrete matrix Fourier transforms of modest sized arrays"; Sec. 2.3:
// the "sines and cosines ... needed in the matrix DFT").
//
//   out = s * A_y . in . A_x^T,   A[u][j] = exp(-+ 2 pi i X_j U_u)
//
// evaluated as two batched GEMMs: on the CUDA cores over even / odd halves with real bases
// (fold.cuh), on the tensor cores over split complex operands. The bases are generated on the
// device in FP64 (the phase X_j U_u = j' u' du / npix is an exact integer times one FP64
// constant, reduced to its fractional cycle before sincospi) and rounded.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "capi_common.h"
#include "fft_engine.cuh"
#include "fold.cuh"
#include "tc_gemm.cuh"
#include "tcx_gemm.cuh"

using namespace coro;

namespace {

coro_status check_mft_wf(const char* fn, const coro_wavefront* wf) {
    if (!wf || !wf->data) { coro::set_error("%s: wavefront or data is NULL", fn); return CORO_EINVAL; }
    if (wf->dtype != CORO_C64 && wf->dtype != CORO_C128) { coro::set_error("%s: bad dtype %d", fn, wf->dtype); return CORO_EINVAL; }
    if (wf->batch < 1 || wf->batch > 65535) { coro::set_error("%s: batch %d", fn, wf->batch); return CORO_ESIZE; }
    if (wf->n < 1 || wf->n > 8192) { coro::set_error("%s: size %d outside [1, 8192]", fn, wf->n); return CORO_ESIZE; }
    return CORO_OK;
}

// Split-precision tensor-core MFT: Y1 = X . W^T written transposed and split, then
// out = s (Y1^T . W^T)^T, with W[r][k] = exp(-+2 pi i r' k' du/npix) the MFT basis.
coro_status mft_tensor_core(coro_ctx ctx, const coro_wavefront* in, int direction, int m, const std::vector<double>& c,
                            bool bf16, coro_wavefront* out) {
    coro_status st = CORO_OK;
    const int batch = in->batch;
    const int nin = in->n;                       // X1 rows = cols
    const int nout = m;                          // W rows, output size
    const size_t es = tc_elem_size(bf16);
    const int ld = tc_ld(nin, bf16);
    const size_t x_bytes = (size_t)4 * batch * nin * ld * es;
    const size_t w_bytes = (size_t)4 * batch * nout * ld * es;
    const size_t z_bytes = w_bytes;
    auto align = [](size_t v) { return (v + 1023) & ~(size_t)1023; };
    unsigned char* work = (unsigned char*)coro::ctx_work(ctx, align(x_bytes) + align(w_bytes) + align(z_bytes), &st);
    if (!work) return st;
    TcOperand X{work, batch, nin, nin, ld};
    TcOperand W{work + align(x_bytes), batch, nout, nin, ld};
    TcOperand Z{work + align(x_bytes) + align(w_bytes), batch, nout, nin, ld};
    void* c_d = coro::upload_async(ctx, c.data(), c.size() * sizeof(double), &st);
    if (!c_d) return st;
    std::vector<TcItem> it1(batch), it2(batch);
    for (int b = 0; b < batch; ++b) {
        it1[b] = TcItem{nin, nout, nin, b, b, 0, 0x7fffffff, 1.0f, 1.0f};
        it2[b] = TcItem{nout, nout, nin, b, b, 0, 0x7fffffff, (float)c[b], 1.0f};
    }
    void* i1 = coro::upload_async(ctx, it1.data(), batch * sizeof(TcItem), &st);
    void* i2 = i1 ? coro::upload_async(ctx, it2.data(), batch * sizeof(TcItem), &st) : nullptr;
    cudaError_t e = (i1 && i2) ? cudaSuccess : cudaErrorMemoryAllocation;
    CUtensorMap mx, mw, mz;
    if (e == cudaSuccess) e = tc_split(bf16, (const float2*)in->data, (long long)nin * nin, nin, X, ctx->stream);
    if (e == cudaSuccess) e = tc_basis(bf16, (const double*)c_d, direction < 0 ? -1 : 1, W, ctx->stream);
    if (e == cudaSuccess) e = tc_make_operand_map(X, bf16, &mx);
    if (e == cudaSuccess) e = tc_make_operand_map(W, bf16, &mw);
    if (e == cudaSuccess) e = tc_make_operand_map(Z, bf16, &mz);
    if (e == cudaSuccess) {
        TcArgs a{};
        a.items = (const TcItem*)i1;
        a.err = ctx->err;
        a.dst = Z.base;
        a.dst_bstride = (long long)4 * nout * ld;
        a.dst_rows = nout;
        a.dst_ld = ld;
        e = tc_launch(bf16, TC_EPI_SPLITT, mx, mw, nin, nout, nin, batch, a, ctx->stream);
    }
    if (e == cudaSuccess) {
        TcArgs a{};
        a.items = (const TcItem*)i2;
        a.err = ctx->err;
        a.dst = out->data;
        a.dst_bstride = (long long)nout * nout;
        a.dst_rows = nout;
        a.dst_ld = nout;
        e = tc_launch(bf16, TC_EPI_C64T, mz, mw, nout, nout, nin, batch, a, ctx->stream);
    }
    coro::free_async(ctx, c_d);
    coro::free_async(ctx, i1);
    coro::free_async(ctx, i2);
    if (e == cudaErrorNotSupported) {
        coro::set_error("coro_propagate_mft: tensor maps unavailable (driver entry point missing)");
        return CORO_ENOTIMPL;
    }
    if (e != cudaSuccess) return coro::cuda_fail(e, "tensor-core MFT");
    return CORO_OK;
}

// Extended-precision tensor-core MFT (CORO_MFT_EXT): the same two GEMMs on sliced BF16
// operands (tcx_gemm.cu), the bases sliced straight from their FP64 values.
coro_status mft_ext(coro_ctx ctx, const coro_wavefront* in, int direction, int m, const std::vector<double>& c,
                    coro_wavefront* out) {
    coro_status st = CORO_OK;
    const int batch = in->batch;
    const int nin = in->n, nout = m;
    const int ld = tcx_ld(nin);
    const size_t x_bytes = (size_t)TCX_X_PLANES * batch * nin * ld * 2;
    const size_t w_bytes = (size_t)TCX_W_PLANES * batch * nout * ld * 2;
    const size_t z_bytes = (size_t)TCX_X_PLANES * batch * nout * ld * 2;
    auto align = [](size_t v) { return (v + 1023) & ~(size_t)1023; };
    unsigned char* work = (unsigned char*)coro::ctx_work(ctx, align(x_bytes) + align(w_bytes) + align(z_bytes), &st);
    if (!work) return st;
    TcOperand X{work, batch, nin, nin, ld};
    TcOperand W{work + align(x_bytes), batch, nout, nin, ld};
    TcOperand Z{work + align(x_bytes) + align(w_bytes), batch, nout, nin, ld};
    std::vector<TcItem> it1(batch), it2(batch);
    for (int b = 0; b < batch; ++b) {
        it1[b] = TcItem{nin, nout, nin, b, b, 0, 0x7fffffff, 1.0f, 1.0f};
        it2[b] = TcItem{nout, nout, nin, b, b, 0, 0x7fffffff, (float)c[b], 1.0f};
        it2[b].scale64 = c[b];
    }
    void* i1 = coro::upload_async(ctx, it1.data(), batch * sizeof(TcItem), &st);
    void* i2 = i1 ? coro::upload_async(ctx, it2.data(), batch * sizeof(TcItem), &st) : nullptr;
    cudaError_t e = (i1 && i2) ? cudaSuccess : cudaErrorMemoryAllocation;
    // the first GEMM writes Z's nin valid columns only; its padding up to ld must read as zeros
    if (e == cudaSuccess) e = cudaMemsetAsync(Z.base, 0, z_bytes, ctx->stream);
    CUtensorMap mx, mw, mz;
    if (e == cudaSuccess) e = tcx_split((const float2*)in->data, (long long)nin * nin, nin, X, ctx->stream);
    for (int b = 0; b < batch && e == cudaSuccess; ++b)
        e = tcx_basis_one(c[b], direction < 0 ? -1 : 1, W, b, nout, nin, ctx->stream);
    if (e == cudaSuccess) e = tcx_make_x_map(X, &mx);
    if (e == cudaSuccess) e = tcx_make_w_map(W, &mw);
    if (e == cudaSuccess) e = tcx_make_x_map(Z, &mz);
    if (e == cudaSuccess) {
        TcArgs a{};
        a.items = (const TcItem*)i1;
        a.err = ctx->err;
        a.dst = Z.base;
        a.dst_bstride = (long long)TCX_X_PLANES * nout * ld;
        a.dst_rows = nout;
        a.dst_ld = ld;
        e = tcx_launch(TC_EPI_SPLITT, mx, mw, nin, nout, batch, a, ctx->stream);
    }
    if (e == cudaSuccess) {
        TcArgs a{};
        a.items = (const TcItem*)i2;
        a.err = ctx->err;
        a.dst = out->data;
        a.dst_bstride = (long long)nout * nout;
        a.dst_rows = nout;
        a.dst_ld = nout;
        e = tcx_launch(TC_EPI_C64T, mz, mw, nout, nout, batch, a, ctx->stream);
    }
    coro::free_async(ctx, i1);
    coro::free_async(ctx, i2);
    if (e == cudaErrorNotSupported) {
        coro::set_error("coro_propagate_mft: tensor maps unavailable (driver entry point missing)");
        return CORO_ENOTIMPL;
    }
    if (e != cudaSuccess) return coro::cuda_fail(e, "extended-precision tensor-core MFT");
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
    // items per round: the contractions carry item x parity (x K split) in grid z
    const int round = batch < 4096 ? batch : 4096;
    auto align = [](size_t v) { return (v + 255) & ~(size_t)255; };
    const size_t f_bytes = align((size_t)round * 4 * hn * hn * sizeof(C)), w_bytes = align((size_t)round * 2 * hn * ldw * sizeof(R));
    const size_t y_bytes = align((size_t)round * 4 * hn * hm * sizeof(C)), t_bytes = align((size_t)round * 4 * hm * hm * sizeof(C));
    size_t part_elems = 0;
    if (std::is_same<C, float2>::value)
        part_elems = std::max(fold_part_elems(2 * hn, hm, hn, round), fold_part_elems(2 * hm, hm, hn, round));
    unsigned char* work = (unsigned char*)coro::ctx_work(ctx, f_bytes + w_bytes + y_bytes + t_bytes + part_elems * sizeof(C), &st);
    if (!work) return st;
    C* F = (C*)work;
    R* W = (R*)(work + f_bytes);
    C* Y = (C*)(work + f_bytes + w_bytes);
    C* T = (C*)(work + f_bytes + w_bytes + y_bytes);
    C* part = part_elems ? (C*)(work + f_bytes + w_bytes + y_bytes + t_bytes) : nullptr;
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
    if (precision == CORO_MFT_EXT) return mft_ext(ctx, in, direction, m, c, out);
    if (precision == CORO_MFT_3XTF32 || precision == CORO_MFT_3XBF16)
        return mft_tensor_core(ctx, in, direction, m, c, precision == CORO_MFT_3XBF16, out);
    return dbl ? mft_cuda_cores<double2>(ctx, in, direction, m, c, out) : mft_cuda_cores<float2>(ctx, in, direction, m, c, out);
}

