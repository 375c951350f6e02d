"""GPU parity of the transforms on even / odd halves (half grids, unpaired edge samples, tiles that
do not divide) against the FP64 oracle's direct sums, at the sizes where the halves can go wrong."""
import numpy as np
import pytest
import torch

from oracle import coronagraph, propagation
from paper_1806_06467_gb300 import coro, inputs

pytestmark = pytest.mark.gpu

# FP32 rounding over at most 2 x 700 terms; the FP64 path against a sum of the same length
TOL = {coro.MFT_FP32: 1e-5, coro.MFT_3XTF32: 1e-5, coro.MFT_3XBF16: 1e-4, coro.MFT_EXT: 2e-7, coro.MFT_FP64: 1e-12}


def rel_l2(got, ref):
    return float(np.linalg.norm(np.asarray(got, np.complex128) - ref) / np.linalg.norm(ref))


@pytest.fixture(scope="module")
def ctx(lib):
    return coro.Context(0)


@pytest.mark.parametrize("prec", sorted(TOL))
@pytest.mark.parametrize("n,m,batch", [(1, 1, 1), (2, 3, 2), (3, 2, 1), (31, 64, 3), (64, 65, 2), (63, 33, 1), (126, 127, 1),
                                       (257, 40, 2), (40, 258, 70), (700, 129, 1), (513, 512, 1)])
def test_mft_halves(ctx, n, m, batch, prec):
    f = inputs.random_field((batch, n, n), seed=n * m)
    du = np.linspace(0.2, 0.6, batch)
    x = torch.from_numpy(f.astype(np.complex128 if prec == coro.MFT_FP64 else np.complex64)).cuda()
    npix = 0.9 * max(n, m)
    y = coro.propagate_mft(ctx, x, npix, -1, m, du, prec).cpu().numpy()
    z = coro.propagate_mft(ctx, x, npix, +1, m, du, prec).cpu().numpy()
    xs = x.cpu().numpy().astype(np.complex128)
    for b in range(0, batch, 23):
        assert rel_l2(y[b], propagation.mft(xs[b], npix, m, du[b])) < TOL[prec]
        assert rel_l2(z[b], propagation.imft(xs[b], npix, m, du[b])) < TOL[prec]


@pytest.mark.parametrize("prec,tol", [(coro.MFT_FP64, 1e-13)])
@pytest.mark.parametrize("n,npix,frac,m_occ,spot,m_det", [
    (64, 60.0, 0.8, 32, 3.0, 48), (65, 65.0, 0.9, 33, 3.9, 47), (130, 130.0, 0.99, 40, 2.0, 50), (131, 120.0, 0.7, 39, 0.0, 129),
    (64, 64.0, 1.0, 32, 3.0, 48),        # the stop reaches the unpaired edge of the pupil array
    (64, 60.0, 0.8, 32, 4.0, 48),        # the spot reaches the unpaired edge of the occulter array
    (66, 66.0, 1.3, 31, 9.0, 33)])       # masks larger than their arrays
def test_lyot_halves(ctx, n, npix, frac, m_occ, spot, m_det, prec, tol):
    """Normalised image, dark-hole sum and peak of two items (even and odd occulters), dark holes
    that end inside and beyond the detector's edge."""
    lam = 550e-9
    items = [dict(m_occ=m_occ, du_occ=0.25, spot_radius=spot, du_det=0.5, dh_in=4.0, dh_out=11.0),
             dict(m_occ=m_occ + 1, du_occ=0.27, spot_radius=spot, du_det=0.45, dh_in=3.0, dh_out=40.0)]
    ph = np.exp(1j * inputs.rng(n).uniform(-0.2, 0.2, (2, n, n)))
    pupil = np.stack([coronagraph.pupil_field(n, npix, lam, None) * p for p in ph])
    x = torch.from_numpy(pupil.astype(np.complex128 if prec == coro.MFT_FP64 else np.complex64)).cuda()
    plan = coro.LyotPlan(ctx, n=n, npix=npix, lyot_frac=frac, m_det=m_det, items=items, precision=prec)
    peak = plan.peak(x)
    img = torch.empty((2, m_det, m_det), dtype=torch.float32, device="cuda")
    fld = torch.empty((2, m_det, m_det), dtype=x.dtype, device="cuda")
    dh = plan.execute(x, peak=peak, intensity=img, field=fld)
    xs = x.cpu().numpy().astype(np.complex128)
    for b, it in enumerate(items):
        p = coronagraph.LyotParams(n, npix, it["m_occ"], it["du_occ"], it["spot_radius"], frac, m_det, it["du_det"])
        ref, s, pk = coronagraph.lyot_psf(xs[b], p, it["dh_in"], it["dh_out"])
        assert abs(peak[b] / pk - 1) < max(10 * tol, 1e-12)
        # the image is held in 32 bits: half a unit in the last place of values up to its maximum
        assert np.max(np.abs(img[b].cpu().numpy() - ref)) < tol + 6e-8 * ref.max()
        assert abs(dh[b] - s) < m_det ** 2 * (tol + 6e-8 * ref.max())
        det = coronagraph.lyot_fields(xs[b], p)["det"]
        assert np.max(np.abs(fld[b].cpu().numpy() - det)) < 30 * (tol + 6e-8) * np.abs(det).max()
    plan.close()


# masks inside their arrays (parity classes) and reaching unpaired edges (complex GEMMs); both dark
# holes end inside the detector, or the second one's reaches its unpaired edge
TC_CASES = [(64, 60.0, 0.8, 32, 3.0, 48, 11.0), (65, 65.0, 0.9, 33, 3.9, 47, 10.0), (130, 130.0, 0.99, 40, 2.0, 50, 11.0),
            (131, 120.0, 0.7, 39, 0.0, 129, 11.0), (257, 240.0, 0.8, 64, 7.0, 131, 25.0), (300, 300.0, 0.5, 33, 1.0, 290, 30.0),
            (64, 64.0, 1.0, 32, 3.0, 48, 11.0), (64, 60.0, 0.8, 32, 4.0, 48, 11.0), (64, 60.0, 0.8, 32, 3.0, 48, 12.0)]


@pytest.mark.parametrize("prec", [coro.MFT_3XTF32, coro.MFT_3XBF16, coro.MFT_EXT])
@pytest.mark.parametrize("n,npix,frac,m_occ,spot,m_det,dh_out", TC_CASES)
def test_lyot_tensor_core_halves(ctx, n, npix, frac, m_occ, spot, m_det, dh_out, prec):
    """Image, peak, field, dark-hole sum and adjoint at the bars of the batched Lyot tests (whole
    image 1e-5 of the peak; peak 1e-5, extended 1e-9; adjoint 1e-3)."""
    from oracle import adjoint
    lam = 550e-9
    items = [dict(m_occ=m_occ, du_occ=0.25, spot_radius=spot, du_det=0.5, dh_in=4.0, dh_out=dh_out),
             dict(m_occ=m_occ + 1, du_occ=0.27, spot_radius=spot, du_det=0.45, dh_in=3.0, dh_out=0.85 * dh_out)]
    ph = np.exp(1j * inputs.rng(n).uniform(-0.2, 0.2, (2, n, n)))
    pupil = np.stack([coronagraph.pupil_field(n, npix, lam, None) * p for p in ph]).astype(np.complex64)
    x = torch.from_numpy(pupil).cuda()
    plan = coro.LyotPlan(ctx, n=n, npix=npix, lyot_frac=frac, m_det=m_det, items=items, precision=prec)
    peak = plan.peak(x)
    img = torch.empty((2, m_det, m_det), dtype=torch.float32, device="cuda")
    fld = torch.empty((2, m_det, m_det), dtype=torch.complex64, device="cuda")
    dh = plan.execute(x, peak=peak, intensity=img, field=fld)
    g, dh_g = plan.gradient(x, peak)
    again = torch.empty_like(img)
    plan.execute(x, peak=peak, intensity=again)          # the gradient leaves nothing behind
    assert torch.equal(img, again)
    for b, it in enumerate(items):
        p = coronagraph.LyotParams(n, npix, it["m_occ"], it["du_occ"], it["spot_radius"], frac, m_det, it["du_det"])
        e = pupil[b].astype(np.complex128)
        ref, s, pk = coronagraph.lyot_psf(e, p, it["dh_in"], it["dh_out"])
        mask = coronagraph.dark_hole_mask(m_det, it["du_det"], it["dh_in"], it["dh_out"])
        assert abs(peak[b] / pk - 1) < (1e-9 if prec == coro.MFT_EXT else 1e-5)
        assert np.max(np.abs(img[b].cpu().numpy() - ref)) < 1e-5
        assert abs(dh[b] - s) < 1e-3 * s + mask.sum() * 1e-7
        assert abs(dh_g[b] - s) < 1e-3 * s + mask.sum() * 1e-7
        det = coronagraph.lyot_fields(e, p)["det"]
        assert rel_l2(fld[b].cpu().numpy(), det) < 1e-3
        assert rel_l2(g[b].cpu().numpy(), adjoint.lyot_adjoint(mask * det / pk, p)) < 1e-3
    plan.close()


@pytest.mark.parametrize("prec", [coro.MFT_FP64, coro.MFT_3XTF32])
def test_lyot_plan_runs_on_a_stream_set_after_its_creation(lib, prec):
    """A plan made behind long work on the context's first stream, executed on another stream at once:
    its bases are complete when creation returns."""
    n, md = 128, 96
    items = [dict(m_occ=40, du_occ=0.25, spot_radius=3.0, du_det=0.5, dh_in=4.0, dh_out=11.0)]
    e = coronagraph.pupil_field(n, 120.0, 550e-9, None)[None]
    x = torch.from_numpy(e.astype(np.complex128 if prec == coro.MFT_FP64 else np.complex64)).cuda()
    img = [torch.empty((1, md, md), dtype=torch.float32, device="cuda") for _ in range(2)]
    busy = torch.ones((4096, 4096), device="cuda")
    first, second = torch.cuda.Stream(), torch.cuda.Stream()
    for k in range(2):
        c = coro.Context(0, stream=first)
        torch.cuda.synchronize()
        if k:
            with torch.cuda.stream(first):
                for _ in range(40):
                    busy = (busy @ busy).clamp_(0.0, 1.0)
        plan = coro.LyotPlan(c, n=n, npix=120.0, lyot_frac=0.8, m_det=md, items=items, precision=prec)
        if k:
            c.lib.check(c.lib.coro_ctx_set_stream(c.handle, second.cuda_stream))
        plan.execute(x, peak=1.0, intensity=img[k], want_dh=False)
        torch.cuda.synchronize()
        plan.close()
    assert torch.equal(img[0], img[1])


@pytest.mark.parametrize("prec", sorted(TOL))
def test_mft_workspace_is_bounded(lib, prec):
    """A batch whose classes would take more than 2 GiB runs in rounds: no more device memory than that is
    taken, and items of every round are the oracle's (the last round is a ragged one)."""
    n, m, batch = 32, 1024, 300
    c = coro.Context(0)
    x = torch.from_numpy(inputs.random_field((batch, n, n), seed=5).astype(np.complex128 if prec == coro.MFT_FP64 else np.complex64)).cuda()
    du = np.linspace(0.1, 0.4, batch)
    coro.propagate_mft(c, x[:1].contiguous(), float(n), -1, m, du[:1], prec)         # modules loaded
    torch.cuda.synchronize()
    out = torch.empty((batch, m, m), dtype=x.dtype, device="cuda")
    before = torch.cuda.mem_get_info()[0]
    coro.propagate_mft(c, x, float(n), -1, m, du, prec, out=out)
    torch.cuda.synchronize()
    assert before - torch.cuda.mem_get_info()[0] <= (2 << 30) + (64 << 20)
    for b in (0, 57, 121, 122, 150, 243, 298, 299):
        assert rel_l2(out[b].cpu().numpy(), propagation.mft(x[b].cpu().numpy().astype(np.complex128), float(n), m, du[b])) < TOL[prec]
    c.close()
