"""Masks of Fresnel plans select: what is not finite under an aperture, stop or occulting spot stays
there, whichever kernels the plan runs."""
import numpy as np
import pytest
import torch

from paper_1806_06467_gb300 import coro, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(lib):
    return coro.Context(0)


def disk(n, r):
    k = np.arange(n) - n // 2
    return k[None, :] ** 2 + k[:, None] ** 2 <= (r * n) ** 2


@pytest.mark.parametrize("layout", ["", "0", "1"])
@pytest.mark.parametrize("n", [1024, 2048, 4096, 1400, 512])
def test_samples_under_masks_that_are_not_finite(ctx, n, layout, monkeypatch):
    """Surfaces with NaN and infinities outside the aperture (and inside an occulting spot) listed
    before it, and a caller's field with NaN in its padding: bitwise the result of zeros there, on
    interleaved, natural and alternating passes and left-out rows alike."""
    if layout == "1" and n not in (1024, 2048, 4096):
        pytest.skip("no alternating layout")
    monkeypatch.setenv("CORO_AUTOTUNE", "0")
    if layout:
        monkeypatch.setenv("CORO_LAYOUT", layout)
    else:
        monkeypatch.delenv("CORO_LAYOUT", raising=False)
    outside, spot = ~disk(n, 0.2003), disk(n, 0.0301)
    g = inputs.rng(n)
    clean = torch.from_numpy((20e-9 * g.standard_normal((n, n))).astype(np.float32)).cuda()
    bad = clean.clone()
    for k, v in enumerate((float("nan"), float("inf"), -float("inf"))):
        at = torch.from_numpy((outside | spot) & (np.add.outer(np.arange(n), 3 * np.arange(n)) % 5 == k)).cuda()
        clean[at] = 0.0
        bad[at] = v
    f = torch.from_numpy(inputs.random_field((1, n, n), seed=n).astype(np.complex64)).cuda()
    out = []
    for m in (clean, bad):
        els = [coro.element(coro.EL_OPD_MAP, plane=0, opd=m), coro.element(coro.EL_APERTURE, plane=0, radius=0.2003),
               coro.element(coro.EL_CIRCLE, plane=0, radius=0.0301, flags=coro.ELF_OPAQUE_INSIDE),
               coro.element(coro.EL_OPD_MAP, plane=1, opd=m), coro.element(coro.EL_CIRCLE, plane=1, radius=0.2003),
               coro.element(coro.EL_CIRCLE, plane=1, radius=0.0301, flags=coro.ELF_OPAQUE_INSIDE),
               coro.element(coro.EL_OPD_MAP, plane=2, opd=m), coro.element(coro.EL_CIRCLE, plane=2, radius=0.2003),
               coro.element(coro.EL_CIRCLE, plane=2, radius=0.0301, flags=coro.ELF_OPAQUE_INSIDE)]
        for uniform in (True, False):
            plan = coro.FresnelPlan(ctx, n=n, batch=1, pixelscale=1.0 / n, wavelength=550e-9, distances=[1.5, 2.0], elements=els,
                                    init_uniform=uniform)
            x = f.clone()
            if m is bad:
                x[0, torch.from_numpy(outside).cuda()] = complex("nan")
            plan.execute(x)
            out.append(x)
            plan.close()
    assert bool(torch.isfinite(torch.view_as_real(out[0])).all())
    assert torch.equal(out[2], out[0]) and torch.equal(out[3], out[1])


@pytest.mark.parametrize("kw", [dict(kind=coro.EL_SCALAR, scalar=float("inf")), dict(kind=coro.EL_SCALAR, scalar=1e300),
                                dict(kind=coro.EL_SINE, sine_freq=2.0, sine_amplitude=float("nan")),
                                dict(kind=coro.EL_ZERNIKE, radius=1.0, coeffs=[1e-8, float("nan")], j_first=4)])
def test_factors_behind_a_mask_that_are_not_finite(ctx, kw, monkeypatch):
    """0 times an infinite or NaN factor is NaN: rows are not left out as zeros behind such an element."""
    n = 1024
    monkeypatch.setenv("CORO_AUTOTUNE", "0")
    els = [coro.element(coro.EL_APERTURE, plane=0, radius=0.2), coro.element(coro.EL_CIRCLE, plane=1, radius=0.1),
           coro.element(kw["kind"], plane=1, **{k: v for k, v in kw.items() if k != "kind"})]
    out = []
    for layout in (None, "0"):
        monkeypatch.delenv("CORO_LAYOUT", raising=False) if layout is None else monkeypatch.setenv("CORO_LAYOUT", layout)
        plan = coro.FresnelPlan(ctx, n=n, batch=1, pixelscale=1.0 / n, wavelength=550e-9, distances=[1.5], elements=els,
                                init_uniform=True)
        x = torch.empty((1, n, n), dtype=torch.complex64, device="cuda")
        plan.execute(x)
        out.append(torch.view_as_real(x))
        plan.close()
    assert bool(torch.isnan(out[1]).any()) and torch.equal(torch.isnan(out[0]), torch.isnan(out[1]))
