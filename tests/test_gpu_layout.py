"""GPU parity: the alternating plane layout of the fused Fresnel plan (a column pass writes its
result transposed into a plan-owned plane, the next row pass reads it back column-wise) against
the FP64 oracle and against the natural in-place layout, through the C ABI.

Tolerance: relative L2 <= 1e-5 against the oracle (complex64), and <= 1e-6 between the two
layouts (the same FP32 arithmetic in another kernel family: rounding order only).
"""
import numpy as np
import pytest
import torch

from paper_1806_06467_gb300 import coro, inputs
from test_gpu_fresnel import rel_l2, relay_elements, relay_oracle, relay_oracle_planes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(lib):
    return coro.Context(0)


def relay_plan(ctx, w, maps_t, batch=1, wavelengths=None, extra=None):
    els = relay_elements(w, maps_t) if extra is None else extra
    return coro.FresnelPlan(ctx, n=w.n, batch=batch, pixelscale=w.dx,
                            wavelength=w.wavelength_m if wavelengths is None else wavelengths,
                            distances=list(w.distances()), elements=els, init_uniform=True)


def names(plan):
    return [plan.pass_kernel(i) for i in range(plan.launch_count)]


@pytest.mark.parametrize("n", [1024, 2048, 4096])
def test_alternating_layout_relay(ctx, n):
    """Six-plane relay on both layouts: the oracle's field to 1e-5 (1024, 2048; 4096 against
    the natural layout only), the layouts within 1e-6 of each other, and the kernels each
    layout reports."""
    w = inputs.RelayWorkload(n=n, npix=n // 2 if n < 4096 else 1024, seed=5)
    maps = [m.astype(np.float32) for m in w.psd_maps()]
    maps_t = [torch.from_numpy(m).cuda() for m in maps]
    plan = relay_plan(ctx, w, maps_t)
    out = {}
    for alt in (True, False):
        plan.set_layout(alt)
        assert plan.layout == alt
        k = names(plan)
        assert any("_pair_t" in x for x in k) == alt, k
        x = torch.full((1, n, n), float("nan"), dtype=torch.complex64, device="cuda")
        plan.execute(x)
        out[alt] = x.cpu().numpy()[0]
    d = rel_l2(out[True], out[False].astype(np.complex128))
    print(f"n {n}: alternating vs natural rel L2 {d:.2e}")
    assert d < 1e-6
    if n < 4096:
        ref = relay_oracle(w, maps)
        assert rel_l2(out[True], ref) < 1e-5


def test_alternating_layout_batch_of_wavelengths(ctx):
    """Two items at different wavelengths (item offsets in the transposed plane and its TMA
    boxes) at 4096^2: alternating equals natural per item."""
    n = 4096
    w = inputs.RelayWorkload(n=n, npix=1024, seed=6)
    maps_t = [torch.from_numpy(m.astype(np.float32)).cuda() for m in w.psd_maps()]
    plan = relay_plan(ctx, w, maps_t, batch=2, wavelengths=[550e-9, 610e-9])
    res = {}
    for alt in (True, False):
        plan.set_layout(alt)
        x = torch.full((2, n, n), float("nan"), dtype=torch.complex64, device="cuda")
        plan.execute(x)
        res[alt] = x.cpu().numpy()
    for b in range(2):
        d = rel_l2(res[True][b], res[False][b].astype(np.complex128))
        assert d < 1e-6, (b, d)
    assert rel_l2(res[True][0], res[True][1].astype(np.complex128)) > 1e-3   # the items differ


def test_alternating_layout_checkpoints_and_taps(ctx):
    """Checkpoints and the phase-gradient tap inside row passes that read the transposed
    plane: stored planes match the oracle's per-plane fields, as on the natural layout."""
    n = 1024
    w = inputs.RelayWorkload(n=n, npix=n // 2, seed=4)
    maps = [m.astype(np.float32) for m in w.psd_maps()]
    maps_t = [torch.from_numpy(m).cuda() for m in maps]
    cps = [torch.zeros((1, n, n), dtype=torch.complex64, device="cuda") for _ in range(3)]
    tap = torch.zeros((1, n, n), dtype=torch.float32, device="cuda")
    g = torch.from_numpy(np.exp(1j * np.linspace(0, 3, n * n)).reshape(1, n, n).astype(np.complex64)).cuda()
    els = relay_elements(w, maps_t)
    els = [els[0], els[1],
           coro.element(coro.EL_CHECKPOINT, plane=2, store=cps[0]), els[2], els[3],
           coro.element(coro.EL_PHASE_GRAD, plane=4, store=tap, ref=g, scalar=1.0),
           els[4], coro.element(coro.EL_CHECKPOINT, plane=4, store=cps[1]), els[5],
           coro.element(coro.EL_CHECKPOINT, plane=5, store=cps[2])]
    plan = relay_plan(ctx, w, maps_t, extra=els)
    ref = relay_oracle_planes(w, maps)
    want = [ref[2][0], ref[4][1], ref[5][1]]
    got = {}
    for alt in (True, False):
        plan.set_layout(alt)
        for c in cps:
            c.fill_(float("nan"))
        tap.fill_(float("nan"))
        x = torch.empty((1, n, n), dtype=torch.complex64, device="cuda")
        plan.execute(x)
        for i, (c, r) in enumerate(zip(cps, want)):
            assert rel_l2(c.cpu().numpy()[0], r) < 1e-5, (alt, i)
        assert torch.equal(cps[2], x)
        got[alt] = tap.cpu().numpy()[0].astype(np.float64)
    assert np.all(np.isfinite(got[True]))
    assert np.linalg.norm(got[True] - got[False]) <= 1e-5 * np.linalg.norm(got[False])


def test_alternating_layout_graph_and_ranges(ctx):
    """Graph replay on the alternating layout is bitwise the eager result; execute_range runs
    every pass in place (natural layout), so the ranges in order agree to rounding; switching
    layouts or kernels resets the plan as documented."""
    n = 1024
    w = inputs.RelayWorkload(n=n, npix=n // 2, seed=7)
    maps_t = [torch.from_numpy(m.astype(np.float32)).cuda() for m in w.psd_maps()]
    plan = relay_plan(ctx, w, maps_t)
    plan.set_layout(True)
    eager = torch.empty((1, n, n), dtype=torch.complex64, device="cuda")
    plan.execute(eager)
    plan.use_graph(True)
    x = torch.empty_like(eager)
    for _ in range(3):
        x.fill_(float("nan"))
        plan.execute(x)
        assert torch.equal(x, eager)
    plan.use_graph(False)
    y = torch.empty_like(eager)
    for i in range(plan.launch_count):
        plan.execute_range(y, i, 1)
    assert rel_l2(y.cpu().numpy()[0], eager.cpu().numpy()[0].astype(np.complex128)) < 1e-6
    plan.set_pass_kernel(1, 0)
    assert not plan.layout and not any("_pair_t" in k for k in names(plan))


def test_alternating_layout_refused_where_unsupported(ctx):
    """complex128 plans and sizes outside 1024-4096 have no alternating layout: CORO_ENOTIMPL
    and the plan stays on the natural layout."""
    for n, dtype in ((512, coro.C64), (1024, coro.C128)):
        w = inputs.RelayWorkload(n=n, npix=n // 2, seed=8)
        maps_t = [torch.from_numpy(m.astype(np.float32)).cuda() for m in w.psd_maps()]
        plan = coro.FresnelPlan(ctx, n=n, batch=1, pixelscale=w.dx, wavelength=w.wavelength_m,
                                distances=list(w.distances()), elements=relay_elements(w, maps_t),
                                init_uniform=True, dtype=dtype)
        with pytest.raises(coro.CoroError):
            plan.set_layout(True)
        assert not plan.layout


def test_plan_tuning_leaves_caller_buffers_alone(ctx):
    """The plan-time tuner (kernel candidates, row variants over every pass, layouts) runs on
    a scratch field with the checkpoint and tap elements left out: buffers those elements
    write keep their contents until the first execute."""
    n = 1024
    w = inputs.RelayWorkload(n=n, npix=n // 2, seed=9)
    maps_t = [torch.from_numpy(m.astype(np.float32)).cuda() for m in w.psd_maps()]
    cp = torch.full((1, n, n), 7.0 + 3.0j, dtype=torch.complex64, device="cuda")
    tap = torch.full((1, n, n), -5.0, dtype=torch.float32, device="cuda")
    els = relay_elements(w, maps_t)
    els = els[:3] + [coro.element(coro.EL_CHECKPOINT, plane=2, store=cp),
                     coro.element(coro.EL_PHASE_GRAD, plane=3, store=tap, scalar=1.0)] + els[3:]
    plan = relay_plan(ctx, w, maps_t, extra=els)
    torch.cuda.synchronize()
    assert bool((cp == (7.0 + 3.0j)).all()) and bool((tap == -5.0).all())
    x = torch.empty((1, n, n), dtype=torch.complex64, device="cuda")
    plan.execute(x)
    assert not bool((cp == (7.0 + 3.0j)).any()) and bool(torch.isfinite(tap).all())


def test_copy_tuning(ctx):
    """A second plan of the same system takes the first one's kernels and layout; plans of
    another size or pass sequence are refused and left unchanged."""
    n = 1024
    w = inputs.RelayWorkload(n=n, npix=n // 2, seed=10)
    maps_t = [torch.from_numpy(m.astype(np.float32)).cuda() for m in w.psd_maps()]
    a = relay_plan(ctx, w, maps_t)
    b = relay_plan(ctx, w, maps_t)
    a.set_pass_kernel(2, -1)                             # units rows, persistent columns
    a.set_layout(True)
    b.copy_tuning(a)
    assert names(b) == names(a) and b.layout
    x, y = (torch.empty((1, n, n), dtype=torch.complex64, device="cuda") for _ in range(2))
    a.execute(x)
    b.execute(y)
    assert torch.equal(x, y)
    a.set_layout(False)
    b.copy_tuning(a)
    assert names(b) == names(a) and not b.layout
    w2 = inputs.RelayWorkload(n=2048, npix=1024, seed=10)
    maps2 = [torch.from_numpy(m.astype(np.float32)).cuda() for m in w2.psd_maps()]
    c = relay_plan(ctx, w2, maps2)
    before = names(c)
    with pytest.raises(coro.CoroError):
        c.copy_tuning(a)
    assert names(c) == before


def test_pass_flops(ctx):
    """FFT arithmetic per pass: two line transforms in every column pass and interior row pass,
    one in the first (uniform start, forward only) and the last (inverse only) row pass."""
    n = 1024
    w = inputs.RelayWorkload(n=n, npix=n // 2, seed=11)
    maps_t = [torch.from_numpy(m.astype(np.float32)).cuda() for m in w.psd_maps()]
    plan = relay_plan(ctx, w, maps_t)
    one = 5.0 * n * np.log2(n) * n
    f = [plan.pass_flops(i) for i in range(plan.launch_count)]
    assert f[0] == one and f[-1] == one
    assert all(x == 2 * one for x in f[1:-1])


@pytest.mark.parametrize("n", [1024, 2048, 4096, 1400, 2800, 4100])
@pytest.mark.parametrize("r_first,r_mid,r_last", [(0.5, 0.13, 0.2), (0.02, 0.0, 0.49), (0.1, 0.3, 0.0)])
def test_rows_left_out_behind_masks(ctx, n, r_first, r_mid, r_last):
    """A uniform beam through an aperture, a stop between two hops, and a last stop (radii in units of
    the grid: single rows, box edges, nearly all rows): transforming only the rows that the masks
    leave gives bitwise the field of all rows, zeros where the last stop blocks, and the same for a
    plan that takes the first one's kernels. A checkpoint behind a mask keeps every row."""
    import os
    lam, dx = np.array([500e-9, 640e-9]), 1.0 / n

    def make(env, check):
        els = [coro.element(coro.EL_APERTURE, plane=0, radius=r_first, obscuration=0.2, n_spiders=4, spider_width=3 * dx),
               coro.element(coro.EL_CIRCLE, plane=1, radius=r_mid), coro.element(coro.EL_LENS, plane=2, focal_length=9.0),
               coro.element(coro.EL_CIRCLE, plane=3, radius=r_last)]
        if check is not None:
            els.append(coro.element(coro.EL_CHECKPOINT, plane=1, store=check))
        os.environ.update(env)
        try:
            return coro.FresnelPlan(ctx, n=n, batch=2, pixelscale=dx, wavelength=lam, distances=[1.5, -2.0, 3.0], elements=els,
                                    init_uniform=True)
        finally:
            for k in env:
                os.environ.pop(k)

    natural = {"CORO_AUTOTUNE": "0", "CORO_LAYOUT": "0"}
    fields = []
    for env, check in ((natural, False), ({"CORO_AUTOTUNE": "0"}, False), ({"CORO_AUTOTUNE": "0"}, True)):
        store = torch.full((2, n, n), float("nan"), dtype=torch.complex64, device="cuda") if check else None
        plan = make(env, store)
        x = torch.full((2, n, n), float("nan"), dtype=torch.complex64, device="cuda")     # not read
        plan.execute(x)
        fields.append(x)
        if check:
            assert bool(torch.isfinite(torch.view_as_real(store)).all())
        elif len(fields) == 2:
            other = make(natural, None)
            other.copy_tuning(plan)
            y = torch.full((2, n, n), float("nan"), dtype=torch.complex64, device="cuda")
            other.execute(y)
            assert torch.equal(x, y)
            y.fill_(1.0)
            plan.execute_range(y, 0, plan.launch_count)
            assert torch.equal(x, y)
    assert torch.equal(fields[0], fields[1]) and torch.equal(fields[0], fields[2])


@pytest.mark.parametrize("n,batch", [(1024, 3), (2048, 2), (4096, 1)])
def test_interleaved_row_pairs_match_natural_layout(ctx, n, batch):
    """A plan as created untuned (row pairs interleaved between passes), with a checkpoint, a direct
    hop of each sign, is bitwise the same kernels on the natural layout."""
    import os
    from oracle import propagation
    lam = np.linspace(500e-9, 600e-9, batch)
    dx, z = 1.0 / n, [1.5, 40.0, -3.0, 2.0]
    meth = [coro.FRESNEL_AS, coro.FRESNEL_DIRECT, coro.FRESNEL_DIRECT, coro.FRESNEL_AS]
    f = inputs.random_field((batch, n, n), seed=n).astype(np.complex64)
    out, stored = [], []
    for env in ({"CORO_AUTOTUNE": "0"}, {"CORO_AUTOTUNE": "0", "CORO_LAYOUT": "0"}):
        store = torch.zeros((batch, n, n), dtype=torch.complex64, device="cuda")
        els = [coro.element(coro.EL_APERTURE, plane=0, radius=0.3), coro.element(coro.EL_CHECKPOINT, plane=1, store=store),
               coro.element(coro.EL_LENS, plane=3, focal_length=7.0)]
        old = {k: os.environ.get(k) for k in env}
        os.environ.update(env)
        try:
            plan = coro.FresnelPlan(ctx, n=n, batch=batch, pixelscale=dx, wavelength=lam, distances=z, methods=meth, elements=els)
        finally:
            for k, v in old.items():
                os.environ.pop(k) if v is None else os.environ.__setitem__(k, v)
        x = torch.from_numpy(f).cuda()
        plan.execute(x)
        out.append(x)
        stored.append(store)
        assert not plan.layout
    assert torch.equal(out[0], out[1]) and torch.equal(stored[0], stored[1])
    if n == 1024:                                        # and against the oracle through the first hop
        from oracle import optics
        ref = propagation.angular_spectrum(f[0] * optics.circular_aperture(n, dx, 0.3), dx, lam[0], z[0])
        assert np.linalg.norm(stored[0][0].cpu().numpy() - ref) < 1e-5 * np.linalg.norm(ref)


@pytest.mark.parametrize("n,box", [(1024, 256), (2048, 256), (4096, 256), (1400, 200), (2800, 200), (4100, 410)])
def test_pass_queries_count_the_rows_that_run(ctx, n, box, monkeypatch):
    """Bytes and lines of the passes of a plan that leaves out rows behind its aperture and stop, and of
    the same plan on every row."""
    monkeypatch.setenv("CORO_AUTOTUNE", "0")
    dx, r_ap, r_stop, batch = 1.0 / n, 0.1251, 0.0601, 2
    m = torch.zeros((n, n), dtype=torch.float32, device="cuda")
    els = [coro.element(coro.EL_OPD_MAP, plane=0, opd=m), coro.element(coro.EL_APERTURE, plane=0, radius=r_ap),
           coro.element(coro.EL_OPD_MAP, plane=1, opd=m, amplitude=m), coro.element(coro.EL_CIRCLE, plane=2, radius=r_stop)]

    def rows(r):                                         # a band of whole boxes around the middle
        k = int(r * n)
        return ((n // 2 + k + box) // box - (n // 2 - k) // box) * box

    row = 8.0 * n * batch
    for layout in (None, "0"):
        monkeypatch.delenv("CORO_LAYOUT", raising=False) if layout is None else monkeypatch.setenv("CORO_LAYOUT", layout)
        a, s = (rows(r_ap), rows(r_stop)) if layout is None else (n, n)
        plan = coro.FresnelPlan(ctx, n=n, batch=batch, pixelscale=dx, wavelength=550e-9, distances=[1.5, 2.0], elements=els,
                                init_uniform=True)
        assert [plan.pass_lines(i) for i in range(plan.launch_count)] == [a, n, n, n, s]
        want = [a * row + 4.0 * a * n,                   # field written, map read
                (a + n) * row, 2 * n * row + 8.0 * n * n, (n + s) * row,
                (s + n) * row]                           # the last pass writes zeros outside the stop's rows
        assert [plan.pass_info(i)[1] for i in range(plan.launch_count)] == want
        plan.close()


@pytest.mark.parametrize("n", [1024, 4096])
def test_layout_that_was_queried_brings_the_plan_back(ctx, n, monkeypatch):
    """layout -> alternating -> the queried layout: the passes, left-out rows and bits the plan was
    created with; a kernel set by hand stays what layout 0 returns to, and a copy follows its source."""
    monkeypatch.setenv("CORO_AUTOTUNE", "0")
    monkeypatch.delenv("CORO_LAYOUT", raising=False)
    w = inputs.RelayWorkload(n=n, npix=n // 4, seed=12)
    maps_t = [torch.from_numpy(m.astype(np.float32)).cuda() for m in w.psd_maps()]
    plan, other = relay_plan(ctx, w, maps_t), relay_plan(ctx, w, maps_t)

    def state(p):
        x = torch.full((1, n, n), float("nan"), dtype=torch.complex64, device="cuda")
        p.execute(x)
        return names(p), [p.pass_lines(i) for i in range(p.launch_count)], [p.pass_info(i) for i in range(p.launch_count)], x

    a, was = state(plan), plan.layout
    assert a[1][0] < n and not was
    plan.set_layout(True)
    assert plan.layout and state(plan)[1] == [n] * plan.launch_count
    other.copy_tuning(plan)
    assert other.layout
    for p in (plan, other):
        p.set_layout(was)
        b = state(p)
        assert a[:3] == b[:3] and torch.equal(a[3], b[3])
    plan.set_pass_kernel(1, 0)
    plan.set_layout(True)
    plan.set_layout(False)
    assert state(plan)[1] == [n] * plan.launch_count and not any("_pair" in k for k in names(plan) if k.startswith("row"))
