"""Workloads of coronagraph modelling, each as one pass through the library's public calls.

`listed()` names them; `draw(rng)` gives another of the same ranges; `prepare` makes what a
program holds before the call (seeded inputs on the GPU, plans), `run` is the pass, `work` what
it has to move and compute at least, `exact` its result in 64 bits by plain torch.

Real values: unit-amplitude beams through obscured apertures, surfaces of 20 nm RMS with a
power-law spectrum, pupils with a few nm of low-order and probe phase, actuator heights of a few
nm. Sums that reach the host in 64 bits but come out of a complex64 chain (dark-hole sums, the
wavefront-control loss) are left out or kept in the chain's own 32 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1806_06467_gb300 import coro, wfc

LAM0 = 550e-9
DEV = "cuda"
MIXED = (150, 1050, 1400, 1500, 2100, 2800, 3000, 4100)   # even lengths that are not powers of two


def listed():
    return [
        # one short free-space hop of a 128-pixel aperture padded to 256: the smallest call, an
        # interactive model or a per-frame step of a control loop
        dict(name="hop_256", kind="hop", n=256, batch=1, dbl=False),
        # a Talbot bench modelled step by step: 256 pixels across the beam, oversampled 8 times,
        # every element and the hop a call of its own, then the detector image
        dict(name="talbot_2048", kind="steps", n=2048, npix=256, batch=1),
        # the six-plane relay (obscured, spidered pupil; lens, surface, lens, surface, stop) at
        # the full grid: the headline propagation workload
        dict(name="relay_4096", kind="relay", n=4096, npix=1024, batch=1, dbl=False, graph=True),
        # the same relay across a band: five wavelengths in one batch at the next smaller grid
        dict(name="relay_2048_band", kind="relay", n=2048, npix=512, batch=5, dbl=False, graph=True),
        # the grid of 700 pixels oversampled 4 times, not a power of two
        dict(name="relay_2800", kind="relay", n=2800, npix=700, batch=1, dbl=False, graph=True),
        # the relay in double precision: the reference run a model is checked against
        dict(name="relay_c128_1024", kind="relay", n=1024, npix=256, batch=1, dbl=True, graph=True),
        # the nine-plane shaped-pupil system through three foci, propagators chosen by the plan
        dict(name="spc_4096", kind="spc", npix=1024, batch=1),
        # broadband image set: 21 wavelengths x 8 sources (the star and seven companions) through
        # the Lyot coronagraph, at the precision that suits companion images
        dict(name="lyot_tf32_168", kind="lyot", precision="tf32", n=1024, npix=1024, m_occ=256, m_det=512, lams=21,
             states=8, companions=True, field=False),
        # one probe state of the same band at extended precision, fields kept for the estimator
        dict(name="lyot_ext_21", kind="lyot", precision="ext", n=1024, npix=1024, m_occ=256, m_det=512, lams=21,
             states=1, companions=False, field=True),
        # one reference image in double precision
        dict(name="lyot_fp64_1", kind="lyot", precision="fp64", n=1024, npix=1024, m_occ=256, m_det=512, lams=1,
             states=1, companions=False, field=True),
        # one matrix Fourier transform of a ragged pupil to a camera field, default precision
        dict(name="mft_1000_301", kind="mft", precision="fp32", direction=-1, n=1000, m=301, batch=1),
        # wavefront control: loss and gradient for two 48 x 48 mirrors over 11 wavelengths
        dict(name="wfc_4096_11", kind="wfc", n=4096, npix=1024, m_occ=256, m_det=512, n_act=48, lams=11),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("hop", "steps", "relay", "relay", "spc", "lyot", "lyot", "mft", "mft", "wfc"))
    if kind == "hop":
        dbl = rng.random() < 0.25
        n = rng.choice((32, 64, 128, 256, 512, 1024, 2048, 4096, 150, 1050, 1400, 2800))
        return dict(kind=kind, n=n, batch=rng.randint(1, max(1, min(9, 4096 * 4096 // (n * n)))), dbl=dbl)
    if kind == "steps":
        n = rng.choice((256, 512, 1024, 2048, 4096))
        return dict(kind=kind, n=n, npix=rng.randint(n // 8, n // 2), batch=rng.randint(1, 3))
    if kind == "relay":
        dbl = rng.random() < 0.2
        n = rng.choice((256, 512, 1024, 2048) if dbl else (256, 512, 1024, 2048, 4096) + MIXED)
        most = max(1, min(7, (2048 * 2048 if dbl else 4100 * 4100) // (n * n)))
        return dict(kind=kind, n=n, npix=rng.randint(n // 6, n // 2), batch=rng.randint(1, most), dbl=dbl,
                    graph=rng.random() < 0.5)
    if kind == "spc":
        return dict(kind=kind, npix=rng.choice((64, 128, 175, 256, 350, 512)), batch=rng.randint(1, 3))
    if kind == "lyot":
        precision = rng.choice(("tf32", "bf16", "ext", "fp64"))
        n = log(130, 1100)
        lams = 1 if precision == "fp64" else rng.randint(1, 21)
        companions = precision in ("tf32", "bf16")
        return dict(kind=kind, precision=precision, n=n, npix=n - rng.randint(0, n // 10), m_occ=log(64, 280),
                    m_det=log(100, 520), lams=lams, states=1 if precision == "fp64" else rng.randint(2, 4),
                    companions=companions, field=rng.random() < 0.5)
    if kind == "mft":
        precision = rng.choice(("fp32", "tf32", "bf16", "ext", "fp64"))
        return dict(kind=kind, precision=precision, direction=rng.choice((-1, 1)), n=log(60, 1500), m=log(40, 1100),
                    batch=rng.randint(1, 2 if precision == "fp64" else 6))
    n = rng.choice((512, 1024, 2048))
    return dict(kind=kind, n=n, npix=n // 4, m_occ=log(64, 256), m_det=log(100, 400), n_act=rng.choice((32, 48)),
                lams=rng.randint(1, 7))


# ------------------------------------------------------------------------------- inputs

def generator(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) & 0x7fffffff)


def uniform(seed, lo, hi, count):
    return np.random.default_rng(int(seed)).uniform(lo, hi, count)


def surface(n, g, rms):
    """A power-law surface (PSD ~ f^-3), metres, float32 [n][n]."""
    white = torch.randn((n, n), generator=g, device=DEV)
    k = torch.fft.fftfreq(n, device=DEV)
    kr = torch.hypot(k[None, :], k[:, None])
    kr[0, 0] = 1.0
    shape = kr ** -1.5
    shape[0, 0] = 0.0
    s = torch.fft.ifft2(torch.fft.fft2(white) * shape).real
    return (s * (rms / s.square().mean().sqrt())).contiguous()


def k2grid(n):
    k = torch.arange(n, device=DEV, dtype=torch.float64) - n // 2
    return k[None, :] ** 2 + k[:, None] ** 2


def band(lams, lo=500e-9, hi=600e-9):
    return np.linspace(lo, hi, lams) if lams > 1 else np.array([LAM0])


CONTEXT = []


def context():
    """One context on torch's current stream, as a program keeps."""
    if not CONTEXT:
        CONTEXT.append(coro.Context(0))
    return CONTEXT[0]


# hop: a random field whose hop keeps its energy
def hop_inputs(c, seed):
    g = generator(seed)
    t = torch.complex128 if c["dbl"] else torch.complex64
    field = torch.randn((c["batch"], c["n"], c["n"]), generator=g, device=DEV, dtype=t)
    return field, 2.0 / c["n"], np.linspace(500e-9, 600e-9, c["batch"]), float(uniform(seed, 0.5, 5.0, 1)[0])


# steps: aperture, a sine phase grating, a surface, a hop, the image
def steps_inputs(c, seed):
    g = generator(seed)
    n, radius = c["n"], 0.02
    dx = 2 * radius / c["npix"]
    u = uniform(seed, 0.5, 1.0, 3)
    return dict(dx=dx, radius=radius, lam=np.linspace(500e-9, 550e-9, c["batch"]), map=surface(n, g, 5e-9),
                amp=10e-9 * u[0], freq=250.0 * u[1], z=8.0 * u[2])


def relay_inputs(c, seed):
    g = generator(seed)
    n = c["n"]
    return dict(dx=1.0 / c["npix"], lam=band(c["batch"], 520e-9, 580e-9), maps=[surface(n, g, 20e-9) for _ in range(2)],
                z=uniform(seed, 0.5, 5.0, 5))


F_LENS = (5.0, 2.0)


def relay_elements(maps):
    return [coro.element(coro.EL_APERTURE, plane=0, radius=0.5, obscuration=0.3, n_spiders=4, spider_width=0.01),
            coro.element(coro.EL_LENS, plane=1, focal_length=F_LENS[0]), coro.element(coro.EL_OPD_MAP, plane=2, opd=maps[0]),
            coro.element(coro.EL_LENS, plane=3, focal_length=F_LENS[1]), coro.element(coro.EL_OPD_MAP, plane=4, opd=maps[1]),
            coro.element(coro.EL_CIRCLE, plane=5, radius=0.45)]


# spc: a 2.37 m f/7.8 telescope, a 20 mm relay at f/20, a ringed shaped pupil, a bow-tie mask
D_TEL, D_RELAY = 2.37, 0.02
F_PRI, F_M3 = 7.8 * 2.37, 20.0 * 0.02
F_M2 = F_PRI * D_RELAY / D_TEL
SPC_LENS = {0: F_PRI, 1: F_M2, 2: F_M3, 3: F_M3, 5: F_M3, 7: F_M3}
SPC_DIST = [F_PRI + F_M2, F_M2 + F_M3, 2 * F_M3, F_M3, F_M3, F_M3, 2 * F_M3, 2 * F_M3]


def spc_lams(c):
    return band(c["batch"], 545e-9, 555e-9)


def shaped_pupil(n, pitch, seed):
    edges = torch.tensor(np.sort(uniform(seed, 0.3, 1.0, 11)) * 0.5 * D_RELAY, device=DEV)
    r = k2grid(n).sqrt() * pitch
    zone = torch.searchsorted(edges, r)
    return (zone % 2 == 0) & (r >= 0.15 * D_RELAY) & (r <= 0.5 * D_RELAY)


def bowtie(n, pitch, lam):
    k = torch.arange(n, device=DEV, dtype=torch.float64) - n // 2
    r = k2grid(n).sqrt() * (pitch / (lam * 20.0))
    return (r >= 2.5) & (r <= 9.0) & (k[:, None].abs() <= math.tan(math.radians(32.5)) * k[None, :].abs())


# lyot: clear pupils with a few nm of low-order phase, and per state either a DM probe or a source
# off the axis (state 0: the star); the spot, the pitches and the dark hole are fixed in angle, so
# in lambda/D they scale with the wavelength
def lyot_items(c, lams):
    items = []
    for lam in lams:
        r = LAM0 / lam
        items.append(dict(m_occ=max(16, int(np.rint(c["m_occ"] * r))), du_occ=12.8 / c["m_occ"] * r, spot_radius=5.0 * r,
                          du_det=128.0 / c["m_det"] * r, dh_in=6.0 * r, dh_out=20.0 * r))
    return items


def lyot_pupils(c, seed):
    lams = np.repeat(band(c["lams"]), c["states"])
    n, npix = c["n"], c["npix"]
    k = (torch.arange(n, device=DEV, dtype=torch.float64) - n // 2) / npix
    disk = (k2grid(n) * ((1.0 / npix) * (1.0 / npix)) <= 0.25)
    u = uniform(seed, -1.0, 1.0, (6, 3))
    opd = sum(5e-9 * a * torch.cos(2 * math.pi * (3 * fx * k[None, :] + 3 * fy * k[:, None]) + 6 * a) for a, fx, fy in u)
    t = torch.complex128 if c["precision"] == "fp64" else torch.complex64
    out = torch.empty((len(lams), n, n), dtype=t, device=DEV)
    tilt = uniform(seed + 1, -9.0, 9.0, (c["states"], 2))            # lambda_c / D
    tilt[0] = 0.0
    for i, lam in enumerate(lams):
        a = i % c["states"]
        if c["companions"]:
            extra = LAM0 * (tilt[a, 0] * k[None, :] + tilt[a, 1] * k[:, None])
        else:
            extra = 20e-9 * torch.sinc(24 * k)[:, None] * (torch.sinc(24 * k) * torch.cos(26 * math.pi * k + a * math.pi / 4))[None, :]
        out[i] = torch.polar(disk.to(torch.float64), (opd + extra) * (2 * math.pi / lam)).to(t)
    return out, lams


PREC = {"fp32": coro.MFT_FP32, "tf32": coro.MFT_3XTF32, "bf16": coro.MFT_3XBF16, "ext": coro.MFT_EXT, "fp64": coro.MFT_FP64}
LYOT_FRAC = 0.8


def mft_inputs(c, seed):
    """Pupil fields on the way out, focal-plane fields on the way back."""
    g = generator(seed)
    t = torch.complex128 if c["precision"] == "fp64" else torch.complex64
    field = torch.randn((c["batch"], c["n"], c["n"]), generator=g, device=DEV, dtype=t)
    npix = float(c["n"] if c["direction"] < 0 else c["m"])
    return field, npix, uniform(seed, 0.1, 0.4, c["batch"])


# wfc: two mirrors 0.3 m apart over a 48 mm pupil
WFC_D, WFC_Z = 0.048, 0.3


def wfc_heights(c, seed):
    h = torch.rand((2, c["n_act"], c["n_act"]), generator=generator(seed), device=DEV)
    return (2 * h - 1) * 5e-9


def wfc_lams(c):
    return band(c["lams"], 525e-9, 575e-9)


# ------------------------------------------------------------------------------- the passes

def prepare(case, seed):
    ctx, kind = context(), case["kind"]
    st = dict(kind=kind, ctx=ctx)
    if kind == "hop":
        st["field"], st["dx"], st["lam"], st["z"] = hop_inputs(case, seed)
    elif kind == "steps":
        st.update(steps_inputs(case, seed))
        n, b = case["n"], case["batch"]
        st["field"] = torch.empty((b, n, n), dtype=torch.complex64, device=DEV)
        st["image"] = torch.empty((b, n, n), dtype=torch.float32, device=DEV)
        st["elements"] = [coro.element(coro.EL_APERTURE, radius=st["radius"]),
                          coro.element(coro.EL_SINE, sine_freq=st["freq"], sine_amplitude=st["amp"], axis=0),
                          coro.element(coro.EL_OPD_MAP, opd=st["map"])]
    elif kind == "relay":
        i = relay_inputs(case, seed)
        n, b = case["n"], case["batch"]
        st["plan"] = coro.FresnelPlan(ctx, n=n, batch=b, pixelscale=i["dx"], wavelength=i["lam"], distances=list(i["z"]),
                                      elements=relay_elements(i["maps"]), dtype=coro.C128 if case["dbl"] else coro.C64,
                                      init_uniform=True)
        st["plan"].use_graph(case["graph"])
        st["field"] = torch.empty((b, n, n), dtype=torch.complex128 if case["dbl"] else torch.complex64, device=DEV)
    elif kind == "spc":
        n, b, lams = 4 * case["npix"], case["batch"], spc_lams(case)
        zero, sp, fpm = (torch.zeros((b, n, n), device=DEV) for _ in range(3))
        els = [coro.element(coro.EL_APERTURE, plane=0, radius=D_TEL / 2, obscuration=0.3, n_spiders=4, spider_width=0.01 * D_TEL)]
        els += [coro.element(coro.EL_LENS, plane=p, focal_length=f) for p, f in SPC_LENS.items()]
        els += [coro.element(coro.EL_OPD_MAP, plane=p, opd=zero, amplitude=m, flags=coro.ELF_MAP_BATCHED) for p, m in ((4, sp), (6, fpm))]
        plan = coro.FresnelSystem(ctx, n=n, batch=b, pixelscale=D_TEL / case["npix"], wavelength=lams, beam_radius=D_TEL / 2,
                                  distances=SPC_DIST, elements=els, init_uniform=True)
        p4, p6 = plan.plane_pitch(4), plan.plane_pitch(6)
        for j, lam in enumerate(lams):
            sp[j] = shaped_pupil(n, p4[j], seed)
            fpm[j] = bowtie(n, p6[j], lam)
        plan.use_graph(True)
        st.update(plan=plan, field=torch.empty((b, n, n), dtype=torch.complex64, device=DEV))
    elif kind == "lyot":
        st["pupil"], lams = lyot_pupils(case, seed)
        b, md, dbl = len(lams), case["m_det"], case["precision"] == "fp64"
        st["plan"] = coro.LyotPlan(ctx, n=case["n"], npix=float(case["npix"]), lyot_frac=LYOT_FRAC, m_det=md,
                                   items=lyot_items(case, lams), precision=PREC[case["precision"]])
        st["peak"] = st["plan"].peak(st["pupil"])
        if not dbl:
            st["plan"].use_graph(True)
        st["image"] = torch.empty((b, md, md), dtype=torch.float32, device=DEV)
        t = torch.complex128 if dbl else torch.complex64
        st["field"] = torch.empty((b, md, md), dtype=t, device=DEV) if case["field"] else None
    elif kind == "mft":
        st["field"], st["npix"], st["du"] = mft_inputs(case, seed)
        st["direction"], st["m"], st["precision"] = case["direction"], case["m"], PREC[case["precision"]]
    else:
        lams = wfc_lams(case)
        st["plan"] = wfc.WfcPlan(ctx, wavelengths=list(lams), n_fresnel=case["n"], diam_m=WFC_D, npix=case["npix"], z_m=WFC_Z,
                                 n_act=case["n_act"], pitch_m=WFC_D / case["n_act"], fwhm_m=WFC_D / case["n_act"],
                                 lyot_frac=LYOT_FRAC, m_det=case["m_det"], items=lyot_items(case, lams),
                                 precision=coro.MFT_3XTF32)
        st["plan"].peak()
        st["heights"] = wfc_heights(case, seed).requires_grad_(True)
    return st


def run(st):
    ctx, kind = st["ctx"], st["kind"]
    if kind == "hop":
        coro.propagate_fresnel(ctx, st["field"], st["dx"], st["lam"], st["z"])
        return st["field"]
    if kind == "steps":
        coro.wavefront_init(ctx, st["field"])
        for el in st["elements"]:
            coro.apply_element(ctx, st["field"], st["dx"], st["lam"], el)
        coro.propagate_fresnel(ctx, st["field"], st["dx"], st["lam"], st["z"])
        coro.intensity(ctx, st["field"], out=st["image"])
        return {"field": st["field"], "image": st["image"]}
    if kind == "relay":
        st["plan"].execute(st["field"])
        return st["field"]
    if kind == "spc":
        return {"pitch": st["plan"].execute(st["field"]), "field": st["field"]}
    if kind == "lyot":
        st["plan"].execute(st["pupil"], peak=st["peak"], intensity=st["image"], field=st["field"], want_dh=False)
        return {"image": st["image"], "field": st["field"]}
    if kind == "mft":
        return coro.propagate_mft(ctx, st["field"], st["npix"], st["direction"], st["m"], st["du"], st["precision"])
    st["heights"].grad = None
    loss = wfc.dark_hole_loss(st["heights"], st["plan"])
    loss.backward()
    return {"loss": loss.detach().float(), "gradient": st["heights"].grad}


# ------------------------------------------------------------------------------- least work

def fft2_flops(n):
    return 5.0 * n * n * math.log2(float(n) * n)


def lyot_flops(n, mo, md):
    """Complex multiply-adds (8 flops) of the MFTs there, back and to the detector."""
    return 8.0 * (2 * (n * mo * n + mo * mo * n) + n * md * n + md * md * n)


def work(case):
    kind, b = case["kind"], case.get("batch", 1)
    cb = 16.0 if case.get("dbl") or case.get("precision") == "fp64" else 8.0
    if kind == "hop":
        n = case["n"]
        return {"bytes": 2 * cb * n * n * b, "flops": 2 * fft2_flops(n) * b}
    if kind == "steps":
        n = case["n"]
        return {"bytes": (cb + 4.0) * n * n * b + 4.0 * n * n, "flops": 2 * fft2_flops(n) * b}
    if kind == "relay":
        n = case["n"]
        return {"bytes": cb * n * n * b + 8.0 * n * n, "flops": 10 * fft2_flops(n) * b}
    if kind == "spc":
        n = 4 * case["npix"]
        return {"bytes": (8.0 + 12.0) * n * n * b, "flops": 13 * fft2_flops(n) * b}
    if kind == "mft":
        n, m = case["n"], case["m"]
        return {"bytes": cb * (n * n + m * m) * b, "flops": 8.0 * (m * n * n + m * m * n) * b}
    lams = wfc_lams(case) if kind == "wfc" else np.repeat(band(case["lams"]), case["states"])
    md = case["m_det"]
    flops = sum(lyot_flops(case["npix"] if kind == "wfc" else case["n"], it["m_occ"], md) for it in lyot_items(case, lams))
    if kind == "wfc":
        return {"bytes": 4.0 * 4 * case["n_act"] ** 2, "flops": 2 * flops + 8 * fft2_flops(case["n"]) * len(lams)}
    n = case["n"]
    return {"bytes": (cb * n * n + 4.0 * md * md + (cb * md * md if case["field"] else 0)) * len(lams), "flops": flops}


# ------------------------------------------------------------------------------- in 64 bits

def dft2(e, inverse=False):
    f = torch.fft.ifft2 if inverse else torch.fft.fft2
    return torch.fft.fftshift(f(torch.fft.ifftshift(e, dim=(-2, -1))), dim=(-2, -1))


def cis(phase):
    return torch.polar(torch.ones_like(phase), phase)


def cycles(c):
    """exp(2 pi i c), the whole cycles dropped first."""
    return cis(2 * math.pi * (c - torch.round(c)))


def hop64(e, dx, lam, z):
    n = e.shape[-1]
    return dft2(dft2(e) * cycles(-0.5 * lam * z / (n * dx) ** 2 * k2grid(n)), inverse=True)


def quad64(n, pitch, lam, z):
    return cycles(0.5 * pitch * pitch / (lam * z) * k2grid(n))


def direct64(e, dx, lam, z, q_in, q_out):
    n = e.shape[-1]
    du = abs(lam * z / (n * dx))
    a = e * quad64(n, dx, lam, z) if q_in else e
    out = (dft2(a) if z > 0 else (n * n) * dft2(a, inverse=True)) * (dx * dx / (1j * lam * z))
    return (out * quad64(n, du, lam, z) if q_out else out), du


def aperture64(n, dx, radius, obscuration, width):
    r2 = k2grid(n) * (dx * dx)
    a = (r2 <= radius * radius) & (r2 >= (obscuration * radius) ** 2)
    if width:
        v = ((torch.arange(n, device=DEV, dtype=torch.float64) - n // 2) * dx).abs() < width / 2
        a &= ~(v[None, :] | v[:, None])
    return a.to(torch.complex128)


def phasor64(opd, lam):
    return cycles(opd.double() / lam)


def basis64(m, du, n, npix, sign):
    u, j = (torch.arange(k, device=DEV, dtype=torch.float64) - k // 2 for k in (m, n))
    return cycles(sign * torch.outer(u, j) * (du / npix))


def mft64(e, npix, m, du):
    a = basis64(m, du, e.shape[-1], npix, -1)
    return (du / npix) * (a @ e @ a.T)


def imft64(e, npix, n, du):
    a = basis64(e.shape[-1], du, n, npix, +1)
    return (du / npix) * (a.T @ e @ a)


def lyot64(e_a, c, n, npix, it, occulter=True):
    if occulter:
        mo = it["m_occ"]
        spot = k2grid(mo) * (it["du_occ"] * it["du_occ"]) <= it["spot_radius"] ** 2
        e_a = e_a - imft64(spot * mft64(e_a, npix, mo, it["du_occ"]), npix, n, it["du_occ"])
    stop = k2grid(n) * ((1.0 / npix) * (1.0 / npix)) <= (0.5 * LYOT_FRAC) ** 2
    return mft64(e_a * stop, npix, c["m_det"], it["du_det"])


def abs2(e):
    return e.real ** 2 + e.imag ** 2


def dm64(h, n, dx):
    na = h.shape[-1]
    pitch = WFC_D / na
    x = (torch.arange(n, device=DEV, dtype=torch.float64) - n // 2) * dx
    xa = (torch.arange(na, device=DEV, dtype=torch.float64) - (na - 1) / 2) * pitch
    g = torch.exp(-(x[:, None] - xa[None, :]) ** 2 * (4 * math.log(2.0) / pitch ** 2))
    return 2.0 * (g @ h @ g.T)


def spc64(c, lam, seed):
    """The nine planes behind a Gaussian pilot beam: inside its Rayleigh range the field is held
    as it is, outside relative to the sphere through the beam's waist."""
    n, pitch = 4 * c["npix"], D_TEL / c["npix"]
    e = aperture64(n, pitch, D_TEL / 2, 0.3, 0.01 * D_TEL)
    q, outside = complex(0.0, -math.pi * (D_TEL / 2) ** 2 / lam), False
    for p in range(9):
        if p == 4:
            e = e * shaped_pupil(n, pitch, seed)
        if p == 6:
            e = e * bowtie(n, pitch, lam)
        if p in SPC_LENS:
            if outside:
                e = e * quad64(n, pitch, lam, q.real)
            e = e * quad64(n, pitch, lam, -SPC_LENS[p])
            q = 1.0 / (1.0 / q - 1.0 / SPC_LENS[p])
            outside = abs(q.real) >= abs(q.imag)
            if outside:
                e = e * quad64(n, pitch, lam, -q.real)
        if p == 8:
            return (e * quad64(n, pitch, lam, q.real) if outside else e), pitch
        qb = q + SPC_DIST[p]
        out_b = abs(qb.real) >= abs(qb.imag)
        if not outside and not out_b:
            e = hop64(e, pitch, lam, SPC_DIST[p])
        else:
            if outside:
                e, pitch = direct64(e, pitch, lam, -q.real, False, True)
            elif q.real != 0.0:
                e = hop64(e, pitch, lam, -q.real)
            if out_b:
                e, pitch = direct64(e, pitch, lam, qb.real, True, False)
            elif qb.real != 0.0:
                e = hop64(e, pitch, lam, qb.real)
        q, outside = qb, out_b


def exact(case, seed):
    kind = case["kind"]
    if kind == "hop":
        field, dx, lams, z = hop_inputs(case, seed)
        return torch.stack([hop64(f.to(torch.complex128), dx, lam, z) for f, lam in zip(field, lams)])
    if kind == "steps":
        i = steps_inputs(case, seed)
        n, out = case["n"], []
        x = (torch.arange(n, device=DEV, dtype=torch.float64) - n // 2) * i["dx"]
        opd = (i["amp"] * torch.sin(2 * math.pi * i["freq"] * x))[None, :] + i["map"].double()
        for lam in i["lam"]:
            e = aperture64(n, i["dx"], i["radius"], 0.0, 0.0) * cycles(opd / lam)
            out.append(hop64(e, i["dx"], lam, i["z"]))
        field = torch.stack(out)
        return {"field": field, "image": abs2(field)}
    if kind == "relay":
        i = relay_inputs(case, seed)
        n, dx, out = case["n"], i["dx"], []
        for lam in i["lam"]:
            e = aperture64(n, dx, 0.5, 0.3, 0.01)
            for p, z in enumerate(i["z"]):
                if p in (1, 3):
                    e = e * quad64(n, dx, lam, -F_LENS[p // 2])
                elif p in (2, 4):
                    e = e * phasor64(i["maps"][p // 2 - 1], lam)
                e = hop64(e, dx, lam, z)
            out.append(e * (k2grid(n) * (dx * dx) <= 0.45 * 0.45))
        return torch.stack(out)
    if kind == "spc":
        both = [spc64(case, lam, seed) for lam in spc_lams(case)]
        return {"pitch": np.array([p for _, p in both]), "field": torch.stack([e for e, _ in both])}
    if kind == "lyot":
        pupil, lams = lyot_pupils(case, seed)
        n, npix, images, fields = case["n"], float(case["npix"]), [], []
        for e, it in zip(pupil, lyot_items(case, lams)):
            e = e.to(torch.complex128)
            det = lyot64(e, case, n, npix, it)
            images.append(abs2(det) / abs2(lyot64(e, case, n, npix, it, occulter=False)).max())
            if case["field"]:
                fields.append(det)
        return {"image": torch.stack(images), "field": torch.stack(fields) if fields else None}
    if kind == "mft":
        field, npix, du = mft_inputs(case, seed)
        to = mft64 if case["direction"] < 0 else imft64
        return torch.stack([to(f.to(torch.complex128), npix, case["m"], float(d)) for f, d in zip(field, du)])
    lams = wfc_lams(case)
    n, npix, dx, total = case["n"], case["npix"], WFC_D / case["npix"], 0.0
    h = wfc_heights(case, seed).double().requires_grad_(True)
    grad = torch.zeros_like(h)
    ap, lo = aperture64(n, dx, WFC_D / 2, 0.0, 0.0), n // 2 - npix // 2
    md = case["m_det"]

    def pupil(hh, lam):
        e = hop64(ap * cycles(dm64(hh[0], n, dx) / lam), dx, lam, WFC_Z) * cycles(dm64(hh[1], n, dx) / lam)
        return hop64(e, dx, lam, -WFC_Z)[lo:lo + npix, lo:lo + npix]

    for lam, it in zip(lams, lyot_items(case, lams)):
        with torch.no_grad():
            peak = abs2(lyot64(pupil(torch.zeros_like(h), lam), case, npix, float(npix), it, occulter=False)).max()
        r2 = k2grid(md) * (it["du_det"] * it["du_det"])
        hole = (r2 >= it["dh_in"] ** 2) & (r2 <= it["dh_out"] ** 2)
        loss = (abs2(lyot64(pupil(h, lam), case, npix, float(npix), it)) * hole).sum() / peak
        grad += torch.autograd.grad(loss, h)[0]
        total += float(loss.detach())
    return {"loss": torch.tensor(total, dtype=torch.float64), "gradient": grad}
