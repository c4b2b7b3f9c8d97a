"""The tile passes over window records (written once per upload) against the
FP64 oracle, and against the form that sets the rows up in the pass, which a
list takes whose records cannot be held (TSP_SIM_FAULT=records).

Grids cover the lane capacities and the two-lanes-per-row form, row counts at
the edge of a warp, odd sizes and unequal pitches, windows clipped by the image
and the kernel's variants.  Bars: the project's own (image 1e-4 relative above 1%
of the maximum; g_rho 1e-4 in norm, g_sigma 1e-3, L 1e-6), for both forms.  Their
gradients differ by float rounding only: with exponents up to some 20 a kernel
value carries some 20 x 2^-24 = 1.2e-6, so 2e-5 between them leaves room for an
order.  (Their images are not held to that: a pixel with a single small term
x = P rho' / D of some 1e-6 carries the accumulator's quantum, 2^-33, at 1e-4
relative.)
"""
import os
from dataclasses import replace

import numpy as np
import pytest

import oracle
from oracle import Setup
from synth import make_workload

pytestmark = pytest.mark.gpu

#        ny,  nz, kwargs                      lanes
GRIDS = [
    (140, 100, {}),                           # 12, one warp
    (171, 121, {}),                           # 12, a row more than a warp would hold
    (350, 250, {}),                           # 24, 64 rows: two warps
    (351, 247, dict(gamma=5e-4, kappa_z=0.1)),
    (361, 251, {}),                           # 24, three warps
    (233, 401, {}),                           # 48, dy = 3 mm, dz = 1.25 mm
    (699, 503, dict(kappa_z=0.2)),            # 64
    (640, 830, {}),                           # two lanes a row
]


def _events(w):
    """The workload's, and some whose windows the image's edges clip."""
    ev = [np.array(x) for x in w.events()]
    k = 40
    rng = np.random.default_rng(5)
    zt = rng.uniform(-1, 1, k) * 0.5 * w.L
    yt = np.where(rng.random(k) < 0.5, -1, 1) * w.R * rng.uniform(0.8, 1.02, k)
    t = rng.uniform(-0.6, 0.6, k)
    ev[0][:k] = zt + (w.R - yt) * t
    ev[1][:k] = zt - (w.R + yt) * t
    ev[2][:k] = -2 * yt * np.sqrt(1 + t * t)
    return ev


def _run(w, ev, rho, kw, records):
    from paper_1502_07478_gb300 import Recon
    if not records:
        os.environ["TSP_SIM_FAULT"] = "records"
    try:
        r = Recon.from_workload(w, **kw)
        r.upload_events(*ev)
    finally:
        os.environ.pop("TSP_SIM_FAULT", None)
    r.iterate(2)
    img = r.read_image().cpu().numpy().astype(np.float64)
    st = r.stats()
    r.set_image(rho)
    L, g, gs = r.loglik_grad()
    out = (img, r.loglik(), L, g.cpu().numpy().astype(np.float64), gs)
    r.close()
    return out, st


@pytest.mark.parametrize("ny,nz,kw", GRIDS)
def test_records_match_oracle_and_general_form(ny, nz, kw):
    w = replace(make_workload("small_5mm"), ny=ny, nz=nz, n_events=300)
    ev = _events(w)
    rng = np.random.default_rng(ny)
    rho = rng.uniform(0.5, 2.0, (ny, nz)).astype(np.float32)
    (img, ll, L, g, gs), st = _run(w, ev, rho, kw, True)
    (img0, ll0, L0, g0, gs0), st0 = _run(w, ev, rho, kw, False)
    for k in ("n_used", "n_empty", "n_outliers", "n_window", "n_qbad", "n_clipped"):
        assert st[k] == st0[k], k
    assert st["n_clipped"] == 0
    setup = Setup.from_workload(w, **kw)
    ref, _ = oracle.mlem(setup, ev, 2)
    Lref, gref, gsref = oracle.loglik_grad(setup, ev, rho.astype(np.float64))
    m = ref > 0.01 * ref.max()
    assert np.max(np.abs(img[m] - ref[m]) / ref[m]) <= 1e-4
    assert np.max(np.abs(img0[m] - ref[m]) / ref[m]) <= 1e-4
    for a, b in ((L, Lref), (ll, Lref), (L0, Lref), (ll0, Lref)):
        assert a == pytest.approx(b, rel=1e-6)
    gref = np.asarray(gref).reshape(ny, nz)
    assert np.linalg.norm(g - gref) <= 1e-4 * np.linalg.norm(gref)
    assert np.linalg.norm(g - g0) <= 2e-5 * np.linalg.norm(gref)
    np.testing.assert_allclose(gs, gsref, rtol=1e-3)


@pytest.mark.parametrize("scale", [1e-12, 1.0, 1e12])
def test_gradient_of_an_image_of_high_contrast(scale):
    """Zero pixels, a cold background and a spot 1e6 times brighter, at any
    scale of the image: events in the cold have P / D far above the fixed-point
    unit and are scattered by float adds.  g_rho is compared where it matters,
    pixel by pixel, at the bar of its norm."""
    from paper_1502_07478_gb300 import Recon
    w = make_workload("small_5mm", n_events=3000)
    ev = w.events()
    rho = np.full((w.ny, w.nz), 1e-3)
    rho[60:70, 40:60] = 1e3
    rho[75:90, 30:50] = 0.0
    rho = (scale * rho).astype(np.float32)
    r = Recon.from_workload(w)
    r.upload_events(*ev)
    r.set_image(rho)
    L, g, gs = r.loglik_grad()
    r.close()
    Lref, gref, gsref = oracle.loglik_grad(Setup.from_workload(w), ev, rho.astype(np.float64))
    gref = np.asarray(gref).reshape(w.ny, w.nz)
    g = g.cpu().numpy().astype(np.float64)
    assert L == pytest.approx(Lref, rel=1e-6)
    assert np.linalg.norm(g - gref) <= 1e-4 * np.linalg.norm(gref)
    hot = np.abs(gref) > 1e-3 * np.abs(gref).max()
    assert np.max(np.abs(g[hot] - gref[hot]) / np.abs(gref[hot])) <= 1e-4
    np.testing.assert_allclose(gs, gsref, rtol=1e-3)
