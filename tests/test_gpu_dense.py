"""Dense lists (64 events over a pixel and more), which the passes over window
records sum in one word of fixed point a pixel, against the FP64 oracle: every lane
capacity, the two-lanes-per-row form, the form whose windows are too large to stage
rho' beside the accumulator, and images whose terms P / D leave the fixed point's
range.  Bars: the project's own (image 1e-4 relative above 1% of the maximum, g_rho
1e-4 in norm, g_sigma 1e-3, L 1e-6)."""
from dataclasses import replace

import numpy as np
import pytest

import oracle
from oracle import Setup
from synth import make_workload

pytestmark = pytest.mark.gpu


def _check(w, ev, rho, kw, lengths=1.0):
    """lengths: the unit of length, in mm (a power of two: the same events)."""
    from paper_1502_07478_gb300 import Recon
    setup = Setup.from_workload(w, **kw)
    r = Recon(w.R / lengths, w.L / lengths, w.ny, w.nz, w.sigma_z / lengths,
              w.sigma_dl / lengths, cut=w.cut, gamma=kw.get("gamma", 0.0) * lengths ** 2,
              kappa_z=kw.get("kappa_z", 0.0))
    r.upload_events(*[e / np.float32(lengths) for e in ev])
    st = r.stats()
    assert st["n_window"] >= 64 * w.ny * w.nz
    r.set_image(rho)
    A = r.backproject().cpu().numpy().astype(np.float64)
    L, g, gs = r.loglik_grad()
    used = r.stats()["n_used"]
    r.close()
    ref = oracle.mlem(setup, ev, 1, rho0=rho.astype(np.float64))[0].reshape(w.ny, w.nz)
    Lref, gref, gsref = oracle.loglik_grad(setup, ev, rho.astype(np.float64))
    gref = np.asarray(gref).reshape(w.ny, w.nz)
    img = rho * A
    m = ref > 0.01 * ref.max()
    assert np.max(np.abs(img[m] - ref[m]) / ref[m]) <= 1e-4
    g = g.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(g - gref) <= 1e-4 * np.linalg.norm(gref)
    if lengths == 1.0:
        assert L == pytest.approx(Lref, rel=1e-6)
        np.testing.assert_allclose(gs, gsref, rtol=1e-3)
    else:
        # the density of an event has the unit of length to the power -3
        assert L == pytest.approx(Lref + 3 * np.log(lengths) * used, rel=1e-6)
        np.testing.assert_allclose(np.asarray(gs) / lengths, gsref, rtol=1e-3)


@pytest.mark.parametrize("ny,nz,kw", [
    (140, 100, {}),
    (171, 121, {}),
    (420, 300, {}),                           # 76 rows, two rows a lane in two warps
    (351, 247, dict(gamma=5e-4, kappa_z=0.1)),
    (233, 401, {}),
    (699, 503, dict(kappa_z=0.2)),
    (640, 830, {}),
    (1151, 820, {}),                          # the last that stages both regions, or near it
    (1399, 1003, {}),                         # 0.5 mm: the accumulator alone
    (1380, 990, dict(gamma=5e-4, kappa_z=0.1)),
])
def test_dense_list_matches_oracle(ny, nz, kw):
    w = replace(make_workload("small_5mm"), ny=ny, nz=nz, n_events=8000)
    rng = np.random.default_rng(ny)
    _check(w, w.events(), rng.uniform(0.5, 2.0, (ny, nz)).astype(np.float32), kw)


@pytest.mark.parametrize("ny,nz", [(140, 100), (1400, 1000)])
@pytest.mark.parametrize("scale,lengths", [(1.0, 1.0), (1e-12, 1.0), (1e12, 1.0), (1.0, 1024.0)])
def test_dense_list_high_contrast(ny, nz, scale, lengths):
    """Zero pixels, a cold background and a spot 1e6 times brighter."""
    w = replace(make_workload("small_5mm"), ny=ny, nz=nz, n_events=8000)
    f = ny // 140
    rho = np.full((ny, nz), 1e-3)
    rho[60 * f:70 * f, 40 * f:60 * f] = 1e3
    rho[75 * f:90 * f, 30 * f:50 * f] = 0.0
    _check(w, w.events(), (scale * rho).astype(np.float32), {}, lengths)


@pytest.mark.parametrize("ny,nz", [(140, 100), (699, 503)])
def test_dense_list_without_records(ny, nz, monkeypatch):
    """A dense list whose records cannot be held is tiled again for the general
    passes, and a later upload for the records."""
    from paper_1502_07478_gb300 import Recon
    w = replace(make_workload("small_5mm"), ny=ny, nz=nz, n_events=8000)
    ev = w.events()
    ref, _ = oracle.mlem(Setup.from_workload(w), ev, 1)
    m = ref > 0.01 * ref.max()
    r = Recon.from_workload(w)
    for fault in ("records", ""):
        monkeypatch.setenv("TSP_SIM_FAULT", fault)
        r.upload_events(*ev)
        r.iterate(1)
        img = r.read_image().cpu().numpy().astype(np.float64)
        assert np.max(np.abs(img[m] - ref[m]) / ref[m]) <= 1e-4
    r.close()
