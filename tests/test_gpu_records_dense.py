"""The passes over window records against the general ones and the FP64 oracle, on lists
that are dense enough for them (64 events over a pixel): every lane capacity, the
two-lanes-per-row form, the accumulator alone, windows clipped by the image, the kernel's
variants; with the general passes' tiles and with the wide ones that only the records have
room for (items of 512 events and more: here by asking for one item an SM).

Bars: the project's own, and 2e-5 between the two forms' gradients (float rounding only:
exponents up to some 20 x 2^-24 = 1.2e-6, and room for an order)."""
import os
from dataclasses import replace

import numpy as np
import pytest

import oracle
from oracle import Setup
from synth import make_workload
from test_gpu_records import GRIDS, _events

pytestmark = pytest.mark.gpu

WIDE = [g for g in GRIDS if g[0] * g[1] < 100_000]
FINE = [(1399, 1003, {})]


def _run(w, ev, rho, kw, fault, wide):
    from paper_1502_07478_gb300 import Recon
    if fault:
        os.environ["TSP_SIM_FAULT"] = fault
    try:
        r = Recon.from_workload(w, **kw)
        if wide:
            r.set_schedule(items_per_sm=1)
        r.upload_events(*ev)
    finally:
        os.environ.pop("TSP_SIM_FAULT", None)
    launches = r.stats()["launches"]
    r.iterate(2)
    img = r.read_image().cpu().numpy().astype(np.float64)
    st = r.stats()
    r.set_image(rho)
    L, g, gs = r.loglik_grad()
    out = (img, r.loglik(), L, g.cpu().numpy().astype(np.float64), gs)
    if fault:
        # once refused, a change of sigma prepares the list without records, too
        r.set_sigma(1.1 * w.sigma_z, w.sigma_dl)
        r.set_sigma(w.sigma_z, w.sigma_dl)
        r.set_image()
        r.iterate(2)
        again = r.read_image().cpu().numpy().astype(np.float64)
        assert np.abs(again - img).max() <= 2e-5 * img.max()
    r.close()
    return out, st, launches


@pytest.mark.parametrize("ny,nz,kw,wide", [(*g, False) for g in GRIDS + FINE] +
                         [(*g, True) for g in WIDE])
def test_records_match_oracle_and_general_passes(ny, nz, kw, wide):
    w = replace(make_workload("small_5mm"), ny=ny, nz=nz, n_events=90_000 if wide else 9000)
    ev = _events(w)
    rho = np.random.default_rng(ny).uniform(0.5, 2.0, (ny, nz)).astype(np.float32)
    (img, ll, L, g, gs), st, n = _run(w, ev, rho, kw, "", wide)
    (img0, ll0, L0, g0, gs0), st0, n0 = _run(w, ev, rho, kw, "records", wide)
    assert st["n_window"] >= 64 * ny * nz
    # which form ran: the records' kernel is a launch of the upload; a list tiled wide
    # and refused is prepared twice
    assert n0 == n + 1 if wide else n0 == n - 1
    for k in ("n_used", "n_empty", "n_outliers", "n_window", "n_qbad", "n_clipped"):
        assert st[k] == st0[k] or (wide and k == "n_outliers"), k
    assert st["n_clipped"] == 0
    setup = Setup.from_workload(w, **kw)
    ref, _ = oracle.mlem(setup, ev, 2)
    Lref, gref, gsref = oracle.loglik_grad(setup, ev, rho.astype(np.float64))
    m = ref > 0.01 * ref.max()
    for x in (img, img0):
        assert np.max(np.abs(x[m] - ref[m]) / ref[m]) <= 1e-4
    for a in (L, ll, L0, ll0):
        assert a == pytest.approx(Lref, rel=1e-6)
    gref = np.asarray(gref).reshape(ny, nz)
    assert np.linalg.norm(g - gref) <= 1e-4 * np.linalg.norm(gref)
    assert np.linalg.norm(g - g0) <= 2e-5 * np.linalg.norm(gref)
    np.testing.assert_allclose(gs, gsref, rtol=1e-3)


def test_streamed_upload_that_is_refused(monkeypatch):
    """begin / append / end in chunks, tiled wide and refused at the end."""
    from paper_1502_07478_gb300 import Recon
    w = make_workload("small_5mm", n_events=90_000)
    ev = w.events()
    ref, _ = oracle.mlem(Setup.from_workload(w), ev, 1)
    m = ref > 0.01 * ref.max()
    r = Recon.from_workload(w)
    r.set_schedule(items_per_sm=1)
    for fault in ("records", ""):
        monkeypatch.setenv("TSP_SIM_FAULT", fault)
        r.begin_events(len(ev[0]))
        for a in range(0, len(ev[0]), 25_000):
            r.append_events(*[x[a:a + 25_000] for x in ev])
        r.end_events()
        r.iterate(1)
        img = r.read_image().cpu().numpy().astype(np.float64)
        assert np.max(np.abs(img[m] - ref[m]) / ref[m]) <= 1e-4
    r.close()


@pytest.mark.parametrize("cut", [3.0, 5.0])
def test_small_radius_and_wide_cut(cut):
    """The paper's own geometry, where Q varies over a window by much."""
    from paper_1502_07478_gb300 import Recon
    w = make_workload("paper_geom_4mm", n_events=20_000, cut=cut)
    ev = w.events()
    r = Recon.from_workload(w)
    r.upload_events(*ev)
    r.iterate(3)
    img = r.read_image().cpu().numpy().astype(np.float64)
    st = r.stats()
    r.close()
    assert st["n_window"] >= 64 * w.ny * w.nz
    ref, rs = oracle.mlem(Setup.from_workload(w), ev, 3)
    m = ref > 0.01 * ref.max()
    assert st["n_used"] == rs.n_used
    assert np.max(np.abs(img[m] - ref[m]) / ref[m]) <= 1e-4


@pytest.mark.parametrize("ny,nz", [(140, 100), (350, 250)])
@pytest.mark.parametrize("n", [20_000, 100_000])
def test_gradient_of_short_and_longer_items(ny, nz, n):
    """At 5 mm a list of 2e4 has fewer than two events an item and group: its gradient goes
    without the records, that of 1e5 over them; at 2 mm both do."""
    from paper_1502_07478_gb300 import Recon
    w = replace(make_workload("small_5mm"), ny=ny, nz=nz, n_events=n)
    ev = w.events()
    r = Recon.from_workload(w)
    r.upload_events(*ev)
    r.iterate(2)
    rho = r.read_image().cpu().numpy().astype(np.float64)
    L, g, gs = r.loglik_grad()
    st = r.stats()
    r.close()
    Lref, gref, gsref = oracle.loglik_grad(Setup.from_workload(w), ev, rho)
    gref = np.asarray(gref).reshape(ny, nz)
    assert st["n_clipped"] == 0
    assert L == pytest.approx(Lref, rel=1e-6)
    assert np.linalg.norm(g.cpu().numpy() - gref) <= 1e-4 * np.linalg.norm(gref)
    np.testing.assert_allclose(gs, gsref, rtol=1e-3)
