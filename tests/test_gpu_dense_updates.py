"""Dense lists (the passes over window records) on the images that updates lead to, against
the FP64 oracle, in every form: half a warp an event, two rows a lane, a row a lane, and
the accumulator alone.

- After ten updates of a phantom with an empty surrounding, events at the body's edge see
  far less than those inside, and their terms leave the range of the plain scatter.
- A point source with a spike for an image: a pixel that is nearly all of D, where the
  terms of all events are equal and their rounding must not add up.

Bars: the project's own (image 1e-4 relative above 1% of the maximum, g_rho 1e-4 in norm).
Counts are conserved up to the float adds to A, one for each of at most some 600 work
items: 600 x 2^-25 = 1.8e-5 if all round alike."""
from dataclasses import replace

import numpy as np
import pytest

import oracle
from oracle import Setup
from synth import make_workload
from synth.phantom import Ellipse, Phantom

pytestmark = pytest.mark.gpu

GRIDS = [(140, 100), (350, 250), (699, 503), (1400, 1000)]


def _image_close(img, ref):
    m = ref > 0.01 * ref.max()
    assert np.max(np.abs(img[m] - ref[m]) / ref[m]) <= 1e-4


@pytest.mark.parametrize("ny,nz", GRIDS)
def test_ten_updates_match_oracle(ny, nz):
    from paper_1502_07478_gb300 import Recon
    w = replace(make_workload("small_5mm"), ny=ny, nz=nz, n_events=8000)
    ev = w.events()
    r = Recon.from_workload(w)
    r.upload_events(*ev)
    assert r.stats()["n_window"] >= 64 * ny * nz
    r.iterate(10)
    img = r.read_image().cpu().numpy().astype(np.float64)
    st = r.stats()
    L, g, gs = r.loglik_grad()
    r.close()
    ref, rs = oracle.mlem(Setup.from_workload(w), ev, 10)
    _image_close(img, ref)
    assert st["n_used"] == rs.n_used
    assert st["sum_s_rho"] == pytest.approx(st["n_used"], rel=2e-5)
    Lref, gref, gsref = oracle.loglik_grad(Setup.from_workload(w), ev, img)
    gref = np.asarray(gref).reshape(ny, nz)
    assert L == pytest.approx(Lref, rel=1e-6)
    assert np.linalg.norm(g.cpu().numpy() - gref) <= 1e-4 * np.linalg.norm(gref)
    np.testing.assert_allclose(gs, gsref, rtol=1e-3)


@pytest.mark.parametrize("ny,nz", GRIDS)
@pytest.mark.parametrize("n", [8000, 20_000])
def test_point_source_from_a_spike(ny, nz, n):
    from paper_1502_07478_gb300 import Recon
    src = Phantom((Ellipse(20.0, -30.0, 2.0, 2.0, 0.0, 1.0),))
    w = replace(make_workload("small_5mm"), ny=ny, nz=nz, n_events=n, phantom_fn=lambda: src)
    ev = w.events()
    iy, iz = int((-30.0 + w.R) / w.dy), int((20.0 + w.L / 2) / w.dz)
    rho0 = np.full((ny, nz), 1e-6, np.float32)
    rho0[iy, iz] = 1e3
    setup = Setup.from_workload(w)
    r = Recon.from_workload(w)
    r.upload_events(*ev)
    assert r.stats()["n_window"] >= 64 * ny * nz
    r.set_image(rho0)
    L, g, gs = r.loglik_grad()
    r.iterate(1)
    img = r.read_image().cpu().numpy().astype(np.float64)
    st = r.stats()
    r.close()
    ref, rs = oracle.mlem(setup, ev, 1, rho0=rho0.astype(np.float64))
    _image_close(img, ref)
    assert st["n_used"] == rs.n_used
    assert st["sum_s_rho"] == pytest.approx(st["n_used"], rel=2e-5)
    Lref, gref, _ = oracle.loglik_grad(setup, ev, rho0.astype(np.float64))
    gref = np.asarray(gref).reshape(ny, nz)
    assert L == pytest.approx(Lref, rel=1e-6)
    assert np.linalg.norm(g.cpu().numpy() - gref) <= 1e-4 * np.linalg.norm(gref)
