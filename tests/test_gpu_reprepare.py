"""A preparation of events that fails (TSP_SIM_FAULT, on the host, before anything
is launched) leaves a context without prepared events: every pass answers
TSP_ESTATE until one has succeeded, since the items and window records of an
earlier preparation belong to another plan."""
import numpy as np
import pytest

from synth import make_workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dense():
    w = make_workload("small_5mm", n_events=20_000)
    return w, w.events()


def _passes(r):
    return [lambda: r.iterate(1), r.loglik, r.loglik_grad, r.backproject]


@pytest.mark.parametrize("kind", ["launch", "oom"])
@pytest.mark.parametrize("call", ["set_sigma", "set_schedule"])
def test_failed_preparation_leaves_nothing_to_run(dense, monkeypatch, kind, call):
    from paper_1502_07478_gb300 import Recon, TspError
    from paper_1502_07478_gb300._lib import TSP_ECUDA, TSP_ENOMEM, TSP_ESTATE
    w, ev = dense
    # wider windows; lower tiles, more than there are bin buffers for
    args = dict(set_sigma=(2.0 * w.sigma_z, 1.5 * w.sigma_dl), set_schedule=(8,))[call]
    if kind == "oom" and call == "set_sigma":
        args = (0.4 * w.sigma_z, 0.4 * w.sigma_dl)      # smaller halo: more tiles
    r = Recon.from_workload(w)
    r.upload_events(*ev)
    r.iterate(1)
    monkeypatch.setenv("TSP_SIM_FAULT", kind)
    try:
        getattr(r, call)(*args)
        failed = False
    except TspError as e:
        failed = True
        assert e.code == (TSP_ECUDA if kind == "launch" else TSP_ENOMEM)
    monkeypatch.delenv("TSP_SIM_FAULT")
    if failed:
        for p in _passes(r):
            with pytest.raises(TspError) as ei:
                p()
            assert ei.value.code == TSP_ESTATE
    else:
        assert kind == "oom"        # every buffer was large enough
    # the same call again prepares the list
    getattr(r, call)(*args)
    r.set_image()
    r.iterate(2)
    img = r.read_image().cpu().numpy().astype(np.float64)
    r.close()
    f = Recon.from_workload(w)
    getattr(f, call)(*args)
    f.upload_events(*ev)
    f.iterate(2)
    ref = f.read_image().cpu().numpy().astype(np.float64)
    f.close()
    assert np.abs(img - ref).max() <= 1e-5 * ref.max()


def test_failed_batch_schedule(dense, monkeypatch):
    from paper_1502_07478_gb300 import Batch, TspError
    from paper_1502_07478_gb300._lib import TSP_ECUDA, TSP_ESTATE
    w, ev = dense
    b = Batch.from_workloads([w, w])
    for i in range(2):
        b.upload_events(i, *ev)
    b.iterate(1)
    monkeypatch.setenv("TSP_SIM_FAULT", "launch")
    with pytest.raises(TspError) as ei:
        b.set_schedule(ty_cap=16)
    assert ei.value.code == TSP_ECUDA
    monkeypatch.delenv("TSP_SIM_FAULT")
    with pytest.raises(TspError) as ei:
        b.iterate(1)
    assert ei.value.code == TSP_ESTATE
    b.set_schedule(ty_cap=16)
    for i in range(2):
        b.set_image(i)
    b.iterate(2)
    a = [b.read_image(i).cpu().numpy().astype(np.float64) for i in range(2)]
    st = b.stats(0)
    b.close()
    assert st["sum_s_rho"] == pytest.approx(st["n_used"], rel=2e-6)
    assert np.abs(a[0] - a[1]).max() <= 1e-5 * a[0].max()
