"""Limits of the window records: the shared memory of their passes and the device
memory that they take."""
from dataclasses import replace

import numpy as np
import pytest

import oracle
from oracle import Setup
from synth import make_workload

pytestmark = pytest.mark.gpu


def test_accumulator_tiles_at_the_shared_memory_limit():
    """2.1 x 0.35 mm pixels: regions whose accumulator alone fits a block, but not
    beside what the passes over window records stage (238 KB of 230)."""
    from paper_1502_07478_gb300 import Recon
    w = replace(make_workload("small_5mm"), ny=333, nz=1429, sigma_dl=170.0, n_events=4000)
    ev = w.events()
    r = Recon.from_workload(w)
    r.upload_events(*ev)
    r.iterate(1)
    img = r.read_image().cpu().numpy().astype(np.float64)
    st = r.stats()
    r.close()
    assert st["n_window"] >= 64 * w.ny * w.nz       # dense enough for records
    ref, rs = oracle.mlem(Setup.from_workload(w), ev, 1)
    m = ref > 0.01 * ref.max()
    assert st["n_used"] == rs.n_used
    assert np.max(np.abs(img[m] - ref[m]) / ref[m]) <= 1e-4


def _free():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_record_memory_is_given_back():
    """2e5 dense events at 2 mm hold some 120 MB of records; a sparse list after them none."""
    from paper_1502_07478_gb300 import Recon
    w = replace(make_workload("small_5mm"), ny=350, nz=250, n_events=200_000)
    ev = w.events()
    few = [x[:1000] for x in ev]
    r = Recon.from_workload(w)
    r.begin_events(200_000)             # (event buffers of the long list, no records)
    r.append_events(*few)
    r.end_events()
    base = _free()
    r.upload_events(*ev)
    held = base - _free()
    assert held >= 100 << 20
    r.upload_events(*few)
    assert base - _free() <= 8 << 20
    r.upload_events(*ev)
    r.iterate(1)
    st = r.stats()
    assert st["sum_s_rho"] == pytest.approx(st["n_used"], rel=2e-6)
    r.close()


def test_a_list_without_room_for_records_is_prepared_once(monkeypatch):
    """A list long enough for wide tiles: refused after the preparation it is prepared
    again for the general passes (two launches more); when the memory report says so
    beforehand it is tiled for them at once."""
    from paper_1502_07478_gb300 import Recon
    w = make_workload("small_5mm", n_events=800_000)
    ev = w.events()
    launches, images = {}, {}
    for fault in ("", "records", "norecords"):
        monkeypatch.setenv("TSP_SIM_FAULT", fault)
        r = Recon.from_workload(w)
        r.upload_events(*ev)
        launches[fault] = r.stats()["launches"]
        r.iterate(1)
        images[fault] = r.read_image().cpu().numpy().astype(np.float64)
        r.close()
    assert launches["norecords"] == launches[""] - 1       # no launch of the records' kernel
    assert launches["records"] == launches["norecords"] + 2
    for f in ("records", "norecords"):
        assert np.abs(images[f] - images[""]).max() <= 2e-5 * images[""].max()


def test_first_upload_does_not_wait_for_other_streams():
    """A fresh context has nothing that its first preparation could disturb: work of
    another stream (a bounded spin of some 0.3 s) is still running when it returns."""
    import torch
    from paper_1502_07478_gb300 import Recon
    w = make_workload("small_5mm", n_events=20_000)
    ev = [torch.from_numpy(x).cuda() for x in w.events()]
    for _ in range(2):                      # (the first time loads the kernels)
        r = Recon.from_workload(w)
        side, mine = torch.cuda.Stream(), torch.cuda.Stream()
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            torch.cuda._sleep(600_000_000)
            done = torch.cuda.Event()
            done.record()
        r.upload_events(*ev, stream=mine)
        running = not done.query()
        torch.cuda.synchronize()
        r.close()
    assert running
