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
