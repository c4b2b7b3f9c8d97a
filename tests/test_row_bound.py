"""The bound of P along a window's row that the fixed-point scatter of the passes over
window records relies on (the very function that the upload compiles for the GPU), against the
largest P of a fine raster of the row, from the vectors o, a, b of Sec. 3 (derived a3,
reading R3) with the full C^-1: random events up to and beyond the strips' ends, at both
of the paper's radii, with wide cuts, the cross term, a z-dependent sigma_z and
another unit of length."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def bound(tmp_path_factory):
    d = tmp_path_factory.mktemp("rowbound")
    (d / "t.cpp").write_text(
        '#include "tsp_row_bound.h"\n'
        'extern "C" float row_bound(float a, float b, float c, float d, float e, float f, float g, '
        "float h, float i) { return tsp::row_p_bound(a, b, c, d, e, f, g, h, i); }\n")
    so = str(d / "t.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_1502_07478_gb300", "csrc"), str(d / "t.cpp"), "-o",
                    so], check=True)
    f = C.CDLL(so).row_bound
    f.restype, f.argtypes = C.c_float, [C.c_float] * 9
    return f


def _row(R, sz, sdl, gamma, yt, t, y, u):
    """(Q, P) along the row: u from the chord's centre."""
    iz, il = 1.0 / sz ** 2, 1.0 / sdl ** 2
    sec, Dy = np.sqrt(1.0 + t * t), y - yt
    b = (u, u, -2.0 * Dy * sec)
    a = (-(y - R) * sec ** 2, -(y + R) * sec ** 2, -2.0 * y * sec * t)
    o = (-(y - R) * t * sec ** 2, -(y + R) * t * sec ** 2, -y * sec * (1.0 + 2.0 * t * t))

    def dot(p, q):
        return iz * (p[0] * q[0] + p[1] * q[1]) + il * p[2] * q[2] + \
            gamma * (p[2] * (q[0] - q[1]) + q[2] * (p[0] - p[1]))

    bcb, acb, Q = dot(b, b), dot(a, b), dot(a, a) + 2.0 * dot(o, b)
    K = np.sqrt(iz * (iz * il - 2.0 * gamma ** 2)) / (2.0 * np.pi ** 2)
    with np.errstate(all="ignore"):
        P = np.where(Q > 0, K / np.sqrt(np.abs(Q)) * np.exp(-0.5 * (bcb - acb ** 2 / Q)), 0.0)
    return Q, acb, P


@pytest.mark.parametrize("R,tmax", [(350.0, 0.9), (130.0, 1.4)])
@pytest.mark.parametrize("cut", [3.0, 5.0])
@pytest.mark.parametrize("gamma", [0.0, 5e-4])
@pytest.mark.parametrize("unit", [1.0, 1024.0])
def test_row_bound_above_the_rows_maximum(bound, R, tmax, cut, gamma, unit):
    rng = np.random.default_rng(7)
    slack, infinite = [], 0
    for _ in range(600):
        f = 1.0 + rng.uniform(0.0, 0.2)              # an event's own sigma_z
        sz, sdl = rng.uniform(8, 12) * f / unit, rng.uniform(30, 50) / unit
        r, gm = R / unit, gamma * unit ** 2
        yt, t = rng.uniform(-1.1, 1.1) * r, rng.uniform(-tmax, tmax)
        hy = 0.5 * cut * sdl / np.sqrt(1.0 + t * t)
        Dy = rng.uniform(-1, 1) * hy
        hu = cut * sz / np.sqrt(2.0) * np.sqrt(1.0 - (Dy / hy) ** 2)
        lo, hi = np.sort(rng.uniform(-hu, hu, 2)) if rng.random() < 0.3 else (-hu, hu)
        y = yt + Dy
        Q, acb, P = _row(r, sz, sdl, gm, yt, t, y, np.linspace(lo, hi, 801))
        # the row's constants as the upload has them, from the row's two ends
        Q2, A2, _ = _row(r, sz, sdl, gm, yt, t, y, np.array([0.0, 1.0]))
        iz, il = 1.0 / sz ** 2, 1.0 / sdl ** 2
        K = np.sqrt(iz * (iz * il - 2.0 * gm ** 2)) / (2.0 * np.pi ** 2)
        shift = np.floor(np.log2(K) - 0.5 * np.log2(2 * iz * r * r) + 12.5)
        b0 = 4.0 * il * Dy * Dy * (1.0 + t * t)
        v = bound(Q2[0], Q2[1] - Q2[0], A2[1] - A2[0], A2[0], lo, hi,
                  np.log2(K) - shift - 0.5 * np.log2(np.e) * b0, iz, 0.5 * np.log2(np.e))
        if Q.min() <= 0.0:
            assert np.isinf(v) or Q.min() > -1e-5 * Q.max()
            infinite += 1
            continue
        pmax = P.max() * 2.0 ** -shift
        assert v >= pmax, (yt, t, Dy, lo, hi)
        if Q.min() > 0.2 * Q.max():
            slack.append(v / pmax)
    assert infinite <= 60
    # close to the row's maximum where Q does not fall to a fifth along the row
    assert np.median(slack) <= 1.3 and len(slack) >= 500, (np.median(slack), len(slack))
