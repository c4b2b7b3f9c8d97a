"""The upper bound of P over an event's window that the fixed-point scatter of the
passes over window records relies on (a sum cannot overflow when every event's
largest term is known), checked against the largest P over a fine raster of the
window, evaluated from the vectors o, a, b of Sec. 3 (derived a3, reading R3) with
the full C^-1, for random events up to and beyond the strips' ends, at both of the
paper's radii, with wide cuts and the cross term."""
import numpy as np
import pytest


def _p_max(R, sz, sdl, cut, gamma, ey, t):
    """Largest P over the window's ellipse (a raster finer than any grid)."""
    iz, il = 1.0 / sz ** 2, 1.0 / sdl ** 2
    sec = np.sqrt(1.0 + t * t)
    hy, hu = cut * sdl / 2.0 / sec, cut * sz / np.sqrt(2.0)
    Dy, u = np.meshgrid(np.linspace(-hy, hy, 161), np.linspace(-hu, hu, 161), indexing="ij")
    y = ey + Dy
    b = (u, u, -2.0 * Dy * sec)
    a = (-(y - R) * sec ** 2, -(y + R) * sec ** 2, -2.0 * y * sec * t)
    o = (-(y - R) * t * sec ** 2, -(y + R) * t * sec ** 2, -y * sec * (1.0 + 2.0 * t * t))

    def dot(p, q):
        return iz * (p[0] * q[0] + p[1] * q[1]) + il * p[2] * q[2] + \
            gamma * (p[2] * (q[0] - q[1]) + q[2] * (p[0] - p[1]))

    bcb, acb, Q = dot(b, b), dot(a, b), dot(a, a) + 2.0 * dot(o, b)
    ok = (bcb <= cut ** 2) & (Q > 0)
    K = np.sqrt(iz * (iz * il - 2.0 * gamma ** 2)) / (2.0 * np.pi ** 2)
    Q = np.where(ok, Q, 1.0)
    return np.where(ok, K / np.sqrt(Q) * np.exp(-0.5 * (bcb - acb ** 2 / Q)), 0.0).max()


def _bound(R, sz, sdl, cut, gamma, ey, t):
    """The upload step's bound, restated in double precision (pixels of size 0)."""
    iz, il, c2i, t = 1.0 / sz ** 2, 1.0 / sdl ** 2, 1.0 + t * t, abs(t)
    hy, umax = cut * sdl / 2.0 / np.sqrt(c2i) * 1.001, cut / np.sqrt(2.0 * iz)
    ymax = abs(ey) + hy
    gam = 8.0 * abs(gamma) * R * t * c2i * np.sqrt(c2i)
    lead = 2.0 * iz * R * R * c2i * c2i
    l1 = 4.0 * il * ymax * (2.0 * t * t + 1.0) * hy * c2i + gam * hy
    l2 = 4.0 * iz * ymax * t * c2i * umax
    m = np.hypot(l1, l2)
    q = lead - gam * ymax - m
    K = np.sqrt(iz * (iz * il - 2.0 * gamma ** 2)) / (2.0 * np.pi ** 2)
    return 1.001 * K / np.sqrt(q) * np.exp(0.5 * cut ** 2 * m / q) if q > 1e-3 * lead else np.inf


@pytest.mark.parametrize("R,tmax", [(350.0, 0.9), (130.0, 1.4)])
@pytest.mark.parametrize("cut", [3.0, 5.0])
@pytest.mark.parametrize("gamma", [0.0, 5e-4])
def test_p_bound_above_window_maximum(R, tmax, cut, gamma):
    rng = np.random.default_rng(11)
    finite = 0
    for _ in range(150):
        args = (R, rng.uniform(8, 12), rng.uniform(30, 50), cut, gamma,
                rng.uniform(-1.1, 1.1) * R, rng.uniform(-tmax, tmax))
        pmax, bound = _p_max(*args), _bound(*args)
        assert bound >= pmax, args
        finite += np.isfinite(bound)
    assert finite >= (150 if R > 200 and cut < 4 and gamma == 0.0 else 1)
