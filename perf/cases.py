"""The work that users of this package have it do, as cases for timing and comparison.

A case is a dict of plain values; prepare() makes what a program has in hand before the call
(events on the GPU or in pinned host memory, a Recon or Batch with its upload done), run() makes
one pass through the public entry points, exact() says what it should have returned, in plain
torch at 64 bits.  Events are drawn on the GPU from seeded random ellipses over the detector of
the paper (two strips at y = +-R, |z| <= L/2), smeared by the stated resolutions; images start
uniform unless a case says otherwise.  Kinds:

  iterate  set the image, n MLEM updates, read the image
  shard    one event-sharded update: back-projection, then the update with it
  grad     log-likelihood with its gradients in image and resolution (LogLik, autograd)
  fit      two evaluations of a resolution fit, each at another sigma
  host     a whole reconstruction from host buffers: streamed upload, updates, log-likelihood,
           image back to the host
  batch    many reconstructions together: updates of all, then all log-likelihoods and gradients
"""
import math

import numpy as np
import torch

from paper_1502_07478_gb300 import Batch, LogLik, Recon


def _case(name, kind, ny, nz, events, iters=1, R=350.0, L=500.0, sz=10.0, sdl=42.0, cut=3.0,
          gamma=0.0, kappa=0.0, k=1, spots=False):
    return dict(name=name, kind=kind, ny=ny, nz=nz, events=events, iters=iters, R=R, L=L, sz=sz,
                sdl=sdl, cut=cut, gamma=gamma, kappa=kappa, k=k, spots=spots)


def listed():
    return [
        # a first look during an acquisition: the events of a moment, one update
        _case("preview_5mm", "iterate", 140, 100, 500),
        # a small study on a coarse grid, few updates
        _case("small_5mm", "iterate", 140, 100, 20_000, iters=5),
        # the paper's own table: its geometry at 4 mm, 1e7 events, one iteration
        _case("table_4mm", "iterate", 65, 75, 10_000_000, R=130.0, L=300.0, sdl=40.0),
        # odd grid, with the paper's set-aside variants: cross term and z-dependent resolution
        _case("variants_2mm", "iterate", 351, 247, 300_000, iters=3, gamma=5e-4, kappa=0.1),
        # a study at 1 mm with a moderate list, several updates
        _case("study_1mm", "iterate", 700, 500, 200_000, iters=5),
        # the paper-scale reconstruction, one of its updates
        _case("paper_1mm", "iterate", 700, 500, 10_000_000),
        # one rank's part of an event-sharded update at 1 mm
        _case("shard_1mm", "shard", 697, 503, 1_000_000),
        # value and gradients of the log-likelihood for an optimiser of one's own
        _case("adjoint_2mm", "grad", 350, 250, 1_000_000),
        # two steps of a resolution fit (5 sigma windows)
        _case("fit_2mm", "fit", 350, 250, 100_000, cut=5.0),
        # very fine pixels with hot spots
        _case("fine_05mm", "iterate", 1400, 1000, 2_000_000, spots=True),
        # list-mode data in host memory to an image in host memory
        _case("host_2mm", "host", 350, 250, 1_000_000, iters=3),
        # independent patients together, pixels of 1, 2 and 4 mm, 1e4 events and up
        _case("batch_mixed", "batch", 700, 500, 500_000, iters=2, k=12),
    ]


# Window pixels of one pass, over all updates, that no case goes beyond (paper_1mm's 4e10).
_MOST_PIXELS = 4.0e10


def _window(ny, nz, R, L, sz, sdl, cut):
    """Mean in-window pixels of an event: the cut ellipse's area (mean cosine 0.9)."""
    return math.pi * cut * cut * sz * sdl * 0.9 / math.sqrt(8.0) / ((2 * R / ny) * (L / nz))


def draw(rng):
    def lg(a, b):
        return math.exp(rng.uniform(math.log(a), math.log(b)))

    kind = rng.choice(["iterate"] * 6 + ["shard", "grad", "grad", "fit", "host", "batch"])
    small = kind == "iterate" and rng.random() < 0.2           # the paper's own geometry
    R, L = (130.0, 300.0) if small else (350.0, 500.0)
    pitch = lg(1.0, 5.0) if kind in ("grad", "fit", "host") or small else lg(0.5, 5.0)
    if kind in ("shard", "batch"):
        pitch = lg(1.0, 4.0)
    pitch_z = pitch * rng.choice([1.0, 1.0, rng.uniform(0.95, 1.2)])
    ny, nz = max(8, round(2 * R / pitch)), max(8, round(L / pitch_z))
    # (windows of at most 256 rows, what an event group of one block holds at the finest pixels)
    sz, sdl = rng.uniform(8.0, 12.0), min(rng.uniform(30.0, 50.0), 84.0 * pitch)
    cut = rng.choice([3.0, 4.0, 5.0]) if kind == "fit" and pitch > 1.9 else 3.0
    iters = {"iterate": rng.randint(1, 5), "host": rng.randint(1, 5), "batch": rng.randint(1, 3)}
    n_it = iters.get(kind, 1)
    k = rng.randint(2, 16) if kind == "batch" else 1
    lo, hi = {"iterate": (500, 1e7), "shard": (1e4, 4e6), "grad": (1e4, 2e6), "fit": (1e4, 5e5),
              "host": (1e4, 4e6), "batch": (2e4, 5e5)}[kind]
    # a gradient costs several updates' time per pixel
    per = {"grad": 4, "fit": 8, "batch": n_it + 4}.get(kind, n_it)
    w = _window(ny, nz, R, L, sz, sdl, cut) * per * k
    n = int(lg(lo, max(lo * 1.5, min(hi, 0.5 * _MOST_PIXELS / w))))
    variants = kind in ("iterate", "shard") and pitch > 0.6 and rng.random() < 0.25
    return _case("", kind, ny, nz, n, iters=n_it, R=R, L=L, sz=sz, sdl=sdl, cut=cut,
                 gamma=rng.uniform(0.0, 5e-4) if variants else 0.0,
                 kappa=rng.uniform(0.0, 0.2) if variants else 0.0, k=k,
                 spots=rng.random() < 0.3)


# ---------------------------------------------------------------------------- events

def _generator(seed, stream):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 1009 + stream)


def _events(R, L, sz, sdl, n, seed, spots=False, stream=0):
    """n events (zu, zd, dl), float32 CUDA tensors: emission points uniform in seeded ellipses
    (a wide background, inner regions, with `spots` small hot ones), angles uniform over those
    that can reach both strips, kept if both hits lie on the strips, then smeared."""
    rng = np.random.default_rng([int(seed), stream])
    ell = [(0.0, 0.0, 0.38 * L, 0.55 * R, 0.0, 1.0)]
    for _ in range(int(rng.integers(2, 6))):
        ell.append((rng.uniform(-0.2, 0.2) * L, rng.uniform(-0.35, 0.35) * R,
                    rng.uniform(0.04, 0.15) * L, rng.uniform(0.04, 0.2) * R,
                    rng.uniform(0.0, math.pi), rng.uniform(0.5, 2.0)))
    for _ in range(4 if spots else 0):
        r = rng.uniform(2.0, 5.0)
        ell.append((rng.uniform(-0.3, 0.3) * L, rng.uniform(-0.4, 0.4) * R, r, r, 0.0, 8.0))
    e = torch.tensor(ell, dtype=torch.float64, device="cuda")
    weight = e[:, 2] * e[:, 3] * e[:, 5]
    g = _generator(seed, stream)
    parts, have = [], 0
    theta_c = math.atan(0.5 * L / R)
    while have < n:
        m = int(2.2 * (n - have)) + 4096
        u = torch.rand(4, m, dtype=torch.float64, device="cuda", generator=g)
        i = torch.searchsorted(torch.cumsum(weight, 0) / weight.sum(), u[0]).clamp_(max=len(ell) - 1)
        rad, ang = u[1].sqrt(), 2 * math.pi * u[2]
        a, b = e[i, 2] * rad * torch.cos(ang), e[i, 3] * rad * torch.sin(ang)
        c, s = torch.cos(e[i, 4]), torch.sin(e[i, 4])
        z, y = e[i, 0] + a * c - b * s, e[i, 1] + a * s + b * c
        t = torch.tan((2 * u[3] - 1) * theta_c)
        zu, zd = z + (R - y) * t, z - (R + y) * t
        dl = -2 * y * torch.sqrt(1 + t * t)
        keep = (y.abs() < R) & (zu.abs() <= 0.5 * L) & (zd.abs() <= 0.5 * L)
        parts.append(torch.stack((zu, zd, dl))[:, keep])
        have += parts[-1].shape[1]
    ev = torch.cat(parts, 1)[:, :n]
    noise = torch.randn(3, n, dtype=torch.float64, device="cuda", generator=g)
    noise *= torch.tensor([[sz], [sz], [sdl]], dtype=torch.float64, device="cuda")
    return (ev + noise).float().contiguous()


def _image(ny, nz, seed, stream=0):
    """A smooth positive image, as an optimiser holds it between steps."""
    g = _generator(seed, 100 + stream)
    y = torch.linspace(-1, 1, ny, device="cuda")[:, None]
    z = torch.linspace(-1, 1, nz, device="cuda")[None, :]
    img = torch.full((ny, nz), 0.2, device="cuda")
    for _ in range(4):
        p = torch.rand(4, device="cuda", generator=g)
        img = img + (0.5 + p[3]) * torch.exp(-(((y - (p[0] - 0.5)) / 0.4) ** 2 +
                                               ((z - (p[1] - 0.5)) / (0.3 + 0.3 * p[2])) ** 2))
    return img.contiguous()


def _members(case):
    """Parameters and event counts of a batch: pixels of 1, 2 or 4 times the case's pitch, event
    counts log-uniform from 1e4 to the case's."""
    rng = np.random.default_rng([7, case["k"], case["ny"], case["events"]])
    out = []
    for i in range(case["k"]):
        f = (1, 2, 4)[int(rng.integers(0, 3))] if i else 1
        n = int(round(math.exp(rng.uniform(math.log(1e4), math.log(max(2e4, case["events"]))))))
        out.append((dict(R=case["R"], L=case["L"], ny=max(8, case["ny"] // f),
                         nz=max(8, case["nz"] // f), sigma_z=float(rng.uniform(8.0, 12.0)),
                         sigma_dl=float(rng.uniform(30.0, 50.0)), cut=case["cut"]), n))
    return out


# ---------------------------------------------------------------------------- the calls

def _recon(case):
    return Recon(case["R"], case["L"], case["ny"], case["nz"], case["sz"], case["sdl"],
                 cut=case["cut"], gamma=case["gamma"], kappa_z=case["kappa"])


def _sigmas(case):
    """The resolutions at which a gradient or a fit's first steps are evaluated: off the true ones."""
    return [(0.85 * case["sz"], 1.2 * case["sdl"]), (0.9 * case["sz"], 1.15 * case["sdl"])]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        members = _members(case)
        b = Batch([p for p, _ in members])
        for i, (p, n) in enumerate(members):
            b.upload_events(i, *_events(p["R"], p["L"], p["sigma_z"], p["sigma_dl"], n, seed,
                                        case["spots"], i))
        return dict(case=case, batch=b)
    ev = _events(case["R"], case["L"], case["sz"], case["sdl"], case["events"], seed, case["spots"])
    r = _recon(case)
    state = dict(case=case, recon=r)
    if kind == "host":
        # list-mode data as an acquisition leaves it: pinned host buffers, in a few chunks
        host = ev.cpu()
        step = -(-case["events"] // 4)
        state["chunks"] = [tuple(x[a:a + step].clone().pin_memory() for x in host)
                           for a in range(0, case["events"], step)]
        state["out"] = np.empty((case["ny"], case["nz"]), dtype=np.float32)
        return state
    r.upload_events(*ev)
    if kind in ("grad", "fit", "shard"):
        state["rho"] = _image(case["ny"], case["nz"], seed)
    if kind in ("grad", "fit"):
        state["sigma"] = [torch.tensor(s, dtype=torch.float32) for s in _sigmas(case)]
    if kind == "grad":
        r.set_sigma(*[float(x) for x in state["sigma"][0]])
    return state


def _value_and_grad(r, rho, sigma):
    """One evaluation of an optimiser's loop, its parameters in 32 bits."""
    rho, sigma = rho.detach().requires_grad_(), sigma.detach().requires_grad_()
    loss = -LogLik.apply(r, rho, sigma)
    loss.backward()
    return [loss.item(), rho.grad, sigma.grad]


def run(state):
    case, r = state["case"], state.get("recon")
    kind = case["kind"]
    if kind == "iterate":
        r.set_image()
        r.iterate(case["iters"])
        return r.read_image()
    if kind == "shard":
        r.set_image(state["rho"])
        A = r.backproject()
        r.apply_update(A)
        return [A, r.read_image()]
    if kind == "grad":
        return _value_and_grad(r, state["rho"], state["sigma"][0])
    if kind == "fit":
        return [_value_and_grad(r, state["rho"], s) for s in state["sigma"]]
    if kind == "host":
        r.begin_events(case["events"])
        for c in state["chunks"]:
            r.append_events(*c)
        r.end_events()
        r.iterate(case["iters"])
        L = r.loglik()
        return [L, r.read_image(out=state["out"])]
    b = state["batch"]
    for i in range(len(b)):
        b.set_image(i)
    b.iterate(case["iters"])
    images = [b.read_image(i) for i in range(len(b))]
    L, gs = b.loglik_grad()
    return [images, [b.read_image(i, which=2) for i in range(len(b))],
            L.astype(np.float32), gs.astype(np.float32)]


# A kernel evaluation: Q, aCb and the exponent along the row (4 multiply-adds), the quotient,
# square root and exponential (6), the denominator's and the scatter's multiply-add (4).  The
# gradient adds the two derivatives (14).  Each list of a pass is read once (12 bytes an event),
# images once per update (read, write, sensitivity).
_FLOPS, _FLOPS_GRAD = 18.0, 32.0


def work(case):
    kind = case["kind"]
    if kind == "batch":
        flops = nbytes = 0.0
        for p, n in _members(case):
            w = n * _window(p["ny"], p["nz"], p["R"], p["L"], p["sigma_z"], p["sigma_dl"], p["cut"])
            flops += w * (_FLOPS * case["iters"] + _FLOPS_GRAD)
            nbytes += (12.0 * n + 16.0 * p["ny"] * p["nz"]) * (case["iters"] + 1)
        return dict(bytes=nbytes, flops=flops)
    n, pix = case["events"], case["ny"] * case["nz"]
    w = n * _window(case["ny"], case["nz"], case["R"], case["L"], case["sz"], case["sdl"],
                    case["cut"])
    passes = {"iterate": case["iters"], "shard": 1, "grad": 1, "fit": 2,
              "host": case["iters"] + 0.5}[kind]
    per = _FLOPS_GRAD if kind in ("grad", "fit") else _FLOPS
    return dict(bytes=passes * (12.0 * n + 16.0 * pix), flops=w * per * passes)


# ---------------------------------------------------------------------------- in 64 bits

_EXACT_MOST = 2.0e10     # padded window pixels, over all passes, that take some 20 seconds


class _Exact:
    """The model in 64 bits: Eq. 2, the windows, the kernel, the sensitivity."""

    def __init__(self, R, L, ny, nz, sz, sdl, cut, ev, gamma=0.0, kappa=0.0):
        self.R, self.L, self.ny, self.nz, self.cut, self.gamma = R, L, ny, nz, cut, gamma
        self.dy, self.dz = 2.0 * R / ny, L / nz
        self.y0, self.z0 = -R + 0.5 * self.dy, -0.5 * L + 0.5 * self.dz
        zu, zd, dl = ev.double()
        self.t = (zu - zd) / (2 * R)
        self.c2 = 1 + self.t ** 2
        self.yt = -0.5 * dl / self.c2.sqrt()
        self.zt = 0.5 * (zu + zd + 2 * self.yt * self.t)
        self.f = 1 + kappa * torch.clamp((2 * self.zt / L) ** 2, max=1.0)
        self.sz, self.sdl = sz, sdl
        self.rows = int(cut * sdl / self.dy) + 3
        self.half = int(cut * sz * (1 + kappa) / math.sqrt(2) / self.dz) + 2
        y = self.y0 + self.dy * torch.arange(ny, dtype=torch.float64, device="cuda")[:, None]
        z = self.z0 + self.dz * torch.arange(nz, dtype=torch.float64, device="cuda")[None, :]
        h = 0.5 * L
        hi = torch.minimum((h - z) / (R - y), (h + z) / (R + y))
        lo = torch.maximum(-(h + z) / (R - y), (z - h) / (R + y))
        self.s = ((torch.atan(hi) - torch.atan(lo)) / math.pi).clamp_(min=0)

    def padded(self):
        return self.t.numel() * float(self.rows) * (2 * self.half + 1)

    def chunks(self):
        n = self.t.numel()
        step = max(1, int(4e7 / (self.rows * (2 * self.half + 1))))
        return [slice(a, min(n, a + step)) for a in range(0, n, step)]

    def window(self, c):
        """(flat pixel indices, inside, y, Dy, u) of a run of events: (events, rows, columns)."""
        t, yt, zt, f = (x[c][:, None] for x in (self.t, self.yt, self.zt, self.f))
        hy = 0.5 * self.cut * self.sdl / self.c2[c][:, None].sqrt()
        iy = torch.floor((yt - hy - self.y0) / self.dy) + torch.arange(self.rows, device="cuda")
        y = self.y0 + iy * self.dy
        Dy = y - yt
        mid = torch.round((zt + t * Dy - self.z0) / self.dz)
        iz = mid[..., None] + torch.arange(-self.half, self.half + 1, device="cuda")
        u = self.z0 + iz * self.dz - (zt + t * Dy)[..., None]
        b = 2 * u * u / (self.sz * f[..., None]) ** 2 + \
            (4 * Dy * Dy * self.c2[c][:, None] / self.sdl ** 2)[..., None]
        ok = (b <= self.cut ** 2) & (iz >= 0) & (iz < self.nz) & \
            ((iy >= 0) & (iy < self.ny))[..., None]
        idx = torch.where(ok, iy[..., None] * self.nz + iz, 0.0).long()
        return idx, ok, y[..., None], Dy[..., None], u

    def kernel(self, c, win, sz, sdl):
        """P over a window for the resolution (sz, sdl); 0 outside."""
        _, ok, y, Dy, u = win
        t, c2, f = (x[c][:, None, None] for x in (self.t, self.c2, self.f))
        iz, il, g, R = 1 / (sz * f) ** 2, 1 / sdl ** 2, self.gamma, self.R
        sec = c2.sqrt()
        Q = 2 * iz * (R * R + y * y) * c2 * c2 + 4 * il * y * y * t * t * c2 + \
            4 * il * y * (1 + 2 * t * t) * Dy * c2 - 8 * g * R * t * c2 * sec * (y + Dy) - \
            4 * iz * y * t * c2 * u
        acb = -2 * iz * y * c2 * u + 4 * il * y * t * Dy * c2 - 4 * g * R * c2 * sec * Dy
        bcb = 2 * iz * u * u + 4 * il * Dy * Dy * c2
        K = (iz * (iz * il - 2 * g * g)).sqrt() / (2 * math.pi ** 2)
        ok = ok & (Q > 0)
        Q = torch.where(ok, Q, 1.0)
        e = torch.where(ok, bcb - acb * acb / Q, 0.0)     # finite outside, for autograd
        return torch.where(ok, K * Q.rsqrt() * torch.exp(-0.5 * e), 0.0)

    def backproject(self, rho):
        """(A, sum log D) at the image rho."""
        w = (self.s * rho).reshape(-1)
        A = torch.zeros_like(w)
        logD = torch.zeros((), dtype=torch.float64, device="cuda")
        for c in self.chunks():
            win = self.window(c)
            P = self.kernel(c, win, self.sz, self.sdl)
            D = (P * w[win[0]]).sum((1, 2))
            pos = D > 0
            inv = torch.where(pos, 1 / D, 0.0)
            logD += torch.log(D[pos]).sum()
            A.index_add_(0, win[0].reshape(-1), (P * inv[:, None, None]).reshape(-1))
        return A.view(self.ny, self.nz), logD

    def iterate(self, rho, n):
        for _ in range(n):
            rho = rho * self.backproject(rho)[0]
        return rho

    def loglik(self, rho):
        return float(self.backproject(rho)[1] - (self.s * rho).sum())

    def value_and_grad(self, rho):
        """(L, dL/drho, dL/d(sz, sdl)), the windows fixed."""
        w = (self.s * rho).reshape(-1)
        A = torch.zeros_like(w)
        L = -float(w.sum())
        sig = torch.tensor([self.sz, self.sdl], dtype=torch.float64, device="cuda",
                           requires_grad=True)
        gs = torch.zeros(2, dtype=torch.float64, device="cuda")
        for c in self.chunks():
            with torch.no_grad():
                win = self.window(c)
            P = self.kernel(c, win, sig[0], sig[1])
            D = (P * w[win[0]]).sum((1, 2))
            logD = torch.log(torch.where(D > 0, D, 1.0)).sum()
            gs += torch.autograd.grad(logD, sig)[0]
            L += float(logD.detach())
            with torch.no_grad():
                inv = torch.where(D > 0, 1 / D, 0.0)
                A.index_add_(0, win[0].reshape(-1), (P * inv[:, None, None]).reshape(-1))
        return L, self.s * (A.view(self.ny, self.nz) - 1), gs


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        members = _members(case)
        models = [_Exact(p["R"], p["L"], p["ny"], p["nz"], p["sigma_z"], p["sigma_dl"], p["cut"],
                         _events(p["R"], p["L"], p["sigma_z"], p["sigma_dl"], n, seed,
                                 case["spots"], i)) for i, (p, n) in enumerate(members)]
        if sum(m.padded() for m in models) * (case["iters"] + 5) > _EXACT_MOST:
            return None
        images, grads, Ls, gss = [], [], [], []
        for m in models:
            rho = m.iterate(torch.ones(m.ny, m.nz, dtype=torch.float64, device="cuda"),
                            case["iters"])
            L, g, gs = m.value_and_grad(rho)
            images.append(rho)
            grads.append(g)
            Ls.append(L)
            gss.append(gs.cpu().numpy())
        return [images, grads, np.array(Ls), np.array(gss)]
    ev = _events(case["R"], case["L"], case["sz"], case["sdl"], case["events"], seed, case["spots"])

    def model(sz, sdl):
        return _Exact(case["R"], case["L"], case["ny"], case["nz"], sz, sdl, case["cut"], ev,
                      case["gamma"], case["kappa"])

    m = model(case["sz"], case["sdl"])
    passes = {"iterate": case["iters"], "shard": 1, "grad": 5, "fit": 10,
              "host": case["iters"] + 1}[kind]
    if m.padded() * passes > _EXACT_MOST:
        return None
    one = torch.ones(case["ny"], case["nz"], dtype=torch.float64, device="cuda")
    if kind == "iterate":
        return m.iterate(one, case["iters"])
    if kind == "host":
        rho = m.iterate(one, case["iters"])
        return [m.loglik(rho), rho.cpu().numpy()]
    rho = _image(case["ny"], case["nz"], seed).double()
    if kind == "shard":
        A = m.backproject(rho)[0]
        return [A, rho * A]
    found = []
    for s in _sigmas(case)[:1 if kind == "grad" else 2]:
        s = [float(x) for x in torch.tensor(s, dtype=torch.float32)]
        L, g, gs = model(*s).value_and_grad(rho)
        found.append([-L, -g, -gs.cpu()])
    return found[0] if kind == "grad" else found
