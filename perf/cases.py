"""The work whose speed this library is judged by: single lattices of every
storage type from the smallest to the largest, a batch, and a served stream,
each through the calls a user's program makes.

A case fixes the sizes, materials and step counts; the seed draws the body
force (plane waves, as in the throughput, batched and served workloads).  All
forces are sums of a few plane waves, so the state after n steps of the
linear scheme has a closed form per wave, which `exact` evaluates.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2208_14870_gb300 as lbm

DEV = "cuda"


# Young's modulus, Poisson's ratio, the fourth-order relaxation times and the
# force correction -(D1, D2, D3) that belongs to them.
ORDER4 = (
    dict(E=0.2, nu=0.5, tau12=0.725, tau22=0.045977011494253386,
         d1=0.16458333333333333, d2=-0.0020833333333333333, d3=0.021666666666666667),
    dict(E=0.11, nu=0.8, tau12=1.4094696969696967, tau22=0.4389597010532247,
         d1=0.0583941, d2=-0.10827257, d3=0.03746528),
)


def listed():
    return [
        # The plain method: a 64 x 64 lattice in double precision, solved to
        # a residual of 1e-10 (the first thing a new user runs).
        dict(name="f64_64_solve", kind="solve", nx=64, ny=64, nu=0.3),
        # Double precision where accuracy matters (convergence studies).
        dict(name="f64_1500x1100", kind="grid", dtype="f64", nx=1500, ny=1100, nu=0.3, steps=100),
        # A small single-precision problem: the low end of the served sizes.
        dict(name="f32_100x75", kind="grid", dtype="f32", nx=100, ny=75, nu=0.2, steps=400),
        # An ordinary problem of odd sides.
        dict(name="f32_333x517", kind="grid", dtype="f32", nx=333, ny=517, nu=0.45, steps=400),
        # A square of the convergence sweep; its state fits the L2 cache.
        dict(name="f32_1024", kind="grid", dtype="f32", nx=1024, ny=1024, nu=0.0, steps=400),
        # The upper end of the served sizes.
        dict(name="f32_4096x3000", kind="grid", dtype="f32", nx=4096, ny=3000, nu=0.4, steps=200),
        # The single-large-lattice throughput workload.
        dict(name="f32_16384", kind="grid", dtype="f32", nx=16384, ny=16384, nu=0.3, steps=100),
        # FP16-shifted storage: an ordinary size, and a large lattice.
        dict(name="f16s_1000x700", kind="grid", dtype="f16s", nx=1000, ny=700, nu=0.3, steps=400),
        dict(name="f16s_8192", kind="grid", dtype="f16s", nx=8192, ny=8192, nu=0.3, steps=100),
        # The fourth-order special case (general relaxation times, corrected
        # force) on host arrays: force in, displacement and stress out.
        dict(name="f32_order4_host_512x384", kind="host", dtype="f32", nx=512, ny=384, **ORDER4[0], steps=400),
        # A batch of uneven problems in one call.
        dict(name="batch_48", kind="batch", count=48, lo=32, hi=1024, layout=1, steps=600),
        # Requests of both storage types to a running server.
        dict(name="served_12", kind="served", count=12, lo=64, hi=1500, layout=2, steps=400),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "f64", "f32", "f32", "f32", "f16s", "f16s", "host", "batch", "served"])
    nu = round(rng.uniform(0.0, 0.45), 3)
    if kind == "solve":
        return dict(kind="solve", nx=rng.randint(40, 96), ny=rng.randint(40, 96), nu=nu)
    if kind == "f64":
        return dict(kind="grid", dtype="f64", nx=_log_int(rng, 32, 1500), ny=_log_int(rng, 32, 1500), nu=nu,
                    steps=rng.randint(60, 200))
    if kind in ("f32", "f16s"):
        nx, ny = _log_int(rng, 32, 8192), _log_int(rng, 32, 8192)
        return dict(kind="grid", dtype=kind, nx=nx, ny=ny, nu=nu,
                    steps=rng.randint(100, 500) if nx * ny < 1 << 22 else rng.randint(60, 150))
    if kind == "host":
        return dict(kind="host", dtype=rng.choice(["f32", "f64"]), nx=_log_int(rng, 48, 1024),
                    ny=_log_int(rng, 48, 1024), **rng.choice(ORDER4), steps=rng.randint(100, 400))
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(8, 48), lo=32, hi=rng.choice([256, 512, 1024]),
                    layout=rng.randint(10, 1 << 30), steps=100 * rng.randint(3, 6))
    return dict(kind="served", count=rng.randint(3, 12), lo=64, hi=rng.choice([400, 1000, 1500]),
                layout=rng.randint(10, 1 << 30), steps=100 * rng.randint(2, 4))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

CHECK = 100          # steps between residual checks


def _lame(E, nu):
    return E * nu / (1.0 - nu * nu), E / (2.0 * (1.0 + nu))


def _problems(case):
    """[(nx, ny, nu, dtype)] of a batch or a served stream."""
    r = np.random.RandomState(case["layout"])
    out = []
    for i in range(case["count"]):
        nx, ny = (int(round(v)) for v in np.exp(r.uniform(math.log(case["lo"]), math.log(case["hi"]), 2)))
        dtype = "f16s" if case["kind"] == "served" and i % 2 else "f32"
        out.append((nx, ny, float(r.uniform(0.0, 0.45)), dtype))
    return out


def _waves(nx, ny, seed, smooth):
    """Plane waves of a body force: integer wave numbers, complex amplitudes
    of g_x and g_y.  smooth: the product field of the plain method (one wave
    per direction); else random waves with amplitudes ~ 1 / |k|^2, the
    fundamental ones among them."""
    r = np.random.RandomState(seed % (1 << 32))
    if smooth:
        k = [(1, 1), (1, -1)]
    else:
        k = [(1, 0), (0, 1)]
        while len(k) < 8:
            a, b = int(r.randint(-4, 5)), int(r.randint(-4, 5))
            if (a, b) != (0, 0):
                k.append((a, b))
    k = np.array(k)
    amp = r.standard_normal((2, len(k))) * np.exp(2j * math.pi * r.uniform(size=(2, len(k))))
    return k, amp / (k ** 2).sum(axis=1) / max(nx, ny) ** 2


def _grid(nx, ny, k, amp):
    """Re sum_m amp[..., m] exp(i k_m . x) on the nodes x = n + 1/2 (FP64)."""
    x = 2 * math.pi / nx * (torch.arange(nx, dtype=torch.float64, device=DEV) + 0.5)
    y = 2 * math.pi / ny * (torch.arange(ny, dtype=torch.float64, device=DEV) + 0.5)
    kx = torch.tensor(k[:, 0], dtype=torch.float64, device=DEV)
    ky = torch.tensor(k[:, 1], dtype=torch.float64, device=DEV)
    ex = torch.exp(1j * kx[:, None] * x[None, :])
    ey = torch.exp(1j * ky[None, :] * y[:, None])
    a = torch.tensor(np.atleast_2d(amp), dtype=torch.complex128, device=DEV)
    right = torch.cat([ex.real, ex.imag])
    out = torch.empty((a.shape[0], ny, nx), dtype=torch.float64, device=DEV)
    for f in range(a.shape[0]):
        e = a[f][None, :] * ey
        torch.matmul(torch.cat([e.real, -e.imag], dim=1), right, out=out[f])
    return out


def _wave_seed(case, seed, i=0):
    return (seed * 1000003 + i * 7919 + 12345) & 0x7FFFFFFF


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("batch", "served"):
        probs = []
        for i, (nx, ny, nu, dtype) in enumerate(_problems(case)):
            g = _grid(nx, ny, *_waves(nx, ny, _wave_seed(case, seed, i), False)).cpu().numpy()
            probs.append((nx, ny, *_lame(1.0, nu), g[0], g[1], dtype))
        st = dict(case=case, probs=probs)
        if kind == "served":
            st["server"] = lbm.Server(2_000_000_000, check_every=CHECK)
        return st
    nx, ny = case["nx"], case["ny"]
    lam, mu = _lame(case.get("E", 1.0), case["nu"])
    lat = lbm.Lattice(nx, ny, lam, mu, case.get("dtype", "f64"), 0.0, case.get("tau12", 0.0),
                      case.get("tau22", 0.0))
    lat.set_stream(torch.cuda.current_stream().cuda_stream)
    g = _grid(nx, ny, *_waves(nx, ny, _wave_seed(case, seed), kind == "solve"))
    if kind == "host":
        g = g.cpu().numpy()
        return dict(case=case, lat=lat, g=g, d=[case["d1"], case["d2"], case["d3"]])
    lat.set_force(g[0], g[1])
    return dict(case=case, lat=lat, out=torch.empty((5, ny, nx), dtype=torch.float64, device=DEV))


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        res, _ = lbm.batch_solve([p[:6] for p in state["probs"]], "f32", 1e-8, CHECK, case["steps"])
        return dict(fields=[r["fields"] for r in res], iters=np.array([r["iters"] for r in res]),
                    status=np.array([r["status"] for r in res]))
    if kind == "served":
        srv = state["server"]
        tickets = [srv.submit(*p, tol=1e-8, max_iters=case["steps"]) for p in state["probs"]]
        res = [srv.wait(t) for t in tickets]
        return dict(fields=[r["fields"] for r in res], iters=np.array([r["iters"] for r in res]),
                    status=np.array([r["status"] for r in res]))
    lat = state["lat"]
    if kind == "host":
        lat.set_force_corrected(state["g"][0], state["g"][1], state["d"])
        lat.reset()
        residual = lat.iterate_checked(case["steps"], CHECK)
        return dict(displacement=lat.displacement(), stress=lat.stress(), residual=residual)
    lat.reset()
    if kind == "solve":
        status, iters, _ = lat.solve(1e-10, 1_000_000, CHECK)
        return dict(fields=lat.fields_device(state["out"]), iters=iters, status=status)
    residual = lat.iterate_checked(case["steps"], CHECK)
    return dict(fields=lat.fields_device(state["out"]), residual=residual)


def _solve_steps(nu, n):
    """A rough count of the steps of a solve, for `work` (the smooth field
    decays at (mu + K) k^2 per step at least at mu k^2)."""
    return 100 * (1 + int(23.0 / (max(100 * 0.35 * 8 * (math.pi / n) ** 2, 1e-9))))


def work(case):
    """Bytes: the force read once, the populations of the final state and the
    five FP64 fields written once.  Flops: 51 per node and step (28 additions,
    5 products, 9 fused multiply-adds)."""
    if case["kind"] in ("batch", "served"):
        lat = [(nx * ny, d, 16) for nx, ny, _, d in _problems(case)]
    else:
        dtype = case.get("dtype", "f64")
        lat = [(case["nx"] * case["ny"], dtype, 16 if dtype == "f64" or case["kind"] == "host" else 8)]
    pop = {"f64": 64, "f32": 32, "f16s": 24}
    steps = case["steps"] if "steps" in case else _solve_steps(case["nu"], max(case["nx"], case["ny"]))
    return dict(bytes=sum(n * (force + pop[d] + 40) for n, d, force in lat),
                flops=sum(51 * n * steps for n, _, _ in lat))


# ---------------------------------------------------------------------------
# The same results in 64 bits, per plane wave
# ---------------------------------------------------------------------------

C = np.array([(1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)])


class _Waves:
    """The scheme on one set of plane waves: amplitudes of the eight
    populations per wave, advanced step by step from zero."""

    def __init__(self, nx, ny, k, amp, lam, mu, tau12=0.5, tau22=0.5, d=None):
        theta, K = 1.0 / 3.0, lam + mu
        w11, ws, wd = (1.0 / (t + 0.5) for t in (mu / theta, 2 * K / (1 + theta), 2 * mu / (1 - theta)))
        w12, w22 = 1.0 / (tau12 + 0.5), 1.0 / (tau22 + 0.5)
        cx, cy = C[:, 0], C[:, 1]
        xx, yy = cx * cx, cy * cy
        M = np.array([cx, cy, cx * cy, xx + yy, xx - yy, cx * yy, xx * cy, xx * yy], dtype=float)
        self.k = 2 * math.pi * k / np.array([nx, ny])
        gx, gy = amp
        if d is not None:
            kx, ky = self.k.T
            dxx, dyy, dxy = 2 * np.cos(kx) - 2, 2 * np.cos(ky) - 2, -np.sin(kx) * np.sin(ky)
            gx, gy = (gx - (d[0] * dxx * gx + d[1] * dxy * gy + d[2] * dyy * gx),
                      gy - (d[2] * dxx * gy + d[1] * dxy * gx + d[0] * dyy * gy))
        R = np.diag([1, 1, 1 - w11, 1 - ws, 1 - wd, 1 - w12, 1 - w12, 1 - w22])
        R[5, 0] = R[6, 1] = w12 * theta
        half = np.zeros((8, 2))
        half[0, 0] = half[1, 1] = 1.0
        half[5, 0] = half[6, 1] = 0.5 * w12 * theta
        self.M, self.g = M, np.stack([gx, gy], axis=1)
        Mi = np.linalg.inv(M)
        S = np.exp(-1j * self.k @ C.T)                     # shift of population i by c_i
        self.A = S[:, :, None] * (Mi @ R @ M)[None]
        self.b = S * (self.g @ (Mi @ half).T)
        self.bare = (1 - w11 / 2, 1 - ws / 2, 1 - wd / 2)
        self.f = np.zeros((len(k), 8), dtype=complex)

    def advance(self, n):
        for _ in range(n):
            self.f = np.einsum("mij,mj->mi", self.A, self.f) + self.b

    def fields(self):
        m = self.f @ self.M.T
        b11, bs, bd = (c * m[:, i] for c, i in zip(self.bare, (2, 3, 4)))
        return np.stack([m[:, 0] + 0.5 * self.g[:, 0], m[:, 1] + 0.5 * self.g[:, 1],
                         -0.5 * (bs + bd), -0.5 * (bs - bd), -b11])


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "served"):
        fields = []
        for i, (nx, ny, nu, _) in enumerate(_problems(case)):
            k, amp = _waves(nx, ny, _wave_seed(case, seed, i), False)
            w = _Waves(nx, ny, k, amp, *_lame(1.0, nu))
            w.advance(case["steps"])
            fields.append(_grid(nx, ny, k, w.fields()).cpu().numpy())
        return dict(fields=fields, iters=None, status=None)
    nx, ny = case["nx"], case["ny"]
    k, amp = _waves(nx, ny, _wave_seed(case, seed), kind == "solve")
    lam, mu = _lame(case.get("E", 1.0), case["nu"])
    if kind == "host":
        w = _Waves(nx, ny, k, amp, lam, mu, case["tau12"], case["tau22"], [case["d1"], case["d2"], case["d3"]])
        w.advance(case["steps"])
        f = _grid(nx, ny, k, w.fields()).cpu().numpy()
        return dict(displacement=f[:2], stress=f[2:], residual=None)
    w = _Waves(nx, ny, k, amp, lam, mu)
    if kind == "solve":
        # the check in the step from t to t + 1 measures u^t; the first one
        # only takes the snapshot
        last = None
        while True:
            w.advance(CHECK - 1)
            u = _grid(nx, ny, k, w.fields()[:2])
            w.advance(1)
            if last is not None and float((u - last).abs().max()) < 1e-10 * CHECK * float(u.abs().max()):
                return dict(fields=_grid(nx, ny, k, w.fields()), iters=None, status=None)
            last = u
    w.advance(case["steps"])
    return dict(fields=_grid(nx, ny, k, w.fields()), residual=None)
