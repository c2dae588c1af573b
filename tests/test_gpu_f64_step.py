"""The bound stated for the FP64 collision in integers, one step against long
double with the rates the device holds (FP64 numbers)."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2208_14870_gb300 import Lattice  # noqa: E402


# In units of 2^-58 of the power of two E above the node's largest value: every
# input is cut by less than 1, a product (factors below 1/4) is off by less than 2.5.
# Standard rates: S 12/4 + 2.5, D 4/4 + 2.5, U 2 + 4 + 1, T U/12 + 2.5, so populations 1-4
# S + D + (U + 1 + 4 T)/2 < 20, 5-8 less.  General rates add (4/4 + 2.5) to T and twice (4/4
# + 2.5) through m_22: < 34.  Then the result's own rounding, 2^-53 of it.
@pytest.mark.parametrize("nx,ny", [(37, 11), (260, 250)])          # k_tile64 or k_one64, as the lattice has it
@pytest.mark.parametrize("spread", [0, 40])
@pytest.mark.parametrize("kw,units", [(dict(), 20), (dict(tau12=0.9, tau22=0.3), 34)])
def test_one_step_within_the_stated_bound(nx, ny, spread, kw, units):
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("needs a long double of 64 bits or more")
    lam, mu = W.lame_2d(1.0, 0.3)
    rng = np.random.RandomState(nx + spread)
    f = rng.standard_normal((8, ny, nx)) * 2.0 ** rng.randint(-spread, 1, (8, ny, nx))
    g = rng.standard_normal((2, ny, nx)) * 2.0 ** rng.randint(-spread, 1, (2, ny, nx))
    with Lattice(nx, ny, lam, mu, "f64", **kw) as lat:
        lat.set_force(g[0], g[1])
        lat.set_populations(f)
        lat.iterate(1)
        got = lat.populations().astype(np.longdouble)
        r = lat.rates
    L = np.longdouble
    q11, qs, qd, q12, q22 = (L(0.25 * (1.0 - r[k])) for k in ("w11", "ws", "wd", "w12", "w22"))
    qt = L(0.25 * (r["w12"] * r["theta"]))
    f, g = f.astype(L), g.astype(L)
    p, q, d, s = f[4] + f[6], f[5] + f[7], f[4] - f[6], f[5] - f[7]
    u, v = f[0] - f[2] + (d - s) + g[0] / 2, f[1] - f[3] + (d + s) + g[1] / 2
    s13, s24 = f[0] + f[2], f[1] + f[3]
    m11, m22 = q11 * (p - q), q22 * (p + q)
    ms, md = qs * (s13 + s24 + 2 * (p + q)), qd * (s13 - s24)
    m12, m21 = qt * u + q12 * (d - s), qt * v + q12 * (d + s)
    A, B = (u + g[0] / 2 - 4 * m12) / 2, (v + g[1] / 2 - 4 * m21) / 2
    P, Q = ms + md - 2 * m22, ms - md - 2 * m22
    o = [P + A, Q + B, P - A, Q - B, m22 + m11 + m12 + m21, m22 - m11 + m21 - m12, m22 + m11 - m12 - m21,
         m22 - m11 - m21 + m12]
    top = np.maximum(abs(f).max(axis=0), abs(g).max(axis=0)).astype(np.float64)
    E = np.ldexp(1.0, np.frexp(top)[1]).astype(L)
    worst = 0.0
    for k, (cx, cy) in enumerate([(1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]):
        want, e = np.roll(o[k], (cy, cx), (0, 1)), np.roll(E, (cy, cx), (0, 1))
        off = np.maximum(abs(got[k] - want) - L(2.0) ** -53 * abs(want), 0) / (e * L(2.0) ** -58)
        worst = max(worst, float(off.max()))
    print("%d x %d spread %d: %.2f units of %d" % (nx, ny, spread, worst, units))
    assert worst <= units
