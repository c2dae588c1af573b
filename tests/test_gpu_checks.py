"""Residual checks of single lattices against states computed another way."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2208_14870_gb300 import Lattice  # noqa: E402


# Checked FP16S strips of a lattice larger than the L2 cache, every launch a
# checked one: the check reads the FP32 state after three of a launch's four steps, which
# an FP32 lattice reaches from the launch's input with the same bits (the scale
# is a power of two), so only the pairs' sums differ (2^-44).
@pytest.mark.parametrize("nx,ny", [(2048, 2048), (2051, 1500)])
def test_f16s_strip_residual_beyond_l2(nx, ny):
    lam, mu = W.lame_2d(1.0, 0.3)
    gx, gy = np.random.RandomState(nx).standard_normal((2, ny, nx)) / max(nx, ny) ** 2
    with Lattice(nx, ny, lam, mu, "f16s") as lat:
        lat.steps_per_launch, lat.wavefront = 4, -1
        lat.set_force(gx, gy)
        got = lat.iterate_checked(8, 4)
        lat.reset()
        lat.iterate(4)
        state = lat.populations()
    u = []
    with Lattice(nx, ny, lam, mu, "f32") as lat:
        lat.set_force(gx, gy)
        for f in (None, state):
            if f is not None:
                lat.set_populations(f)
            lat.iterate(3)
            u.append(lat.displacement())
    d = u[1] - u[0]
    want = [np.abs(d).max() / (4 * np.abs(u[1]).max()), np.sqrt((d ** 2).sum() / (u[1] ** 2).sum()) / 4,
            np.abs(u[1]).max(), np.sqrt((u[1] ** 2).sum())]
    assert np.allclose(got[:4], want, rtol=1e-12, atol=0.0) and got[4] == 0.0


# Norms whose squares sum to more than FP32 holds over a block, but not over a
# thread's nodes: a lattice scaled by a power of two has the same residuals and
# scaled norms.  A uniform force (u = 7.5 at the last check) and a little noise;
# 2^122 per node, at most 16 nodes a thread.
@pytest.mark.parametrize("nx,ny,plan", [(100, 75, None), (333, 100, None), (300, 40, (4, 8)), (257, 64, (4, 8))])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_norms_beyond_fp32_squares(nx, ny, plan, dtype):
    if dtype == "f64" and plan:
        pytest.skip("no schedules for FP64 storage")
    lam, mu = W.lame_2d(1.0, 0.3)
    g = np.random.RandomState(nx).standard_normal((2, ny, nx)) * 2.0 ** -10
    g[0] += 1.0
    got = []
    for e in (0, 58):
        with Lattice(nx, ny, lam, mu, dtype) as lat:
            if plan:
                lat.steps_per_launch, lat.wavefront = plan
            lat.set_force(*(g * 2.0 ** e))
            r = lat.iterate_checked(8, 4)
            got.append(np.concatenate([r[:2], r[2:4] * 2.0 ** -e, r[4:]]))
    assert np.isfinite(got[0]).all() and got[0][2] > 7.0
    assert np.allclose(got[1], got[0], rtol=1e-14, atol=0.0)
