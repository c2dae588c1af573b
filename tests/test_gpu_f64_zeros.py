"""FP64 lattices that are zero but for a part (a localised force and its first
steps): nodes of zeros stay zero at no more than the cost of others."""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2208_14870_gb300 import Lattice  # noqa: E402


# Against the FP64 oracle (a hundred roundings of the largest population), at a
# subnormal force's scale too, which no zero may be taken for.
@pytest.mark.parametrize("nx,ny", [(7, 5), (64, 64), (300, 200)])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -1060])
def test_one_node_forced(nx, ny, scale):
    lam, mu = W.lame_2d(1.0, 0.3)
    rates = oracle.relaxation_rates(lam, mu)
    g = np.zeros((2, ny, nx))
    g[:, ny // 2, nx // 3] = (1.0, -0.5)
    with Lattice(nx, ny, lam, mu, "f64") as lat:
        for steps in (1, 2, 4):
            lat.reset()
            lat.set_force(*(g * scale))
            lat.iterate(steps)
            got = lat.populations()
            want = oracle.run(oracle.zero_state(nx, ny), g[0], g[1], rates, steps)
            tol = 100 * 2.0 ** -53 if scale == 1.0 else 100 * 2.0 ** -14
            assert np.abs(got / scale - want).max() <= tol * np.abs(want).max(), steps
            assert (got[want == 0.0] == 0.0).all()
            f = lat.fields()
            reach = np.abs(want).sum(0) > 0.0
            assert (f[:, ~reach & (g[0] == 0.0)] == 0.0).all() and np.abs(f).max() > 0.0


def test_zeros_cost_no_more_than_others():
    nx, ny = 1500, 1100
    stream = torch.cuda.current_stream()
    ms = []
    for zeros in (False, True):
        g = np.random.RandomState(1).standard_normal((2, ny, nx))
        if zeros:
            g[:, :, np.arange(nx) % 32 != 0] = 0.0
        with Lattice(nx, ny, *W.lame_2d(1.0, 0.3), "f64") as lat:
            lat.set_stream(stream.cuda_stream)
            lat.set_force(*g)
            best = np.inf
            for _ in range(6):
                lat.reset()
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record(stream)
                lat.iterate(12)
                b.record(stream)
                b.synchronize()
                best = min(best, a.elapsed_time(b))
            ms.append(best)
    assert ms[1] < 1.5 * ms[0], ms     # (both paths in every warp: four times)
