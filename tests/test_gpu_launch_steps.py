"""lbm_get_launch_steps: that many plain steps are one launch, and one step more is
not, for every storage type, schedule and plan."""
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2208_14870_gb300 as P  # noqa: E402
from paper_2208_14870_gb300 import Lattice  # noqa: E402


# default plans: register tiles, strips, FP64 tiles and single steps; set schedules
@pytest.mark.parametrize("nx,ny", [(5, 3), (63, 30), (64, 64), (100, 75), (300, 300), (1500, 1100), (63, 8000)])
@pytest.mark.parametrize("dtype,plan", [("f64", None), ("f32", None), ("f16s", None), ("f32", (4, -1)), ("f16s", (4, -1)),
                                        ("f32", (3, 0)), ("f16s", (3, 0)), ("f32", (1, 0)), ("f16s", (2, 0))])
def test_one_launch(nx, ny, dtype, plan):
    lam, mu = W.lame_2d(1.0, 0.3)
    with Lattice(nx, ny, lam, mu, dtype) as lat:
        if plan:
            lat.steps_per_launch, lat.wavefront = plan
        k = P.lbm_get_launch_steps(lat.ctx)
        assert k >= 1
        for n, one in ((k, True), (k + 1, False)):
            before = P.lbm_get_launches(lat.ctx)
            lat.iterate(n)
            assert (P.lbm_get_launches(lat.ctx) - before == 1) == one, (k, n)
