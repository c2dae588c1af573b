"""Lattices at the limit of the device's memory: one that fits only without ghost
columns is laid out without them and advances on register tiles, with the same
states."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2208_14870_gb300 as P  # noqa: E402
from paper_2208_14870_gb300 import Lattice  # noqa: E402

BYTES = {"f32": 88, "f16s": 72}      # populations twice, force, snapshot


# widths with ghost columns: 64 (a quarter more memory), 70, and 300 (wavefront groups of four)
@pytest.mark.parametrize("nx,ny", [(64, 60000), (70, 50000), (300, 20000)])
@pytest.mark.parametrize("dtype", ["f32", "f16s"])
def test_fits_only_without_ghost_columns(nx, ny, dtype):
    lam, mu = W.lame_2d(1.0, 0.3)
    plain = BYTES[dtype] * nx * ny
    padded = BYTES[dtype] * ((nx + 23) // 8 * 8) * ny
    rng = np.random.RandomState(nx)
    g = torch.from_numpy(rng.standard_normal((2, ny, nx)) / nx ** 2)
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    filler = torch.empty(free - (plain + padded) // 2, dtype=torch.uint8, device="cuda")
    lat = Lattice(nx, ny, lam, mu, dtype)
    try:
        del filler
        torch.cuda.empty_cache()
        assert plain <= P.lbm_get_device_bytes(lat.ctx) < padded
        gd = g.cuda()
        for plan, steps, every in ((None, 8, 4), (None, 21, 7), ((4, -1), 21, 7), ((3, -1), 13, 6), ((2, 0), 5, 2)):
            res = []
            with Lattice(nx, ny, lam, mu, dtype) as full:
                assert P.lbm_get_device_bytes(full.ctx) >= padded
                for one in (full, lat):
                    if plan:
                        one.steps_per_launch, one.wavefront = plan
                    one.set_force(gd[0], gd[1])
                    one.reset()
                    r = one.iterate_checked(steps, every)
                    out = torch.empty((5, ny, nx), dtype=torch.float64, device="cuda")
                    res.append((one.fields_device(out), r))
            assert torch.equal(res[0][0], res[1][0]), plan
            assert np.allclose(res[0][1], res[1][1], rtol=1e-12, atol=0.0), plan
    finally:
        lat.close()
