"""Strip kernel (two to six steps per launch, one warp per strip of 64 slot
columns) against one step per launch, at the sizes where its copies, halos
and pairs can go wrong: widths that are no multiple of a 16-byte chunk (every
remainder of eight), odd widths, whole numbers of strips and one column more,
heights of one segment row, and every step count a launch can take.  FP32
states must be equal; FP16-shifted states are compared with the three-step
tile kernel, which rounds to FP16 at the same steps."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2208_14870_gb300 as P  # noqa: E402
from paper_2208_14870_gb300 import Lattice  # noqa: E402

# 280 and 364: whole strips of 56 and 52 output columns (five and six steps)
SIZES = [(256, 8), (257, 9), (258, 31), (259, 40), (260, 13), (261, 8), (262, 21), (263, 17),
         (280, 33), (281, 10), (364, 12), (365, 25), (1000, 61)]


def _state(nx, ny, dtype, spl, wave, steps, check_every=None, **kw):
    lam, mu = W.lame_2d(1.0, 0.3)
    rng = np.random.RandomState(nx * 1000 + ny)
    gx, gy = rng.standard_normal((2, ny, nx)) / max(nx, ny) ** 2
    with Lattice(nx, ny, lam, mu, dtype, **kw) as lat:
        lat.steps_per_launch = spl
        lat.wavefront = wave
        lat.set_force(gx, gy)
        if check_every:
            lat.iterate_checked(steps, check_every)
        else:
            lat.iterate(steps)
        return lat.populations()


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("rows", [1, 6, -1])
def test_f32_equals_single_steps(nx, ny, rows):
    for steps in (2, 3, 4, 5, 6, 7, 8, 15):
        ref = _state(nx, ny, "f32", 1, 0, steps)
        assert np.array_equal(_state(nx, ny, "f32", 4, rows, steps), ref), steps


@pytest.mark.parametrize("nx,ny", [(257, 9), (364, 40)])
def test_f32_general_rates_and_checks(nx, ny):
    kw = dict(tau12=0.9, tau22=0.3, theta=0.25)
    for steps in (2, 5, 6, 7, 20):
        ref = _state(nx, ny, "f32", 1, 0, steps, **kw)
        assert np.array_equal(_state(nx, ny, "f32", 4, -1, steps, **kw), ref), steps
    ref = _state(nx, ny, "f32", 1, 0, 37, **kw)
    assert np.array_equal(_state(nx, ny, "f32", 4, -1, 37, check_every=9, **kw), ref)


# Checked launches of four and of five steps (windows of five steps end in one
# launch), with the residual of the last check.
@pytest.mark.parametrize("nx,ny", [(256, 8), (257, 9), (364, 40), (261, 8)])
@pytest.mark.parametrize("every", [4, 5, 9, 10])
def test_f32_checked_launches(nx, ny, every):
    lam, mu = W.lame_2d(1.0, 0.3)
    gx, gy = np.random.RandomState(nx + ny).standard_normal((2, ny, nx)) / max(nx, ny) ** 2
    res = []
    for spl, wave in ((1, 0), (4, -1), (4, 3)):
        with Lattice(nx, ny, lam, mu, "f32") as lat:
            lat.steps_per_launch, lat.wavefront = spl, wave
            lat.set_force(gx, gy)
            r = lat.iterate_checked(4 * every, every)
            res.append((lat.populations(), r))
    for pops, r in res[1:]:
        assert np.array_equal(pops, res[0][0])
        assert np.allclose(r, res[0][1], rtol=1e-12, atol=0.0)


# Recovery of the fields from FP32 states: subnormal populations, and populations
# whose sums leave FP32's range, give the same fields as their multiples by a
# power of two in the middle of it.
@pytest.mark.parametrize("nx,ny", [(5, 3), (33, 9), (256, 8)])
def test_f32_fields_at_the_ends_of_the_range(nx, ny):
    lam, mu = W.lame_2d(1.0, 0.3)
    k = np.random.RandomState(nx).randint(-5, 6, (8, ny, nx)).astype(np.float64)
    with Lattice(nx, ny, lam, mu, "f32") as lat:
        got = []
        for e in (-149, -60, 0, 125):
            lat.set_populations(k * 2.0 ** e)
            got.append(lat.fields() * 2.0 ** -e)
    assert np.isfinite(got[2]).all() and np.abs(got[2]).max() > 0.0
    for f in got:
        assert np.allclose(f, got[2], rtol=2.0 ** -50, atol=2.0 ** -50)


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("kw", [dict(), dict(tau12=0.9, tau22=0.3)])
def test_f16s_equals_tiles(nx, ny, kw):
    ny = max(ny, 16)
    for rows in (5, -1):
        ref = _state(nx, ny, "f16s", 3, 0, 6, **kw)
        assert np.array_equal(_state(nx, ny, "f16s", 3, rows, 6, **kw), ref)


# Register tiles (k_tile; the default of small FP32 lattices): lattices smaller
# than a tile, ragged last tiles, odd and unpadded widths, every step count of
# a window with its checked last launch.
@pytest.mark.parametrize("nx,ny", [(1, 1), (2, 3), (5, 1), (1, 40), (31, 7), (33, 64), (64, 64), (100, 75), (257, 30),
                                   (333, 100)])
@pytest.mark.parametrize("kw", [dict(), dict(tau12=0.9, tau22=0.3)])
def test_default_plan_equals_single_steps(nx, ny, kw):
    lam, mu = W.lame_2d(1.0, 0.3)
    rng = np.random.RandomState(nx * 1000 + ny)
    gx, gy = rng.standard_normal((2, ny, nx)) / max(nx, ny) ** 2
    for steps, check in ((1, 0), (2, 0), (3, 0), (13, 0), (29, 1), (40, 7), (41, 20)):
        res = []
        for plain in (True, False):
            with Lattice(nx, ny, lam, mu, "f32", **kw) as lat:
                if plain:
                    lat.steps_per_launch, lat.wavefront = 1, 0
                lat.set_force(gx, gy)
                r = lat.iterate_checked(steps, check) if check else lat.iterate(steps)
                res.append((lat.populations(), r))
        assert np.array_equal(res[0][0], res[1][0]), (steps, check)
        if check:   # sums of pairs in another order: about 2^-44 relative
            assert np.allclose(res[0][1], res[1][1], rtol=1e-12, atol=0.0), (steps, check)


# FP16S: the default plan (tiles that round where a group of steps ends, strips)
# against the same groups, one launch each: every group length (one, two, three
# and four steps), lattices smaller than a tile, ragged ones, windows whose
# groups do not divide them.
@pytest.mark.parametrize("nx,ny", [(1, 1), (5, 3), (33, 64), (63, 30), (64, 23), (70, 24), (100, 15), (100, 75), (200, 300),
                                   (255, 40), (256, 8), (300, 300), (90, 2413)])
@pytest.mark.parametrize("kw", [dict(), dict(tau12=0.9, tau22=0.3)])
def test_f16s_default_plan_equals_groups(nx, ny, kw):
    lam, mu = W.lame_2d(1.0, 0.3)
    rng = np.random.RandomState(nx * 1000 + ny)
    gx, gy = rng.standard_normal((2, ny, nx)) / max(nx, ny) ** 2
    for steps, check in ((1, 0), (2, 0), (7, 0), (29, 0), (29, 1), (40, 7), (41, 20)):
        res = []
        for groups in (True, False):
            with Lattice(nx, ny, lam, mu, "f16s", **kw) as lat:
                if groups:
                    lat.steps_per_launch = lat.steps_per_launch
                lat.set_force(gx, gy)
                r = lat.iterate_checked(steps, check) if check else lat.iterate(steps)
                res.append((lat.populations(), r))
        assert np.array_equal(res[0][0], res[1][0]), (steps, check)
        if check:
            assert np.allclose(res[0][1], res[1][1], rtol=1e-12, atol=0.0), (steps, check)


# FP64 tiles (k_tile64): several steps per launch against one step per launch
# (an iterate call of one step is one), on lattices smaller than a tile, ragged
# ones and large ones.
@pytest.mark.parametrize("nx,ny", [(1, 1), (3, 2), (7, 5), (33, 1), (64, 64), (100, 75), (130, 257)])
@pytest.mark.parametrize("kw", [dict(), dict(tau12=0.9, tau22=0.3), dict(theta=0.1)])
def test_f64_tiles_equal_single_steps(nx, ny, kw):
    lam, mu = W.lame_2d(1.0, 0.3)
    rng = np.random.RandomState(nx * 1000 + ny)
    gx, gy = rng.standard_normal((2, ny, nx)) / max(nx, ny) ** 2
    with Lattice(nx, ny, lam, mu, "f64", **kw) as a, Lattice(nx, ny, lam, mu, "f64", **kw) as b:
        a.set_force(gx, gy)
        b.set_force(gx, gy)
        for _ in range(11):
            a.iterate(1)
        b.iterate(11)
        assert np.array_equal(a.populations(), b.populations())
        for _ in range(10):
            a.iterate_checked(1, 10)
        ra = a.iterate_checked(9, 10)
        rb = b.iterate_checked(19, 10)
        assert np.array_equal(a.populations(), b.populations())
        assert np.allclose(ra, rb, rtol=1e-13, atol=0.0)


# FP64 collision in integers (step_f64) against long double, one step: populations
# of mixed magnitudes, zeros, and scales on either side of the lines to FP64
# arithmetic (2^-923 and 2^977).  Integers: the last rounding and eight units of
# 2^-58 of the largest value's power of two, so 2^-54 of the largest value; FP64:
# at most 32 roundings of sums of twelve populations.
@pytest.mark.parametrize("scale,integers", [(0, True), (-880, True), (940, True), (-990, False), (1000, False)])
@pytest.mark.parametrize("kw", [dict(), dict(tau12=0.9, tau22=0.3)])
def test_f64_step_against_long_double(scale, integers, kw):
    nx, ny = 37, 11
    lam, mu = (np.longdouble(v) for v in W.lame_2d(1.0, 0.3))
    rng = np.random.RandomState(scale + 2000)
    f = rng.standard_normal((8, ny, nx)) * 2.0 ** rng.randint(-40, 1, (8, ny, nx))
    f[rng.random_sample(f.shape) < 0.1] = 0.0
    f[:, 3, :5] = 0.0
    g = rng.standard_normal((2, ny, nx)) * 2.0 ** rng.randint(-60, 1, (2, ny, nx))
    g[:, 3, :3] = 0.0
    f, g = np.ldexp(f, scale), np.ldexp(g, scale)
    with Lattice(nx, ny, float(lam), float(mu), "f64", **kw) as lat:
        lat.set_force(g[0], g[1])
        lat.set_populations(f)
        lat.iterate(1)
        got = lat.populations()
    one = np.longdouble(1)
    th, t12, t22 = one / 3, np.longdouble(kw.get("tau12", 0.5)), np.longdouble(kw.get("tau22", 0.5))
    w11, w12, w22 = one / (mu / th + one / 2), one / (t12 + one / 2), one / (t22 + one / 2)
    ws, wd = one / (2 * (lam + mu) / (1 + th) + one / 2), one / (2 * mu / (1 - th) + one / 2)
    f, g = np.ldexp(f, -scale).astype(np.longdouble), np.ldexp(g, -scale).astype(np.longdouble)
    p, q, r, s = f[4] + f[6], f[5] + f[7], f[4] - f[6], f[5] - f[7]
    u, v = f[0] - f[2] + (r - s) + g[0] / 2, f[1] - f[3] + (r + s) + g[1] / 2
    s13, s24 = f[0] + f[2], f[1] + f[3]
    m11, m22 = (1 - w11) * (p - q) / 4, (1 - w22) * (p + q) / 4
    ms, md = (1 - ws) * (s13 + s24 + 2 * (p + q)) / 4, (1 - wd) * (s13 - s24) / 4
    m12, m21 = (w12 * th * u + (1 - w12) * (r - s)) / 4, (w12 * th * v + (1 - w12) * (r + s)) / 4
    A, B = (u + g[0] / 2 - 4 * m12) / 2, (v + g[1] / 2 - 4 * m21) / 2
    P_, Q_ = ms + md - 2 * m22, ms - md - 2 * m22
    o = [P_ + A, Q_ + B, P_ - A, Q_ - B, m22 + m11 + m12 + m21, m22 - m11 + m21 - m12, m22 + m11 - m12 - m21,
         m22 - m11 - m21 + m12]
    top = np.maximum(abs(f).max(axis=0), abs(g).max(axis=0))
    for k, (cx, cy) in enumerate([(1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]):
        want, big = np.roll(o[k], (cy, cx), (0, 1)), np.roll(top, (cy, cx), (0, 1))
        err = abs(np.ldexp(got[k].astype(np.longdouble), -scale) - want)
        # (the rates are FP64 numbers: 2^-53 of sums of up to twelve populations)
        tol = 2.0 ** -53 * abs(want) + (2.0 ** -54 + 2.0 ** -50) * big if integers else 2.0 ** -44 * big + 2.0 ** -70
        assert (err <= tol).all(), k


# Steps that hold no check: the residual of a fresh context is infinite and its
# norms are zero, whatever an earlier context left in the memory.
@pytest.mark.parametrize("dtype", ["f64", "f32", "f16s"])
def test_residual_before_the_first_check(dtype):
    lam, mu = W.lame_2d(1.0, 0.3)
    g = np.random.RandomState(3).standard_normal((2, 200, 300)) * 1e-5
    for steps in (300, 86, 0):
        with Lattice(300, 200, lam, mu, dtype) as lat:
            lat.set_force(g[0], g[1])
            r = lat.iterate_checked(steps, 100)
            lat.fields()
        if steps < 100:
            assert np.array_equal(r, [np.inf, np.inf, 0.0, 0.0, 0.0])


def _problems(sizes):
    out = []
    for i, (nx, ny) in enumerate(sizes):
        gx, gy = np.random.RandomState(i).standard_normal((2, ny, nx)) / max(nx, ny) ** 2
        out.append((nx, ny, *W.lame_2d(1.0, 0.1 + 0.02 * i), gx, gy))
    return out


def _alone(prob, steps, transposed):
    """Fields of the problem as a single FP32 lattice, in the arena's orientation."""
    nx, ny, lam, mu, gx, gy = prob
    if transposed:
        nx, ny, gx, gy = ny, nx, gy.T, gx.T
    with Lattice(nx, ny, lam, mu, "f32") as lat:
        lat.set_force(gx, gy)
        lat.iterate(steps)
        f = lat.fields()
    return f.transpose(0, 2, 1)[[1, 0, 3, 2, 4]] if transposed else f


# Strip items of the arena: widths without ghost columns (below 16), narrower
# than a strip, whole strips of 56 columns and one more, with every chunk length
# that leaves another rest of five.
@pytest.mark.parametrize("k", [4, 8, 12, 16, 100])
def test_arena_strips_equal_single_lattices(k, monkeypatch):
    monkeypatch.setenv("LBM_BATCH_TILE_V", str(P.LBM_TILE_WAVE))
    probs = _problems([(1, 1), (5, 9), (15, 40), (16, 16), (17, 30), (56, 20), (57, 20), (112, 33), (113, 70), (64, 300),
                       (255, 9), (257, 64), (300, 31)])
    steps = 2 * k
    res, rep = P.batch_solve(probs, "f32", 0.0, k, steps)
    assert rep["tile_v"] == P.LBM_TILE_WAVE
    for p, r in zip(probs, res):
        assert r["iters"] == steps
        assert np.array_equal(r["fields"], _alone(p, steps, r["transposed"])), p[:2]


def test_arena_f16s_strips_round_where_tiles_do(monkeypatch):
    # below 256 x 8 both round the state to FP16 every second step
    probs = _problems([(1, 1), (15, 40), (16, 16), (57, 20), (112, 33), (113, 70), (64, 300), (255, 9)])
    res = []
    for v in (P.LBM_TILE_WAVE, P.LBM_TILE_TWO_STEP):
        monkeypatch.setenv("LBM_BATCH_TILE_V", str(v))
        res.append(P.batch_solve(probs, "f16s", 0.0, 8, 24)[0])
    for a, b in zip(*res):
        if a["fields"].shape[2] < 256 and a["fields"].shape[1] < 256:
            assert np.array_equal(a["fields"], b["fields"])


def test_arena_problem_that_fits_only_without_ghost_columns():
    # 32 columns and eight ghost columns per side take half as much again: a
    # budget between the two
    prob = _problems([(32, 200)])[0]
    n = 32 * 200
    with P.Server(max(1 << 20, 2 * int(n * 88 * 1.2)), check_every=100) as srv:
        r = srv.wait(srv.submit(*prob, dtype="f32", tol=0.0, max_iters=200))
    assert np.array_equal(r["fields"], _alone(prob, 200, r["transposed"]))
