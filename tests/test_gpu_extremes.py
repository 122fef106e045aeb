"""Finite elevations so large that single-precision differences overflow: any
finite DEM is accepted, so every decision on it is the FP64 definition's."""
import numpy as np
import pytest

import paper_2003_02200_gb300 as tvs
from paper_2003_02200_gb300 import terrain

pytestmark = pytest.mark.gpu

BIG = np.float32(3.4028234663852886e38)


@pytest.fixture(scope="module", params=[1, 0], ids=["pruned", "unpruned"])
def ctx(request):
    with tvs.Context(0) as c:
        c.set_tuning(prune=request.param)
        yield c


def _check(ctx, orc, dem, h0, n, rng, ks):
    rows, cols = dem.shape
    for k in ks:
        got = ctx.debug_direction_cv(dem, 10.0, h0, n, rng, k)
        d = orc.direction(n, k, rows, cols)
        want = np.stack([orc.line_cv(dem, 10.0, h0, n, rng, 64, k, p - d["D"]) for p in range(d["H"] + d["D"])])
        bad = np.argwhere(got != want)
        assert bad.size == 0, f"k {k}: {len(bad)} samples differ, first {bad[:4].tolist()}"


def _towers(rows, cols, seed):
    """Fractal ground with cells of either sign whose differences pass FLT_MAX."""
    r = np.random.default_rng(seed)
    dem = terrain.fractal_dem(rows, cols, 0.7, 1200.0, seed)
    for v in (-3e38, 0.5e38, 3.4e38, -1e38, 2e38, -3.4e38, 3e38, -0.25e38):
        dem[r.integers(rows), r.integers(cols)] = v
    return dem


def test_rise_after_an_overflowed_slope(ctx, orc):
    """From -3e38, 0.5e38 at 20 steps overflows a single-precision difference;
    3.4e38 at 34 steps is higher still, and 3.3e38 at 35 is not."""
    dem = np.zeros((2, 96), np.float32)
    dem[:, 8] = -3e38
    dem[:, 28], dem[:, 42], dem[:, 43] = 0.5e38, 3.4e38, 3.3e38
    _check(ctx, orc, dem, 1.5, 4, 0.0, (0,))


def test_falls_past_the_lowest_float(ctx, orc):
    """From 3e38, a near target at 2e38 and farther ones below -0.5e38: their
    differences overflow downward, their slopes lie above the near one's."""
    dem = np.full((2, 96), -1e38, np.float32)
    dem[:, 8], dem[:, 9] = 3e38, 2e38
    dem[:, 28:40] = -0.5e38
    _check(ctx, orc, dem, 1.5, 4, 0.0, (0,))


# packed rows, one row per warp, rows shared by 2, 4 and 16 warps
@pytest.mark.parametrize("rows,cols", [(40, 61), (5, 300), (4, 900), (3, 2100), (2, 3300), (2, 9000)])
@pytest.mark.parametrize("h0,rng", [(1.5, 0.0), (0.0, 405.0)])
def test_towers(ctx, orc, rows, cols, h0, rng):
    _check(ctx, orc, _towers(rows, cols, 70 + cols), h0, 8, rng, (0, 3))


@pytest.mark.parametrize("value", [-BIG, np.float32(1e20), np.float32(-(2.0 ** 59))])
@pytest.mark.parametrize("rows,cols", [(40, 61), (9, 700), (3, 2100)])
def test_no_data_cells(ctx, orc, rows, cols, value):
    """One cell in fifty holds a no-data value, so that most rows do (and the
    flag buffer fills), two neighbours of a blend among them; the last value
    is just below where rows are handed over whole."""
    r = np.random.default_rng(cols)
    dem = terrain.fractal_dem(rows, cols, 0.7, 1200.0, 8)
    dem[r.random(dem.shape) < 0.02] = value
    dem[:2, 11] = value
    _check(ctx, orc, dem, 1.5, 8, 0.0, (0, 3))


@pytest.mark.parametrize("h0", [2.0 ** 60, 3e38, 1e300])
def test_huge_observer_heights(ctx, orc, h0):
    _check(ctx, orc, terrain.fractal_dem(5, 130, 0.7, 1200.0, 7), h0, 8, 0.0, (0, 3))


def _points(ctx, orc, dem, povs, n, h0=1.5):
    """Areas in both readings and the map of each POV."""
    import torch
    cols = dem.shape[1]
    d = torch.tensor(dem, device="cuda")
    p = np.asarray(povs, np.int32)
    want = ctx.total_viewshed(dem, 10.0, h0, n)[p[:, 0], p[:, 1]]
    np.testing.assert_array_equal(ctx.viewshed_points(d, 10.0, h0, n, 0.0, p).cpu().numpy(), want)
    want = orc.direct_viewshed(dem, 10.0, h0, n, 0.0, cells=p[:, 0].astype(np.int64) * cols + p[:, 1])
    got = ctx.viewshed_points(d, 10.0, h0, n, 0.0, p, mode="direct").cpu().numpy()
    # FP32 blend and sums of 8 directions
    np.testing.assert_allclose(got, want, rtol=4e-6, atol=4e-4)
    for q in p:
        seen = ctx.visibility_map(d, 10.0, h0, n, 0.0, q[None]).cpu().numpy()
        ref = orc.visibility_map(dem, 10.0, h0, n, 0.0, povs=q[None])
        # cells on a sector boundary may fall to either side (two atan2 implementations)
        assert np.mean(seen != ref) < 1e-3


@pytest.mark.parametrize("rows,cols", [(40, 61), (130, 170)])
def test_points_among_towers(ctx, orc, rows, cols):
    """Short walks and walks by tile maxima, from the towers and beside them."""
    dem = _towers(rows, cols, 5)
    ii, jj = np.nonzero(np.abs(dem) > 1e37)
    p = np.concatenate([np.stack([ii, jj], 1), np.stack([ii, (jj + 1) % cols], 1), [[0, 0], [rows - 1, cols - 1]]])
    _points(ctx, orc, dem, p, 7)


def test_points_above_a_fall_past_the_lowest_float(ctx, orc):
    """A tile's bound overflows downward: from 3e38 over 2e38 the ground at
    -1e38 is hidden at first and rises into view far out."""
    dem = np.full((40, 300), -1e38, np.float32)
    dem[:, :48] = 2e38        # three whole tiles
    dem[20, 8] = 3e38
    _points(ctx, orc, dem, [(20, 8), (20, 7), (3, 299)], 4)


def test_points_beside_a_fall_at_the_first_target(ctx, orc):
    """The first target's slope overflows in double-float."""
    dem = np.full((9, 60), 100.0, np.float32)
    dem[4, 8], dem[4, 9], dem[4, 10], dem[4, 11] = -3.4e38, 3.4e38, 1e37, 3.4e38
    _points(ctx, orc, dem, [(4, 8), (4, 9), (4, 10), (4, 7)], 4)


@pytest.mark.parametrize("h0", [2.0 ** 60, 3e38, 1e300])
def test_points_at_huge_observer_heights(ctx, orc, h0):
    _points(ctx, orc, terrain.fractal_dem(60, 150, 0.7, 1200.0, 7), [(0, 0), (30, 60), (59, 149)], 4, h0)


@pytest.mark.parametrize("value", [-BIG, BIG, np.float32(1e30), np.float32(-1e9), np.float32(-9999.0), np.float32(1e-30)])
@pytest.mark.parametrize("rows,cols,rng", [(40, 61, 0.0), (6, 900, 0.0), (3, 2100, 4567.0), (2, 5000, 0.0)])
@pytest.mark.parametrize("base", [0.0, -3e6])
def test_skipping_beside_no_data_changes_no_bit(rows, cols, rng, value, base):
    """The lines that blocks are tested against, on ground whose heights are far
    below (or above) the row's largest: FP32 and certified decisions, skipping
    or not."""
    r = np.random.default_rng(cols)
    dem = terrain.fractal_dem(rows, cols, 0.7, 1200.0, 8) + np.float32(base)
    dem[r.random(dem.shape) < 0.02] = value
    with tvs.Context(0) as c:
        for fp32 in (1, 0):
            c.set_tuning(fp32_decisions=fp32, prune=1)
            got = c.total_viewshed(dem, 10.0, 1.5, 8, rng)
            c.set_tuning(prune=0)
            np.testing.assert_array_equal(got, c.total_viewshed(dem, 10.0, 1.5, 8, rng))


@pytest.mark.parametrize("value", [-BIG, np.float32(-1e9), np.float32(1e20)])
@pytest.mark.parametrize("rows,cols", [(40, 61), (60, 600)])
def test_points_beside_no_data(ctx, orc, rows, cols, value):
    """From inside a corner without data, its edge and beyond it."""
    dem = terrain.fractal_dem(rows, cols, 0.7, 600.0, 3)
    dem[:rows // 3, :cols // 3] = value
    i, j = rows // 3, cols // 3
    _points(ctx, orc, dem, [(0, 0), (i - 1, j - 1), (i - 1, 3), (i, 3), (i + 1, j + 1), (rows - 1, cols - 1)], 7)
