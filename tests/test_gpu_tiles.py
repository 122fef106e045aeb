"""Point walks by tile maxima (walks of 128 targets and more): POVs at corners,
edges and tile borders of ragged DEMs, on terrain that rises, falls and ties.
The sDEM area of a cell is the total viewshed map's value bit for bit; the
direct reading and the visibility map are held to the FP64 oracle."""
import numpy as np
import pytest

import paper_2003_02200_gb300 as tvs
from paper_2003_02200_gb300 import terrain

pytestmark = pytest.mark.gpu

# areas: FP32 blend and sums of 8 directions
RTOL = 4e-6


@pytest.fixture(scope="module")
def ctx():
    with tvs.Context(0) as c:
        yield c


def _dem(kind, rows, cols):
    i, j = np.mgrid[0:rows, 0:cols].astype(np.float64)
    if kind == "fractal":
        return terrain.fractal_dem(rows, cols, 0.7, 900.0, 3, spike_frac=0.02)
    if kind == "ridge":
        return (-500.0 - 0.02 * (i - rows / 3) ** 2 - 0.01 * (j - cols / 2) ** 2).astype(np.float32)
    if kind == "level":
        return np.zeros((rows, cols), np.float32)
    raise ValueError(kind)


def _povs(rows, cols):
    ii = [0, 1, 15, 16, 17, rows // 2, rows - 17, rows - 16, rows - 1]
    jj = [0, 1, 15, 16, 31, cols // 2, cols - 17, cols - 16, cols - 1]
    return np.array([(i, j) for i in ii for j in jj], np.int32)


@pytest.mark.parametrize("kind,h0", [("fractal", 1.5), ("ridge", 3.0), ("level", 1.5), ("level", 0.0)])
@pytest.mark.parametrize("rows,cols,n,rng", [(129, 200, 12, 0.0), (257, 143, 8, 0.0), (160, 333, 16, 1450.0)])
def test_sdem_points_equal_the_map(ctx, kind, h0, rows, cols, n, rng):
    import torch
    dem = _dem(kind, rows, cols)
    p = _povs(rows, cols)
    want = ctx.total_viewshed(dem, 10.0, h0, n, rng)[p[:, 0], p[:, 1]]
    got = ctx.viewshed_points(torch.tensor(dem, device="cuda"), 10.0, h0, n, rng, p).cpu().numpy()
    np.testing.assert_array_equal(got, want)


@pytest.mark.parametrize("kind,h0", [("fractal", 1.5), ("ridge", 3.0), ("level", 0.0)])
@pytest.mark.parametrize("rows,cols,n,rng", [(129, 200, 12, 0.0), (257, 143, 7, 0.0), (160, 333, 16, 1450.0)])
def test_direct_points_and_visibility_map(ctx, orc, kind, h0, rows, cols, n, rng):
    import torch
    dem = _dem(kind, rows, cols)
    d = torch.tensor(dem, device="cuda")
    p = _povs(rows, cols)
    want = orc.direct_viewshed(dem, 10.0, h0, n, rng, cells=p[:, 0].astype(np.int64) * cols + p[:, 1])
    got = ctx.viewshed_points(d, 10.0, h0, n, rng, p, mode="direct").cpu().numpy()
    np.testing.assert_allclose(got, want, rtol=RTOL, atol=RTOL * 100.0)
    q = p[[0, 10, 40, 60, 80]]
    seen = ctx.visibility_map(d, 10.0, h0, n, rng, q).cpu().numpy()
    ref = orc.visibility_map(dem, 10.0, h0, n, rng, povs=q)
    # cells on a sector boundary may fall to either side (two atan2 implementations)
    assert np.mean(seen != ref) < 1e-3


@pytest.mark.parametrize("npov,n", [(1, 4), (63, 8), (64, 8)])
@pytest.mark.parametrize("rows,cols", [(40, 767), (40, 768), (769, 40), (127, 128), (128, 90), (120, 127)])
def test_either_side_of_the_rule(ctx, orc, npov, n, rows, cols):
    """Walks of 127, 128, 767, 768 targets of fewer and more lines than the tile
    maxima are taken for, in both readings, and their visibility map."""
    import torch
    dem = _dem("fractal", rows, cols)
    d = torch.tensor(dem, device="cuda")
    p = np.random.default_rng(rows + cols).integers(0, (rows, cols), (npov, 2)).astype(np.int32)
    want = ctx.total_viewshed(dem, 10.0, 1.5, n)[p[:, 0], p[:, 1]]
    np.testing.assert_array_equal(ctx.viewshed_points(d, 10.0, 1.5, n, 0.0, p).cpu().numpy(), want)
    want = orc.direct_viewshed(dem, 10.0, 1.5, n, 0.0, cells=p[:, 0].astype(np.int64) * cols + p[:, 1])
    got = ctx.viewshed_points(d, 10.0, 1.5, n, 0.0, p, mode="direct").cpu().numpy()
    np.testing.assert_allclose(got, want, rtol=RTOL, atol=RTOL * 100.0)
    seen = ctx.visibility_map(d, 10.0, 1.5, n, 0.0, p).cpu().numpy()
    ref = orc.visibility_map(dem, 10.0, 1.5, n, 0.0, povs=p)
    # cells on a sector boundary may fall to either side (two atan2 implementations)
    assert np.mean(seen != ref) < 1e-3 * npov
