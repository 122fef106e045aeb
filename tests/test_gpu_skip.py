"""The pruned certified walk (blocks skipped by their window maxima, flagged
work handed over or marked): per-sample measures are integers and must equal
the FP64 oracle's exactly, at row lengths around the group, block and chunk
sizes, on terrain that falls away from every observer (negative slopes, the
falling lines of the skip test), on ties, and with the flag buffer full."""
import numpy as np
import pytest

import paper_2003_02200_gb300 as tvs
from paper_2003_02200_gb300 import terrain

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    with tvs.Context(0) as c:
        yield c


def _terrain(kind, rows, cols, seed):
    r = np.random.default_rng(seed)
    j = np.arange(cols, dtype=np.float64)[None, :].repeat(rows, 0)
    if kind == "fractal":
        return terrain.fractal_dem(rows, cols, 0.7, 1200.0, seed)
    if kind == "valley":        # every walk looks down first, then up a far slope
        z = 0.004 * (j - 0.6 * cols) ** 2
    elif kind == "ridge":       # slopes stay negative: the lines of the test fall
        z = -0.01 * (j - 0.4 * cols) ** 2 - 300.0
    elif kind == "sawtooth":    # many equal crests: near ties block after block
        z = (j % 37) * 4.0 + 1000.0
        return z.astype(np.float32)
    else:
        raise ValueError(kind)
    return (z + r.uniform(0.0, 3.0, (rows, cols))).astype(np.float32)


def _check(ctx, orc, dem, h0, n, rng, ks, prec=64):
    rows, cols = dem.shape
    for k in ks:
        got = ctx.debug_direction_cv(dem, 10.0, h0, n, rng, k)
        d = orc.direction(n, k, rows, cols)
        want = np.stack([orc.line_cv(dem, 10.0, h0, n, rng, prec, k, p - d["D"]) for p in range(d["H"] + d["D"])])
        bad = np.argwhere(got != want)
        assert bad.size == 0, f"k {k}: {len(bad)} samples differ, first {bad[:4].tolist()}"


@pytest.mark.parametrize("cols", [2, 3, 4, 5, 15, 16, 17, 18, 19, 20, 21, 31, 33, 35, 63, 64, 66, 127, 129, 131, 513])
@pytest.mark.parametrize("kind", ["fractal", "ridge"])
def test_row_lengths(ctx, orc, cols, kind):
    _check(ctx, orc, _terrain(kind, 5, cols, cols), 1.5, 8, 0.0, (0, 1, 7))


@pytest.mark.parametrize("rng", [0.0, 9.0, 25.0, 159.0, 165.0, 175.0, 335.0, 700.0])
@pytest.mark.parametrize("kind", ["fractal", "valley", "ridge", "sawtooth"])
def test_walk_limits(ctx, orc, kind, rng):
    """Limits inside, at and past a 16-step block."""
    _check(ctx, orc, _terrain(kind, 6, 150, 5), 2.0, 12, rng, (0, 2, 11))


# rows of more than about 1200 samples are shared by two warps, shorter ones are a warp's own
@pytest.mark.parametrize("cols", [1000, 1351, 2003, 2300])
@pytest.mark.parametrize("kind", ["fractal", "valley", "ridge", "sawtooth"])
def test_long_rows(ctx, orc, kind, cols):
    _check(ctx, orc, _terrain(kind, 3, cols, 9), 1.5, 8, 0.0, (0, 7))


@pytest.mark.parametrize("limit", list(range(1, 21)) + [31, 32, 33, 34, 47, 48, 49])
@pytest.mark.parametrize("cols", [71, 1500])
def test_every_place_of_a_limit_in_a_block(ctx, orc, cols, limit):
    """Walks of 1 to 49 steps: the block that the limit ends, for one row per
    warp and for shared rows, certified and with FP32 decisions."""
    dem = _terrain("fractal", 3, cols, 40 + limit)
    _check(ctx, orc, dem, 1.5, 4, 10.0 * limit + 1.0, (0,))
    with tvs.Context(0) as c:
        c.set_tuning(fp32_decisions=1)
        _check(c, orc, dem, 1.5, 4, 10.0 * limit + 1.0, (0,), prec=32)


# rows that 2, 4, 8 and 16 warps share, and walks long enough to flush their measures
@pytest.mark.parametrize("cols,rng", [(2500, 0.0), (3300, 0.0), (3300, 12345.0), (5000, 0.0), (5000, 45678.0),
                                      (9000, 0.0), (16384, 0.0)])
def test_rows_shared_by_many_warps(ctx, orc, cols, rng):
    _check(ctx, orc, _terrain("fractal", 2, cols, 17), 1.5, 4, rng, (0,))


@pytest.mark.parametrize("rows,cols", [(260, 300), (3, 2100), (2, 9000)])
def test_full_flag_buffer(ctx, rows, cols):
    """Level ground seen from its own height: every target ties with the
    running maximum, so nearly every walk is flagged and the buffer (one entry
    per 64 walks) overflows.  A half-line of two or more targets sees the
    first one only and measures 4; those of the inner cells all have them."""
    n = 16
    dem = np.zeros((rows, cols), np.float32)
    got = ctx.total_viewshed(dem, 10.0, 0.0, n)
    with tvs.Context(0) as c:
        c.set_tuning(prune=0)
        np.testing.assert_array_equal(got, c.total_viewshed(dem, 10.0, 0.0, n))
    if rows > 10:
        g = [1.0 + tvs.direction(n, k, rows, cols)["t"] ** 2 for k in range(n)]
        np.testing.assert_allclose(got[20:-20, 20:-20], 8.0 * sum(g) * np.pi / (2 * n) * 100.0, rtol=4e-6)


@pytest.mark.parametrize("rows,cols,n,rng", [(33, 41, 1500, 0.0), (64, 97, 720, 0.0), (130, 61, 360, 333.0),
                                             (5, 300, 500, 0.0), (16, 16, 4096, 45.0), (250, 250, 90, 0.0)])
@pytest.mark.parametrize("kind", ["fractal", "ridge", "sawtooth"])
def test_packed_rows(ctx, kind, rows, cols, n, rng):
    """Launches with enough short rows pack several of them, of both walk
    directions and across direction boundaries, into a warp: every area equals
    the unpruned sweep's, which takes one row per warp."""
    dem = _terrain(kind, rows, cols, 21)
    got = ctx.total_viewshed(dem, 10.0, 2.5, n, rng)
    with tvs.Context(0) as c:
        c.set_tuning(prune=0)
        np.testing.assert_array_equal(got, c.total_viewshed(dem, 10.0, 2.5, n, rng))


@pytest.mark.parametrize("rows,cols", [(40, 61), (5, 300), (4, 900), (3, 2100)])
@pytest.mark.parametrize("value", [-3.4028234663852886e38, 1e30, -1e9])
@pytest.mark.parametrize("h0,rng", [(1.5, 0.0), (0.0, 700.0)])
def test_rest_of_a_walk(ctx, orc, rows, cols, value, h0, rng):
    """One cell so high or low that no margin settles anything on its rows:
    block after block of a walk is flagged, and its second flag hands over all
    that is left of it, pruned and unpruned."""
    dem = _terrain("fractal", rows, cols, 33)
    dem[rows // 2, cols // 3] = value
    _check(ctx, orc, dem, h0, 8, rng, (0, 3))
    with tvs.Context(0) as c:
        c.set_tuning(prune=0)
        _check(c, orc, dem, h0, 8, rng, (0, 3))


@pytest.mark.parametrize("rows,cols,rng", [(60, 90, 0.0), (9, 1500, 0.0), (2, 3300, 9000.0), (2, 6000, 0.0)])
def test_every_cta_size_gives_the_same_map(ctx, rows, cols, rng):
    dem = _terrain("fractal", rows, cols, 4)
    want = ctx.total_viewshed(dem, 10.0, 1.5, 8, rng)
    with tvs.Context(0) as c:
        for most in (1, 2, 3, 5, 11, 13):
            c.set_tuning(sweep_max_warps=most)
            np.testing.assert_array_equal(c.total_viewshed(dem, 10.0, 1.5, 8, rng), want, err_msg=f"{most} warps")


@pytest.mark.parametrize("prune", [1, 0])
def test_walks_beside_an_outlier_are_handed_over_once(orc, prune):
    """A cell of -1e9 spoils the reference of the groups around its samples:
    every decision of their walks is inside its margin.  The cell enters one
    sample of two rows per direction, so a group of four POVs in each, walked
    both ways; each of those walks reaches the exact pass once."""
    n, rows, cols = 8, 60, 90
    dem = _terrain("fractal", rows, cols, 12)
    with tvs.Context(0) as c:
        c.set_tuning(prune=prune)
        c.total_viewshed(dem, 10.0, 1.5, n)
        tvs.sweep_stats(clear=True)
        c.total_viewshed(dem, 10.0, 1.5, n)
        usual = tvs.sweep_stats(clear=True)["exact_walks"]
        dem[rows // 2, cols // 2] = -1e9
        c.total_viewshed(dem, 10.0, 1.5, n)
        assert tvs.sweep_stats(clear=True)["exact_walks"] <= usual + n * 2 * 4 * 2
        _check(c, orc, dem, 1.5, n, 0.0, (0, 1, 3))


@pytest.mark.parametrize("cols", [33, 34, 65, 97, 129, 256, 257, 258, 259, 289, 513, 515, 2100, 9000])
@pytest.mark.parametrize("kind", ["level", "steps"])
def test_exact_walks_of_every_length(ctx, orc, kind, cols):
    """Ties block after block at lengths around the exact walks' chunks (32 to
    256 targets), with more flagged walks than the buffer has entries (one per
    64 walks, more for long rows, 4096 at least): the rest are found by the scan
    and walked whole.  Per sample against the FP64 oracle."""
    rows = 2 if cols > 2000 else 5000 // cols + 4
    dem = np.zeros((rows, cols), np.float32)
    if kind == "steps":
        dem += (2 * np.random.default_rng(cols).integers(0, 3, (rows, cols))).astype(np.float32)
    tvs.sweep_stats(clear=True)
    _check(ctx, orc, dem, 0.0, 4, 0.0, (0,))
    if kind == "level":
        cap = max(4096, 2 * rows * cols * max(1.0, max(rows, cols) / 1024) / 64)
        assert tvs.sweep_stats(clear=True)["exact_walks"] > cap
