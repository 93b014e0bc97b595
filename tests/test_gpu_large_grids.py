"""Grids that reach the limits of a launch's dimensions with the automatic
strip heights: 65535 blocks along y and z."""
import numpy as np
import pytest

from paper_2302_08341_gb300 import synth
from tests.gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def capi():
    return require_gpu()


def _fields(ny, nx, seed):
    """A bed that repeats every 1000 rows, its roughness, and shallow water."""
    rng = np.random.default_rng(seed)
    reps = (ny + 999) // 1000
    z = np.tile(rng.uniform(0.0, 1.0, (1000, nx)).astype(np.float32), (reps, 1))[:ny].copy()
    n = np.tile(rng.uniform(0.02, 0.08, (1000, nx)).astype(np.float32), (reps, 1))[:ny].copy()
    h0 = np.tile(rng.uniform(0.0, 0.3, (1000, nx)).astype(np.float32), (reps, 1))[:ny].copy()
    return z, n, h0


@pytest.mark.parametrize("track", [False, True])
def test_a_grid_of_more_than_65535_short_strips(capi, track):
    """1.6 million rows: in strips of 24 or 9 rows more than a launch holds.
    The automatic shape steps it, as strips of 64 rows do."""
    ny, nx = 1_600_000, 5
    z, n, h0 = _fields(ny, nx, 5)
    hy = synth.hyetograph_constant(60.0, 600.0)
    res = []
    for fixed in (False, True):
        with capi.Grid(z, n) as g:
            g.ensemble_init(1, np.ones(1, np.float32), np.ones(1, np.float32), hy, h0=h0)
            if track:
                g.track_max_depth(True)
            if fixed:
                g.set_launch(64, 1)
            rows = g.get_launch()[0]
            assert (ny + rows - 1) // rows <= 65535
            g.step(3)
            g.sync()
            res.append(g.get_state(0))
    for a, b in zip(*res):
        assert np.array_equal(a, b)
    assert res[0][0].max() > 0.0 and np.abs(res[0][2]).max() > 0.0


def test_a_domain_of_more_than_65535_tiles(capi):
    """Land cover with cells outside the domain: the step launches the tiles
    that hold a cell of it, here 33 thousand strips of two spans.  The same
    step, bit for bit, as with direct loads, which leave no tile out."""
    ny, nx = 800_000, 129
    z, n, h0 = _fields(ny, nx, 7)
    cls = np.zeros((ny, nx), np.int32)
    cls[::7, ::3] = 1
    cls[400_000:400_100] = 3
    classes = [c[:3] + (1 if i == 3 else 0,) for i, c in enumerate(synth.LAND_CLASSES)]
    hy = synth.hyetograph_constant(60.0, 600.0)
    res = []
    for engine in (1, 0):
        with capi.Grid(z, n) as g:
            g.set_land_cover(cls, classes)
            g.ensemble_init(1, np.ones(1, np.float32), np.ones(1, np.float32), hy, h0=h0)
            rows = g.get_launch()[0]
            assert 2 * ((ny - 100) // rows) > 65535
            g.set_engine(engine)
            g.step(2)
            g.sync()
            res.append(g.get_state(0))
    for a, b in zip(*res):
        assert np.array_equal(a, b)
    assert res[0][0].max() > 0.0 and not res[0][0][400_000:400_100].any()
