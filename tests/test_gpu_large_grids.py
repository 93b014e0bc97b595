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
