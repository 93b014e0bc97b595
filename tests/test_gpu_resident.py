"""GPU steps that stay on the chip: ensembles that fit there take another
kernel, which gives the states, clocks and rain of the ordinary march bit for
bit (a launch shape that is set keeps an ensemble on the march), over sizes at
the edges of its bands and quads, every option of the step and numbers of steps
on both sides of a run."""
import numpy as np
import pytest

from paper_2302_08341_gb300 import synth
from tests.gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def capi():
    return require_gpu()


def _run(capi, ny, nx, M, march, land=False, track=False, inflow=False, deep=False, steps=(1, 24, 31, 290)):
    terr = synth.make_terrain(ny, nx, seed=91)
    rm, sc = synth.ensemble_prior(91, M)
    rng = np.random.default_rng(91)
    h0 = rng.uniform(0.0, 2.0 if deep else 0.1, (M, ny, nx)).astype(np.float32)
    h0[:, ::3, ::2] = 0.0
    p = capi.Params.default(east_outflow=1, south_outflow=1)
    with capi.Grid(terr.z, terr.n, p) as g:
        if land:
            g.set_land_cover(rng.integers(0, 4, (ny, nx)), [c[:3] + (0,) for c in synth.LAND_CLASSES])
        g.ensemble_init(M, rm, sc, synth.hyetograph_triangular(60.0, 30.0, 60.0), h0=h0)
        if inflow:
            g.set_inflow(ny // 3, max(ny // 3 + 1, ny // 2), np.array([3.0, 5.0, 1.0], np.float32))
        if track:
            g.track_max_depth(True)
        if march:
            g.set_launch(8, 1)
        for n in steps:
            g.step(n)
        g.advance_to(450.0)
        out = [np.array(g.get_state(m)) for m in range(M)]
        if track:
            out += [g.max_depth(m) for m in range(M)]
        mem = g.members()
        out += [mem["t"], mem["steps"], mem["hmax"]]
        vol = g.volumes()
        out += [vol["storage"], vol["rain"]]
        if inflow:
            out.append(g.inflow_volume())
        return out, vol


@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 9, 3), (3, 4, 2), (153, 5, 1), (64, 131, 7), (40, 129, 76),
                                   (30, 33, 152), (30, 33, 153), (305, 310, 1)])
@pytest.mark.parametrize("options", [dict(), dict(land=True, track=True), dict(inflow=True, deep=True),
                                     dict(land=True, inflow=True), dict(track=True, deep=True)])
def test_resident_steps_equal_the_march(capi, shape, options):
    a, va = _run(capi, *shape, march=False, **options)
    b, vb = _run(capi, *shape, march=True, **options)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
    # outflow and clamp: sums of compensated FP32 partials that round by 2^-24
    # of each row's terms, which have one sign
    for k in ("outflow", "clamp"):
        assert np.all(np.abs(va[k] - vb[k]) <= 2.0 ** -22 * np.abs(vb[k]))
