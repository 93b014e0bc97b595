"""GPU steps that stay on the chip, further: that they are the ones that ran,
options beside those of test_gpu_resident.py, and the volumes they sum over
many steps at once."""
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2302_08341_gb300 import synth
from tests.gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def capi():
    return require_gpu()


@pytest.mark.parametrize("shape", [(1, 9, 3), (3, 4, 2), (64, 131, 7)])
def test_drained_volume_of_many_steps_in_one_launch(capi, shape):
    """A rain that changes every second and drains away at once.  With strips of
    one row the march adds up the same rows' drained depths without rounding
    before its two-word sums, step by step in FP64.  The resident steps keep two
    words over a whole launch, 2^-48 for each of up to 4800 additions a thread:
    2^-34 covers both."""
    ny, nx, M = shape
    rng = np.random.default_rng(97)
    terr = synth.make_terrain(ny, nx, seed=97)
    rm, sc = synth.ensemble_prior(97, M)
    hy = (1e-5 * rng.lognormal(0.0, 2.0, 320)).astype(np.float32)
    res = []
    for march in (False, True):
        with capi.Grid(terr.z, terr.n, capi.Params.default(rain_block=1.0)) as g:
            g.set_land_cover(np.full((ny, nx), 2), [c[:3] + (0,) for c in synth.LAND_CLASSES])
            g.ensemble_init(M, rm, sc, hy)
            g.set_land_params(synth.land_prior(97, M)[0], np.full(M, 1.0, np.float32))
            if march:
                g.set_launch(1, 1)
            g.step(300)
            res.append((g.drained(), [np.stack(g.get_state(m)) for m in range(M)]))
    for a, b in zip(res[0][1], res[1][1]):
        assert np.array_equal(a, b)
    assert res[1][0].min() > 0.0
    assert np.all(np.abs(res[0][0] - res[1][0]) <= 2.0 ** -34 * res[1][0])


def _forms(capi, shape, march, params, land, track, stream=None):
    import torch
    ny, nx, M = shape
    rng = np.random.default_rng(101)
    terr = synth.make_terrain(ny, nx, seed=101)
    rm, sc = synth.ensemble_prior(101, M)
    h0 = rng.uniform(0.0, 1.5, (M, ny, nx)).astype(np.float32)
    h0[:, ::3, ::2] = 0.0
    with capi.Grid(terr.z, terr.n, capi.Params.default(**params)) as g:
        if land:
            cls = rng.integers(0, 4, (ny, nx))
            cls[: max(1, ny // 5)] = 3                          # outside the domain, and scattered cells
            g.set_land_cover(cls, synth.LAND_CLASSES)
        with torch.cuda.stream(stream) if stream else torch.cuda.stream(torch.cuda.current_stream()):
            g.ensemble_init(M, rm, sc, synth.hyetograph_triangular(60.0, 30.0, 60.0), h0=h0)
            if land:
                g.set_land_params(*synth.land_prior(101, M))
            if track:
                g.track_max_depth(True)
            if march:
                g.set_launch(8, 1)
            n0 = g.launch_count
            g.step(31)
            launches = g.launch_count - n0
            g.advance_to(90.0)
            g.sync()
            out = [x for m in range(M) for x in g.get_state(m)]
            if track:
                out += [g.max_depth(m) for m in range(M)]
            y = g.gauge_sample(np.array([0, ny * nx // 2, ny * nx - 1], np.int32))
        mem = g.members()
        out += [y, mem["t"], mem["steps"], mem["hmax"], g.volumes()["storage"], g.volumes()["rain"]]
        # resident: 31 steps are at most a launch to the ring's first slot, one of 24 and the rest
        assert launches == 62 if march else launches <= 3
        return out


@pytest.mark.parametrize("shape", [(1, 9, 3), (64, 131, 7), (40, 129, 76), (305, 310, 1)])
@pytest.mark.parametrize("options", [dict(params=dict(limiter=0)), dict(params=dict(east_outflow=0)),
                                     dict(params=dict(east_outflow=0, south_outflow=1, limiter=0)),
                                     dict(params=dict(), land=True),
                                     dict(params=dict(south_outflow=1, limiter=0), land=True, track=True)])
def test_resident_steps_ran_and_equal_the_march(capi, shape, options):
    """The limiter off, closed and open edges, land cover with cells and whole
    rows outside the domain: states, clocks, maxima, gauges, storage and rain
    bit for bit, and the launches counted are those of resident steps."""
    if options.get("land") and shape[0] < 5:
        pytest.skip("no row would be inside the domain")
    o = dict(dict(land=False, track=False), **options)
    a = _forms(capi, shape, False, **o)
    b = _forms(capi, shape, True, **o)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("march", [False, True])
def test_every_call_on_a_side_stream(capi, march):
    """An ensemble made, stepped and read on a non-blocking stream while the
    default stream is busy: as on the default stream."""
    import torch
    shape, o = (64, 131, 7), dict(params=dict(), land=True, track=True)
    ref = _forms(capi, shape, march, **o)
    side = torch.cuda.Stream()
    torch.cuda._sleep(200_000_000)
    got = _forms(capi, shape, march, stream=side, **o)
    for x, y in zip(ref, got):
        assert np.array_equal(x, y)


_REFUSED = """
import sys
sys.modules["torch"] = None
import numpy as np
from paper_2302_08341_gb300 import capi, synth
terr = synth.make_terrain(64, 131, seed=98)
rm, sc = synth.ensemble_prior(98, 7)
res = []
for march, graphs in ((True, False), (False, False), (False, True)):
    with capi.Grid(terr.z, terr.n) as g:
        g.ensemble_init(7, rm, sc, synth.hyetograph_constant(60.0, 600.0))
        g.set_graphs(graphs)
        if march:
            g.set_launch(8, 1)
        n0 = g.launch_count
        g.step(60)
        g.advance_to(90.0)
        assert g.launch_count - n0 >= 2 * 90, "the steps did not march"
        res.append([np.stack(g.get_state(m)) for m in range(7)])
for r in res[1:]:
    for a, b in zip(res[0], r):
        assert np.array_equal(a, b)
print("done")
"""


def test_a_refused_cooperative_launch_falls_back_to_the_march(capi, tmp_path):
    """The runtime's cooperative launch replaced by one that returns its error
    (cudaErrorCooperativeLaunchTooLarge): the steps march, plainly and from a
    graph, with the same results."""
    shim = tmp_path / "refuse.c"
    shim.write_text("int cudaLaunchCooperativeKernel() { return 720; }\n")
    lib = tmp_path / "refuse.so"
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(lib), str(shim)], check=True)
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", _REFUSED], cwd=root, capture_output=True, text=True, timeout=120,
                       env=dict(os.environ, LD_PRELOAD=str(lib)))
    assert r.returncode == 0 and "done" in r.stdout, r.stderr
