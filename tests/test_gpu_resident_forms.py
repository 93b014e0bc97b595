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
