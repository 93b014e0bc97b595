"""Steps on a stream of the caller's own: a non-blocking stream is not ordered
with the default stream, so whatever a step needs cleared or copied has to be
so on the step's own stream."""
import numpy as np
import pytest

from paper_2302_08341_gb300 import synth
from tests.gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def capi():
    return require_gpu()


def _grid(capi, ny, nx, M):
    terr = synth.make_terrain(ny, nx, seed=83)
    rm, sc = synth.ensemble_prior(83, M)
    g = capi.Grid(terr.z, terr.n)
    g.ensemble_init(M, rm, sc, synth.hyetograph_constant(90.0, 600.0))
    return g


def _march(capi, ny, nx, M, steps):
    with _grid(capi, ny, nx, M) as g:
        g.set_launch(8, 1)
        for n in steps:
            g.step(n)
        return [np.stack(g.get_state(m)) for m in range(M)], g.members()["t"]


@pytest.mark.parametrize("shape", [(1, 9, 1), (64, 131, 7), (305, 310, 1)])
def test_the_first_step_on_a_side_stream_while_the_default_stream_is_busy(capi, shape):
    """An ensemble whose steps stay on the chip takes its first steps on a
    non-blocking stream, with about a tenth of a second of work queued on the
    default stream before them."""
    import torch
    steps = (5, 30)
    ref, t = _march(capi, *shape, steps)
    side = torch.cuda.Stream()
    with _grid(capi, *shape) as g:
        torch.cuda._sleep(200_000_000)
        with torch.cuda.stream(side):
            for n in steps:
                g.step(n)
            g.sync()
            for m in range(shape[2]):
                assert np.array_equal(np.stack(g.get_state(m)), ref[m])
        assert np.array_equal(g.members()["t"], t)


@pytest.mark.parametrize("shape", [(64, 131, 7), (40, 129, 200)])
def test_the_first_steps_may_be_recorded_into_a_graph(capi, shape):
    """flood_step(n) only launches: it may be an ensemble's first call inside
    the capture of the caller's stream, on the chip (7 members) as on the march
    (200), and the graph's replays step the ensemble."""
    import torch
    n, replays = 6, 3
    ref, t = _march(capi, *shape, (n,) * replays)
    stream = torch.cuda.Stream()
    with _grid(capi, *shape) as g:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            g.step(n)
        with torch.cuda.stream(stream):
            for _ in range(replays):
                graph.replay()
            g.sync()
            for m in range(shape[2]):
                assert np.array_equal(np.stack(g.get_state(m)), ref[m])
        assert np.array_equal(g.members()["t"], t)
