"""GPU readout: states into device memory (odd sizes, arrays off the 16-byte
boundary, overlapping arrays), gauge lists on both sides of the launch-argument
limit, the filter's outputs in host or device memory, and the batch's volumes,
each bit for bit what the host copies say."""
import numpy as np
import pytest

import oracle
from paper_2302_08341_gb300 import synth
from tests.gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def capi():
    return require_gpu()


@pytest.mark.parametrize("shape", [(1, 1), (3, 4), (5, 257), (65, 128)])
@pytest.mark.parametrize("shift", [0, 1])
def test_state_into_device_memory(capi, shape, shift):
    import torch
    ny, nx = shape
    n = ny * nx
    terr = synth.make_terrain(ny, nx, seed=5)
    M = 3
    rm, sc = synth.ensemble_prior(5, M)
    h0 = np.random.default_rng(5).uniform(0.0, 0.2, (M, ny, nx)).astype(np.float32)
    L, s = capi.lib(), capi.stream_handle(None)
    with capi.Grid(terr.z, terr.n) as g:
        g.ensemble_init(M, rm, sc, synth.hyetograph_constant(60.0, 600.0), h0=h0)
        for _ in range(2):
            g.step(3)
            for m in range(M):
                host = g.get_state(m)
                buf = torch.full((3 * n + 8,), -1.0, device="cuda")
                outs = [buf[shift + k * n:shift + (k + 1) * n] for k in range(3)]
                assert L.flood_get_state(g.h, m, *(capi.ptr(o) for o in outs), s) == capi.FLOOD_OK
                torch.cuda.synchronize()
                for o, want in zip(outs, host):
                    assert np.array_equal(o.cpu().numpy().reshape(ny, nx), want)
                assert float(buf[:shift].sum() + buf[shift + 3 * n:].sum()) == -8.0
                # one array for all three: the last one stays, as with copies
                one = torch.empty(n, device="cuda")
                assert L.flood_get_state(g.h, m, *[capi.ptr(one)] * 3, s) == capi.FLOOD_OK
                torch.cuda.synchronize()
                assert np.array_equal(one.cpu().numpy().reshape(ny, nx), host[2])


@pytest.mark.parametrize("G", [1, 64, 65])
def test_gauges_and_filter_outputs(capi, G):
    import torch
    ny, nx, M = 20, 30, 7
    terr = synth.make_terrain(ny, nx, seed=6)
    rm, sc = synth.ensemble_prior(6, M)
    rng = np.random.default_rng(6)
    cells = rng.integers(0, ny * nx, G).astype(np.int32)
    y = rng.uniform(0.05, 0.15, (M, G)).astype(np.float32)
    d = rng.uniform(0.08, 0.12, G)
    h0 = rng.uniform(0.0, 0.2, (M, ny, nx)).astype(np.float32)
    got = []
    for device in (False, True):
        with capi.Grid(terr.z, terr.n) as g:
            g.ensemble_init(M, rm, sc, synth.hyetograph_constant(60.0, 600.0), h0=h0)
            assert np.array_equal(g.gauge_sample(cells), h0.reshape(M, -1)[:, cells])
            out = None
            if device:
                out = dict(weights=torch.zeros(M, dtype=torch.float64, device="cuda"),
                           idx=torch.zeros(M, dtype=torch.int32, device="cuda"),
                           neff=torch.zeros(1, dtype=torch.float64, device="cuda"),
                           resampled=torch.zeros(1, dtype=torch.int32, device="cuda"))
            u, beta = synth.pf_draws(6, 1, M)
            r = g.pf_assimilate(d, 0.05, u, beta, y=y, outputs=out)
            torch.cuda.synchronize()
            r = out if device else r
            got.append([np.asarray(r[k].cpu() if device else r[k]).ravel()
                        for k in ("weights", "idx", "neff", "resampled")])
            mem = g.members()
            assert np.array_equal(mem["steps"], np.zeros(M)) and mem["weights"].shape == (M,)
    for a, b in zip(*got):
        assert np.array_equal(a, b)


def test_batch_volumes_and_states_on_the_device(capi):
    import torch
    shapes = [(16, 20), (17, 33), (1, 5), (100, 129)]
    terrs = [synth.make_terrain(ny, nx, seed=60 + k) for k, (ny, nx) in enumerate(shapes)]
    hys = [synth.hyetograph_constant(60.0, 120.0)] * len(shapes)
    one = np.ones(len(shapes), np.float32)
    with capi.Batch([t.z for t in terrs], [t.n for t in terrs]) as b:
        b.init(hys, one, one, np.full(len(shapes), 60.0))
        b.step(30.0)
        mem = b.members()
        for i, (ny, nx) in enumerate(shapes):
            host = b.get_state(i)
            outs = [torch.empty(ny, nx, device="cuda") for _ in range(3)]
            assert capi.lib().flood_batch_get_member_state(b.h, i, 0, *(capi.ptr(o) for o in outs),
                                                           capi.stream_handle(None)) == capi.FLOOD_OK
            for o, want in zip(outs, host):
                assert np.array_equal(o.cpu().numpy(), want)
            # FP64 sums of at most 1.3e4 values in another order: 1.3e4 * 2^-53
            want = oracle.storage(host[0].astype(np.float64), 1.0) * capi.Params.default().dx ** 2
            assert abs(mem["storage"][i] - want) <= 2e-12 * max(want, 1e-30)
