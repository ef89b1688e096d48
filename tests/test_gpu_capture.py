"""Calls on a stream that the caller captures into a CUDA graph: what is recorded does not run, so
the state's planes stay as they were, and a replay works on the populations it finds."""
from __future__ import annotations

import numpy as np
import pytest

import scenarios as S

pytestmark = pytest.mark.gpu

FP32, FP64, AB, AA = 0, 1, 0, 1
KINDS = [(FP32, AB, S.FORCE_CHEMPOT), (FP32, AA, S.FORCE_CHEMPOT), (FP32, AB, S.FORCE_PSEUDO), (FP64, AB, S.FORCE_CHEMPOT)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_04508_gb300 import build
    build.build()


def _scenario(force):
    sc = S.small_parity()
    if force == S.FORCE_PSEUDO:
        sc = sc.with_(dmu_w=[0.15, -0.15], force_model=S.FORCE_PSEUDO, k=1.0, kappa=0.0, T_over_Tc=0.7)
    return sc


def _lattice(sc, precision, layout):
    import paper_2203_04508_gb300 as G
    lat = G.Lattice(sc.physics(), precision=precision, layout=layout)
    lat.init_droplets(sc.droplets())
    return lat


@pytest.mark.parametrize("precision,layout,force", KINDS)
@pytest.mark.parametrize("steps", [0, 2])
def test_a_recorded_read_out_leaves_the_state_and_reads_what_it_finds(precision, layout, force, steps):
    import torch
    sc = _scenario(force)
    a, b = (_lattice(sc, precision, layout) for _ in range(2))
    for lat in (a, b):
        lat.step(steps)
        lat.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=a.stream):
        out = a.fields(on_device=True)
    # the steps that follow start from the state, not from planes that were only recorded
    a.step(4)
    b.step(4)
    assert np.array_equal(a.populations(), b.populations())
    # another state in the same place, not stepped or read before the replay
    drops = sc.droplets()
    drops = dict(drops, r0=[0.8 * r for r in drops["r0"]])
    for lat in (a, b):
        lat.init_droplets(drops)
    torch.cuda.synchronize()
    graph.replay()
    torch.cuda.synchronize()
    for u, v in zip(out, b.fields()):
        assert np.array_equal(u.cpu().numpy(), v)
    a.step(3)
    b.step(3)
    assert np.array_equal(a.populations(), b.populations())


@pytest.mark.parametrize("warm", [0, 4])
@pytest.mark.parametrize("precision", [FP32, FP64])
def test_a_recorded_batch_step(precision, warm):
    """lbm_batch_step under the caller's capture, replayed between steps that are not recorded."""
    import paper_2203_04508_gb300 as G
    import torch
    scs = [S.small_parity(), S.small_parity(seed=11, nx=97, ny=83)]
    a, b = (G.Batch([sc.physics() for sc in scs], precision=precision) for _ in range(2))
    for batch in (a, b):
        batch.init([sc.droplets() for sc in scs])
        batch.step(warm)
        batch.synchronize()

    def same():
        for x, y in zip(a.instances, b.instances):
            assert np.array_equal(x.populations(), y.populations())
            for u, v in zip(x.fields(), y.fields()):
                assert np.array_equal(u, v)

    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=a.stream):
        a.step(4)
    for between in (0, 6, 2):
        graph.replay()
        torch.cuda.synchronize()
        b.step(4)
        same()
        a.step(between)
        b.step(between)
        same()
    a.check()
