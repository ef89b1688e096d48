"""The FP64 step of four overlapping kernels against the separate passes and the batched kernel, bit for
bit: every product that meets a sum is rounded explicitly, and the compensation sums are added in one
order.  So a reverse sweep, which recomputes its segments by the separate passes, sweeps the states
that the forward pass went through."""
from __future__ import annotations

import numpy as np
import pytest

import scenarios as S
from harness import make_lattice
from test_gpu_fp64_step import CASES

pytestmark = pytest.mark.gpu

SHAPES = dict(CASES)
SHAPES.update({
    # more boundary nodes than one block of 128 threads sums up in one round (2 x 17001 > 32768)
    "long_channel_17001x21": lambda: S.Scenario(name="l", nx=17001, ny=21, T_over_Tc=0.9, gx=3e-6, gy=-1e-6, r0=[4.0] * 30,
                                                 x0=list(np.random.default_rng(4).uniform(10, 16990, 30)),
                                                 y0=list(np.random.default_rng(5).uniform(5, 15, 30))),
    "interpolated": lambda: S.small_parity().with_(bc=S.BC_MIBC),
    "half_way": lambda: S.small_parity().with_(bc=S.BC_HBB, coll=S.COLL_BGK, tau=0.9),
    "gravity": lambda: S.c3_impact(128, 256),
})


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_04508_gb300 import build
    build.build()


@pytest.mark.parametrize("name", list(SHAPES))
def test_fp64_paths_give_the_same_bits(name):
    import paper_2203_04508_gb300 as G
    sc = SHAPES[name]()
    a, b = make_lattice(sc, fp64=True), make_lattice(sc, fp64=True)
    batch = G.Batch([sc.physics()], precision=G.LBM_FP64)
    batch.init([sc.droplets()])
    b.set_collide_kernel(0)
    for n in (1, 2, 11, 16):
        a.step(n)
        b.step(n)
        batch.step(n)
        pops = a.populations()
        assert np.array_equal(pops, b.populations()), n
        assert np.array_equal(pops, batch.instances[0].populations()), n
        assert a.mass() == b.mass()
        for u, v in zip(a.fields(), b.fields()):
            assert np.array_equal(u, v)
    assert np.array_equal(a.dM_history(), b.dM_history())
