"""The fused step of one lattice in AA order against the one of two lattices: the same populations,
masses and compensation histories bit for bit, on lattices at the edges of its strips (56 columns) and
bands, and on lattices that are walked, whose strips hand their outermost columns' populations on
(a last strip of one column; nx a multiple of 56; walls and periodic)."""
from __future__ import annotations

import numpy as np
import pytest

import scenarios as S
from harness import make_lattice
from test_gpu_fused_step import CASES, PSEUDO, _box

pytestmark = pytest.mark.gpu

SHAPES = dict(CASES)
SHAPES.update({
    "walked_a_column_more_2297x2301": lambda: _box(2297, 2301),
    "walked_whole_strips_2296x2310": lambda: _box(2296, 2310, walls=1),
    "walked_pseudo": lambda: _box(2360, 2290, **PSEUDO),
    "walked_two_narrow_strips_57x10701": lambda: _box(57, 10701, walls=1, x0=[28.0], y0=[60.0], r0=[9.0], cx=[30.2],
                                                      cy=[5000.4], r=[11.0], dmu_w=[0.02]),
    "walked_narrowest_5x21300": lambda: _box(5, 21300, r0=[3.0]),
})


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_04508_gb300 import build
    build.build()


@pytest.mark.parametrize("name", list(SHAPES))
def test_aa_step_equals_two_lattices(name):
    import paper_2203_04508_gb300 as G
    sc = SHAPES[name]()
    a = make_lattice(sc, fp64=False)
    b = G.Lattice(sc.physics(), precision=G.LBM_FP32, layout=G.LBM_LAYOUT_AA)
    b.init_droplets(sc.droplets())
    assert b.launches_per_step() <= 3
    for n in (1, 2, 10) if a.nx * a.ny > 100000 else (1, 2, 11, 16):
        a.step(n)
        b.step(n)
        assert np.array_equal(a.populations(), b.populations()), n
        assert a.mass() == b.mass()
        for u, v in zip(a.fields(), b.fields()):
            assert np.array_equal(u, v)
    assert np.array_equal(a.dM_history(), b.dM_history())
    # to the separate passes and on
    b.set_collide_kernel(0)
    a.step(3)
    b.step(3)
    assert np.array_equal(a.populations(), b.populations())
