"""The FP64 step of four overlapping kernels (the default of FP64 lattices on two population
lattices) against the separate passes, on lattices at the edges of its blocks of 128 x 1 and 32 x 4
nodes: populations, masses, compensation histories and read-outs.

Both form the same sums; a compiler may contract the link rule's differently, so they may differ by
roundings: 2^-53 times some 60 roundings a step over 30 steps, 2e-13 of the largest value; bound 1e-12."""
from __future__ import annotations

import numpy as np
import pytest

import scenarios as S
from harness import make_lattice
from test_gpu_fused_step import _box

pytestmark = pytest.mark.gpu

CASES = {
    "smallest_5x5": lambda: S.Scenario(name="s", nx=5, ny=5, walls=0, T_over_Tc=0.9, x0=[2.1], y0=[2.6], r0=[1.5]),
    "walls_5x21": lambda: S.Scenario(name="w", nx=5, ny=21, T_over_Tc=0.9, x0=[2.5], y0=[10.3], r0=[2.0]),
    "blocks_128x48": lambda: _box(128, 48, coll=S.COLL_BGK, tau=1.0),
    "a_column_and_a_row_more_129x49": lambda: _box(129, 49, walls=1),
    "peng_robinson_ibc": lambda: S.e1_flat_drop(0.3, 60.0, nx=200, ny=120, r0=25.0).with_(bc=S.BC_IBC),
    "parity_131x97": lambda: S.small_parity(),
}


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_04508_gb300 import build
    build.build()


def _close(a, b):
    a, b = np.asarray(a), np.asarray(b)
    assert (np.abs(a - b) <= 1e-12 * np.abs(b).max()).all(), np.abs(a - b).max()


@pytest.mark.parametrize("name", list(CASES))
def test_fp64_step_equals_the_separate_passes(name):
    sc = CASES[name]()
    a, b = make_lattice(sc, fp64=True), make_lattice(sc, fp64=True)
    b.set_collide_kernel(0)
    assert a.launches_per_step() < b.launches_per_step()
    for n in (1, 2, 11, 16):
        a.step(n)
        b.step(n)
        _close(a.populations(), b.populations())
        assert a.mass()[0] == pytest.approx(b.mass()[0], rel=1e-12)
        for u, v in zip(a.fields(), b.fields()):
            assert (np.abs(u - v) <= 1e-11 * max(np.abs(v).max(), 1e-3)).all()   # v: a difference of populations
    scale = np.abs(a.populations()).max() * sc.nx
    assert (np.abs(a.dM_history() - b.dM_history()) <= 1e-12 * scale).all()
    # from one path to the other and on
    a.set_collide_kernel(0)
    a.step(3)
    b.step(3)
    _close(a.populations(), b.populations())
