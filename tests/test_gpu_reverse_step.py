"""The FP32 reverse step (four kernels, recomputation by the fused step) against the FP64 one (the
separate kernels) from the same state and seeds, on lattices at the edges of its blocks; a repeated
sweep (replayed) against the first (issued); the forward state after a sweep.

Bounds: a step and its reverse are about 60 roundings deep, so after 4 + 4 steps FP32 is
2^-24 * 480 = 3e-5 of the largest value off at the most; 1e-4 leaves a factor of three.  dJ/dc comes
from differences of neighbouring populations a thousandth of the populations' size: 1e-3 of the
largest."""
from __future__ import annotations

import numpy as np
import pytest

import scenarios as S
from harness import make_lattice
from test_gpu_fused_step import _box

pytestmark = pytest.mark.gpu

CASES = {
    "walls_131x97": lambda: S.small_parity(),
    "smallest_5x5": lambda: S.Scenario(name="s", nx=5, ny=5, walls=0, T_over_Tc=0.9, x0=[2.1], y0=[2.6], r0=[1.5]),
    "walls_5x21": lambda: S.Scenario(name="w", nx=5, ny=21, T_over_Tc=0.9, x0=[2.5], y0=[10.3], r0=[2.0]),
    "one_block_56x48": lambda: _box(56, 48),
    "a_column_and_a_row_more_57x49": lambda: _box(57, 49, walls=1),
    "bgk_periodic": lambda: _box(170, 66, coll=S.COLL_BGK, tau=1.0),
    "peng_robinson": lambda: S.e1_flat_drop(0.3, 60.0, nx=200, ny=120, r0=25.0),
    "ibc": lambda: _box(90, 70, walls=1, bc=S.BC_IBC),
    "mibc": lambda: _box(90, 70, bc=S.BC_MIBC),
    "hbb": lambda: _box(113, 70, bc=S.BC_HBB),
    "no_eos": lambda: _box(60, 50, eos=S.EOS_NONE, walls=1),
}


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_04508_gb300 import build
    build.build()


def _close(a, b, rel, what):
    scale = np.abs(b).max() if b.size else 0.0
    assert (np.abs(a - b) <= rel * scale).all(), (what, np.abs(a - b).max() if a.size else 0, scale)


@pytest.mark.parametrize("name", list(CASES))
def test_fp32_reverse_step_against_fp64(name):
    import torch
    sc = CASES[name]()
    rng = np.random.default_rng(3)
    drho, df = rng.standard_normal((sc.ny, sc.nx)), rng.standard_normal((9, sc.ny, sc.nx))
    out = {}
    for fp64 in (False, True):
        lat = make_lattice(sc, fp64=fp64)
        lat.step(2)
        lat.forward_checkpointed(4, 3)     # a segment of three steps and one of one
        before = lat.populations().copy()
        runs = [lat.adjoint(drho=torch.tensor(drho), df=torch.tensor(df), want_df0=True) for _ in range(2)]
        assert np.array_equal(lat.populations(), before)
        lat.step(3)
        ref = make_lattice(sc, fp64=fp64)
        ref.step(9)
        assert np.array_equal(lat.populations(), ref.populations())
        out[fp64] = [(g, d.cpu().numpy().astype(np.float64)) for g, d in runs]
    n = len(sc.cx)
    for g, d in out[False]:
        g64, d64 = out[True][0]
        _close(d, d64, 1e-4, "dJ/df0")
        _close(g[:n + 1], g64[:n + 1], 1e-4, "dJ/d dmu")
        if sc.eos != S.EOS_NONE:   # (a uniform fluid at rest: dJ/dc is zero, FP64's 1e-16 its rounding)
            _close(g[n + 1:], g64[n + 1:], 1e-3, "dJ/dc")
