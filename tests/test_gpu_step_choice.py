"""Choosing the kernels of the separate passes, and going back to the step lbm_build_links chose."""
from __future__ import annotations

import numpy as np
import pytest

import scenarios as S

pytestmark = pytest.mark.gpu

FP32, FP64, AB, AA = 0, 1, 0, 1
PSEUDO = dict(dmu_w=[0.15, -0.15], force_model=S.FORCE_PSEUDO, k=1.0, kappa=0.0, T_over_Tc=0.7)


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_04508_gb300 import build
    build.build()


@pytest.mark.parametrize("precision,layout,over", [(FP32, AB, {}), (FP32, AA, {}), (FP32, AB, PSEUDO), (FP32, AA, PSEUDO),
                                                   (FP64, AB, {}), (FP32, AB, dict(eos=S.EOS_NONE))])
def test_reset_goes_back_to_the_default_step(precision, layout, over):
    import paper_2203_04508_gb300 as G
    sc = S.small_parity().with_(**over)
    a, b = (G.Lattice(sc.physics(), precision=precision, layout=layout) for _ in range(2))
    for lat in (a, b):
        lat.init_droplets(sc.droplets())
    launches, kind = a.launches_per_step(), a.collide_kernel()
    choices = [lambda: b.set_collide_kernel(0), lambda: b.set_mu_kernel(1)]
    if precision == FP32:
        choices.append(lambda: b.set_collide_kernel(1))
        if layout == AB and not over:
            choices.append(lambda: b.set_mu_kernel(3))
    for choose in choices:
        for n in (3, 8):
            choose()
            a.step(n)
            b.step(n)
            b.reset_kernels()
            assert b.launches_per_step() == launches and b.collide_kernel() == kind
            a.step(n)
            b.step(n)
            assert np.array_equal(a.populations(), b.populations())
            assert a.mass() == b.mass()
            for u, v in zip(a.fields(), b.fields()):
                assert np.array_equal(u, v)
    b.reset_kernels()   # nothing to undo
    assert b.launches_per_step() == launches
