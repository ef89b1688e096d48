"""Choosing the kernels of the separate passes, and going back to the step lbm_build_links chose."""
from __future__ import annotations

import numpy as np
import pytest

import scenarios as S
from test_gpu_fused_step import _box

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


@pytest.mark.parametrize("precision,layout,over", [(FP32, AB, {}), (FP32, AA, {}), (FP32, AB, PSEUDO), (FP64, AB, {})])
def test_profiled_steps_run_the_kernels_of_the_step(precision, layout, over):
    """lbm_profile_steps times what lbm_step runs: the fused step has no density or chemical-potential
    kernel of its own, the FP64 one no layer kernel; the values and the state are lbm_step's."""
    import paper_2203_04508_gb300 as G
    sc = S.small_parity().with_(**over)
    a, b = (G.Lattice(sc.physics(), precision=precision, layout=layout) for _ in range(2))
    for lat in (a, b):
        lat.init_droplets(sc.droplets())
    for n in (3, 4, 1):
        a.step(n)
        ms = b.profile_steps(n)
        zero = {0, 2} if precision == FP32 else {1}
        assert all((v == 0.0) == (k in zero) for k, v in enumerate(ms)), ms
        assert np.array_equal(a.populations(), b.populations())
        assert a.mass() == b.mass()
        a.step(2)
        b.step(2)
        assert np.array_equal(a.populations(), b.populations())
    assert np.array_equal(a.dM_history(), b.dM_history())
    b.set_collide_kernel(0)      # the separate passes' five phases
    ms = b.profile_steps(2)
    assert (ms[[0, 1, 3, 4]] > 0).all()


def _batch(precision=FP32, layout=AB, walked=False):
    import paper_2203_04508_gb300 as G
    scs = [S.small_parity(), S.small_parity(seed=11, nx=97, ny=83)]
    if walked:   # large enough for the batch's walks
        scs = [_box(2100, 2001, walls=1), _box(2000, 2100), _box(1999, 2300)]
    b = G.Batch([sc.physics() for sc in scs], precision=precision, layout=layout)
    b.init([sc.droplets() for sc in scs])
    return scs, b


def test_a_poll_budget_does_not_choose_the_batch_kernel():
    """Any budget but zero leaves the fused step, which waits for nothing, in place."""
    _, b = _batch()
    assert b.kernel() == 0
    for polls in (1, 100, (1 << 22) - 1, (1 << 22) + 1, 1 << 30):
        b.set_spin_limit(polls)
        assert b.kernel() == 0
    b.step(3)
    b.check()
    b.set_spin_limit(0)
    assert b.kernel() == 1
    b.set_spin_limit(1 << 22)
    assert b.kernel() == 0
    b.instances[1].set_mu_kernel(1)
    assert b.kernel() == 1
    b.instances[1].reset_kernels()
    assert b.kernel() == 0
    for kw in (dict(precision=FP64), dict(layout=AA)):
        assert _batch(**kw)[1].kernel() == 1


@pytest.mark.parametrize("walked", [False, True])
def test_the_persistent_kernel_by_choice_and_after_a_timeout(walked):
    """The persistent kernel against the fused step (tiles and walks) over changes between them, and
    again after its barriers gave up."""
    from paper_2203_04508_gb300 import LbmError
    scs, a = _batch(walked=walked)
    b = _batch(walked=walked)[1]
    if b.info()["grid"] >= 2:
        b.set_spin_limit(0)
        b.step(3)
        with pytest.raises(LbmError):
            b.check()
        b.set_spin_limit(1 << 22)
        b.init([sc.droplets() for sc in scs])
    for n, kind in ((1, 1), (13, 0), (2, 1), (5, 1), (8, 0)):
        b.set_kernel(kind)
        assert b.kernel() == kind
        a.step(n)
        b.step(n)
        b.check()
        for x, y in zip(a.instances, b.instances):
            assert np.array_equal(x.populations(), y.populations())
            assert x.mass() == y.mass()
            for u, v in zip(x.fields(), y.fields()):
                assert np.array_equal(u, v)
    for x, y in zip(a.instances, b.instances):
        assert np.array_equal(x.dM_history(), y.dM_history())
    with pytest.raises(LbmError):
        b.set_kernel(2)


def test_the_autotuner_times_the_persistent_kernel():
    """Its shapes are the persistent kernel's: on a batch whose steps are fused the trials run that
    kernel all the same -- with a budget of one poll its barriers give up, which only they can."""
    from paper_2203_04508_gb300 import LbmError
    scs, b = _batch()
    if b.info()["grid"] < 2:
        pytest.skip("a one-block grid never waits")
    b.set_spin_limit(1)
    assert b.kernel() == 0
    with pytest.raises(LbmError) as e:
        b.autotune(2)
    assert e.value.status == 6
    assert b.kernel() == 0
    b.set_spin_limit(1 << 22)
    b.init([sc.droplets() for sc in scs])
    r = b.autotune(2)
    assert b.kernel() == 0
    tiles = {k: v for k, v in r["ms"].items() if "x" in k}
    assert r["ms"][r["tile"]] == min(tiles.values())
    b.init([sc.droplets() for sc in scs])
    a = _batch()[1]
    a.step(9)
    b.step(9)
    for x, y in zip(a.instances, b.instances):
        assert np.array_equal(x.populations(), y.populations())
