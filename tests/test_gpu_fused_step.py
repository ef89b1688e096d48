"""The fused step (the default of FP32 lattices on two population lattices) against the separate
passes: the same populations, masses and compensation histories bit for bit, on lattices at the
edges of its strips (56 or 60 columns a warp) and bands, walled and periodic, for both force
models, both equations of state and both collisions; and switching between the two paths."""
from __future__ import annotations

import numpy as np
import pytest

import scenarios as S
from harness import make_lattice

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_04508_gb300 import build
    build.build()


def _box(nx, ny, walls=0, **kw):
    """A drop beside a cylinder (where one fits) in an nx x ny box."""
    base = dict(name=f"box_{nx}x{ny}", nx=nx, ny=ny, walls=walls, T_over_Tc=0.7, x0=[0.3 * nx], y0=[0.45 * ny],
                r0=[max(2.0, 0.12 * min(nx, ny))])
    if min(nx, ny) >= 40:
        base.update(cx=[0.62 * nx + 0.21], cy=[0.55 * ny + 0.37], r=[0.17 * min(nx, ny)], dmu_w=[0.02])
    base.update(kw)
    return S.Scenario(**base)


PSEUDO = dict(force_model=S.FORCE_PSEUDO, k=1.0, kappa=0.0, T_over_Tc=0.7, dmu_w=[0.15])
CASES = {
    "walls_131x97": lambda: S.small_parity(),
    "smallest_5x5": lambda: S.Scenario(name="s", nx=5, ny=5, walls=0, T_over_Tc=0.9, x0=[2.1], y0=[2.6], r0=[1.5]),
    "walls_5x21": lambda: S.Scenario(name="w", nx=5, ny=21, T_over_Tc=0.9, x0=[2.5], y0=[10.3], r0=[2.0]),
    "one_strip_56": lambda: _box(56, 45),
    "one_strip_and_a_column": lambda: _box(57, 41, walls=1),
    "first_whole_strip_116": lambda: _box(116, 50),      # strip 1 ends at the lattice's last column but four
    "last_strip_of_one_column_113": lambda: _box(113, 47),
    "strips_of_60": lambda: _box(120, 43, **PSEUDO),
    "strips_of_60_and_a_column": lambda: _box(181, 49, walls=1, **PSEUDO),
    "bgk_periodic": lambda: _box(170, 66, coll=S.COLL_BGK, tau=1.0),
    "peng_robinson": lambda: S.e1_flat_drop(0.3, 60.0, nx=200, ny=120, r0=25.0),
    "ibc": lambda: _box(90, 70, walls=1, bc=S.BC_IBC),
    "gravity_impact": lambda: S.c3_impact(256, 512),
    "drops_1024": lambda: S.c2_fp32_single(),
}


@pytest.mark.parametrize("name", list(CASES))
def test_fused_step_equals_the_separate_passes(name):
    sc = CASES[name]()
    a, b = make_lattice(sc, fp64=False), make_lattice(sc, fp64=False)
    b.set_collide_kernel(0)
    assert a.launches_per_step() < b.launches_per_step()
    for n in (1, 2, 11, 16):
        a.step(n)
        b.step(n)
        assert np.array_equal(a.populations(), b.populations()), n
        assert a.mass() == b.mass()
    assert np.array_equal(a.dM_history(), b.dM_history())
    for u, v in zip(a.fields(), b.fields()):
        assert np.array_equal(u, v)


def test_full_size_impact():
    a, b = make_lattice(S.c3_impact(), fp64=False), make_lattice(S.c3_impact(), fp64=False)
    b.set_collide_kernel(1)
    for n in (1, 24):
        a.step(n)
        b.step(n)
    assert np.array_equal(a.populations(), b.populations())
    assert a.mass() == b.mass()


def test_switching_paths_and_reading_out_between_steps(tmp_path):
    """Read-outs, a checkpoint and changes of path between steps leave the fused step's values."""
    sc = S.small_parity()
    a, b, c = (make_lattice(sc, fp64=False) for _ in range(3))
    b.set_collide_kernel(0)
    for n in (3, 4, 9):
        a.step(n)
        a.fields()
        a.max_speed()
        a.column_density(5)
        b.step(n)
    c.step(3)
    c.profile_steps(4)
    c.save(str(tmp_path / "c.ckpt"))
    d = make_lattice(sc, fp64=False)
    d.load(str(tmp_path / "c.ckpt"))
    c.set_mu_kernel(3)
    c.step(9)
    d.step(9)
    assert np.array_equal(a.populations(), b.populations())
    assert np.array_equal(a.populations(), c.populations())
    assert np.array_equal(a.populations(), d.populations())


@pytest.mark.parametrize("walk", [False, True])
def test_fused_batch_equals_the_persistent_kernel_and_single_lattices(walk):
    """Instances of mixed sizes advanced by the fused step over flat item lists (tiles, and the walks
    that large batches take) against the persistent batched kernel (which a batch whose waits are
    bounded by the caller runs) and against a lattice of its own, bit for bit."""
    import paper_2203_04508_gb300 as G
    scs = [S.small_parity(), _box(64, 70, walls=1), _box(117, 61), S.e1_flat_drop(0.3, 60.0, nx=90, ny=75, r0=18.0)]
    if walk:
        scs = [_box(2100, 2001, walls=1), _box(2000, 2100), _box(1999, 2300)]
    a, b = (G.Batch([sc.physics() for sc in scs]) for _ in range(2))
    b.set_spin_limit((1 << 22) + 1)
    for batch in (a, b):
        batch.init([sc.droplets() for sc in scs])
    for n in (1, 13, 2):
        a.step(n)
        b.step(n)
        b.check()
    for k in range(len(scs)):
        one = make_lattice(scs[k], fp64=False)
        one.step(16)
        pops = one.populations()
        assert np.array_equal(a.instances[k].populations(), pops), k
        assert np.array_equal(b.instances[k].populations(), pops), k
        assert a.instances[k].mass() == one.mass() == b.instances[k].mass()
        assert np.array_equal(a.instances[k].dM_history(), one.dM_history())


@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("steps", [4, 7])
def test_a_stored_lattice_holds_the_bytes_of_the_separate_passes(layout, steps, tmp_path):
    """A checkpoint keeps the lattice as stored, padding and solid nodes' slots too."""
    import paper_2203_04508_gb300 as G
    files = []
    for k, sc in enumerate((S.small_parity(), _box(121, 60))):
        for kind in (None, 0):
            lat = G.Lattice(sc.physics(), precision=G.LBM_FP32, layout=layout)
            lat.init_droplets(sc.droplets())
            if kind is not None:
                lat.set_collide_kernel(kind)
            lat.step(steps)
            path = tmp_path / f"{k}_{kind}.ckpt"
            lat.save(str(path))
            files.append(path.read_bytes())
    assert files[0] == files[1]
    assert files[2] == files[3]
