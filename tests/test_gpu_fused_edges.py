"""The fused step's read-outs and its lattices' edges: arrays that are not 8-byte aligned and streams
other than the default one, diagnostics between steps, strips of 56 columns with the pseudopotential
force, and walked lattices whose rows are not whole 16-byte pieces -- against the separate passes, bit for
bit."""
from __future__ import annotations

import ctypes as C

import numpy as np
import pytest

import scenarios as S
from harness import make_lattice
from test_gpu_fused_step import PSEUDO, _box

pytestmark = pytest.mark.gpu

AB, AA = 0, 1


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_04508_gb300 import build
    build.build()


def _pair(sc, layout=AB):
    """A lattice on its default step and one on the separate passes."""
    import paper_2203_04508_gb300 as G
    a, b = (G.Lattice(sc.physics(), precision=G.LBM_FP32, layout=layout) for _ in range(2))
    for lat in (a, b):
        lat.init_droplets(sc.droplets())
    b.set_collide_kernel(0)
    return a, b


def _same(a, b):
    assert np.array_equal(a.populations(), b.populations())
    assert a.mass() == b.mass()
    for u, v in zip(a.fields(), b.fields()):
        assert np.array_equal(u, v)


@pytest.mark.parametrize("layout", [AB, AA])
@pytest.mark.parametrize("over", [{}, PSEUDO])
@pytest.mark.parametrize("misaligned", [(1, 0, 0), (0, 0, 1), (1, 1, 1)])
def test_read_out_into_arrays_that_are_not_8_byte_aligned(layout, over, misaligned):
    """At both lattice parities; a step after it starts from the same state."""
    import torch
    a, b = _pair(_box(93, 61, walls=1, **over), layout)
    n = a.nx * a.ny
    for steps in (0, 1, 2, 5):
        a.step(steps)
        b.step(steps)
        raw = [torch.full((n + 2,), -7.0, dtype=torch.float32, device="cuda") for _ in range(3)]
        torch.cuda.synchronize()
        a._c(a.lib.lbm_fields(a.ctx, *[C.c_void_p(t.data_ptr() + 4 * m) for t, m in zip(raw, misaligned)], 1))
        a.synchronize()
        for t, m, want in zip(raw, misaligned, b.fields()):
            got = t.cpu().numpy()
            assert np.array_equal(got[m:m + n].reshape(want.shape), want)
            assert (got[:m] == -7.0).all() and (got[m + n:] == -7.0).all()
    a.step(3)
    b.step(3)
    _same(a, b)


def test_read_out_on_another_stream():
    """The read-out runs after what that stream has queued and before what it queues next."""
    import torch
    a, b = _pair(S.small_parity())
    other = torch.cuda.Stream()
    for steps in (0, 3, 4):
        a.step(steps)
        b.step(steps)
        with torch.cuda.stream(other):
            busy = torch.randn(4096, 4096, device="cuda")
            for _ in range(8):
                busy = busy @ busy * 1e-3
            got = a.fields(on_device=True)
            copies = [2.0 * t for t in got]
            for t in got:
                t.zero_()
        other.synchronize()
        for u, v in zip(copies, b.fields()):
            assert np.array_equal(u.cpu().numpy(), 2.0 * v)
    a.step(2)
    b.step(2)
    _same(a, b)


@pytest.mark.parametrize("layout", [AB, AA])
def test_diagnostics_between_steps_with_the_pseudopotential_force(layout):
    a, b = _pair(_box(113, 61, walls=1, **PSEUDO), layout)
    for steps in (1, 4, 2, 9):
        a.step(steps)
        b.step(steps)
        assert a.max_speed() == b.max_speed()
        assert np.array_equal(a.column_density(56), b.column_density(56), equal_nan=True)   # NaN: solid
    _same(a, b)


@pytest.mark.parametrize("nx,walls", [(112, 0), (113, 1), (113, 0), (169, 1), (57, 0)])
def test_pseudopotential_strips(nx, walls):
    """Whole strips only, and a last strip of one column."""
    a, b = _pair(_box(nx, 47, walls=walls, **PSEUDO))
    for steps in (1, 2, 11):
        a.step(steps)
        b.step(steps)
        _same(a, b)


@pytest.mark.parametrize("layout", [AB, AA])
@pytest.mark.parametrize("over", [{}, PSEUDO])
@pytest.mark.parametrize("nx,ny,walls", [(2297, 2301, 0), (2302, 2290, 1)])
def test_walked_lattices_of_ragged_rows(layout, over, nx, ny, walls):
    """Strips at the edges load column by column (nx % 4 != 0)."""
    a, b = _pair(_box(nx, ny, walls=walls, **over), layout)
    for steps in (1, 4, 9):
        a.step(steps)
        b.step(steps)
        assert np.array_equal(a.populations(), b.populations())
    _same(a, b)
