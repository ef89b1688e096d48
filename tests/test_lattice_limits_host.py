"""The largest lattices that 32-bit plane offsets reach.  No GPU is needed."""
import ctypes as C

import pytest

import scenarios as S


@pytest.mark.parametrize("precision,per_line", [(0, 32), (1, 16)])
def test_padded_planes_beyond_32_bit_offsets_are_refused(precision, per_line):
    """Rows are padded to 128 bytes: nine planes of a narrow lattice pass 2^31 values long before it has
    2e8 nodes, and the kernels' offsets would wrap.  The largest that fits is accepted."""
    from paper_2203_04508_gb300 import _abi, build
    from paper_2203_04508_gb300.lattice import make_config
    build.build()
    lib = _abi.load()

    def status(nx, ny):
        c, keep = make_config(S.Scenario(name="narrow", nx=nx, ny=ny, walls=0).physics(), precision)
        n = C.c_size_t()
        return lib.lbm_workspace_size(C.byref(c), C.byref(n))

    most = (2 ** 31 - 1) // (9 * per_line)
    assert status(5, most) == _abi.LBM_OK
    assert status(5, most + 1) == _abi.LBM_EINVAL
    assert status(5, 40000000) == _abi.LBM_EINVAL
    assert status(20000, 10000) == _abi.LBM_OK
