"""The cached choice of kernels: a mesh whose factors have no fixed-point form must not decide for those that have one."""

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,nx", [(6, 600), (8, 150)])
def test_a_mesh_out_of_range_does_not_choose_for_others(N, nx):
    import paper_2109_03592_gb300 as sem
    far = sem.Mesh(dict(kind="box", nx=nx, ny=1, nz=1, N=N, lx=1e75 * nx, ly=1e75, lz=1e75))  # factors above 2^200
    near = sem.Mesh(dict(kind="box", nx=nx, ny=1, nz=1, N=N, lx=1.0 * nx, ly=1.0, lz=1.0))
    assert far.ax_variant(sem.FP64) in (0, 1)
    assert near.ax_variant(sem.FP64) in (4, 5) and not near.fp64_double_float()
    assert sem.Mesh(dict(kind="box", nx=nx, ny=1, nz=1, N=N, lx=1e75 * nx, ly=1e75, lz=1e75)).ax_variant(sem.FP64) in (0, 1)
