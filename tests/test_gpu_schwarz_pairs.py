"""The FP32 local solves with two lines per thread (large meshes, n a multiple of 4) against the FP64 application, which
has one line per thread, on meshes on both sides of the rule's line, the last CTA partly filled."""

import pytest

pytestmark = pytest.mark.gpu

TOL32 = 2e-5  # relative L2, as for the FP32 application elsewhere


@pytest.mark.parametrize("N", [3, 7])
@pytest.mark.parametrize("shape", [(21, 21, 23), (22, 21, 21), (23, 19, 23)])  # 10,143, 9702 and 10,051 elements
def test_fp32_against_fp64(N, shape):
    import torch

    import paper_2109_03592_gb300 as sem
    m = sem.Mesh(dict(kind="box", nx=shape[0], ny=shape[1], nz=shape[2], N=N))
    sw = sem.Schwarz(m, h2=3.0)
    g = torch.Generator(device="cuda").manual_seed(N)
    f = torch.randn(m.shape, generator=g, dtype=torch.float64, device="cuda")
    r = m.rhs(f, torch.empty_like(f))
    r /= r.norm()
    z, z32 = torch.empty_like(r), torch.empty(m.shape, dtype=torch.float32, device="cuda")
    sw.apply(r, z, prec=sem.FP64)
    sw.apply(r.float(), z32, prec=sem.FP32)
    assert float((z32.double() - z).norm() / z.norm()) < TOL32
