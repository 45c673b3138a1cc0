"""Device memory of a mesh: the FP64 factors are kept in one form, whichever kernels read them, also while it is built."""

import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# per local point: coordinates 24, factors 48 (FP64 or fixed point), 24 (FP32), mass 8, 4 and (fixed point) 8, assembled
# diagonals 16, flags 1, gather-scatter ids at most 5
MESH = 138
COEF = 80 + 28  # factors 48 and 24, diagonal 8; mass 8, 4 and 8, diagonal 8


def _bytes(m):
    import paper_2109_03592_gb300 as sem
    info = sem.sem.MeshInfo()
    assert sem.lib().sem_mesh_info(m._h, ctypes.byref(info)) == 0
    return info.dev_bytes


def _mesh(monkeypatch, variant, n=20, N=7):
    import paper_2109_03592_gb300 as sem
    if variant is not None:
        monkeypatch.setenv("SEM_FP64_VARIANT", str(variant))
    return sem.Mesh(dict(kind="box", nx=n, ny=n, nz=n, N=N))


@pytest.mark.parametrize("variant", [None, 0, 1, 4, 5])
def test_one_form_of_the_factors(variant, monkeypatch):
    import torch
    m = _mesh(monkeypatch, variant)
    small = 64 * m.E + (1 << 20)  # per element, tables
    base = _bytes(m)
    assert base <= MESH * m.n_local + small
    one = torch.ones(m.shape, dtype=torch.float64, device="cuda")
    for h1, h2 in [(one, one), (one, None), (None, one), (one * 1e80, one), (None, one * 1e80), (one, one * 1e80)]:
        m.set_coefficients(h1, h2)
        assert _bytes(m) <= base + COEF * m.n_local + small
    m.set_coefficients(None, None)
    assert _bytes(m) == base


def test_build_needs_little_more_than_the_mesh(monkeypatch):
    import torch
    import paper_2109_03592_gb300 as sem
    n, N = 40, 7
    _mesh(monkeypatch, None, 2)  # the library's own start-up
    points = n ** 3 * (N + 1) ** 3
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    hold = torch.empty(free - 165 * points - (400 << 20), dtype=torch.uint8, device="cuda")
    try:
        m = _mesh(monkeypatch, None, n, N)
        assert m.ax_variant(sem.FP64) in (4, 5)
        u = torch.from_numpy(np.random.default_rng(0).standard_normal(1 << 10)).cuda()
        assert float(u.norm()) > 0
    finally:
        del hold
        torch.cuda.empty_cache()


def test_one_form_of_the_pressure_factors(monkeypatch):
    import torch
    m = _mesh(monkeypatch, None, 12, 5)
    small = 64 * m.E + (1 << 20)
    base, points = _bytes(m), m.pressure_size()
    p = torch.ones(m.pressure_shape, dtype=torch.float64, device="cuda")
    m.pressure_apply(p, torch.empty_like(p))
    assert _bytes(m) <= base + 72 * points + 8 * m.n_local + small
    m.pressure_diag(torch.empty_like(p))
    assert _bytes(m) <= base + 80 * points + 8 * m.n_local + small
    m.pressure_apply_f32(p.float(), torch.empty(m.pressure_shape, dtype=torch.float32, device="cuda"))
    assert _bytes(m) <= base + 116 * points + 12 * m.n_local + small


def test_an_allocation_failure_is_reported_once(monkeypatch):
    import torch
    import paper_2109_03592_gb300 as sem
    _mesh(monkeypatch, None, 2)
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (1 << 30), dtype=torch.uint8, device="cuda")
    try:
        with pytest.raises(sem.SemError):
            _mesh(monkeypatch, None, 40)  # 4.5 GB
        _mesh(monkeypatch, None, 4)  # the next call knows nothing of it
    finally:
        del hold
        torch.cuda.empty_cache()
