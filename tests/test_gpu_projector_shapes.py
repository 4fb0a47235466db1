"""The projector's kernels at the sizes where their tiling can go wrong, through
the C ABI: volumes whose axes differ, detectors that end inside a set of 32 rows
or a block of columns, one-voxel axes, scans whose columns change major axis
inside a view, and non-finite voxels."""
import ctypes
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import torch
    from paper_2008_01567_gb300 import build, msf
    build.build()
    assert torch.cuda.is_available()
    return msf


def _geometry(M, nx, ny, nz, nt, nu, nv, views, fine=1.0):
    """A plan over any volume shape (unit voxels), the detector covering it with
    a margin; fine < 1 leaves the volume partly outside the fan."""
    R = 0.5 * math.hypot(nx, ny)
    dso, dsd = 4.0 * R + 1.0, 8.0 * R + 4.0
    du = fine * 2.2 * dsd * math.tan(math.asin(R / dso)) / nu
    dv = fine * 1.1 * nz * dsd / (dso - R) / nv
    dv = min(dv, 1.9 * dsd / math.sqrt(2.0) / max(1, nv - 1))
    ang = np.ascontiguousarray(0.37 + 2.0 * math.pi * np.arange(nt * views) / (nt * views) * 1.13)
    geom = M.msf_geom(nu, nv, views, du, dv, dso, dsd, ang.ctypes.data_as(ctypes.POINTER(ctypes.c_double)))
    return geom, M.msf_vol(nx, ny, nz, nt, 1.0), ang


SHAPES = [  # nx, ny, nz, nt, nu, nv, views, fine
    (1, 1, 1, 1, 1, 1, 1, 1.0), (33, 7, 5, 2, 9, 31, 3, 1.0), (8, 40, 31, 1, 65, 33, 7, 1.0), (40, 33, 64, 2, 7, 160, 4, 1.0),
    (17, 16, 129, 1, 30, 161, 5, 1.0), (24, 24, 3, 3, 40, 8, 6, 1.0), (31, 45, 26, 1, 50, 193, 5, 0.6), (20, 21, 70, 1, 12, 325, 3, 0.5)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("bad", [False, True], ids=["finite", "nonfinite"])
def test_forward_equals_the_direct_kernel(M, shape, bad):
    # the direct kernel reads the volume in its own layout, one ray per thread,
    # with the same operations in the same order: equal bit for bit, and a
    # non-finite voxel reaches the same rays
    import torch
    geom, vol, ang = _geometry(M, *shape)
    g = torch.Generator("cuda").manual_seed(5)
    x = torch.randn((vol.nt, vol.nz, vol.ny, vol.nx), device="cuda", generator=g)
    if bad:
        x.view(-1)[torch.tensor([0, x.numel() // 2, x.numel() - 1], device="cuda")] = float("inf")
    y, ref = (torch.full((vol.nt, geom.views, geom.nv, geom.nu), -1.0, device="cuda") for _ in range(2))
    L = M.lib()
    h = ctypes.c_void_p()
    assert L.msf_projector_create(ctypes.byref(geom), ctypes.byref(vol), ctypes.byref(h)) == 0, L.msf_last_error()
    try:
        assert L.msf_project_static(ctypes.byref(geom), ctypes.byref(vol), x.data_ptr(), ref.data_ptr(), None) == 0
        for cols, rows in ((16, 8), (32, 4), (64, 2)):
            assert L.msf_projector_set_tuning(h, cols, rows, 16) == 0
            assert L.msf_project(h, x.data_ptr(), y.data_ptr(), None) == 0
            torch.cuda.synchronize()
            assert torch.equal(torch.isnan(y), torch.isnan(ref))
            assert torch.equal(torch.nan_to_num(y, 7.0), torch.nan_to_num(ref, 7.0)), (cols, rows)
    finally:
        L.msf_projector_destroy(h)


def _oracle_At(y, geom, vol, ang):
    """A^T in FP64: the oracle's scatter over the plan's own shape."""
    import oracle
    out = np.zeros((vol.nt, vol.nz, vol.ny, vol.nx))
    for t in range(vol.nt):
        a = np.ascontiguousarray(ang[t * geom.views:(t + 1) * geom.views])
        oracle._L().or_project(oracle._p(out[t]), oracle._p(np.ascontiguousarray(y[t])), vol.nx, vol.ny, vol.nz, 1.0, geom.nu,
                               geom.nv, geom.du, geom.dv, geom.dso, geom.dsd, oracle._p(a), geom.views, 1)
    return out


# detectors of fine rows (up to 16 rows per voxel), of coarse rows (several voxels per row) and of fine columns
ADJ_SHAPES = SHAPES + [(12, 9, 33, 1, 20, 400, 3, 0.4), (15, 18, 96, 1, 25, 6, 4, 1.0), (13, 11, 40, 2, 250, 37, 3, 0.8)]


@pytest.mark.parametrize("shape", ADJ_SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_adjoint_matches_oracle_at_ragged_sizes(M, shape):
    import torch
    geom, vol, ang = _geometry(M, *shape)
    y = np.random.default_rng(6).standard_normal((vol.nt, geom.views, geom.nv, geom.nu)).astype(np.float32)
    ref = _oracle_At(y.astype(np.float64), geom, vol, ang)
    yg = torch.from_numpy(y).cuda()
    L = M.lib()
    h = ctypes.c_void_p()
    assert L.msf_projector_create(ctypes.byref(geom), ctypes.byref(vol), ctypes.byref(h)) == 0, L.msf_last_error()
    try:
        first = None
        for zrun in (8, 16, 32, 64):
            assert L.msf_projector_set_tuning(h, 32, 4, zrun) == 0
            x = torch.full((vol.nt, vol.nz, vol.ny, vol.nx), -1.0, device="cuda")
            assert L.msf_backproject(h, yg.data_ptr(), x.data_ptr(), None) == 0
            torch.cuda.synchronize()
            got = x.cpu().numpy().astype(np.float64)
            assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref), zrun   # the projector's tolerance
            first = x if first is None else first
            assert torch.equal(x, first), zrun
    finally:
        L.msf_projector_destroy(h)


def test_nonfinite_reading_reaches_its_own_footprint_only(M):
    import torch
    geom, vol, ang = _geometry(M, 20, 21, 30, 1, 24, 27, 4)
    y = np.zeros((1, geom.views, geom.nv, geom.nu), np.float32)
    y[0, 1, 13, 11] = 1.0
    ref = _oracle_At(y.astype(np.float64), geom, vol, ang)
    y[0, 1, 13, 11] = np.inf
    L = M.lib()
    h = ctypes.c_void_p()
    assert L.msf_projector_create(ctypes.byref(geom), ctypes.byref(vol), ctypes.byref(h)) == 0, L.msf_last_error()
    try:
        x = torch.zeros((1, vol.nz, vol.ny, vol.nx), device="cuda")
        assert L.msf_backproject(h, torch.from_numpy(y).cuda().data_ptr(), x.data_ptr(), None) == 0
        torch.cuda.synchronize()
        hit = ~np.isfinite(x.cpu().numpy())
    finally:
        L.msf_projector_destroy(h)
    w = ref / ref.max()
    assert hit[w > 1e-3].all() and not hit[w < -1e-9].any() and not (hit & (w == 0)).any()
