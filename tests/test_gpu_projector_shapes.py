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
