"""The plan's lines along z share their margins: a volume of few slices takes no more
than the 16 bytes per voxel of a z-paired copy, and the margins keep a line's taps and
windows from its neighbours (against the oracle and the direct kernel in
test_gpu_projector_shapes.py; here the sizes at which a line fills its pitch)."""
import ctypes

import numpy as np
import pytest

from tests.test_gpu_projector_shapes import _geometry, _oracle_At

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import torch
    from paper_2008_01567_gb300 import build, msf
    build.build()
    assert torch.cuda.is_available()
    return msf


# two zeros between lines of 4k + 2 voxels and four between lines of 4k rows, the least there are
@pytest.mark.parametrize("nz,nv", [(1, 1), (2, 4), (3, 5), (6, 8), (10, 12), (34, 36)])
def test_plans_of_few_slices(M, nz, nv):
    import torch
    shape = (21, 18, nz, 2, 26, nv, 5)
    geom, vol, ang = _geometry(M, *shape)
    L, h = M.lib(), ctypes.c_void_p()
    assert L.msf_projector_create(ctypes.byref(geom), ctypes.byref(vol), ctypes.byref(h)) == 0, L.msf_last_error()
    try:
        N, G = 21 * 18 * nz * 2, 2 * 5
        assert L.msf_projector_bytes(h) <= 16 * N + 4 * G * 26 * (nv + 7) + G * (8 + 8 + 4 + 32 * 26) + 4 * (nz + 24)
        g = torch.Generator("cuda").manual_seed(9)
        x = torch.randn((2, nz, 18, 21), device="cuda", generator=g)
        y, ref = (torch.full((2, 5, nv, 26), -1.0, device="cuda") for _ in range(2))
        assert L.msf_project_static(ctypes.byref(geom), ctypes.byref(vol), x.data_ptr(), ref.data_ptr(), None) == 0
        assert L.msf_project(h, x.data_ptr(), y.data_ptr(), None) == 0
        torch.cuda.synchronize()
        assert torch.equal(y, ref)
        e = torch.randn(y.shape, device="cuda", generator=g)
        assert L.msf_backproject(h, e.data_ptr(), x.data_ptr(), None) == 0
        torch.cuda.synchronize()
        at = _oracle_At(e.cpu().numpy().astype(np.float64), geom, vol, ang)
        assert np.linalg.norm(x.cpu().numpy() - at) <= 1e-5 * np.linalg.norm(at)   # the projector's tolerance
    finally:
        L.msf_projector_destroy(h)
