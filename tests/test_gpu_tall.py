"""Tall volumes of a small cross-section, which take the launches that cubes of test
size do not: every number of voxels per lane, several blocks along z and several chunks
of detector rows, for A, A^T and the ICD agent, against FP64."""
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


def _plan(M, shape, **kw):
    geom, vol, ang = _geometry(M, *shape, **kw)
    h = ctypes.c_void_p()
    assert M.lib().msf_projector_create(ctypes.byref(geom), ctypes.byref(vol), ctypes.byref(h)) == 0, M.lib().msf_last_error()
    return geom, vol, ang, h


def test_autotuner_times_each_launch_once(M):
    # 64 slices: every z-run is the same launch, so the first; 224: three launches
    import torch
    for nz, allowed in ((64, (8,)), (224, (8, 16, 64))):
        geom, vol, ang, h = _plan(M, (20, 18, nz, 2, 30, nz + 10, 6))
        L, choice = M.lib(), (ctypes.c_int * 3)()
        try:
            e = torch.randn((2, 6, nz + 10, 30), device="cuda", generator=torch.Generator("cuda").manual_seed(1))
            x = torch.empty((2, 2, nz, 18, 20), device="cuda")
            assert L.msf_backproject(h, e.data_ptr(), x[0].data_ptr(), None) == 0
            assert L.msf_projector_autotune(h, None, choice) == 0
            assert choice[2] in allowed and choice[0] * choice[1] == 128
            assert L.msf_backproject(h, e.data_ptr(), x[1].data_ptr(), None) == 0
            torch.cuda.synchronize()
            assert torch.equal(x[0], x[1])
        finally:
            L.msf_projector_destroy(h)
