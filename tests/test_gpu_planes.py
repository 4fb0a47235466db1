"""Thin volumes and detectors, whose plans take lanes along the detector columns and
along x (planes of z-pairs) instead of lines along z: against the direct kernel and FP64
references, and, since the choice of A^T and the agents does not depend on the number of
frames, plans of one frame bit for bit.  Through the C ABI."""
import ctypes

import numpy as np
import pytest

from tests.test_gpu_projector_shapes import _geometry, _oracle_At
from tests.test_gpu_tall import _icd, _matrix

pytestmark = pytest.mark.gpu
CONFIGS = [(32, 4, 16), (64, 2, 8), (16, 8, 32), (32, 4, 64)]


@pytest.fixture(scope="module")
def M():
    import torch
    from paper_2008_01567_gb300 import build, msf
    build.build()
    assert torch.cuda.is_available()
    return msf


class _Plan:
    def __init__(self, M, shape):
        self.geom, self.vol, self.ang = _geometry(M, *shape)
        self.L, self.h = M.lib(), ctypes.c_void_p()
        assert self.L.msf_projector_create(ctypes.byref(self.geom), ctypes.byref(self.vol), ctypes.byref(self.h)) == 0

    def __enter__(self):
        return self

    def __exit__(self, *a):
        self.L.msf_projector_destroy(self.h)

    def volume(self, fill=-1.0):
        import torch
        return torch.full((self.vol.nt, self.vol.nz, self.vol.ny, self.vol.nx), fill, device="cuda")

    def sino(self, fill=-1.0):
        import torch
        return torch.full((self.vol.nt, self.geom.views, self.geom.nv, self.geom.nu), fill, device="cuda")


# nx, ny, nz, nt, nu, nv, views, ragged in every axis: one slice and one row; few of both; few
# slices under a tall detector, and a volume under few rows; ICD in lines beside CG in planes;
# nine slices, ICD in planes; A alone in planes.  The first, third and last take A in planes.
SHAPES = [(45, 41, 1, 3, 300, 1, 10), (47, 44, 2, 2, 66, 5, 8), (70, 66, 7, 3, 250, 11, 16), (50, 47, 5, 2, 70, 70, 6),
          (130, 121, 30, 1, 180, 9, 5), (90, 85, 13, 2, 120, 19, 6), (150, 140, 9, 1, 210, 12, 5), (40, 38, 40, 5, 340, 30, 24)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_plan_holds_no_more_than_pairs(M, shape):
    # 16 bytes per voxel, 4 per ray (and the margins of calls that take lines), the column table
    nx, ny, nz, nt, nu, nv, views = shape
    with _Plan(M, shape) as P:
        G = nt * views
        assert P.L.msf_projector_bytes(P.h) <= 16 * nx * ny * nz * nt + 4 * G * nu * (nv + 7) + G * (8 + 8 + 4 + 32 * nu) + 4 * (nz + 24)


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("bad", [False, True], ids=["finite", "nonfinite"])
def test_forward_equals_the_direct_kernel(M, shape, bad):
    import torch
    with _Plan(M, shape) as P:
        x = torch.randn(P.volume().shape, device="cuda", generator=torch.Generator("cuda").manual_seed(5))
        if bad:
            x.view(-1)[torch.tensor([0, x.numel() // 2, x.numel() - 1], device="cuda")] = float("inf")
        ref = P.sino()
        assert P.L.msf_project_static(ctypes.byref(P.geom), ctypes.byref(P.vol), x.data_ptr(), ref.data_ptr(), None) == 0
        for c in CONFIGS:
            assert P.L.msf_projector_set_tuning(P.h, *c) == 0
            y = P.sino()
            assert P.L.msf_project(P.h, x.data_ptr(), y.data_ptr(), None) == 0
            torch.cuda.synchronize()
            assert torch.equal(torch.isnan(y), torch.isnan(ref))
            assert torch.equal(torch.nan_to_num(y, 7.0), torch.nan_to_num(ref, 7.0)), c


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_adjoint_matches_oracle(M, shape):
    import torch
    with _Plan(M, shape) as P:
        y = np.random.default_rng(6).standard_normal(P.sino().shape).astype(np.float32)
        ref = _oracle_At(y.astype(np.float64), P.geom, P.vol, P.ang)
        yg, first = torch.from_numpy(y).cuda(), None
        for c in CONFIGS:
            assert P.L.msf_projector_set_tuning(P.h, *c) == 0
            x = P.volume()
            assert P.L.msf_backproject(P.h, yg.data_ptr(), x.data_ptr(), None) == 0
            torch.cuda.synchronize()
            got = x.cpu().numpy().astype(np.float64)
            assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref), c   # the projector's tolerance
            first = x if first is None else first
            assert torch.equal(x, first), c


def _prox(P, y, lam, v, x, icd, tuning):
    """Two CG steps or one sweep on copies of x; with other calls of the plan in between."""
    import torch
    d, out = ctypes.c_void_p(), x.clone()
    assert P.L.msf_projector_set_tuning(P.h, *tuning) == 0
    assert P.L.msf_dataprox_create(P.h, ctypes.byref(d)) == 0
    try:
        f = P.L.msf_prox_data_icd if icd else P.L.msf_prox_data
        for _ in range(2):
            s = P.sino()
            assert P.L.msf_project(P.h, x.data_ptr(), s.data_ptr(), None) == 0
            out.copy_(x)
            assert f(d, y.data_ptr(), lam.data_ptr(), v.data_ptr(), out.data_ptr(), 0.3, 1 if icd else 2, None) == 0
            torch.cuda.synchronize()
    finally:
        P.L.msf_dataprox_destroy(d)
    return out


def _cg(A, y, lam, v, z, sigma, n):
    r = A.T @ (lam * (y - A @ z)) + (v - z) / sigma ** 2
    p, z = r.copy(), z.copy()
    for _ in range(n):
        q = A.T @ (lam * (A @ p)) + p / sigma ** 2
        alpha = (r @ r) / (p @ q)
        z, r0 = z + alpha * p, r
        r = r - alpha * q
        p = r + (r @ r) / (r0 @ r0) * p
    return z


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("icd", [False, True], ids=["cg", "icd"])
def test_data_agents(M, shape, icd):
    # the last frame against FP64, to the agents' tolerance (1e-5 per A and A^T pair, twice); the
    # first and the last in plans of their own, bit for bit
    import torch
    nx, ny, nz, nt, nu, nv, views = shape
    with _Plan(M, shape) as P:
        g = torch.Generator("cuda").manual_seed(8)
        v, x = (torch.rand(P.volume().shape, device="cuda", generator=g) for _ in range(2))
        lam, y = torch.rand(P.sino().shape, device="cuda", generator=g) + 0.1, P.sino()
        assert P.L.msf_project(P.h, v.data_ptr(), y.data_ptr(), None) == 0
        y += torch.randn(y.shape, device="cuda", generator=g)
        got = _prox(P, y, lam, v, x, icd, (32, 4, 16))
        assert torch.equal(got, _prox(P, y, lam, v, x, icd, (32, 4, 16)))
        for t in (0, nt - 1):
            ang = np.ascontiguousarray(P.ang[t * views:(t + 1) * views])
            one = _Plan.__new__(_Plan)
            one.L, one.h, one.geom, one.vol = P.L, ctypes.c_void_p(), M.msf_geom.from_buffer_copy(P.geom), M.msf_vol.from_buffer_copy(P.vol)
            one.geom.angles, one.vol.nt = ang.ctypes.data_as(ctypes.POINTER(ctypes.c_double)), 1
            assert P.L.msf_projector_create(ctypes.byref(one.geom), ctypes.byref(one.vol), ctypes.byref(one.h)) == 0
            with one:
                assert torch.equal(got[t], _prox(one, *(a[t:t + 1].contiguous() for a in (y, lam, v, x)), icd, (32, 4, 16))[0])
        if views * nu * nv * max(nx, ny) > 4e6:
            return                            # (too many taps for a sparse matrix here; in lines both times)
        A = _matrix(P.geom, P.vol, ang)
        yn, ln, vn, xn = (a[-1].cpu().numpy().astype(np.float64).ravel() for a in (y, lam, v, x))
        ref = _icd(A, yn, ln, vn, xn, 0.3, 1, (nz, ny, nx)) if icd else _cg(A, yn, ln, vn, xn, 0.3, 2)
        out = got[-1].cpu().numpy().astype(np.float64).ravel()
        assert np.linalg.norm(out - ref) <= (2 * 8 if icd else 2 * 2) * 1e-5 * np.linalg.norm(ref)
        assert np.linalg.norm(xn - ref) > 1e-2 * np.linalg.norm(ref)


@pytest.mark.parametrize("shape", [SHAPES[2], SHAPES[5], SHAPES[7]], ids=lambda s: "x".join(map(str, s)))
def test_autotune_keeps_results(M, shape):
    # plans of planes, of both layouts for the agents, and with A alone in planes
    import torch
    with _Plan(M, shape) as P:
        g = torch.Generator("cuda").manual_seed(8)
        x, e = torch.rand(P.volume().shape, device="cuda", generator=g), torch.rand(P.sino().shape, device="cuda", generator=g)
        outs, choice = [], (ctypes.c_int * 3)()
        for tuned in (False, True):
            if tuned:
                assert P.L.msf_projector_autotune(P.h, None, choice) == 0
                assert choice[0] * choice[1] == 128 and choice[2] in (8, 16, 32, 64)
            y, b = P.sino(), P.volume()
            assert P.L.msf_project(P.h, x.data_ptr(), y.data_ptr(), None) == 0
            assert P.L.msf_backproject(P.h, e.data_ptr(), b.data_ptr(), None) == 0
            torch.cuda.synchronize()
            outs.append((y, b))
        assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])
