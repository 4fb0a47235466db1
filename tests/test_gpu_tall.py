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


# 7, 10 and 12 sets of 32 slices: 8, 10 and 12 voxels per lane with z-runs of 64, other
# numbers and up to six blocks along z with the shorter ones
@pytest.mark.parametrize("shape", [(9, 11, 201, 1, 16, 213, 3), (10, 9, 303, 1, 15, 335, 3), (8, 9, 382, 1, 14, 401, 3)],
                         ids=lambda s: "x".join(map(str, s)))
def test_adjoint_of_tall_volumes(M, shape):
    import torch
    geom, vol, ang, h = _plan(M, shape)
    L, first = M.lib(), None
    y = np.random.default_rng(6).standard_normal((1, geom.views, geom.nv, geom.nu)).astype(np.float32)
    ref, yg = _oracle_At(y.astype(np.float64), geom, vol, ang), torch.from_numpy(y).cuda()
    try:
        for zrun in (8, 16, 32, 64):
            assert L.msf_projector_set_tuning(h, 32, 4, zrun) == 0
            x = torch.full((1, vol.nz, vol.ny, vol.nx), -1.0, device="cuda")
            assert L.msf_backproject(h, yg.data_ptr(), x.data_ptr(), None) == 0
            torch.cuda.synchronize()
            got = x.cpu().numpy().astype(np.float64)
            assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref), zrun   # the projector's tolerance
            first = x if first is None else first
            assert torch.equal(x, first), zrun
    finally:
        L.msf_projector_destroy(h)


def _matrix(geom, vol, ang):
    """A of one frame in FP64, sparse: rows (view, iv, iu), columns (z, y, x)."""
    from scipy import sparse
    nx, ny, nz, rows, cols, vals = vol.nx, vol.ny, vol.nz, [], [], []
    u = (np.arange(geom.nu) - 0.5 * (geom.nu - 1)) * geom.du
    v = (np.arange(geom.nv) - 0.5 * (geom.nv - 1))[:, None] * geom.dv
    for j, th in enumerate(ang):
        c, s = np.cos(th), np.sin(th)
        dx, dy = -geom.dsd * c - u * s, -geom.dsd * s + u * c
        step = np.sqrt(dx ** 2 + dy ** 2 + v ** 2)
        for xmaj in (True, False):
            on = (np.abs(dx) >= np.abs(dy)) == xmaj
            dm, da, sm, sa = (dx, dy, geom.dso * c, geom.dso * s) if xmaj else (dy, dx, geom.dso * s, geom.dso * c)
            nm, na = (nx, ny) if xmaj else (ny, nx)
            for k in range(nm):
                lam = ((k - 0.5 * (nm - 1)) - sm) / dm
                fa = np.broadcast_to(sa + lam * da + 0.5 * (na - 1), v.shape[:1] + u.shape)
                fz = lam * v + 0.5 * (nz - 1)
                a0, z0 = np.floor(fa).astype(int), np.floor(fz).astype(int)
                for p in (0, 1):
                    for q in (0, 1):
                        a, z = a0 + p, z0 + q
                        w = np.where(p, fa - a0, 1 - (fa - a0)) * np.where(q, fz - z0, 1 - (fz - z0)) * step / np.abs(dm)
                        ok = on & (a >= 0) & (a < na) & (z >= 0) & (z < nz) & (w != 0)
                        iv, iu = np.nonzero(ok)
                        y, x = (a[ok], k) if xmaj else (k, a[ok])
                        rows.append((j * geom.nv + iv) * geom.nu + iu)
                        cols.append((z[ok] * ny + y) * nx + x)
                        vals.append(w[ok])
    return sparse.csr_matrix((np.concatenate(vals), (np.concatenate(rows), np.concatenate(cols))),
                             shape=(len(ang) * geom.nv * geom.nu, nz * ny * nx))


def _icd(A, y, lam, v, z, sigma, sweeps, shape):
    iz, iy, ix = np.indices(shape).reshape(3, -1)
    group, z, e = ((iz % 2) * 2 + iy % 2) * 2 + ix % 2, z.copy(), y - A @ z
    theta2 = (A.multiply(A)).T @ lam + 1 / sigma ** 2
    for _ in range(sweeps):
        for g in range(8):
            on = group == g
            if not on.any():
                continue              # a volume of one slice
            th1 = np.where(on, -(A.T @ (lam * e)) + (z - v) / sigma ** 2, 0.0)
            d = -th1 / theta2
            ad = A @ d
            alpha = -(th1 @ d) / (lam @ ad ** 2 + d @ d / sigma ** 2)
            z, e = z + alpha * d, e - alpha * ad
    return z


# group voxels along z in two, two, three and eleven sets of 32, the last beside two sets of warps
# that share a tile's views; more rows than one chunk of five sets takes
@pytest.mark.parametrize("shape,zruns", [((5, 6, 67, 1, 11, 75, 4), (8, 64)), ((6, 5, 131, 2, 11, 190, 3), (8, 16, 64)),
                                         ((4, 5, 391, 1, 9, 420, 2), (8, 16, 64)), ((3, 4, 643, 1, 7, 655, 2), (32, 64)),
                                         ((75, 73, 13, 1, 110, 21, 4), (16,))], ids=lambda s: "x".join(map(str, s)))
def test_icd_agent_of_tall_volumes(M, shape, zruns):
    import torch
    geom, vol, ang, h = _plan(M, shape)
    L, d, sigma, sweeps = M.lib(), ctypes.c_void_p(), 0.4, 2
    r = np.random.default_rng(9)
    f32 = lambda a: a.astype(np.float32).astype(np.float64)
    v, z0 = f32(r.random((vol.nt, vol.nz * vol.ny * vol.nx))), f32(r.random((vol.nt, vol.nz * vol.ny * vol.nx)))
    lam = f32(r.random((vol.nt, geom.views * geom.nv * geom.nu)) + 0.1)
    y, ref = np.empty_like(lam), np.empty_like(v)
    for t in range(vol.nt):
        A = _matrix(geom, vol, ang[t * geom.views:(t + 1) * geom.views])
        y[t] = f32(A @ v[t] + 0.3 * r.standard_normal(A.shape[0]))
        ref[t] = _icd(A, y[t], lam[t], v[t], z0[t], sigma, sweeps, (vol.nz, vol.ny, vol.nx))
    yg, lg, vg = (torch.from_numpy(a.astype(np.float32)).cuda() for a in (y, lam, v))
    assert L.msf_dataprox_create(h, ctypes.byref(d)) == 0
    try:
        for zrun in zruns:
            assert L.msf_projector_set_tuning(h, 16, 8, zrun) == 0
            z = torch.from_numpy(z0.astype(np.float32)).cuda()
            assert L.msf_prox_data_icd(d, yg.data_ptr(), lg.data_ptr(), vg.data_ptr(), z.data_ptr(), sigma, sweeps, None) == 0
            torch.cuda.synchronize()
            got = z.cpu().numpy().astype(np.float64)
            # two projections and gathers of 1e-5 per group step, as in test_gpu_icd.py
            assert np.linalg.norm(got - ref) <= 2 * 8 * sweeps * 1e-5 * np.linalg.norm(ref), zrun
            assert np.linalg.norm(z0 - ref) > 1e-2 * np.linalg.norm(ref)
    finally:
        L.msf_dataprox_destroy(d)
        L.msf_projector_destroy(h)
