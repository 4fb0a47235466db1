"""The q-GGMRF agents at the ends of their arithmetic's range, against the FP64 oracle
through the C ABI."""
import numpy as np
import pytest

import oracle
from paper_2008_01567_gb300 import synth
from tests._problems import f32

pytestmark = pytest.mark.gpu
SHAPES = [(3, 5, 6, 40), (3, 18, 22, 70)]   # all sweeps in one launch, a launch per colour


@pytest.fixture(scope="module")
def M():
    import torch
    from paper_2008_01567_gb300 import build, msf
    build.build()
    assert torch.cuda.is_available()
    return msf


def _sweeps(M, v, z, sigma, q, T, sx, n, alias=False):
    import torch
    nt, nz, ny, nx = v.shape
    zg = torch.from_numpy(z.astype(np.float32)).cuda()
    vg = zg if alias else torch.from_numpy(v.astype(np.float32)).cuda()
    M.msf_prox_qggmrf(M.msf_vol(nx, ny, nz, nt, 1.0), M.msf_mrf(2.0, q, T, sx, 0.5), vg, zg, sigma, n)
    torch.cuda.synchronize()
    return zg.cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_two_far_outliers_keep_their_influence(M, shape):
    # with q = 1 an outlier's weight falls as its distance grows and its influence stays: two
    # whose weights' product would be below FP32's normal numbers, of equal and of uneven size
    v, z = f32(synth.normal(53, shape) + 1.0), f32(synth.normal(54, shape) + 1.0)
    z[1, 2, 3, 9] = z[1, 2, 3, 11] = 1.2e18
    z[1, 2, 3, 20], z[1, 2, 3, 22] = 1e12, -1e30
    z[1, 3, 3, 30], z[1, 1, 3, 30] = 2e25, 3e25
    out = np.abs(z) > 1e11
    v[out] = z[out] = f32(z)[out]
    got, ref = _sweeps(M, v, z, 0.2, 1.0, 1.0, 0.1, 1), oracle.prox_qggmrf(v, z, 0.2, 2.0, 1.0, 1.0, 0.1, 0.5, 1)
    ok = ~out
    # their influence, b / (2 sx) beside v / sigma^2, carries the logarithm's 2^-22 times
    # log2(1e32) times ln 2: 2e-5 of it, 1e-5 of a voxel
    assert np.abs(got - ref)[ok].max() <= 1e-5 * max(1.0, np.abs(ref[ok]).max())
