"""The q-GGMRF kernels at the sizes where their launch can go wrong: rows that end
inside a warp, axes of one or two voxels (no inner voxels), and extreme potentials,
against the FP64 oracle through the C ABI."""
import numpy as np
import pytest

import oracle
from paper_2008_01567_gb300 import synth
from tests._problems import f32, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import torch
    from paper_2008_01567_gb300 import build, msf
    build.build()
    assert torch.cuda.is_available()
    return msf


def _sweeps(M, v, z, sigma, q, sx, bt, n):
    import torch
    nt, nz, ny, nx = v.shape
    vg, zg = (torch.from_numpy(a.astype(np.float32)).cuda() for a in (v, z))
    M.msf_prox_qggmrf(M.msf_vol(nx, ny, nz, nt, 1.0), M.msf_mrf(2.0, q, 1.0, sx, bt), vg, zg, sigma, n)
    torch.cuda.synchronize()
    return zg.cpu().numpy().astype(np.float64), oracle.prox_qggmrf(v, z, sigma, 2.0, q, 1.0, sx, bt, n)


@pytest.mark.parametrize("shape", [(1, 1, 1, 1), (1, 2, 1, 2), (3, 3, 3, 3), (2, 5, 9, 67), (4, 3, 2, 64), (3, 7, 4, 65), (1, 4, 33, 130),
                                   # the largest volume of one launch (4096 voxels per colour), and the next that takes sixteen
                                   (2, 32, 32, 32), (2, 32, 32, 33), (3, 21, 34, 70)],
                         ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("q", [1.0, 1.2, 2.0])
def test_sweeps_match_oracle_at_ragged_sizes(M, shape, q):
    # 1e-5: the bound of the agent's parity test for up to four sweeps
    v, z = f32(synth.normal(51, shape) + 1.0), f32(synth.normal(52, shape) + 1.0)
    got, ref = _sweeps(M, v, z, 0.2, q, 0.1, 0.5, 2)
    assert rel_l2(got, ref) <= 1e-5


def test_outliers_leave_their_neighbours_weights(M):
    # two far outliers beside one voxel, as a pair of opposite neighbours and as
    # neighbours of two pairs: the weights of the others must not be lost
    shape = (3, 5, 6, 40)
    v, z = f32(synth.normal(53, shape) + 1.0), f32(synth.normal(54, shape) + 1.0)
    z[1, 2, 3, 9] = z[1, 2, 3, 11] = 1e12
    z[1, 3, 3, 20] = z[1, 2, 4, 20] = -1e12
    v[z > 1e11], v[z < -1e11] = 1e12, -1e12
    got, ref = _sweeps(M, v, z, 0.2, 1.2, 0.1, 0.5, 1)
    ok = np.abs(ref) < 1e6
    assert ok.sum() >= ok.size - 4
    # an outlier's weight is about |D/sx|^-0.8 relative to a near neighbour's and
    # multiplies 1e12: its 2^-21 relative error bounds what a voxel may be off
    assert np.abs(got - ref)[ok].max() <= 1e-5 * max(1.0, np.abs(ref[ok]).max())
