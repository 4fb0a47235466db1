"""What a non-finite value, or a sum that overflows, must reach and must not: through
the C ABI."""
import numpy as np
import pytest

from paper_2008_01567_gb300 import synth
from tests._problems import f32

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import torch
    from paper_2008_01567_gb300 import build, msf
    build.build()
    assert torch.cuda.is_available()
    return msf


def test_infinite_loss_gradient_at_a_corner_misses_the_taps_outside(M):
    # dR is infinite at pixel (0, 0) of the first image: the last layer's taps that would
    # read the row above or the column before it have no term there, and stay finite
    import torch
    B, H, W = 2, 9, 21
    c = M.Cnn(4096)
    c.set_params(M.pack_params(*synth.cnn_weights(61)))
    c.train_reserve(B * H * W)
    clean = f32(synth.uniform(62, (B, H, W), 0.0, 2.0)).astype(np.float32)
    noisy = np.repeat(clean[:, None], 5, 1) + f32(synth.normal(63, (B, 5, H, W), 0.1)).astype(np.float32)
    clean[0, 0, 0] = np.inf
    M.msf_train_step(c, torch.from_numpy(noisy).cuda(), torch.from_numpy(clean).cuda(), 1e-3, want_loss=False)
    torch.cuda.synchronize()
    g = M.unpack_params(c.get_grads())[0][9][0].reshape(64, 3, 3)
    assert np.isfinite(g[:, 0, :]).all() and np.isfinite(g[:, :, 0]).all()
    assert not np.isfinite(g[:, 1:, 1:]).any()


@pytest.mark.parametrize("n_cg", [1, 2])
def test_residual_that_overflows_in_the_last_step_is_reported(M, n_cg):
    # readings of 1e12 with weights of 1e8: the residual's values are near 1e21, their
    # squares beyond FP32, the state stays near 1e12
    import torch
    scan = synth.Scan(n=16, nt=2, nu=24, nv=22, views=5)
    shape = (2, scan.nt, scan.n, scan.n, scan.n)
    W, X = torch.zeros(shape, device="cuda"), torch.zeros(shape, device="cuda")
    y = torch.full((scan.nt, scan.views, scan.nv, scan.nu), 1e12, device="cuda")
    y *= 1 + torch.rand(y.shape, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    m = M.Mace(M.Projector(scan), W, X, y, torch.full_like(y, 1e8), M.MSF_PRIOR_QGGMRF, mrf=M.msf_mrf(2.0, 1.2, 1.0, 0.1, 0.5))
    with pytest.raises(M.MsfError) as e:
        M.msf_mace_step(m, 0.5, 1.0, [0.5, 0.5], n_cg, 1)
    assert e.value.status == 5 and "CG" in str(e.value)
    assert n_cg > 1 or torch.isfinite(X).all()
