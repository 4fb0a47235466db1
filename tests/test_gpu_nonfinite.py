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
