"""The channel sums that the training step's backward kernels form as they store dz (the conv
bias gradients), where a thread has no element, one, or more than one run of 32: against
FP64 sums of the stored dz, through the C ABI."""
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


# 311296 threads of 8 channels: 38912 pixels per element of a thread, 1245184 for a run of 32
@pytest.mark.parametrize("B,H,W", [(1, 8, 17), (19, 32, 64), (20, 250, 250)])
def test_bias_gradients_are_the_sums_of_the_stored_dz(M, B, H, W):
    # FP32 runs of at most 32 BF16 values (31 roundings of 2^-24), then FP64: 2e-6 of sum |dz|
    import torch
    P = B * H * W
    c = M.Cnn(4096)
    c.set_params(M.pack_params(*synth.cnn_weights(61)))
    c.train_reserve(P)
    c.train_trace(True)
    clean = f32(synth.uniform(62, (B, H, W), 0.0, 2.0)).astype(np.float32)
    noisy = np.repeat(clean[:, None], 5, 1) + f32(synth.normal(63, (B, 5, H, W), 0.1)).astype(np.float32)
    M.msf_train_step(c, torch.from_numpy(noisy).cuda(), torch.from_numpy(clean).cuda(), 1e-3)
    grads, _, _ = M.unpack_params(c.get_grads())
    for layer in (0, 4, 8):
        dz = c.train_tensor(c.TT_DZ, layer, P).reshape(P, 64)
        assert np.abs(dz).sum() > 0
        err = np.abs(grads[layer][1] - dz.sum(0, dtype=np.float64))
        assert (err <= 2e-6 * np.abs(dz).sum(0, dtype=np.float64) + 1e-30).all(), layer
