"""The CNN agents' ring of transposed frames where it wraps: handles of one and two
frames against one that holds every frame, in both turned orientations, at slice widths
that take staged patches (a multiple of four) and that read the frames directly."""
import pytest

from paper_2008_01567_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import torch
    from paper_2008_01567_gb300 import build, msf
    build.build()
    assert torch.cuda.is_available()
    return msf


# nx, ny, nz: slices of the yz agent are nz x ny, of the zx agent nx x nz
@pytest.mark.parametrize("nx,ny,nz", [(16, 12, 20), (14, 13, 19)], ids=["staged", "direct"])
@pytest.mark.parametrize("orient", [1, 2], ids=["yz", "zx"])
@pytest.mark.parametrize("frames", [1, 2])
def test_small_handles_equal_a_large_one(M, nx, ny, nz, orient, frames):
    import torch
    nt = 15
    vol, x = M.msf_vol(nx, ny, nz, nt, 1.0), torch.rand((nt, nz, ny, nx), device="cuda",
                                                       generator=torch.Generator("cuda").manual_seed(12))
    flat, outs = M.pack_params(*synth.cnn_weights(67)), []
    for n in (frames, nt):
        c = M.Cnn(n * nx * ny * nz)
        c.set_params(flat)
        for _ in range(2):                # a second call finds the first one's frames in the ring
            out = torch.full_like(x, -5.0)
            M.msf_denoise(c, orient, vol, x, out)
            torch.cuda.synchronize()
            outs.append(out)
        out = torch.full_like(x, -5.0)    # other frames through the same handle
        M.msf_denoise(c, orient, vol, x.flip(0).contiguous(), out)
        torch.cuda.synchronize()
        outs.append(out)
    assert torch.equal(outs[0], outs[3]) and torch.equal(outs[1], outs[4]) and torch.equal(outs[2], outs[5])
    assert torch.equal(outs[0], outs[1])
