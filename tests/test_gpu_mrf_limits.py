"""The q-GGMRF agents at the ends of their arithmetic's range, against the FP64 oracle
through the C ABI."""
import numpy as np
import pytest

import oracle
from paper_2008_01567_gb300 import synth
from tests._problems import I0, f32, measurement, rel_l2

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


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("q", [1.8, 1.99, 2.0])
def test_ratios_below_the_normal_numbers(M, shape, q):
    # |D / (T sx)| near 1e-39, which p - q near 0 brings back to 0.4: 1e-5, the agent's bound
    v, z = f32(1e-19 * synth.normal(55, shape)), f32(1e-19 * synth.normal(56, shape))
    got = _sweeps(M, v, z, 1.0, q, 1e20, 1.0, 2)
    assert rel_l2(1e19 * got, 1e19 * oracle.prox_qggmrf(v, z, 1.0, 2.0, q, 1e20, 1.0, 0.5, 2)) <= 1e-5


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_in_place_on_its_own_input(M, shape):
    # d_v == d_x: every sweep takes the voxel's present value as v
    z = f32(synth.normal(57, shape) + 1.0)
    got, ref = _sweeps(M, z, z, 0.2, 1.2, 1.0, 0.1, 3, alias=True), z
    for _ in range(3):
        ref = oracle.prox_qggmrf(ref, ref, 0.2, 2.0, 1.2, 1.0, 0.1, 0.5, 1)
    assert rel_l2(got, ref) <= 1e-5


def test_captured_sweeps_equal_eager_ones(M):
    # a captured call of a small volume takes a launch per colour, an eager one a launch for all:
    # the same bits, also where colours are empty
    import torch
    for shape in ((1, 1, 9, 40), (2, 6, 7, 40), (1, 32, 32, 32)):
        nt, nz, ny, nx = shape
        vol, mrf = M.msf_vol(nx, ny, nz, nt, 1.0), M.msf_mrf(2.0, 1.2, 1.0, 0.1, 0.5)
        g = torch.Generator("cuda").manual_seed(6)
        v, z = (torch.randn(shape, device="cuda", generator=g) for _ in range(2))
        a, b = z.clone(), z.clone()
        M.msf_prox_qggmrf(vol, mrf, v, a, 0.2, 2)
        graph, st = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=st):
            M.msf_prox_qggmrf(vol, mrf, v, b, 0.2, 2)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(a, b) and not torch.equal(a, z), shape


def test_direct_map_with_ratios_below_the_normal_numbers(M):
    # the surrogate's Laplacian of the direct MAP solve, T = 1e39; the bound of test_gpu_map.py
    import torch
    scan, n_outer, n_cg = synth.TINY, 2, 4
    x0, counts, y, lam = measurement(scan, 51)
    P, c = M.Projector(scan), torch.from_numpy(counts.astype(np.float32)).cuda()
    yg, lg = torch.zeros_like(c), torch.zeros_like(c)
    M.msf_weights(c, yg, lg, I0, I0)
    xs = f32(0.5 * x0)
    x = torch.from_numpy(xs.astype(np.float32)).cuda()
    M.msf_map_solve(M.MapSolver(P), M.msf_mrf(2.0, 1.99, 1e39, 0.2, 0.5), 30.0, yg, lg, x, n_outer, n_cg)
    ref = oracle.map_mm(f32(y), f32(lam), xs, scan, 2.0, 1.99, 1e39, 0.2, 0.5, 30.0, n_outer, n_cg)
    assert rel_l2(x.cpu().numpy(), ref) <= 2 * n_outer * (n_cg + 1) * 1e-5
    assert rel_l2(xs, ref) > 1e-2
