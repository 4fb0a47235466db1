"""Handles created and used at once on a stream that is not ordered after the default
stream (every torch.cuda.Stream): a create call leaves none of its clears pending, so
the results equal those of handles that had come to rest, bit for bit.  The workspaces
are large, so that clears left behind would still run when the first kernels do."""
import pytest

from paper_2008_01567_gb300 import synth

pytestmark = pytest.mark.gpu
SCAN = synth.Scan(n=192, nt=10, nu=256, nv=200, views=6)


@pytest.fixture(scope="module")
def M():
    import torch
    from paper_2008_01567_gb300 import build, msf
    build.build()
    assert torch.cuda.is_available()
    return msf


@pytest.fixture(scope="module")
def data():
    import torch
    g = torch.Generator("cuda").manual_seed(71)
    shape = (SCAN.nt, SCAN.n, SCAN.n, SCAN.n)
    v = torch.rand(shape, device="cuda", generator=g)
    y = torch.rand((SCAN.nt, SCAN.views, SCAN.nv, SCAN.nu), device="cuda", generator=g)
    return v, y, torch.rand(y.shape, device="cuda", generator=g)


def _on_a_side_stream(call):
    """call(True), which lets the new handle come to rest, and call(False), at once on a new stream."""
    import torch
    torch.cuda.synchronize()
    ref = call(True)
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream()):
        got = call(False)
    torch.cuda.synchronize()
    assert torch.equal(got, ref)


@pytest.mark.parametrize("icd", [False, True], ids=["cg", "icd"])
def test_data_agent_runs_at_once_on_a_side_stream(M, data, icd):
    import torch
    v, y, lam = data
    P = M.Projector(SCAN)
    xs = [torch.zeros_like(v), torch.zeros_like(v)]

    def call(rest):
        x = xs.pop()
        dp = M.DataProx(P)
        if rest:
            torch.cuda.synchronize()
        if icd:
            M.msf_prox_data_icd(dp, y, lam, v, x, 0.2, 1)
        else:
            M.msf_prox_data(dp, y, lam, v, x, 0.2, 2)
        torch.cuda.synchronize()
        return x

    _on_a_side_stream(call)


def test_mace_runs_at_once_on_a_side_stream(M, data):
    import torch
    v, y, lam = data
    P = M.Projector(SCAN)
    states = [tuple(torch.stack([v, v]) for _ in range(2)) for _ in range(2)]

    def call(rest):
        W, X = states.pop()
        m = M.Mace(P, W, X, y, lam, M.MSF_PRIOR_QGGMRF, mrf=M.msf_mrf(2.0, 1.2, 1.0, 0.1, 0.5))
        if rest:
            torch.cuda.synchronize()
        M.msf_mace_step(m, 0.5, 0.2, [0.5, 0.5], 2, 1)
        torch.cuda.synchronize()
        return torch.cat([W, X])

    _on_a_side_stream(call)
