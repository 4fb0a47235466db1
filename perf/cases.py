"""What the library is timed on: its agents and whole iterations, through its public entry points.

listed() names the calls that stand for its use; draw() gives more of the same
kinds, over the same ranges of sizes, views and scan protocols.  Every case is a
dict of plain values; prepare() makes what a user's program holds before the
call (inputs on the GPU, plan and handles), run() makes one pass, exact() says
what that pass computes, in FP64 and without the library.

Inputs follow the paper's set-up: a phantom of uniform ellipsoids that moves one
voxel per time-point, its exact line integrals, Poisson photon counts at 1e4.
"""
import math
import types

import numpy as np
import torch

from paper_2008_01567_gb300 import msf

I0 = 1e4
SIGMA, Q, T, SX, BT = 0.2, 1.2, 1.0, 0.1, 0.5        # plain runs: prox scale and 4D MRF (p = 2)
MRF = (2.0, Q, T, SX, BT)
SCAN_KINDS = ("project", "backproject", "prox_cg", "prox_icd", "mace_plain", "mace_learned")


def _scan_case(kind, n, nt, nu, nv, views, mode, **more):
    return dict(kind=kind, n=n, nt=nt, nu=nu, nv=nv, views=views, mode=mode, **more)


def listed():
    return [
        # one forward projection of the tiny workload: latency and launches
        _scan_case("project", 24, 4, 32, 32, 12, "sparse360", name="project_24"),
        # the projector workload: a 128^3 x 8 volume, 32 views per time-point over 360 degrees
        _scan_case("project", 128, 8, 192, 160, 32, "sparse360", cols=16, rows=8, zrun=32, name="project_128"),
        # its adjoint for the limited-angle protocol (a 90 degree wedge per time-point)
        _scan_case("backproject", 128, 8, 192, 160, 32, "wedge90", cols=16, rows=8, zrun=32, name="backproject_128_wedge"),
        # the data agent on a volume, detector and view count that fit no tile (a plan as created, not tuned)
        _scan_case("prox_cg", 101, 5, 143, 117, 21, "wedge90", n_cg=3, name="prox_cg_odd"),
        # the data agent of the full workload: 384^3 x 16, five CG iterations (the launch shapes its autotuner picks)
        _scan_case("prox_cg", 384, 16, 512, 384, 24, "sparse360", n_cg=5, cols=64, rows=2, zrun=64, name="prox_cg_full"),
        # the paper's own data agent: three grouped coordinate-descent sweeps
        _scan_case("prox_icd", 96, 6, 160, 128, 24, "sparse360", n_icd=3, name="prox_icd_96"),
        # the plain prior agent on the largest volume of the problem queue
        dict(kind="qggmrf", nx=192, ny=192, nz=192, nt=12, n_sweeps=2, name="qggmrf_192"),
        # a learned prior agent at the projector workload's volume, slices across the fastest axis
        dict(kind="denoise", nx=128, ny=128, nz=128, nt=8, orient=1, name="denoise_128_yz"),
        # the same agent on slices of odd height and width
        dict(kind="denoise", nx=77, ny=85, nz=63, nt=5, orient=2, name="denoise_odd_zx"),
        # one training step of the benchmark's recipe: batch 128 of 64 x 64 patches
        dict(kind="train", batch=128, h=64, w=64, name="train_128x64x64"),
        # the tiny workload whole: ten plain iterations from zero, as the benchmark runs them
        _scan_case("mace_plain", 24, 4, 32, 32, 12, "sparse360", iters=10, graph=False, name="mace_plain_24"),
        # one learned multi-slice-fusion iteration from a stored state, replayed as a graph
        _scan_case("mace_learned", 192, 8, 256, 192, 24, "sparse360", iters=1, graph=True, name="mace_learned_192"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(SCAN_KINDS + ("prox_cg", "qggmrf", "denoise", "denoise", "train"))
    if kind == "train":
        return dict(kind=kind, batch=_log_int(rng, 4, 128), h=_log_int(rng, 16, 64), w=_log_int(rng, 16, 64))
    if kind in ("qggmrf", "denoise"):
        n = _log_int(rng, 24, 192 if kind == "qggmrf" else 128)
        c = dict(kind=kind, nx=n, ny=max(8, n + rng.randint(-n // 4, n // 4)), nz=max(8, n + rng.randint(-n // 3, n // 6)),
                 nt=rng.randint(1, 10))
        c.update(dict(n_sweeps=rng.randint(1, 3)) if kind == "qggmrf" else dict(orient=rng.randint(0, 2)))
        return c
    n = _log_int(rng, 24, {"project": 320, "backproject": 320, "prox_cg": 256, "prox_icd": 128, "mace_plain": 160,
                           "mace_learned": 144}[kind])
    c = _scan_case(kind, n, rng.randint(3, 12), max(16, int(n * rng.uniform(1.1, 1.6))), max(16, int(n * rng.uniform(0.9, 1.4))),
                   rng.randint(8, 40), rng.choice(["sparse360", "wedge90", "wedge180"]))
    if kind in ("prox_cg", "prox_icd"):
        c.update({"n_cg" if kind == "prox_cg" else "n_icd": rng.randint(1, 5 if kind == "prox_cg" else 3)})
    if kind.startswith("mace"):
        c.update(iters=rng.randint(2, 6) if kind == "mace_plain" else 1, graph=rng.random() < 0.5)
    return c


# ------------------------------------------------------------------ inputs


def _scan(c):
    """Volume one unit wide, source at 4, detector at 8, 5% margin around the projected volume."""
    r = 0.5 * math.sqrt(2.0)
    pitch = 1.05 * max(2.0 * 8.0 * math.tan(math.asin(r / 4.0)) / c["nu"], 8.0 / (4.0 - r) / c["nv"])
    t = np.arange(c["nt"])[:, None]
    j = np.arange(c["views"])[None, :]
    if c["mode"] == "sparse360":
        ang = 2.0 * math.pi * (j + t / c["nt"]) / c["views"]
    else:
        ang = math.radians(float(c["mode"][5:])) * (t + j / c["views"])
    return types.SimpleNamespace(n=c["n"], nt=c["nt"], nu=c["nu"], nv=c["nv"], views=c["views"], vox=1.0 / c["n"], pitch=pitch,
                                 dso=4.0, dsd=8.0, angles=lambda: np.asarray(ang, dtype=np.float64))


def _gen(seed, k=0):
    return torch.Generator("cuda").manual_seed(int(seed) * 1009 + 17 * k + 1)


def _ellipsoids(seed, count=6):
    """Centres in the inner half, semi-axes 0.08 to 0.3, random rotations, attenuation 0.5 to 2."""
    r = np.random.RandomState(int(seed) % (2 ** 31 - 1))
    return [(r.uniform(-0.25, 0.25, 3), np.linalg.qr(r.standard_normal((3, 3)))[0] / r.uniform(0.08, 0.3, 3)[:, None],
             r.uniform(0.5, 2.0)) for _ in range(count)]


def _phantom(seed, nx, ny, nz, nt, vox):
    ax = [(torch.arange(m, device="cuda", dtype=torch.float32) - 0.5 * (m - 1)) * vox for m in (nx, ny, nz)]
    x = torch.zeros((nt, nz, ny, nx), device="cuda")
    for centre, R, mu in _ellipsoids(seed):
        for t in range(nt):
            p = [ax[0] - centre[0], (ax[1] - centre[1])[:, None], (ax[2] - centre[2] - t * vox)[:, None, None]]
            d2 = sum((R[k, 0] * p[0] + R[k, 1] * p[1] + R[k, 2] * p[2]) ** 2 for k in range(3))
            x[t] += (d2 <= 1.0).float() * mu
    return x


def _counts(seed, s):
    """Photon counts [nt][views][nv][nu] of the phantom's exact line integrals."""
    u = (torch.arange(s.nu, device="cuda", dtype=torch.float32) - 0.5 * (s.nu - 1)) * s.pitch
    v = ((torch.arange(s.nv, device="cuda", dtype=torch.float32) - 0.5 * (s.nv - 1)) * s.pitch)[:, None]
    out = torch.empty((s.nt, s.views, s.nv, s.nu), device="cuda")
    ell, g = _ellipsoids(seed), _gen(seed, 1)
    for t, row in enumerate(s.angles()):
        for j, th in enumerate(row):
            c, n = math.cos(th), math.sin(th)
            src = np.array([s.dso * c, s.dso * n, 0.0])
            d = [-s.dsd * c - u * n, -s.dsd * n + u * c, v]
            length = torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
            line = 0.0
            for centre, R, mu in ell:
                o = R @ (src - centre - np.array([0.0, 0.0, t * s.vox]))
                m = [R[k, 0] * d[0] + R[k, 1] * d[1] + R[k, 2] * d[2] for k in range(3)]
                a = m[0] ** 2 + m[1] ** 2 + m[2] ** 2
                b = m[0] * o[0] + m[1] * o[1] + m[2] * o[2]
                line = line + mu * length * 2.0 * torch.sqrt(torch.clamp(b * b - a * (float(o @ o) - 1.0), min=0.0)) / a
            out[t, j] = torch.poisson(I0 * torch.exp(-line), generator=g)
    return out


def _measured(seed, s):
    lam = _counts(seed, s).clamp_(min=1.0)
    return -torch.log(lam / I0), lam          # y = -ln(n / I0), Lambda = I0 exp(-y) = n


def _noisy(seed, x, k, scale=0.05):
    return x + scale * torch.randn(x.shape, device="cuda", generator=_gen(seed, k))


def _network(seed):
    """A 10-layer network (5 -> 64 -> ... -> 1, BatchNorm in layers 2 to 9) of He-normal
    weights whose last layer is small, as a denoiser's correction is: [(w, b)], [(gamma, beta, mean, var)]."""
    r = np.random.RandomState((int(seed) * 7 + 3) % (2 ** 31 - 1))
    convs, bns = [], []
    for l in range(10):
        cin, cout = (5 if l == 0 else 64), (1 if l == 9 else 64)
        convs.append((r.standard_normal((cout, cin, 3, 3)) * math.sqrt(2.0 / (9 * cin)) * (0.02 if l == 9 else 1.0),
                      r.normal(0.0, 0.02, cout)))
        if 0 < l < 9:
            bns.append((r.uniform(0.8, 1.2, 64), r.normal(0.0, 0.1, 64), r.normal(0.0, 0.1, 64), r.uniform(0.5, 1.5, 64)))
    return convs, bns


def _flat(convs, bns):
    return np.concatenate([a.ravel() for p in convs for a in p] + [a.ravel() for p in bns for a in p]).astype(np.float32)


def _inputs(c, seed):
    """The inputs alone: tensors on the GPU, from the seed."""
    kind = c["kind"]
    if kind == "train":
        x = torch.rand((c["batch"], 1, c["h"], c["w"]), device="cuda", generator=_gen(seed, 2))
        clean = torch.nn.functional.avg_pool2d(x, 9, stride=1, padding=4)[:, 0] * 2.0
        sigma = 0.02 + 0.18 * torch.rand((c["batch"], 1, 1, 1), device="cuda", generator=_gen(seed, 3))
        noise = torch.randn((c["batch"], 5, c["h"], c["w"]), device="cuda", generator=_gen(seed, 4))
        return dict(noisy=(clean[:, None] + sigma * noise).contiguous(), clean=clean.contiguous())
    if kind in ("qggmrf", "denoise"):
        x = _phantom(seed, c["nx"], c["ny"], c["nz"], c["nt"], 1.0 / max(c["nx"], c["ny"], c["nz"]))
        v = _noisy(seed, x, 5)
        return dict(v=v, x=_noisy(seed, x, 6)) if kind == "qggmrf" else dict(v=v)
    s = _scan(c)
    if kind == "backproject":
        return dict(e=torch.randn((s.nt, s.views, s.nv, s.nu), device="cuda", generator=_gen(seed, 7)) + 0.5)
    x = _phantom(seed, s.n, s.n, s.n, s.nt, s.vox)
    if kind == "project":
        return dict(x=_noisy(seed, x, 8))
    y, lam = _measured(seed, s)
    if kind.startswith("prox"):
        return dict(y=y, lam=lam, v=_noisy(seed, x, 9), x=0.9 * x)
    if kind == "mace_plain":
        return dict(y=y, lam=lam)
    return dict(y=y, lam=lam, W=torch.stack([_noisy(seed, x, 10 + k) for k in range(4)]), X=torch.stack([0.95 * x] * 4))


# ------------------------------------------------------------------ one pass


def prepare(case, seed):
    c = dict(case)
    st = types.SimpleNamespace(c=c, i=_inputs(c, seed))
    kind = c["kind"]
    if kind in SCAN_KINDS:
        st.scan = _scan(c)
        st.P = msf.Projector(st.scan)
        if "zrun" in c:
            msf.msf_projector_set_tuning(st.P, c["cols"], c["rows"], c["zrun"])
        shape = (st.scan.nt,) + (st.scan.n,) * 3
    if kind == "project":
        st.y = torch.empty((st.scan.nt, st.scan.views, st.scan.nv, st.scan.nu), device="cuda")
    elif kind == "backproject":
        st.x = torch.empty(shape, device="cuda")
    elif kind.startswith("prox"):
        st.dp = msf.DataProx(st.P)
        st.x = torch.empty(shape, device="cuda")
    elif kind == "qggmrf":
        st.vol, st.mrf = msf.msf_vol(c["nx"], c["ny"], c["nz"], c["nt"], 1.0 / c["nx"]), msf.msf_mrf(*MRF)
        st.x = torch.empty_like(st.i["x"])
    elif kind == "denoise":
        st.vol = msf.msf_vol(c["nx"], c["ny"], c["nz"], c["nt"], 1.0 / c["nx"])
        st.cnn = msf.Cnn(c["nx"] * c["ny"] * c["nz"])
        st.cnn.set_params(_flat(*_network(seed)))
        st.out = torch.empty_like(st.i["v"])
    elif kind == "train":
        st.cnn = msf.Cnn(c["batch"] * c["h"] * c["w"])
        st.cnn.train_reserve(c["batch"] * c["h"] * c["w"])
        st.cnn.set_params(_flat(*_network(seed)))
    else:
        K1 = 2 if kind == "mace_plain" else 4
        st.W, st.X = (torch.zeros((K1,) + shape, device="cuda") for _ in range(2))
        if K1 == 2:
            st.m = msf.Mace(st.P, st.W, st.X, st.i["y"], st.i["lam"], msf.MSF_PRIOR_QGGMRF, mrf=msf.msf_mrf(*MRF))
        else:
            st.cnn = msf.Cnn(st.scan.n ** 3)
            st.cnn.set_params(_flat(*_network(seed)))
            st.m = msf.Mace(st.P, st.W, st.X, st.i["y"], st.i["lam"], msf.MSF_PRIOR_CNN, cnn=st.cnn)
    return st


def run(st):
    c, i, kind = st.c, st.i, st.c["kind"]
    if kind == "project":
        msf.msf_project(st.P, i["x"], st.y)
        return st.y
    if kind == "backproject":
        msf.msf_backproject(st.P, i["e"], st.x)
        return st.x
    if kind == "prox_cg":
        st.x.copy_(i["x"])                     # the warm start, which the call overwrites
        msf.msf_prox_data(st.dp, i["y"], i["lam"], i["v"], st.x, SIGMA, c["n_cg"])
        return st.x
    if kind == "prox_icd":
        st.x.copy_(i["x"])
        msf.msf_prox_data_icd(st.dp, i["y"], i["lam"], i["v"], st.x, SIGMA, c["n_icd"])
        return st.x
    if kind == "qggmrf":
        st.x.copy_(i["x"])
        msf.msf_prox_qggmrf(st.vol, st.mrf, i["v"], st.x, SIGMA, c["n_sweeps"])
        return st.x
    if kind == "denoise":
        msf.msf_denoise(st.cnn, c["orient"], st.vol, i["v"], st.out)
        return st.out
    if kind == "train":
        loss = msf.msf_train_step(st.cnn, i["noisy"], i["clean"], 1e-3)
        return dict(loss=loss, params=st.cnn.get_params())
    if kind == "mace_plain":
        st.W.zero_()
        st.X.zero_()
        for _ in range(c["iters"]):
            msf.msf_mace_step(st.m, 0.5, SIGMA, [0.25, 0.75], 5, 1, want_residual=False, use_graph=c["graph"])
        return dict(W=st.W, X=st.X)
    st.W.copy_(i["W"])                         # a stored state, resumed
    st.X.copy_(i["X"])
    r = msf.msf_mace_step(st.m, 0.8, 0.4, [0.25] * 4, 5, use_graph=c["graph"])
    return dict(W=st.W, X=st.X, residual=r)


def work(case):
    """Inputs read once, outputs written once; per ray and plane about 12 operations each way, 2 per weight and pixel of a
    network.  Iterations of a solver each apply their operators, whose volumes and sinograms count once per application."""
    c, kind = case, case["kind"]
    if kind == "train":
        px = c["batch"] * c["h"] * c["w"]
        return dict(bytes=4.0 * 6 * px + 3 * 4.0 * 340000, flops=3.0 * px * 2 * 9 * (5 * 64 + 8 * 64 * 64 + 64))
    if kind in ("qggmrf", "denoise"):
        N = c["nx"] * c["ny"] * c["nz"] * c["nt"]
        if kind == "denoise":
            return dict(bytes=8.0 * N, flops=2.0 * 9 * (5 * 64 + 8 * 64 * 64 + 64) * N)
        return dict(bytes=12.0 * N, flops=28.0 * 12 * N * c["n_sweeps"])
    N, M = c["nt"] * c["n"] ** 3, c["nt"] * c["views"] * c["nv"] * c["nu"]
    cross = 12.0 * 0.42 * c["n"] * M           # about 42% of the rays' planes lie in the volume
    one = 4.0 * (N + M)
    if kind in ("project", "backproject"):
        return dict(bytes=one, flops=cross)
    if kind == "prox_cg":
        return dict(bytes=2 * (c["n_cg"] + 1) * one, flops=2 * (c["n_cg"] + 1) * cross)
    if kind == "prox_icd":
        return dict(bytes=(2 + 2 * c["n_icd"]) * one, flops=(2 + 2 * c["n_icd"]) * cross)
    agent = 28.0 * 12 if kind == "mace_plain" else 3 * 2.0 * 9 * (5 * 64 + 8 * 64 * 64 + 64)
    return dict(bytes=c["iters"] * (12 * one + 40.0 * N), flops=c["iters"] * (12 * cross + agent * N))


# ------------------------------------------------------------------ the same in FP64, in torch


def _taps(s, th):
    """One view: the four (flat index into the zero-padded frame, weight) pairs of every ray on every plane, [plane][nv][nu]."""
    f64 = dict(device="cuda", dtype=torch.float64)
    n, c, w = s.n, math.cos(th), math.sin(th)
    u = (torch.arange(s.nu, **f64) - 0.5 * (s.nu - 1)) * s.pitch
    v = (torch.arange(s.nv, **f64) - 0.5 * (s.nv - 1))[:, None] * s.pitch
    dx, dy = -s.dsd * c - u * w, -s.dsd * w + u * c
    xm = dx.abs() >= dy.abs()
    dmaj, da = torch.where(xm, dx, dy), torch.where(xm, dy, dx)
    smaj = torch.where(xm, torch.full_like(dx, s.dso * c), torch.full_like(dx, s.dso * w))
    sa = torch.where(xm, torch.full_like(dx, s.dso * w), torch.full_like(dx, s.dso * c))
    k = torch.arange(n, **f64)[:, None]
    lam = ((k - 0.5 * (n - 1)) * s.vox - smaj) / dmaj                     # [plane][nu]
    fa = ((sa + lam * da) / s.vox + 0.5 * (n - 1)).clamp(-1.0, n)[:, None, :]
    fz = (lam[:, None, :] * v / s.vox + 0.5 * (n - 1)).clamp(-1.0, n)
    a0, z0 = fa.floor().clamp(max=n - 1), fz.floor().clamp(max=n - 1)
    wa, wz = fa - a0, fz - z0
    step = torch.sqrt(dx ** 2 + dy ** 2 + v ** 2) * s.vox / dmaj.abs()
    p = n + 2
    kk = (torch.arange(n, device="cuda") + 1)[:, None, None]
    base = (z0.long() + 1) * (p * p) + torch.where(xm, (a0.long() + 1) * p + kk, kk * p + a0.long() + 1)
    sm = torch.where(xm, p, 1)
    return [(base, (1 - wa) * (1 - wz) * step), (base + sm, wa * (1 - wz) * step),
            (base + p * p, (1 - wa) * wz * step), (base + p * p + sm, wa * wz * step)]


def _A(x, s):
    y = torch.empty((s.nt, s.views, s.nv, s.nu), device="cuda", dtype=torch.float64)
    for t, row in enumerate(s.angles()):
        f = torch.nn.functional.pad(x[t], (1,) * 6).reshape(-1)
        for j, th in enumerate(row):
            y[t, j] = sum((f[i] * w).sum(0) for i, w in _taps(s, th))
    return y


def _At(y, s, square=False):
    p = s.n + 2
    x = torch.empty((s.nt, s.n, s.n, s.n), device="cuda", dtype=torch.float64)
    for t, row in enumerate(s.angles()):
        f = torch.zeros(p ** 3, device="cuda", dtype=torch.float64)
        for j, th in enumerate(row):
            for i, w in _taps(s, th):
                f.index_add_(0, i.reshape(-1), ((w * w if square else w) * y[t, j]).reshape(-1))
        x[t] = f.reshape(p, p, p)[1:-1, 1:-1, 1:-1]
    return x


def _dots(a, b):
    return (a * b).sum((1, 2, 3), keepdim=True)


def _prox_cg(y, lam, v, x, s, sigma, n_cg):
    """n_cg conjugate-gradient steps on (A^T Lambda A + I/sigma^2) z = A^T Lambda y + v/sigma^2, per time-point."""
    z = x.clone()
    r = _At(lam * (y - _A(z, s)), s) + (v - z) / sigma ** 2
    p, rr = r.clone(), _dots(r, r)
    for _ in range(n_cg):
        q = _At(lam * _A(p, s), s) + p / sigma ** 2
        alpha = rr / _dots(p, q)
        z, r = z + alpha * p, r - alpha * q
        new = _dots(r, r)
        p, rr = r + new / rr * p, new
    return z


def _prox_icd(y, lam, v, x, s, sigma, n_sweeps):
    """Coordinate descent in eight parity groups: a Newton step per voxel, an exact line search per group and time-point."""
    z, e = x.clone(), y - _A(x, s)
    theta2 = _At(lam, s, square=True) + 1.0 / sigma ** 2
    k = torch.arange(s.n, device="cuda") % 2
    key = (k[:, None, None] * 2 + k[None, :, None]) * 2 + k[None, None, :]
    for _ in range(n_sweeps):
        for g in range(8):
            theta1 = -_At(lam * e, s) + (z - v) / sigma ** 2
            delta = torch.where(key == g, -theta1 / theta2, torch.zeros_like(z))
            ad = _A(delta, s)
            alpha = -_dots(theta1, delta) / (_dots(lam * ad, ad) + _dots(delta, delta) / sigma ** 2)
            z, e = z + alpha * delta, e - alpha * ad
    return z


def _qggmrf(v, x, sigma, n_sweeps):
    """Sweeps of 16 parity colours; each voxel takes the minimiser of the symmetric-bound surrogate."""
    pad = (1, 1) * 4
    z = torch.nn.functional.pad(x, pad)
    inside = torch.nn.functional.pad(torch.ones_like(x), pad)
    norm = 6.0 + 12.0 / math.sqrt(2.0) + 8.0 / math.sqrt(3.0)
    near = [((0, a, b, d), 1.0 / (math.sqrt(a * a + b * b + d * d) * norm)) for a in (-1, 0, 1) for b in (-1, 0, 1) for d in (-1, 0, 1)
            if a or b or d] + [((-1, 0, 0, 0), BT), ((1, 0, 0, 0), BT)]
    for _ in range(n_sweeps):
        for col in range(16):
            first = [(col >> k) & 1 for k in (3, 2, 1, 0)]
            if any(f >= m for f, m in zip(first, x.shape)):
                continue

            def at(a, off, p=1):
                return a[tuple(slice(p + f + o, p + m + o, 2) for f, o, m in zip(first, off, x.shape))]

            zs, num, den = at(z, (0,) * 4), at(v, (0,) * 4, 0) / sigma ** 2, 1.0 / sigma ** 2
            for off, b in near:
                zr = at(z, off)
                r = ((zs - zr).abs() / (T * SX)) ** (2.0 - Q)
                a = 2.0 * b * at(inside, off) * (1.0 + Q / 2.0 * r) / (2.0 * SX ** 2 * (1.0 + r) ** 2)
                num, den = num + a * zr, den + a
            zs.copy_(num / den)
    return z[1:-1, 1:-1, 1:-1, 1:-1]


def _double(a):
    return torch.as_tensor(a, device="cuda").double()


def _net(x, convs, bns, training=False):
    """centre - R of the network on [B][5][H][W]; BatchNorm with batch or running statistics."""
    a = x
    for l, (w, b) in enumerate(convs):
        z = torch.nn.functional.conv2d(a, w, b, padding=1)
        if 0 < l < 9:
            g, be, mean, var = bns[l - 1]
            z = torch.nn.functional.batch_norm(z, mean, var, g, be, training, 0.1, 1e-5)
        a = z if l == 9 else torch.relu(z)
    return x[:, 2] - a[:, 0]


_ORDER = [(0, 1, 2, 3), (0, 3, 1, 2), (0, 2, 3, 1)]    # [nt][z][y][x] -> [nt][slice][row][col]


def exact(case, seed):
    c, kind = dict(case), case["kind"]
    if kind in SCAN_KINDS:
        applications = {"project": 1, "backproject": 1, "prox_cg": 2 * c.get("n_cg", 0) + 2, "prox_icd": 16 * c.get("n_icd", 0) + 2,
                        "mace_plain": 12 * c.get("iters", 0)}.get(kind)
        rays = c["nt"] * c["views"] * (c["nv"] * c["nu"] * c["n"] + 4e5)
        if applications is None or applications * rays > 2e10:
            return None                        # the learned iteration in FP64, or more than about 20 s of projections
    elif kind == "train" and c["batch"] * c["h"] * c["w"] > 6e5:
        return None
    elif kind == "denoise" and c["nx"] * c["ny"] * c["nz"] * c["nt"] > 3e6:
        return None                            # FP64 convolutions of tens of TFLOP
    elif kind == "qggmrf" and c["nx"] * c["ny"] * c["nz"] * c["nt"] * c["n_sweeps"] > 3e8:
        return None
    i = _inputs(c, seed)
    if kind == "train":
        convs, bns = _network(seed)
        n = lambda a: _double(a.astype(np.float32))  # noqa: E731
        convs = [[n(a).requires_grad_() for a in p] for p in convs]
        bns = [[n(g).requires_grad_(), n(b).requires_grad_(), n(m), n(v)] for g, b, m, v in bns]
        loss = ((_net(i["noisy"].double(), convs, bns, True) - i["clean"].double()) ** 2).mean()
        loss.backward()

        def adam(p):
            if p.grad is None:
                return p
            return p - 1e-3 * p.grad / (p.grad.abs() + 1e-8)       # the first step: m / (sqrt(v) + eps), bias-corrected

        flat = [adam(a).detach().reshape(-1) for p in convs + bns for a in p]
        return dict(loss=float(loss.detach()), params=torch.cat(flat))
    if kind == "denoise":
        convs, bns = _network(seed)
        n = lambda a: _double(a.astype(np.float32))  # noqa: E731
        convs, bns = [[n(a) for a in p] for p in convs], [[n(a) for a in p] for p in bns]
        s4 = i["v"].double().permute(*_ORDER[c["orient"]])
        out = torch.empty_like(s4, memory_format=torch.contiguous_format)
        for t in range(c["nt"]):
            x = torch.stack([s4[min(max(t + k, 0), c["nt"] - 1)] for k in range(-2, 3)], 1)
            for b in range(0, x.shape[0], 16):
                out[t, b:b + 16] = _net(x[b:b + 16], convs, bns)
        return out.permute(*np.argsort(_ORDER[c["orient"]]).tolist()).contiguous()
    d = {k: a.double() for k, a in i.items()}
    if kind == "qggmrf":
        return _qggmrf(d["v"], d["x"], SIGMA, c["n_sweeps"]).contiguous()
    s = _scan(c)
    if kind == "project":
        return _A(d["x"], s)
    if kind == "backproject":
        return _At(d["e"], s)
    if kind == "prox_cg":
        return _prox_cg(d["y"], d["lam"], d["v"], d["x"], s, SIGMA, c["n_cg"])
    if kind == "prox_icd":
        return _prox_icd(d["y"], d["lam"], d["v"], d["x"], s, SIGMA, c["n_icd"])
    W = [torch.zeros((s.nt,) + (s.n,) * 3, device="cuda", dtype=torch.float64) for _ in range(2)]
    X = [w.clone() for w in W]
    for _ in range(c["iters"]):
        X = [_prox_cg(d["y"], d["lam"], W[0], X[0], s, SIGMA, 5), _qggmrf(W[1], X[1], SIGMA, 1)]
        z = 0.25 * (2 * X[0] - W[0]) + 0.75 * (2 * X[1] - W[1])
        W = [w + 2 * 0.5 * (z - x) for w, x in zip(W, X)]
    return dict(W=torch.stack(W), X=torch.stack(X))
