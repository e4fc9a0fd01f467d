"""GPU parity of the differentiable leapfrog (FP32 forward, hand-written
adjoint, checkpointed reverse pass, torch.autograd) against the FP64
oracle's exact discrete adjoint.  Bar: relative L2 <= 1e-3 for each of
dL/dx0, dL/dv0, dL/dm (FP32 arithmetic against FP64)."""
import numpy as np
import pytest

from paper_0909_0879_gb300 import ics

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0909_0879_gb300 import _lib

    _lib.load()
    return torch


def rel_l2(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def test_acc_and_vjp_kernels_match_oracle(torch_cuda, oracle_mod):
    torch = torch_cuda
    from paper_0909_0879_gb300 import _lib

    for n, eps in ((1, 1e-3), (37, 1e-3), (257, 0.0), (3000, 1e-3)):
        m, x, v = ics.plummer(n, 900 + n) if n > 1 else (np.ones(1), np.zeros((1, 3)), np.zeros((1, 3)))
        g = np.random.default_rng(n).normal(size=(n, 3))
        dx = torch.tensor(x, dtype=torch.float32, device="cuda")
        dm = torch.tensor(m, dtype=torch.float32, device="cuda")
        dg = torch.tensor(g, dtype=torch.float32, device="cuda")
        acc = torch.empty((n, 3), dtype=torch.float32, device="cuda")
        gx = torch.empty_like(acc)
        gm = torch.empty(n, dtype=torch.float32, device="cuda")
        _lib.lf_acc(n, dx, dm, acc, eps=eps)
        _lib.lf_acc_vjp(n, dx, dm, dg, gx, gm, eps=eps)
        torch.cuda.synchronize()
        # the oracle sees the same float32-rounded inputs
        xr = dx.double().cpu().numpy()
        mr = dm.double().cpu().numpy()
        gr = dg.double().cpu().numpy()
        ra = oracle_mod.acc(mr, xr, eps)
        rgx, rgm = oracle_mod.acc_vjp(mr, xr, gr, eps)
        if n == 1:
            assert np.all(acc.cpu().numpy() == 0) and np.all(gm.cpu().numpy() == 0)
            continue
        assert rel_l2(acc.double().cpu().numpy(), ra) < 1e-5
        assert rel_l2(gx.double().cpu().numpy(), rgx) < 1e-4
        assert rel_l2(gm.double().cpu().numpy(), rgm) < 1e-4


@pytest.mark.parametrize("n", [65536, 131101, 262401])
@pytest.mark.parametrize("eps", [1e-3, 0.0])
def test_wide_acc_shape_large_n(torch_cuda, oracle_mod, eps, n):
    """N >= 65,536 takes the wide acceleration shape (4 particles per
    thread, packed pairs, 4 or 8 threads per particle group): the smallest
    such N, and two ragged ones, n = 131,101 (8 threads per group on 152
    SMs) and 262,401 (4 threads), against the FP64 oracle on 512 sampled
    particles, same float32-rounded inputs."""
    torch = torch_cuda
    from paper_0909_0879_gb300 import _lib

    m, x, v = ics.plummer(n, 905)
    dx = torch.tensor(x, dtype=torch.float32, device="cuda")
    dm = torch.tensor(m, dtype=torch.float32, device="cuda")
    acc = torch.empty((n, 3), dtype=torch.float32, device="cuda")
    _lib.lf_acc(n, dx, dm, acc, eps=eps)
    torch.cuda.synchronize()
    xr = dx.double().cpu().numpy()
    mr = dm.double().cpu().numpy()
    sample = np.sort(np.random.default_rng(6).choice(n, 512, replace=False)).astype(np.int32)
    ra, _ = oracle_mod.force_jerk(mr, xr, np.zeros_like(xr), eps, idx=sample)
    got = acc.double().cpu().numpy()[sample]
    assert np.all(np.isfinite(got))
    assert rel_l2(got, ra) < 1e-5


def test_leapfrog_adjoint_n4096(torch_cuda, oracle_mod):
    """N = 4096 Plummer, eps = 1e-3, 64 KDK steps of dt = 1/128 in FP32,
    checkpoints every 8 steps; L = sum |x(T) - y|^2 with y = x0 + N(0,0.05^2)
    (seed 5).  (a) The GPU gradient against the oracle's FP64 reverse sweep
    along the GPU's own FP32 trajectory: relative L2 <= 1e-4 (adjoint
    arithmetic).  (b) Against the oracle's fully FP64 run: relative L2 <=
    1e-2; the FP32 and FP64 trajectories separate through close encounters
    over the 64 steps, which bounds this agreement (about 4e-3 measured)."""
    torch = torch_cuda
    from paper_0909_0879_gb300 import _lib
    from paper_0909_0879_gb300.autograd import leapfrog

    n, eps, dt, steps = 4096, 1e-3, 1.0 / 128, 64
    m, x, v = ics.plummer(n, 1005)
    y = x + np.random.default_rng(5).normal(0.0, 0.05, x.shape)
    x0 = torch.tensor(x, dtype=torch.float32, device="cuda", requires_grad=True)
    v0 = torch.tensor(v, dtype=torch.float32, device="cuda", requires_grad=True)
    mm = torch.tensor(m, dtype=torch.float32, device="cuda", requires_grad=True)
    yt = torch.tensor(y, dtype=torch.float32, device="cuda")
    xT, vT = leapfrog(x0, v0, mm, steps, dt, eps, ckpt_every=8)
    loss = ((xT - yt) ** 2).sum()
    loss.backward()
    torch.cuda.synchronize()
    g_gpu = [t.grad.double().cpu().numpy() for t in (x0, v0, mm)]
    # the GPU's own trajectory, every step (checkpoint interval 1)
    xw = x0.detach().clone()
    vw = v0.detach().clone()
    acc = torch.empty_like(xw)
    ck = torch.empty(_lib.lf_ckpt_floats(n, steps, 1), dtype=torch.float32, device="cuda")
    _lib.lf_forward(n, mm.detach(), xw, vw, acc, steps, dt, ck, eps=eps, ckpt_every=1)
    torch.cuda.synchronize()
    path = ck.view(steps, 2, n, 3)[:, 0].double().cpu().numpy()
    xs = np.concatenate([path, xw.double().cpu().numpy()[None]], axis=0)
    assert np.array_equal(xs[-1], xT.detach().double().cpu().numpy())
    mr = mm.detach().double().cpu().numpy()
    lx_T = 2.0 * (xs[-1] - yt.double().cpu().numpy())
    g_path = oracle_mod.leapfrog_adjoint_path(mr, xs, lx_T, np.zeros((n, 3)), eps, dt)
    e_path = [rel_l2(a, b) for a, b in zip(g_gpu, g_path)]
    xr = x0.detach().double().cpu().numpy()
    vr = v0.detach().double().cpu().numpy()
    L, gx, gv, gm = oracle_mod.leapfrog_loss_grad(mr, xr, vr, y, eps, dt, steps)
    e_full = [rel_l2(a, b) for a, b in zip(g_gpu, (gx, gv, gm))]
    print("loss gpu %.8e oracle %.8e; same-path rel L2 %s; FP64-run rel L2 %s"
          % (loss.item(), L, ["%.2e" % e for e in e_path], ["%.2e" % e for e in e_full]))
    assert abs(loss.item() - L) <= 1e-4 * L
    assert max(e_path) <= 1e-4
    assert max(e_full) <= 1e-2


def test_checkpoint_interval_does_not_change_gradients(torch_cuda):
    """Recomputing from checkpoints reproduces the forward pass exactly, so
    the gradient is bit-identical for any checkpoint interval."""
    torch = torch_cuda
    from paper_0909_0879_gb300.autograd import leapfrog

    n = 500
    m, x, v = ics.plummer(n, 3)
    grads = []
    for ck in (1, 3, 8, 64):
        x0 = torch.tensor(x, dtype=torch.float32, device="cuda", requires_grad=True)
        v0 = torch.tensor(v, dtype=torch.float32, device="cuda", requires_grad=True)
        mm = torch.tensor(m, dtype=torch.float32, device="cuda", requires_grad=True)
        xT, vT = leapfrog(x0, v0, mm, 20, 1.0 / 128, 1e-3, ckpt_every=ck)
        (xT.square().sum() + 0.5 * vT.square().sum()).backward()
        grads.append([t.grad.cpu().numpy() for t in (x0, v0, mm)])
    for g in grads[1:]:
        for a, b in zip(g, grads[0]):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("n", [31, 511, 512, 513, 1025, 2049, 4864, 4865, 9729])
@pytest.mark.parametrize("eps", [0.05, 0.0])
def test_acc_and_vjp_at_tile_and_group_edges(torch_cuda, oracle_mod, n, eps):
    """Record tiles of 512 (force) and 1,024 (vector-Jacobian product), 32
    particles per group, one group per SM up to n = 4,864 on 152 SMs: sizes
    at and just past those edges against the oracle, same float32 inputs."""
    torch = torch_cuda
    from paper_0909_0879_gb300 import _lib

    m, x, v = ics.plummer(n, 910 + n)
    g = np.random.default_rng(n).normal(size=(n, 3))
    dx, dm, dg = (torch.tensor(a, dtype=torch.float32, device="cuda") for a in (x, m, g))
    acc = torch.full((n, 3), np.nan, dtype=torch.float32, device="cuda")
    gx = torch.full_like(acc, np.nan)
    gm = torch.full((n,), np.nan, dtype=torch.float32, device="cuda")
    _lib.lf_acc(n, dx, dm, acc, eps=eps)
    _lib.lf_acc_vjp(n, dx, dm, dg, gx, gm, eps=eps)
    xr, mr, gr = (t.double().cpu().numpy() for t in (dx, dm, dg))
    ra = oracle_mod.acc(mr, xr, eps)
    rgx, rgm = oracle_mod.acc_vjp(mr, xr, gr, eps)
    assert rel_l2(acc.double().cpu().numpy(), ra) < 1e-5
    assert rel_l2(gx.double().cpu().numpy(), rgx) < 1e-4
    assert rel_l2(gm.double().cpu().numpy(), rgm) < 1e-4


@pytest.mark.parametrize("nsteps,ckpt", [(1, 1), (1, 8), (2, 1), (3, 2), (5, 3), (6, 3)])
def test_short_runs_and_segments(torch_cuda, oracle_mod, nsteps, ckpt):
    """Odd and even step counts (the positions alternate between two
    buffers), one or several segments, full or short last one: end state,
    final acceleration and gradients against the oracle."""
    torch = torch_cuda
    from paper_0909_0879_gb300 import _lib
    from paper_0909_0879_gb300.autograd import leapfrog

    n, eps, dt = 300, 0.05, 1.0 / 64
    m, x, v = ics.plummer(n, 77)
    y = x + np.random.default_rng(7).normal(0.0, 0.05, x.shape)
    leaves = [torch.tensor(a, dtype=torch.float32, device="cuda", requires_grad=True)
              for a in (x, v, m)]
    xT, vT = leapfrog(*leaves, nsteps, dt, eps, ckpt_every=ckpt)
    ((xT - torch.tensor(y, dtype=torch.float32, device="cuda")) ** 2).sum().backward()
    xr, vr, mr = (t.detach().double().cpu().numpy() for t in leaves)
    _, gx, gv, gm = oracle_mod.leapfrog_loss_grad(mr, xr, vr, y, eps, dt, nsteps)
    for t, r in zip(leaves, (gx, gv, gm)):
        assert rel_l2(t.grad.double().cpu().numpy(), r) < 1e-4
    # the acceleration left behind is A(x) at the returned positions
    xw, vw = leaves[0].detach().clone(), leaves[1].detach().clone()
    acc = torch.empty_like(xw)
    _lib.lf_forward(n, leaves[2].detach(), xw, vw, acc, nsteps, dt, None, eps=eps)
    assert torch.equal(xw, xT.detach()) and torch.equal(vw, vT.detach())
    ra = oracle_mod.acc(mr, xw.double().cpu().numpy(), eps)
    assert rel_l2(acc.double().cpu().numpy(), ra) < 1e-5


@pytest.mark.parametrize("n", [16384, 16385, 17 * 1024 + 300])
@pytest.mark.parametrize("eps", [0.05, 0.0])
def test_lent_scratch_takes_each_pair_once(torch_cuda, n, eps):
    """The forward steps with scratch on loan: accelerations against FP64 sums
    of the same FP32 inputs (a term is off by at most ~15 u, a chain of 64
    terms by 64 u of their absolute sum, u = 2^-24), two steps and their
    gradient against the run without it (a kick is off by twice that, plus
    the roundings of x and v; a pair's tidal tensor by a few of the offset in
    x over its distance), and too little scratch changes no bit."""
    torch = torch_cuda
    from paper_0909_0879_gb300 import _lib

    m, x, v = ics.plummer(n, 7, masses=ics.salpeter_masses(n, 7))
    X, V, M = [torch.tensor(a, dtype=torch.float32, device="cuda") for a in (x, v, m)]
    size = _lib.lf_scratch_bytes(n)
    assert size > 0 and _lib.lf_scratch_bytes(16383) == 0
    u, dt = 2.0**-24, 2.0**-9
    idx = torch.cat([torch.arange(64), torch.arange(n - 64, n),
                     torch.arange(100, n, 97)]).cuda()
    d = X.double()[None] - X.double()[idx][:, None]
    s2 = (d * d).sum(-1) + eps * eps
    t = torch.where(s2 > 0, M.double() * s2**-1.5, 0.0)[..., None] * d
    ref, size_of = t.sum(1), t.abs().sum(1)
    out = {}
    for side, lent in (("one", None), ("pairs", size), ("little", size - 256)):
        sc = None if lent is None else torch.empty(lent, dtype=torch.uint8, device="cuda")
        acc, xs, vs = torch.empty_like(X), X.clone(), V.clone()
        _lib.lf_forward(n, M, xs, vs, acc, 0, dt, None, eps=eps, scratch=sc)
        a0 = acc.clone()
        ck = torch.empty(_lib.lf_ckpt_floats(n, 2, 2), dtype=torch.float32, device="cuda")
        _lib.lf_forward(n, M, xs, vs, acc, 2, dt, ck, eps=eps, ckpt_every=2, scratch=sc)
        lx, lv, lm = X.clone(), V.clone(), torch.empty_like(M)
        work = torch.empty(_lib.lf_work_floats(n, 2), dtype=torch.float32, device="cuda")
        _lib.lf_backward(n, M, ck, 2, dt, lx, lv, lm, work, eps=eps, ckpt_every=2, scratch=sc)
        out[side] = [a.double() for a in (a0, xs, vs, acc, lx, lv, lm)]
    assert all(torch.equal(a, b) for a, b in zip(out["one"], out["little"]))
    assert not torch.equal(out["one"][0], out["pairs"][0])
    err = (out["pairs"][0][idx] - ref).abs()
    assert bool((err <= 80 * u * size_of).all()), (err / size_of).max().item() / u
    da = 2 * 80 * u * size_of.max().item()
    dv = 2 * dt * da + 8 * u * V.abs().max().item()
    assert (out["pairs"][2] - out["one"][2]).abs().max().item() <= dv
    dx = 2 * dt * dv + 8 * u * X.abs().max().item()
    assert (out["pairs"][1] - out["one"][1]).abs().max().item() <= dx
    gap = min(torch.where(r > 0, r, 9.0).min().item()
              for r in (torch.cdist(c, X.double()) for c in X.double().split(1024)))
    bar = 1e-5 + 12 * dx / np.hypot(gap, eps)
    for a, b in zip(out["pairs"][4:], out["one"][4:]):
        assert ((a - b).norm() <= bar * b.norm()).item()


@pytest.mark.parametrize("mass,length", [(2e30, 1e17), (2e33, 3e18), (1.0, 1.0), (1e-30, 1e-8)])
def test_lent_scratch_in_other_units(torch_cuda, mass, length):
    """Masses and lengths in SI and cgs units (stars, a parsec), masses of 1 and
    tiny ones: the pair-symmetric forward steps against FP64 sums of the same
    FP32 inputs and the run without scratch, with the bars of the test above;
    masses and lengths on powers of two of N-body units scale every bit."""
    torch = torch_cuda
    from paper_0909_0879_gb300 import _lib

    n, u = 16384, 2.0**-24
    m, x, v = ics.plummer(n, 7, masses=ics.salpeter_masses(n, 7))
    m = m * n * mass
    x = x * (length / np.abs(x).max())
    X, M = [torch.tensor(a, dtype=torch.float32, device="cuda") for a in (x, m)]
    eps = float(np.float32(1e-3 * length))
    idx = torch.arange(0, n, 97, device="cuda")
    d = X.double()[None] - X.double()[idx][:, None]
    t = (M.double() * ((d * d).sum(-1) + eps * eps)**-1.5)[..., None] * d
    ref, size_of = t.sum(1), t.abs().sum(1)
    sc = torch.empty(_lib.lf_scratch_bytes(n), dtype=torch.uint8, device="cuda")
    # a fourth of the softening in a step of this length from rest
    dt = float(np.sqrt(0.25 * eps / size_of.max().item()))
    out = []
    for lent in (sc, None):
        acc, xs, vs = torch.empty_like(X), X.clone(), torch.zeros_like(X)
        _lib.lf_forward(n, M, xs, vs, acc, 0, dt, None, eps=eps, scratch=lent)
        a0 = acc.clone()
        _lib.lf_forward(n, M, xs, vs, acc, 2, dt, None, eps=eps, scratch=lent)
        out.append([a.double() for a in (a0, xs, vs)])
    err = (out[0][0][idx] - ref).abs()
    assert bool((err <= 80 * u * size_of).all()), (err / size_of).max().item() / u
    da = 2 * 80 * u * size_of.max().item()
    dv = 2 * dt * da + 8 * u * out[1][2].abs().max().item()
    assert (out[0][2] - out[1][2]).abs().max().item() <= dv
    dx = 2 * dt * dv + 8 * u * X.abs().max().item()
    assert (out[0][1] - out[1][1]).abs().max().item() <= dx


@pytest.mark.parametrize("n", [16384, 65537])
def test_lent_scratch_scales_exactly(torch_cuda, n):
    """Powers of two on masses and lengths change no other bit of the
    acceleration (four and eight i-particles per thread)."""
    torch = torch_cuda
    from paper_0909_0879_gb300 import _lib

    m, x, v = ics.plummer(n, 7, masses=ics.salpeter_masses(n, 7))
    sc = torch.empty(_lib.lf_scratch_bytes(n), dtype=torch.uint8, device="cuda")
    res = []
    for pm, px in ((0, 0), (100, 50), (110, 61), (-40, -20)):
        X, M = [torch.tensor(a, dtype=torch.float32, device="cuda") for a in (x, m)]
        X, M = X * 2.0**px, M * 2.0**pm
        acc = torch.empty_like(X)
        _lib.lf_forward(n, M, X, torch.zeros_like(X), acc, 0, 0.0, None, eps=2.0**(px - 10),
                        scratch=sc)
        res.append(acc.double() * 2.0**(2 * px - pm))
    for a in res[1:]:
        assert torch.equal(a, res[0])


def test_backward_lends_only_what_forward_had(torch_cuda, monkeypatch):
    """The forward pass found no room for scratch and the backward pass does: the
    segments are re-run without it, so the gradients are those of a run that never
    had any."""
    torch = torch_cuda
    from paper_0909_0879_gb300 import autograd

    n = 16384
    m, x, v = ics.plummer(n, 7)
    real, grads = autograd._scratch, []
    for room in ((False, False), (False, True), (True, True)):
        asked = iter(room)
        monkeypatch.setattr(autograd, "_scratch",
                            lambda *a: real(*a) if next(asked, False) else None)
        leaves = [torch.tensor(a, dtype=torch.float32, device="cuda", requires_grad=True)
                  for a in (x, v, m)]
        xT, vT = autograd.leapfrog(*leaves, 6, 2.0**-9, 1e-2, ckpt_every=3)
        (xT.square().sum() + 0.5 * vT.square().sum()).backward()
        grads.append([t.grad for t in leaves])
    assert all(torch.equal(a, b) for a, b in zip(grads[0], grads[1]))
    assert not all(torch.equal(a, b) for a, b in zip(grads[0], grads[2]))
