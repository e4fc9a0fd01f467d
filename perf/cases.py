"""What a user of this framework has it do, as cases that can be timed and
compared: integrating star clusters (Hermite with shared and block steps,
the symplectic schemes with and without the Galactic field, many clusters at
once), evaluating forces on an active list or on caller-owned device memory,
differentiating through the leapfrog, and the energy check of a run.

Every case goes through the package's public entry points.  The integrators
hand back what a snapshot holds, positions and velocities, in the arrays a
program keeps for it in pinned memory; force calls hand back their
acceleration and jerk, the adjoint its gradients, the diagnostic its
energies.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_0909_0879_gb300 import _lib, ics
from paper_0909_0879_gb300.autograd import leapfrog


def listed():
    return [
        # A small cluster driven step by step from the host (the shared-step
        # N = 1024 configuration): launches, synchronisations and a snapshot.
        dict(name="hermite_1k", kind="hermite", model="plummer", n=1024, prec="ds", eps=1e-3,
             lev=8, steps=8),
        # A mid-size, ragged run of the paper's own system (uniform sphere
        # with a mass spectrum) in FP32, shared steps.
        dict(name="hermite_sphere_100k_fp32", kind="hermite", model="sphere", n=100003,
             prec="fp32", eps=-1.0, lev=12, steps=1),
        # The headline configuration: one shared Hermite step of a million
        # particles of a King cluster, stored in the library's spatial order, with
        # a step that resolves the softening length at the cluster's velocities.
        dict(name="hermite_king_1m", kind="hermite", model="king", n=1048576, prec="ds",
             eps=1e-4, lev=12, steps=1),
        # Individual (block) time steps: a checkpoint is resumed, advanced by
        # some hundred block steps on the device and read back.
        dict(name="blocks_64k", kind="blocks", n=65536, prec="ds", eps=1e-4, blocks=512),
        # The paper's sixth-order integrator on its own system.
        dict(name="symplectic6_64k", kind="symplectic", model="sphere", n=65536, prec="ds",
             eps=-1.0, order=6, dt=2.0**-11, steps=1, field=False),
        # A cluster on its orbit in the Galactic field, leapfrog, FP32, an
        # odd number of particles.
        dict(name="leapfrog_field_20k_fp32", kind="symplectic", model="galactic", n=20011,
             prec="fp32", eps=1e-4, order=2, dt=2.0**-12, steps=4, field=True),
        # Forces on an active list far shorter than the system, as a
        # block-step driver outside the library asks for them.
        dict(name="active_3k_of_262k", kind="active", n=262147, n_act=3001, prec="ds", eps=1e-4),
        # Forces of a whole small unsoftened system in caller-owned memory.
        dict(name="noalloc_8k_eps0", kind="noalloc", n=8000, prec="ds", eps=0.0),
        # A population study: a thousand clusters of 16..1024 stars.
        dict(name="batched_1000", kind="batched", clusters=1000, prec="ds", steps=50),
        # Fitting initial conditions: gradients through 64 leapfrog steps.
        dict(name="adjoint_4k", kind="adjoint", n=4096, eps=0.05, steps=64, ckpt=8),
        # The differentiable leapfrog run forward only, at a large odd size.
        dict(name="forward_131k", kind="forward", n=131101, eps=0.01, steps=4),
        # The energy check around any run.
        dict(name="energy_64k", kind="energy", n=65536, prec="ds", eps=1e-4),
    ]


def _log(rng, lo, hi):
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return max(lo, min(hi, n))


def draw(rng):
    kind = rng.choice(["hermite", "hermite", "blocks", "symplectic", "symplectic", "active",
                       "noalloc", "batched", "adjoint", "forward", "energy"])
    prec = rng.choice(["ds", "fp32"])
    soft = rng.choice([0.0, 1e-4, 1e-3, 1e-2])
    if kind == "hermite":
        n = _log(rng, 300, 900000)
        model = rng.choice(["plummer", "sphere", "king"])
        eps = -1.0 if model == "sphere" else max(soft, 1e-4)
        if n <= 2048:
            return dict(kind=kind, model=model, n=n, prec=prec, eps=eps, lev=8, steps=8)
        return dict(kind=kind, model=model, n=n, prec=prec, eps=eps, lev=12, steps=1)
    if kind == "blocks":
        return dict(kind=kind, n=_log(rng, 2000, 65536), prec="ds", eps=max(soft, 1e-4),
                    blocks=rng.choice([64, 256, 512]))
    if kind == "symplectic":
        model = rng.choice(["sphere", "galactic"])
        return dict(kind=kind, model=model, n=_log(rng, 1000, 300000), prec=prec,
                    eps=-1.0 if model == "sphere" else 1e-4, order=rng.choice([2, 6]),
                    dt=2.0**-11 if model == "sphere" else 2.0**-12, steps=1,
                    field=model == "galactic")
    if kind == "active":
        n = _log(rng, 20000, 600000)
        return dict(kind=kind, n=n, n_act=min(n, _log(rng, 10, 30000)), prec=prec, eps=soft)
    if kind == "noalloc":
        return dict(kind=kind, n=_log(rng, 500, 60000), prec=prec, eps=soft)
    if kind == "batched":
        return dict(kind=kind, clusters=_log(rng, 50, 1500), prec=prec,
                    steps=rng.choice([10, 20, 50]))
    if kind == "adjoint":
        return dict(kind=kind, n=_log(rng, 200, 16000), eps=0.05,
                    steps=rng.choice([10, 32, 50, 64]), ckpt=rng.choice([1, 8, 16]))
    if kind == "forward":
        return dict(kind=kind, n=_log(rng, 1000, 400000), eps=0.01, steps=rng.choice([1, 4]))
    return dict(kind=kind, n=_log(rng, 1000, 130000), prec=prec, eps=max(soft, 1e-4))


def _eps(case):
    """A negative softening stands for a tenth of the mean distance, the
    paper's choice of a fraction of it."""
    e = case["eps"]
    return e if e >= 0 else 0.1 * (4.0 * math.pi / (3.0 * case["n"])) ** (1.0 / 3.0)


def _model(case, seed):
    """Masses, positions and velocities of the case's system (host, FP64)."""
    n, model = case["n"], case.get("model", "plummer")
    if model == "king":
        m, x, v = ics.king(n, 7.0, seed)
    elif model == "sphere":
        m, x, v = ics.uniform_sphere(n, seed, Q=1.0, masses=ics.salpeter_masses(n, seed + 1))
    elif model == "galactic":
        # 1e5 solar masses, virial radius 10 pc, at 8.5 kpc on a circular orbit
        m, x, v = ics.plummer(n, seed)
        mass, length = 0.00431, 0.01
        m, x = m * mass, x * length + np.array([8.5, 0.0, 0.0])
        v = v * math.sqrt(mass / length) + np.array([0.0, 22.0, 0.0])
    elif case["kind"] in ("blocks", "active", "energy"):
        m, x, v = ics.plummer(n, seed, masses=ics.salpeter_masses(n, seed + 1))
    else:
        m, x, v = ics.plummer(n, seed)
    if model == "king" and n >= 65536:
        p = _lib.spatial_order(x, 256)
        m, x, v = m[p], x[p], v[p]
    return m, x, v


def _active(case, seed):
    return ics.random_active_subset(case["n"], case["n_act"], seed + 7)


def _clusters(case, seed):
    """Offsets, masses, positions and velocities of the case's clusters:
    Plummer spheres of unit mass; the case fixes their sizes."""
    sizes = ics.cluster_sizes(case["clusters"], 1004)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    parts = [ics.plummer(int(k), (seed, c)) for c, k in enumerate(sizes)]
    return (off, np.concatenate([p[0] for p in parts]), np.concatenate([p[1] for p in parts]),
            np.concatenate([p[2] for p in parts]))


def _pinned(n, keys):
    return {k: torch.empty((n, 3), dtype=torch.float64, pin_memory=True).numpy() for k in keys}


def _gpu(a, dtype=torch.float64):
    return torch.tensor(a, dtype=dtype, device="cuda")


def prepare(case, seed):
    kind, st = case["kind"], dict(case=case)
    if kind == "batched":
        off, m, x, v = _clusters(case, seed)
        st["batch"] = _lib.Batch(off, m, x, v, eps=1e-2, lev_shared=8, precision=case["prec"])
        return st
    m, x, v = _model(case, seed)
    n, eps = case["n"], _eps(case)
    if kind in ("adjoint", "forward"):
        f = torch.float32
        st["leaf"] = [_gpu(a, f).requires_grad_(kind == "adjoint") for a in (x, v, m)]
        if kind == "adjoint":
            g = np.random.default_rng(seed + 3)
            st["cot"] = [_gpu(g.normal(size=(n, 3)), f) for _ in range(2)]
        return st
    if kind == "noalloc":
        st["in"] = [_gpu(a) for a in (m, x, v)]
        st["out"] = [torch.empty((n, 3), dtype=torch.float64, device="cuda") for _ in range(2)]
        return st
    kw = dict(eps=eps, precision=case["prec"])
    if kind == "hermite":
        kw.update(block_steps=False, lev_shared=case["lev"])
    elif kind == "blocks":
        kw.update(eta=0.01, lev_min=3, lev_max=20)
    s = st["sys"] = _lib.NBody(m, x, v, **kw)
    if kind == "active":
        st["idx"] = torch.from_numpy(_active(case, seed)).cuda()
        st["out"] = [torch.empty((case["n_act"], 3), dtype=torch.float64, device="cuda")
                     for _ in range(2)]
        s.predict(0.0)
    elif kind == "symplectic":
        if case["field"]:
            s.set_external({})
    if kind == "blocks":
        st["checkpoint"] = s.get_state()
    if kind in ("hermite", "blocks", "symplectic"):
        st["snap"] = _pinned(n, ("x", "v"))
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "hermite":
        s = state["sys"]
        for _ in range(case["steps"]):
            s.step()
        return s.get_state(want=("x", "v"), out=state["snap"])
    if kind == "blocks":
        s = state["sys"]
        s.set_state(state["checkpoint"])
        done, t = s.run_blocks(1.0, max_blocks=case["blocks"])
        return dict(s.get_state(want=("x", "v"), out=state["snap"]), done=done, t=t)
    if kind == "symplectic":
        s = state["sys"]
        s.symplectic(case["order"], case["dt"], case["steps"])
        return s.get_state(want=("x", "v"), out=state["snap"])
    if kind == "active":
        acc, jerk = state["out"]
        state["sys"].force_jerk_dev(state["idx"], case["n_act"], acc, jerk)
        return acc, jerk
    if kind == "noalloc":
        (m, x, v), (acc, jerk) = state["in"], state["out"]
        _lib.force_jerk_noalloc(case["n"], m, x, v, None, case["n"], acc, jerk, eps=_eps(case),
                                precision=case["prec"])
        return acc, jerk
    if kind == "batched":
        b = state["batch"]
        b.run(case["steps"])
        st = b.get_state()
        return st["x"], st["v"]
    if kind == "adjoint":
        x0, v0, m = state["leaf"]
        xT, vT = leapfrog(x0, v0, m, case["steps"], 1.0 / 128, case["eps"],
                          ckpt_every=case["ckpt"])
        return (xT, vT) + torch.autograd.grad((xT, vT), (x0, v0, m), state["cot"])
    if kind == "forward":
        x0, v0, m = state["leaf"]
        return leapfrog(x0, v0, m, case["steps"], 1.0 / 1024, case["eps"])
    return state["sys"].energy()


# Operations of a pair of particles: the acceleration on one of them, the
# acceleration and jerk on one of them, and the same for both at once.
_A1, _AJ1, _A2, _AJ2 = 19, 44, 26, 54


def work(case):
    n = case.get("n", 0)
    kind = case["kind"]
    if kind == "hermite":
        # (x, v, a, jerk, m) read and all but m written, once per pass
        return dict(bytes=n * 8.0 * 25, flops=case["steps"] * _AJ2 * n * (n - 1) / 2.0)
    if kind == "blocks":
        # a block step advances about 1 % of the particles on average
        return dict(bytes=n * 8.0 * 25, flops=case["blocks"] * 0.01 * _AJ1 * float(n) * n)
    if kind == "symplectic":
        evals = 1 + case["steps"] * (7 if case["order"] == 6 else 1)
        return dict(bytes=n * 8.0 * 13, flops=evals * _A2 * n * (n - 1) / 2.0)
    if kind == "active":
        return dict(bytes=n * 48.0 + case["n_act"] * 52.0, flops=_AJ1 * float(n) * case["n_act"])
    if kind == "noalloc":
        return dict(bytes=n * 8.0 * 13, flops=_AJ2 * n * (n - 1) / 2.0)
    if kind == "batched":
        # sizes are log-uniform on 16..1024: mean 242, mean square 1.26e5
        c = case["clusters"]
        return dict(bytes=c * 242 * 8.0 * 25, flops=case["steps"] * _AJ2 * c * 1.26e5 / 2)
    if kind in ("adjoint", "forward"):
        evals = case["steps"] + 1
        pair = evals * _A2
        if kind == "adjoint":
            pair = evals * (2 * _A2 + 70)  # recomputed forces and the adjoint's pair sum
        return dict(bytes=n * 4.0 * (28 if kind == "adjoint" else 13),
                    flops=pair * n * (n - 1) / 2.0)
    return dict(bytes=n * 8.0 * 7, flops=13.0 * n * (n - 1) / 2.0)


# ---- the same results in plain FP64 torch


def _pairs(x, m, eps, v=None, rows=None):
    """Acceleration (and jerk, with v) on the rows' particles."""
    xi = x if rows is None else x[rows]
    vi = v if rows is None or v is None else v[rows]
    chunk = max(1, int(6e7) // x.shape[0])
    acc, jerk = [], []
    for b in range(0, xi.shape[0], chunk):
        d = [x[None, :, c] - xi[b:b + chunk, None, c] for c in range(3)]
        r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + eps * eps
        y = torch.where(r2 > 0, r2, torch.inf).rsqrt_()
        y2 = y * y
        f = m[None, :] * y * y2
        acc.append(torch.stack([(f * d[c]).sum(1) for c in range(3)], 1))
        if v is not None:
            w = [v[None, :, c] - vi[b:b + chunk, None, c] for c in range(3)]
            q = 3.0 * (d[0] * w[0] + d[1] * w[1] + d[2] * w[2]) * y2
            jerk.append(torch.stack([(f * (w[c] - q * d[c])).sum(1) for c in range(3)], 1))
    acc = torch.cat(acc)
    return acc if v is None else (acc, torch.cat(jerk))


def _hermite(x, v, a, j, force, dt):
    """One shared Hermite step; force(x, v) gives acceleration and jerk."""
    xp = x + dt * (v + dt / 2 * (a + dt / 3 * j))
    vp = v + dt * (a + dt / 2 * j)
    an, jn = force(xp, vp)
    a2 = (-6 * (a - an) - dt * (4 * j + 2 * jn)) / dt**2
    a3 = (12 * (a - an) + 6 * dt * (j + jn)) / dt**3
    return (xp + dt**4 * (a2 / 24 + dt * a3 / 120), vp + dt**3 * (a2 / 6 + dt * a3 / 24), an, jn)


def _galaxy(x):
    """Acceleration of Allen & Santillan's (1991) Galaxy."""
    r2 = (x * x).sum(1, keepdim=True)
    r = r2.sqrt()
    a = -606.0 * x / (r2 + 0.3873**2) ** 1.5
    z = x[:, 2:]
    zeta = (z * z + 0.25**2).sqrt()
    d3 = (x[:, :1] ** 2 + x[:, 1:2] ** 2 + (5.3178 + zeta) ** 2) ** 1.5
    a = a - 3690.0 / d3 * torch.cat([x[:, :2], z * (5.3178 + zeta) / zeta], 1)
    q = r.clamp(max=100.0) / 12.0
    u = q**1.02
    return a - 4615.0 * q * u / (1.0 + u) * x / (r2 * r)


def _weights(order):
    if order == 2:
        return [1.0]
    w1, w2, w3 = -1.17767998417887100695, 0.235573213359358133684, 0.784513610477557263820
    return [w3, w2, w1, 1.0 - 2.0 * (w1 + w2 + w3), w1, w2, w3]


def _vjp(x, m, g, eps):
    """Gradients of sum(g * acc(x, m)) with respect to x and m."""
    gx, gm, chunk = [], [], max(1, int(6e7) // x.shape[0])
    for b in range(0, x.shape[0], chunk):
        k = slice(b, b + chunk)
        d = [x[None, :, c] - x[k, None, c] for c in range(3)]
        y2 = 1.0 / (d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + eps * eps)
        y3 = y2 * y2.sqrt()
        u = [m[k, None] * g[None, :, c] - m[None, :] * g[k, None, c] for c in range(3)]
        q = 3.0 * (d[0] * u[0] + d[1] * u[1] + d[2] * u[2]) * y2
        gx.append(torch.stack([(y3 * (u[c] - q * d[c])).sum(1) for c in range(3)], 1))
        gm.append(-(y3 * sum(g[None, :, c] * d[c] for c in range(3))).sum(1))
    return torch.cat(gx), torch.cat(gm)


def _exact_batched(case, seed):
    off, m, x, v = (torch.from_numpy(a).cuda() for a in _clusters(case, seed))
    size = off[1:] - off[:-1]
    out = [torch.empty_like(x), torch.empty_like(v)]
    order = torch.argsort(size).tolist()
    dt = 2.0**-8
    while order:
        # clusters of like size as one padded stack (massless padding)
        cl = order[-48:]
        order = order[:-48]
        k = int(size[cl].max())
        at = off[cl][:, None] + torch.arange(k, device="cuda")[None, :]
        real = torch.arange(k, device="cuda")[None, :] < size[cl][:, None]
        at = torch.where(real, at, off[cl][:, None])
        mm, xx, vv = m[at] * real, x[at], v[at]

        def force(p, q):
            d, w = p[:, None] - p[:, :, None], q[:, None] - q[:, :, None]
            y2 = 1.0 / ((d * d).sum(-1, keepdim=True) + 1e-4)
            f = mm[:, None, :, None] * y2 * y2.sqrt()
            w = w - 3.0 * (d * w).sum(-1, keepdim=True) * y2 * d
            return (f * d).sum(2), (f * w).sum(2)

        a, j = force(xx, vv)
        for _ in range(case["steps"]):
            xx, vv, a, j = _hermite(xx, vv, a, j, force, dt)
        out[0][at[real]], out[1][at[real]] = xx[real], vv[real]
    return tuple(o.cpu() for o in out)


def exact(case, seed):
    kind = case["kind"]
    n = case.get("n", 0)
    if kind == "batched":
        return _exact_batched(case, seed)
    if kind == "blocks":
        return None  # a schedule of its own; the library's is compared with itself
    pairs = {"hermite": 2 * n * n * case.get("steps", 1), "active": n * case.get("n_act", 0),
             "symplectic": 8 * n * n, "adjoint": 5 * n * n * case.get("steps", 1),
             "forward": 5 * n * n}.get(kind, n * n)
    if pairs > 1.2e11:
        return None
    m, x, v = (_gpu(a) for a in _model(case, seed))
    eps = _eps(case)
    if kind == "hermite":
        def force(p, q):
            return _pairs(p, m, eps, q)

        a, j = force(x, v)
        for _ in range(case["steps"]):
            x, v, a, j = _hermite(x, v, a, j, force, 2.0 ** -case["lev"])
        return dict(x=x, v=v)
    if kind == "symplectic":
        def acc(p):
            return _pairs(p, m, eps) + (_galaxy(p) if case["field"] else 0.0)

        a = acc(x)
        for _ in range(case["steps"]):
            for w in _weights(case["order"]):
                h = w * case["dt"]
                v = v + 0.5 * h * a
                x = x + h * v
                a = acc(x)
                v = v + 0.5 * h * a
        return dict(x=x, v=v)
    if kind == "active":
        return _pairs(x, m, eps, v, torch.from_numpy(_active(case, seed)).cuda().long())
    if kind == "noalloc":
        return _pairs(x, m, eps, v)
    if kind in ("adjoint", "forward"):
        # the FP32 inputs, in 64 bits
        x, v, m = (t.float().double() for t in (x, v, m))
        h = 1.0 / 128 if kind == "adjoint" else 1.0 / 1024
        path, a = [x], _pairs(x, m, eps)
        for _ in range(case["steps"]):
            v = v + 0.5 * h * a
            x = x + h * v
            a = _pairs(x, m, eps)
            v = v + 0.5 * h * a
            path.append(x)
        if kind == "forward":
            return x, v
        g = np.random.default_rng(seed + 3)
        lx, lv = (_gpu(g.normal(size=(n, 3)), torch.float32).double() for _ in range(2))
        lm = torch.zeros_like(m)
        for k in range(case["steps"], 0, -1):
            dx, dm = _vjp(path[k], m, 0.5 * h * lv, eps)
            lx, lm = lx + dx, lm + dm
            lv = lv + h * lx
            dx, dm = _vjp(path[k - 1], m, 0.5 * h * lv, eps)
            lx, lm = lx + dx, lm + dm
        return x, v, lx, lv, lm
    if kind == "energy":
        kin = 0.5 * (m * (v * v).sum(1)).sum().item()
        pot, chunk = 0.0, max(1, int(6e7) // n)
        for b in range(0, n, chunk):
            d = [x[None, :, c] - x[b:b + chunk, None, c] for c in range(3)]
            y = (d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + eps * eps).rsqrt_()
            pot -= 0.5 * (m[b:b + chunk] * ((m[None, :] * y).sum(1) - m[b:b + chunk] / eps)
                          ).sum().item()
        return kin, pot, kin + pot
    return None
