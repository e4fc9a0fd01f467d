"""The pair-symmetric force of all particles (contexts with shared steps,
symplectic steps) against the FP64 oracle and the one-sided kernel, at the
edges of its block ring; bars as for the one-sided kernel (FP32 pair
arithmetic: condition-relative and norm-wise, 1e-6 / 1e-5 in split
precision)."""
import os

import numpy as np
import pytest

from paper_0909_0879_gb300 import ics

pytestmark = pytest.mark.gpu

TOL = {"ds": (1e-6, 1e-5), "fp32": (1e-3, 1e-3)}
MIN_N = 16384  # smallest n of the pair-symmetric kernel


@pytest.fixture(scope="module")
def nb():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0909_0879_gb300 import _lib

    _lib.load()
    return _lib


def _system(nb, n, sort, seed=31, equal=False):
    m, x, v = ics.plummer(n, seed, masses=None if equal else ics.salpeter_masses(n, seed))
    if sort:
        p = nb.spatial_order(x, 256)
        m, x, v = m[p], x[p], v[p]
    return m, x, v


# 16 whole blocks (even ring), one particle more (17 blocks, the last one
# with one particle), a last block of two tiles, an odd ring of whole
# blocks; in spatial order most tiles take the far field
@pytest.mark.parametrize("n", [MIN_N, MIN_N + 1, 17 * 1024 + 300, 21 * 1024])
@pytest.mark.parametrize("prec", ["ds", "fp32"])
@pytest.mark.parametrize("eps", [1e-3, 0.0])
@pytest.mark.parametrize("sort", [False, True])
@pytest.mark.parametrize("equal", [False, True])
def test_matches_oracle_and_one_sided(nb, oracle_mod, n, prec, eps, sort, equal):
    """(equal: one mass for all takes a shorter pair loop where no record or
    lane past n is met)"""
    m, x, v = _system(nb, n, sort, equal=equal)
    with nb.NBody(m, x, v, eps=eps, precision=prec, block_steps=False, lev_shared=10) as s:
        got = s.get_state(want=("a", "jerk"))
    with nb.NBody(m, x, v, eps=eps, precision=prec) as s:
        one = s.get_state(want=("a", "jerk"))  # block steps: one-sided
        s.set_symplectic_layout("as_given")
        s.symplectic(2, 0.0, 1)  # the acceleration-only kernel, x unchanged
        acc = s.get_state(want=("a", "x"))
    assert np.array_equal(acc["x"], x)
    idx = np.unique(np.concatenate([np.arange(64), np.arange(n - 64, n),
                                    np.random.default_rng(n).integers(0, n, 900)])).astype(np.int32)
    ra, rj = oracle_mod.force_jerk(m, x, v, eps, idx=idx)
    ca, cj = oracle_mod.force_jerk_abs(m, x, v, eps, idx=idx)
    ta, tj = TOL[prec]
    for a in (got["a"], acc["a"]):
        assert np.max(np.linalg.norm(a[idx] - ra, axis=1) / ca) <= ta
        assert np.linalg.norm(a[idx] - ra) <= ta * np.linalg.norm(ra)
        assert np.linalg.norm(a - one["a"]) <= 2 * ta * np.linalg.norm(one["a"])
    assert np.max(np.linalg.norm(got["jerk"][idx] - rj, axis=1) / cj) <= tj
    assert np.linalg.norm(got["jerk"] - one["jerk"]) <= 2 * tj * np.linalg.norm(one["jerk"])
    # it is the pair-symmetric kernel that ran, not the one-sided one
    assert not np.array_equal(got["a"], one["a"])


@pytest.mark.parametrize("prec,eps", [("ds", 1e-3), ("fp32", 1e-3), ("ds", 0.0)])
def test_step_loop_and_device_steps_agree_bitwise(nb, prec, eps):
    """nb_step, the fused and the general device-resident steps take the same
    kernel for steps of all particles, with the same bits, run after run."""
    n = MIN_N + 1
    m, x, v = _system(nb, n, True)
    kw = dict(eps=eps, precision=prec, block_steps=False, lev_shared=10)
    res = []
    for mode in ("step", "step", "auto", "general"):
        with nb.NBody(m, x, v, **kw) as s:
            if mode == "step":
                for _ in range(3):
                    s.step()
            else:
                s.set_block_mode(mode)
                assert s.run_blocks(3 * 2.0**-10)[0] == 3
            res.append(s.get_state())
    for st in res[1:]:
        for k in st:
            assert np.array_equal(st[k], res[0][k]), k


def test_one_sided_where_rows_or_shapes_are_asked_for_and_without_scratch(nb):
    """Rows of the active list handed to the caller are those an index list
    gives; a forced shape is the shape that runs; without room for the
    partial sums the one-sided kernel runs and the call succeeds."""
    n = MIN_N
    m, x, v = _system(nb, n, False)
    kw = dict(eps=1e-3, block_steps=False, lev_shared=10)
    with nb.NBody(m, x, v, **kw) as s:
        t, na = s.next_block()
        s.predict(t)
        a, j = s.force_jerk()
        ai, ji = s.force_jerk(np.arange(n))
        assert np.array_equal(a, ai) and np.array_equal(j, ji)
        s.correct(t)
        rows = s.get_state(want=("a",))["a"]
        assert np.array_equal(rows, a)
    with nb.NBody(m, x, v, **kw) as s:
        s.set_force_variant(26)
        s.step()
        forced = s.get_state(want=("a",))["a"]
        assert np.array_equal(forced, a) or np.linalg.norm(forced - a) <= 2e-6 * np.linalg.norm(a)
    os.environ["NB_TEST_MAX_BYTES"] = str(32 << 20)
    try:
        with nb.NBody(m, x, v, **kw) as s, nb.NBody(m, x, v, eps=1e-3) as o:
            assert np.array_equal(s.get_state(want=("a",))["a"], o.get_state(want=("a",))["a"])
            s.step()
            o.symplectic(2, 2.0**-10, 1)
            assert np.isfinite(s.get_state(want=("x",))["x"]).all()
    finally:
        del os.environ["NB_TEST_MAX_BYTES"]


@pytest.mark.parametrize("n", [MIN_N + 1, 17 * 1024 + 300])
@pytest.mark.parametrize("order", [2, 6])
@pytest.mark.parametrize("prec", ["ds", "fp32"])
@pytest.mark.parametrize("field", [False, True])
def test_symplectic_steps_match_one_sided(nb, n, order, prec, field):
    """Records written by the kick-drift and field and closing kick in the
    fix-up: two steps against the one-sided path, which keeps them in
    launches of their own (no room for the pair-symmetric scratch).  The pair
    sums differ by at most 2 TOL of the largest pair acceleration, and a
    velocity by the sum of its kicks (|h| adds up to at most 6 dt per step)."""
    m, x, v = _system(nb, n, False)
    m, x = m * 0.00431, x * 0.01 + np.array([8.5, 0.0, 0.0])
    v = v * 0.65 + np.array([0.0, 22.0, 0.0])
    dt, res = 2.0**-12, {}
    for side in ("pairs", "one"):
        if side == "one":
            os.environ["NB_TEST_MAX_BYTES"] = str(32 << 20)
        try:
            with nb.NBody(m, x, v, eps=1e-4, precision=prec) as s:
                pair = np.abs(s.get_state(want=("a",))["a"]).max()
                if field:
                    s.set_external({})
                s.set_symplectic_layout("as_given")
                s.symplectic(order, dt, 2)
                res[side] = s.get_state(want=("x", "v", "a"))
        finally:
            os.environ.pop("NB_TEST_MAX_BYTES", None)
    da = 2 * TOL[prec][0] * pair
    dv = 2 * 6 * dt * da
    for k, bar in (("a", 2 * da), ("v", dv), ("x", 2 * 6 * dt * dv + 1e-15 * 9)):
        err = np.abs(res["pairs"][k] - res["one"][k]).max()
        assert err <= bar, (k, err, bar)
    assert not np.array_equal(res["pairs"]["a"], res["one"]["a"])  # two routes


@pytest.mark.parametrize("prec", ["ds", "fp32"])
@pytest.mark.parametrize("equal", [False, True])
@pytest.mark.parametrize("power", [-60, 30, 90])
def test_scaled_masses_scale_the_sums_exactly(nb, prec, equal, power):
    """Masses times a power of two take another internal scale of positions
    and masses; every operation scales exactly, so the sums do too."""
    m, x, v = _system(nb, MIN_N + 1, False, equal=equal)
    res = []
    for mm in (m, m * 2.0**power):
        with nb.NBody(mm, x, v, eps=1e-3, precision=prec, block_steps=False, lev_shared=10) as s:
            a = s.get_state(want=("a", "jerk"))
            s.set_symplectic_layout("as_given")
            s.symplectic(2, 0.0, 1)
            res.append((a["a"], a["jerk"], s.get_state(want=("a",))["a"]))
    for one, two in zip(*res):
        assert np.array_equal(one * 2.0**power, two)


# whole blocks of 2,048 (even ring), one particle more, a last block of two tiles
@pytest.mark.parametrize("n", [65536, 65537, 67 * 1024 + 300])
@pytest.mark.parametrize("equal", [False, True])
def test_wide_blocks_against_fp64_sums(nb, n, equal):
    """FP32 acceleration with eight i-particles per thread, sums of the same
    FP32 inputs: a term is off by at most ~15 u, a chain of 256 terms by
    256 u of their absolute sum (u = 2^-24)."""
    import torch

    m, x, v = (a.astype(np.float32).astype(np.float64) for a in _system(nb, n, False, equal=equal))
    eps = 1e-2
    with nb.NBody(m, x, v, eps=eps, precision="fp32") as s:
        s.set_symplectic_layout("as_given")
        s.symplectic(2, 0.0, 1)
        got = torch.from_numpy(s.get_state(want=("a",))["a"]).cuda()
    X, M = torch.from_numpy(x).cuda(), torch.from_numpy(m).cuda()
    idx = torch.cat([torch.arange(64), torch.arange(n - 64, n), torch.arange(100, n, 401)]).cuda()
    for part in idx.split(128):
        d = X[None] - X[part][:, None]
        t = (M * ((d * d).sum(-1) + eps * eps)**-1.5)[..., None] * d
        err, size = (got[part] - t.sum(1)).abs(), t.abs().sum(1)
        assert bool((err <= 271 * 2.0**-24 * size).all()), (err / size).max().item() * 2.0**24


# below MIN_N the pair-symmetric kernel runs where its units divide well:
# (7,168 and 8,192: one per CTA; 9,000: two for 180 units on 152 SMs, left to
# the one-sided kernel; 12,289: a last block of one particle)
@pytest.mark.parametrize("n,taken", [(6000, False), (7168, True), (8192, True), (9000, False),
                                     (12289, True), (MIN_N - 1, True)])
@pytest.mark.parametrize("prec", ["ds", "fp32"])
def test_middle_sizes(nb, oracle_mod, n, taken, prec):
    m, x, v = _system(nb, n, False)
    with nb.NBody(m, x, v, eps=1e-3, precision=prec, block_steps=False, lev_shared=10) as s:
        got = s.get_state(want=("a", "jerk"))
    with nb.NBody(m, x, v, eps=1e-3, precision=prec) as s:
        one = s.get_state(want=("a", "jerk"))
    import torch

    if torch.cuda.get_device_properties(0).multi_processor_count == 152:
        assert np.array_equal(got["a"], one["a"]) != taken
    idx = np.arange(0, n, 7, dtype=np.int32)
    ra, rj = oracle_mod.force_jerk(m, x, v, 1e-3, idx=idx)
    ta, tj = TOL[prec]
    assert np.linalg.norm(got["a"][idx] - ra) <= ta * np.linalg.norm(ra)
    assert np.linalg.norm(got["jerk"][idx] - rj) <= tj * np.linalg.norm(rj)


@pytest.mark.parametrize("prec", ["ds", "fp32"])
def test_one_mass_far_above_the_others(nb, prec):
    """A black hole among stars in units of a solar mass and a kilometre: its
    pull at some parsecs is a normal float, the mean mass over the cube of that
    distance is not."""
    n = MIN_N
    m, x, v = ics.plummer(n, 31)
    m, x, v = np.ones(n), x * 3e13, np.zeros((n, 3))
    m[0], x[0] = 4e6, 0.0
    r = np.linalg.norm(x, axis=1)
    x[r > 2e14] *= 0.05
    kw = dict(eps=1e9, precision=prec)
    with nb.NBody(m, x, v, block_steps=False, lev_shared=10, **kw) as s:
        got = s.get_state(want=("a",))["a"]
    with nb.NBody(m, x, v, **kw) as s:
        one = s.get_state(want=("a",))["a"]  # block steps: one-sided
        s.set_symplectic_layout("as_given")
        s.symplectic(2, 0.0, 1)
        acc = s.get_state(want=("a",))["a"]
    assert (np.linalg.norm(one, axis=1)[1:] > 0).all()
    for a in (got, acc):
        d = np.linalg.norm(a - one, axis=1) / np.linalg.norm(one, axis=1)
        assert d[1:].max() <= 2 * TOL[prec][0]  # the hole's pull is nearly all of it


def test_path_does_not_follow_free_memory(nb):
    """A context made while most of the device is in use takes the same kernel,
    and so gives the same bits, as one made on an empty device."""
    import torch

    n = 262144
    m, x, v = ics.plummer(n, 31)
    p = nb.spatial_order(x, 256)
    m, x, v = m[p], x[p], v[p]
    kw = dict(eps=1e-3, block_steps=False, lev_shared=10)
    with nb.NBody(m, x, v, **kw) as s:
        want = s.get_state(want=("a",))["a"]
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    # the partial sums take 1 GB at this n, the context 0.2 GB
    hold = torch.empty(max(0, free - (7 << 28)), dtype=torch.uint8, device="cuda")
    try:
        with nb.NBody(m, x, v, **kw) as s:
            got = s.get_state(want=("a",))["a"]
    finally:
        del hold
        torch.cuda.empty_cache()
    assert np.array_equal(got, want)


# a shape, a cap of the grid (below the built-in grid of either size), both, a table
@pytest.mark.parametrize("force", [lambda s: s.set_force_variant(26),
                                   lambda s: s.set_force_variant(-1, 7),
                                   lambda s: s.set_force_variant(1, 7),
                                   lambda s: s.set_force_table([(4096, 0), (0, 3)])])
@pytest.mark.parametrize("n", [1000, MIN_N])
def test_a_forced_shape_is_the_shape_that_steps(nb, n, force):
    """nb_step under a forced shape, grid or table takes the rows that the same
    setting hands out, bit for bit, and not the pair-symmetric sums (the one launch
    of a small step has the separate kernels' bits)."""
    m, x, v = _system(nb, n, False)
    kw = dict(eps=1e-3, block_steps=False, lev_shared=10)
    with nb.NBody(m, x, v, **kw) as s, nb.NBody(m, x, v, **kw) as o, nb.NBody(m, x, v, **kw) as d:
        force(s)
        force(o)
        s.step()
        d.step()
        t, na = o.next_block()
        o.predict(t)
        a, j = o.force_jerk()
        got, built_in = s.get_state(want=("a", "jerk")), d.get_state(want=("a", "jerk"))
    assert np.array_equal(got["a"], a) and np.array_equal(got["jerk"], j)
    assert n < MIN_N or not np.array_equal(built_in["a"], a)
