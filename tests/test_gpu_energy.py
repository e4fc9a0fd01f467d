"""The energy of a state against a sum in extended precision, around the size
where the split-precision pair sum takes over from the FP64 one (n = 1,024)
and at ragged sizes.  Bar: 2e-15 of the pair energy; a term carries 2^-46 =
1.4e-14 at most, independent from pair to pair, so that n >= 1,024 particles
(5e5 pairs) leave less than an ulp, and the FP64 sums a few."""
import math
import os

import numpy as np
import pytest

from paper_0909_0879_gb300 import ics

pytestmark = pytest.mark.gpu

BAR = 2e-15


@pytest.fixture(scope="module")
def nb():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0909_0879_gb300 import _lib

    _lib.load()
    return _lib


def _reference(m, x, v, eps):
    """Kinetic and pair energy: FP64 terms, exact sums (each term's own
    rounding is 1e-16 and averages over the pairs)."""
    w = []
    for i in range(len(m) - 1):
        d = x[i + 1:] - x[i]
        r2 = d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1] + d[:, 2] * d[:, 2] + eps * eps
        w.append(m[i] * math.fsum(m[i + 1:] / np.sqrt(r2)))
    return math.fsum((0.5 * m[:, None] * v * v).ravel()), -math.fsum(w)


def _system(n, kind):
    m, x, v = ics.plummer(n, 71, masses=ics.salpeter_masses(n, 72))
    if kind == "offset":  # a small cluster far from the origin
        x = 0.01 * x + np.array([8.5, -3.0, 0.25])
    if kind == "binaries":  # hard binaries that hold most of the energy
        for k in range(0, 12, 2):
            x[k + 1] = x[k] + 1e-6 * (1 + k) * np.array([0.3, 0.5, -0.7])
    if kind == "massless":
        m[1::3] = 0.0
        x[4] = x[3] + 1e-17
    return m, x, v


@pytest.mark.parametrize("n", [1023, 1024, 1025, 1279, 3000])
@pytest.mark.parametrize("eps", [0.0, 1e-4])
@pytest.mark.parametrize("kind", ["plain", "offset", "binaries", "massless"])
def test_energy_against_exact_sum(nb, n, eps, kind):
    m, x, v = _system(n, kind)
    if eps == 0.0 and kind == "massless":
        pytest.skip("a coincident pair")
    k_ref, w_ref = _reference(m, x, v, eps)
    with nb.NBody(m, x, v, eps=eps) as s:
        k, w, e = s.energy()
    assert abs(k / k_ref - 1.0) <= BAR
    assert abs(w / w_ref - 1.0) <= BAR
    assert e == k + w


@pytest.mark.parametrize("scale", [1e-30, 1e30])
def test_energy_in_other_units(nb, scale):
    """Lengths and masses far from 1: the sum is scaled by powers of two."""
    n = 1100
    m, x, v = _system(n, "plain")
    k0, w0 = _reference(m, x, v, 1e-3)
    with nb.NBody(m, x, v, eps=1e-3) as s:
        st = s.get_state()
        st["x"] = x * 2.0**60 if scale > 1 else x * 2.0**-60
        # the context keeps its own softening, so the reference does too
        s.set_state(st)
        k, w, _ = s.energy()
    k_ref, w_ref = _reference(m, st["x"], v, 1e-3)
    assert abs(k / k0 - 1.0) <= BAR
    # (2^-60: every distance far below the softening, hardly any of the
    # roundings are independent)
    assert abs(w / w_ref - 1.0) <= (BAR if scale > 1 else 1e-14)


def test_energy_of_coincident_particles_and_without_scratch(nb):
    n = 1200
    m, x, v = _system(n, "plain")
    with nb.NBody(m, x, v, eps=0.0) as s:
        st = s.get_state()
        w0 = s.energy()[1]
        st["x"][700] = st["x"][20]
        s.set_state(st)
        with pytest.raises(nb.NBodyError) as e:
            s.energy()
        assert e.value.status == nb.NB_ERR_NUMERIC
    with nb.NBody(m, x, v, eps=0.0) as s:
        os.environ["NB_TEST_MAX_BYTES"] = "1000"
        try:
            w1 = s.energy()[1]  # the FP64 sum
        finally:
            del os.environ["NB_TEST_MAX_BYTES"]
        w2 = s.energy()[1]
    assert abs(w1 / w0 - 1.0) <= BAR and w2 == w0


@pytest.mark.parametrize("n", [1024, 1500, 5000])
@pytest.mark.parametrize("mass", [0.5000000149518913, 0.1])
def test_energy_of_equal_masses(nb, n, mass):
    """One mass for all, of which two FP32 words leave out 1.8e-15 and 2.8e-16:
    the terms' errors average out, this one would not.  Bar: a few FP64 roundings
    of the result."""
    m, x, v = ics.plummer(n, 70)
    m[:] = mass
    _, w_ref = _reference(m, x, v, 1e-3)
    with nb.NBody(m, x, v, eps=1e-3) as s:
        assert abs(s.energy()[1] / w_ref - 1.0) <= 8e-16


@pytest.mark.parametrize("sep", [1e-13, 1e-12, 1e-10, 1e-8])
def test_energy_of_close_light_pairs(nb, sep):
    """Close pairs of light particles, each 1e-5 of the pair energy, at
    separations near the last bits of the coordinates."""
    n = 1100
    for seed in range(4):
        m, x, v = ics.plummer(n, 71 + seed)
        r = np.random.default_rng(seed)
        for k in range(10, 20, 2):
            m[k] = m[k + 1] = np.sqrt(1e-5 * sep)
            d = r.normal(size=3)
            x[k + 1] = x[k] + sep / np.linalg.norm(d) * d
        _, w_ref = _reference(m, x, v, 0.0)
        with nb.NBody(m, x, v, eps=0.0) as s:
            assert abs(s.energy()[1] / w_ref - 1.0) <= BAR


def _without_scratch(s):
    os.environ["NB_TEST_MAX_BYTES"] = "1000"
    try:
        return s.energy()  # the FP64 sum
    finally:
        del os.environ["NB_TEST_MAX_BYTES"]


@pytest.mark.parametrize("ratio", [1e-6, 1e-18, 5e-31, 1e-37, 1e-45, 0.0])
@pytest.mark.parametrize("first", [True, False])
def test_energy_around_a_dominant_particle(nb, ratio, first):
    """Far lighter particles before or after a heavy one: the FP64 sum, whose
    chain of n additions is good to n / 2 ulps."""
    n = 1100
    m, x, v = ics.plummer(n, 71, masses=ics.salpeter_masses(n, 72))
    m *= ratio * n
    m[0 if first else n - 1] = 1.0
    m[1 if first else 0] = 0.0
    _, w_ref = _reference(m, x, v, 1e-4)
    with nb.NBody(m, x, v, eps=1e-4) as s, nb.NBody(m, x, v, eps=1e-4) as o:
        w, w64 = s.energy()[1], _without_scratch(o)[1]
    assert w == w64
    assert abs(w - w_ref) <= n * 2.0**-53 * abs(w_ref)


def test_energy_of_two_light_particles_around_a_heavy_one(nb):
    """Their own term is most of the pair energy, and small beside the square of
    the total mass."""
    n = 1024
    for seed in range(16):
        r = np.random.default_rng(seed)
        m, x, v = np.full(n, 1e-13), r.uniform(-1, 1, (n, 3)), np.zeros((n, 3))
        m[0] = 1.0
        m[5], m[700] = 2.9e-6, 2.9e-6
        d = r.normal(size=3)
        x[700] = x[5] + 6.3e-8 * d / np.linalg.norm(d)
        _, w_ref = _reference(m, x, v, 0.0)
        with nb.NBody(m, x, v, eps=0.0) as s, nb.NBody(m, x, v, eps=0.0) as o:
            w, w64 = s.energy()[1], _without_scratch(o)[1]
        assert w == w64
        assert abs(w - w_ref) <= n * 2.0**-53 * abs(w_ref)


# a twentieth of the harmonic mean distance, more than half of it, and far more
@pytest.mark.parametrize("eps,fp64", [(0.05, False), (1.0, True), (4.0, True), (1e4, True)])
@pytest.mark.parametrize("n", [1024, 1300])
def test_energy_where_softening_dominates(nb, eps, fp64, n):
    """Softening as long as the separations and longer: hardly any of the
    roundings are independent, and the FP64 sum is taken."""
    same = []
    for seed in range(3):
        m, x, v = ics.plummer(n, 71 + seed, masses=ics.salpeter_masses(n, 72))
        x = x + np.array([30.0, 0.0, 0.0])
        _, w_ref = _reference(m, x, v, eps)
        with nb.NBody(m, x, v, eps=eps) as s, nb.NBody(m, x, v, eps=eps) as o:
            w, w64 = s.energy()[1], _without_scratch(o)[1]
        assert abs(w / w_ref - 1.0) <= BAR
        same.append(w == w64)
    assert all(same) or not fp64
