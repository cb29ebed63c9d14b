"""Spatial order in integrations beyond a fixed era of equal masses (dynamic
eras, unequal masses, a system away from the origin, a resumed run) and with
bodies whose speed or mass is no number in a force call.

Integrations against their FP64 run over at most 2^-10 time units: forces that
agree to 1e-6 of the pair magnitudes (a below 1e3 at the softening used) move
v by at most 1e-6 and r by 1e-9; a step estimate within 1e-6 of a power of two
may fall on its other side for a body or two of 40000. A resumed run repeats
the bits of the one that was not interrupted: the order comes from the state
at the era's start. A speed that is no number touches no other body's results;
an infinite one gives every other body an infinite criterion."""
import numpy as np
import pytest

from paper_1205_2288_gb300 import inputs, tsbts
from test_gpu_force import (gpu_force, pair_magnitude_sum,  # noqa: F401
                            torch_cuda)

pytestmark = pytest.mark.gpu


def _system(kind, n):
    if kind == "salpeter":
        m = inputs.salpeter_masses(n, 6)
        return inputs.plummer(n, 5, masses=m)
    m, r, v = inputs.plummer(n, 5)
    if kind == "shifted":
        r = r + np.array([100.0, -60.0, 30.0])
    return m, r, v


@pytest.mark.parametrize("kind,n,era_mode,span", [
    ("salpeter", 40001, 1, 11), ("shifted", 40000, 0, 11),
    ("plummer", 36864, 1, 10)])
def test_eras_match_fp64(torch_cuda, kind, n, era_mode, span):  # noqa: F811
    m, r, v = _system(kind, n)
    out = []
    for prec in (tsbts.TSBTS_FP64, tsbts.TSBTS_MIXED):
        with tsbts.Simulation(m, r, v, eps=1 / 256, eta=0.01,
                              dt_max=2.0 ** -(span + 2), era_mode=era_mode,
                              era_log2=span + 2, precision=prec) as sim:
            sim.step_era(2.0 ** -span)
            out.append((sim.state(), sim.stats()))
    (s0, t0), (s1, t1) = out
    assert t1["eras"] >= 2
    assert np.abs(s0["r"] - s1["r"]).max() < 1e-9
    assert np.abs(s0["v"] - s1["v"]).max() < 1e-6
    assert (s0["dt"] != s1["dt"]).sum() <= 2


def test_resume_repeats_the_bits(torch_cuda):  # noqa: F811
    m, r, v = _system("salpeter", 40001)
    kw = dict(eps=1 / 256, eta=0.01, dt_max=2.0 ** -12, era_mode=0,
              era_log2=12, precision=tsbts.TSBTS_MIXED)
    with tsbts.Simulation(m, r, v, **kw) as sim:
        sim.step_era(2.0 ** -12)
        mid = sim.checkpoint()
        sim.step_era(2.0 ** -11)
        want = sim.state()
    with tsbts.Simulation(m, r, v, **kw) as sim:
        sim.set_state(mid)
        sim.step_era(2.0 ** -11)
        got = sim.state()
    for k in ("r", "v", "a", "tau", "dt"):
        np.testing.assert_array_equal(got[k], want[k])


@pytest.mark.parametrize("what,value", [
    ("speed", np.nan), ("speed", np.inf), ("speed", 1e30), ("mass", 0.0)])
def test_odd_bodies_in_a_sorted_call(torch_cuda, what, value):  # noqa: F811
    n, eps, odd = 66000, 1 / 512, 12345
    m, r, v = inputs.plummer(n, 11)
    if what == "speed":
        v[odd] = [value, 0.1, -0.2]
    else:
        m[odd] = value
    a, phi, q = gpu_force(torch_cuda, tsbts.TSBTS_MIXED, m, r, v, eps,
                          np.arange(n, dtype=np.int32))
    near = np.argsort(((r - r[odd]) ** 2).sum(1))[1:40]  # its subtile and on
    pick = np.unique(np.concatenate([near, np.linspace(0, n - 1, 60,
                                                       dtype=int)]))
    pick = pick[pick != odd]
    scale = pair_magnitude_sum(m, r, eps, pick)
    for k, i in enumerate(pick):
        d = r - r[i]
        s2 = (d * d).sum(1) + eps * eps
        f = m / (s2 * np.sqrt(s2))
        f[i] = 0.0
        assert np.abs(a[i] - (f[:, None] * d).sum(0)).max() < 1e-6 * scale[k]
        p = m / np.sqrt(s2)
        p[i] = 0.0
        np.testing.assert_allclose(phi[i], -p.sum(), rtol=1e-6)
        with np.errstate(invalid="ignore", over="ignore"):
            c = ((v - v[i]) ** 2).sum(1) / s2
        c[i] = 0.0
        want = max(np.nanmax(c), f.max())
        if want > 3.4e38 * (1 - 2e-6):  # beyond FP32: the mixed path's inf
            assert np.isinf(q[i])
        else:
            np.testing.assert_allclose(q[i], want, rtol=2e-6)
    assert np.isfinite(a).all() and np.isfinite(phi).all()
