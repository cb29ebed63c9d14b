"""Mixed force on spatially sorted bodies (large calls and large systems):
single-subtraction coordinates about a group's centre for far pairs, and
subtiles whose criterion cannot exceed what the bodies have left out.

Against the oracle on sampled bodies, with the tolerances of
test_gpu_force.py (a 1e-6 of the pair magnitudes, phi 1e-6, q 2e-6: the
roundings of a far pair are 3/2 units against one, both far below). Systems
off the origin, of two distant clumps, with unequal masses, repeated active
bodies and a ragged last subtile. The integrator's sorted path against its
FP64 path: the same block schedule, positions to 1e-9 (forces agree to 1e-6,
and the span is 2^-11 time units)."""
import numpy as np
import pytest

from paper_1205_2288_gb300 import inputs, tsbts
from test_gpu_force import (gpu_force, pair_magnitude_sum,  # noqa: F401
                            torch_cuda)

pytestmark = pytest.mark.gpu


def _system(kind, n):
    m, r, v = inputs.plummer(n, 5)
    if kind == "salpeter":
        m = inputs.salpeter_masses(n, 6)
    elif kind == "off_origin":
        r = r * 1e-2 + np.array([30.0, -20.0, 10.0])
    elif kind == "two_clumps":
        r = r * 0.05
        r[::2] += 40.0
    return m, r, v


@pytest.mark.parametrize("kind,n,n_act,eps", [
    ("plummer", 65537, 65537, 1 / 512), ("salpeter", 70001, 40000, 1e-4),
    ("off_origin", 65600, 65600, 1e-3), ("two_clumps", 65555, 50001, 1e-3),
    ("plummer", 131072, 20000, 1 / 512)])
def test_sorted_calls(torch_cuda, orc, kind, n, n_act, eps):  # noqa: F811
    m, r, v = _system(kind, n)
    idx = inputs.active_subset(n, n_act, 7)
    g = np.random.default_rng(8)
    g.shuffle(idx)
    idx[10] = idx[n_act - 1]
    a, phi, q = gpu_force(torch_cuda, tsbts.TSBTS_MIXED, m, r, v, eps, idx)
    pick = np.unique(np.linspace(0, n_act - 1, 700).astype(int))
    orc.set_threads(8)
    ao, phio, qo = orc.forces(m, r, v, eps, idx[pick])
    scale = pair_magnitude_sum(m, r, eps, idx[pick])
    assert (np.abs(a[pick] - ao).max(1) / scale).max() < 1e-6
    np.testing.assert_allclose(phi[pick], phio, rtol=1e-6)
    np.testing.assert_allclose(q[pick], qo, rtol=2e-6)
    np.testing.assert_array_equal(a[10], a[n_act - 1])
    assert np.isfinite(a).all() and (q > 0).all()


def test_sorted_integration_matches_fp64(torch_cuda):  # noqa: F811
    n, t = 33000, 2.0 ** -11
    m, r, v = inputs.plummer(n, 9)
    kw = dict(eps=1 / 256, eta=0.01, dt_max=1 / 8, era_log2=3)
    out = []
    for prec in (tsbts.TSBTS_FP64, tsbts.TSBTS_MIXED):
        with tsbts.Simulation(m, r, v, precision=prec, **kw) as sim:
            sim.schedule_log(2_000_000)
            sim.step_era(t)
            out.append((sim.state(), sim.schedule()))
    (s0, l0), (s1, l1) = out
    np.testing.assert_array_equal(l0["tau"], l1["tau"])
    np.testing.assert_array_equal(l0["n_act"], l1["n_act"])
    off = np.concatenate([[0], np.cumsum(l0["n_act"])])
    for k in range(0, len(l0["tau"]), 7):
        np.testing.assert_array_equal(np.sort(l0["idx"][off[k]:off[k + 1]]),
                                      np.sort(l1["idx"][off[k]:off[k + 1]]))
    np.testing.assert_array_equal(s0["dt"], s1["dt"])
    assert np.abs(s0["r"] - s1["r"]).max() < 1e-9
    assert np.abs(s0["v"] - s1["v"]).max() < 1e-6
