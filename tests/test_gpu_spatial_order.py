"""Force calls at and beyond the line from which a mixed call puts its bodies
in spatial order (2^32 interactions, a quarter of the bodies active): systems
away from the origin, of clumps, with unequal masses and with a body far
outside, partial and shuffled active lists with repeats, longer than the body
count, ragged last subtiles, and the calls just below the line.

Against the oracle on sampled bodies, with the tolerances of
test_gpu_force.py (a 1e-6 of the pair magnitudes, phi 1e-6, q 2e-6)."""
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
    elif kind == "shifted":
        r = r + np.array([10.0, 0.0, 0.0])
    elif kind == "far_away":
        r = r + np.array([3000.0, -1800.0, 900.0])
    elif kind == "clumps":
        r = r * 0.05
        r[::3] += 40.0
    elif kind == "escaper":
        r[7] = [1e5, -3e4, 2e4]
    return m, r, v


@pytest.mark.parametrize("kind,n,n_act,eps", [
    ("plummer", 65536, 65536, 1 / 512), ("plummer", 65536, 65535, 1 / 512),
    ("shifted", 65601, 65601, 1e-3), ("far_away", 65539, 65539, 1 / 512),
    ("salpeter", 90001, 60000, 1e-4), ("clumps", 90017, 50001, 1e-3),
    ("escaper", 66000, 66000, 1 / 512), ("plummer", 131072, 32768, 1 / 512),
    ("plummer", 131073, 32767, 1 / 512), ("salpeter", 70001, 90000, 1e-3)])
def test_calls(torch_cuda, orc, kind, n, n_act, eps):  # noqa: F811
    m, r, v = _system(kind, n)
    g = np.random.default_rng(8)
    idx = inputs.active_subset(n, min(n, n_act), 7)
    idx = np.concatenate([idx, g.choice(idx, n_act - len(idx))])
    idx = idx.astype(np.int32)
    g.shuffle(idx)
    idx[10] = idx[n_act - 1]
    a, phi, q = gpu_force(torch_cuda, tsbts.TSBTS_MIXED, m, r, v, eps, idx)
    pick = np.unique(np.linspace(0, n_act - 1, 500).astype(int))
    orc.set_threads(8)
    ao, phio, qo = orc.forces(m, r, v, eps, idx[pick])
    scale = pair_magnitude_sum(m, r, eps, idx[pick])
    assert (np.abs(a[pick] - ao).max(1) / scale).max() < 1e-6
    np.testing.assert_allclose(phi[pick], phio, rtol=1e-6)
    np.testing.assert_allclose(q[pick], qo, rtol=2e-6)
    np.testing.assert_array_equal(a[10], a[n_act - 1])
    assert np.isfinite(a).all() and (q > 0).all()
