"""Mixed force over the widths and tiles of its tiled work items: active
counts around the group widths (8 .. 256 bodies, two per thread), j ranges
that end inside a quad, a lane round or a 512-body tile, eps = 0 (every
iteration in the masked form) and repeated bodies. The tolerances of
test_gpu_force.py: they bound FP32 pair terms and compensated sums of any
order, which every width shares."""
import numpy as np
import pytest

from paper_1205_2288_gb300 import inputs, tsbts
from test_gpu_force import (gpu_force, pair_magnitude_sum,  # noqa: F401
                            torch_cuda)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,n_act,eps", [
    (511, 511, 0.01), (513, 257, 0.01), (1025, 1000, 0.0), (2047, 129, 0.01),
    (4097, 513, 0.01), (8191, 2049, 0.01), (8193, 8193, 1 / 256)])
def test_widths_and_tile_edges(torch_cuda, orc, n, n_act, eps):  # noqa: F811
    m, r, v = inputs.plummer(n, n)
    idx = inputs.active_subset(n, n_act, n_act)
    idx[-1] = idx[0]
    a, phi, q = gpu_force(torch_cuda, tsbts.TSBTS_MIXED, m, r, v, eps, idx)
    ao, phio, qo = orc.forces(m, r, v, eps, idx)
    with np.errstate(divide="ignore"):
        scale = pair_magnitude_sum(m, r, eps, idx)
    assert (np.abs(a - ao).max(1) / scale).max() < 1e-6
    np.testing.assert_allclose(phi, phio, rtol=1e-6)
    np.testing.assert_allclose(q, qo, rtol=2e-6)
    np.testing.assert_allclose(a[-1], a[0], rtol=1e-6)
