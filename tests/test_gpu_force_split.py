"""FP64 j-split force over the ranges of its reciprocal square root: squared
distances inside 2^-119 .. 2^119 take the refined FP32 estimate, others the
correctly rounded form. Same tolerances as the j-split test of
test_gpu_force.py (a 1e-13 of the pair magnitudes, phi 1e-13, q 1e-14): the
terms are the same to a few ulps at every scale."""
import numpy as np
import pytest

from paper_1205_2288_gb300 import inputs, tsbts
from test_gpu_force import (gpu_force, pair_magnitude_sum,  # noqa: F401
                            torch_cuda)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1e-30, 2.0 ** -60, 2.0 ** -58, 1.0,
                                   2.0 ** 58, 2.0 ** 60, 1e30])
@pytest.mark.parametrize("eps", [0.0, 0.01])
def test_scales(torch_cuda, orc, scale, eps):  # noqa: F811
    n = 257
    m, r, v = inputs.plummer(n, 3)
    r = r * scale
    idx = inputs.active_subset(n, 200, 4)
    a, phi, q = gpu_force(torch_cuda, tsbts.TSBTS_FP64, m, r, v, eps * scale,
                          idx, exact_order=0)
    ao, phio, qo = orc.forces(m, r, v, eps * scale, idx)
    with np.errstate(divide="ignore"):
        w = pair_magnitude_sum(m, r, max(eps * scale, 1e-3 * scale), idx)
    assert (np.abs(a - ao).max(1) / np.maximum(
        w, np.abs(ao).max(1))).max() < 1e-13
    np.testing.assert_allclose(phi, phio, rtol=1e-13)
    np.testing.assert_allclose(q, qo, rtol=1e-14)
