"""FP64 force with ascending-j sums where one block per SM (152) is full with
32 bodies (4864 active ones) and takes a second group beyond. Bit-identical to
the oracle."""
import numpy as np
import pytest

from paper_1205_2288_gb300 import inputs, tsbts
from test_gpu_force import gpu_force, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_act", [4864, 4865])
def test_one_and_two_groups_per_block(torch_cuda, orc, n_act):  # noqa: F811
    n = 5003
    m, r, v = inputs.plummer(n, n)
    idx = inputs.active_subset(n, n_act, n_act)
    orc.set_threads(8)
    ref = orc.forces(m, r, v, 0.01, idx)
    got = gpu_force(torch_cuda, tsbts.TSBTS_FP64, m, r, v, 0.01, idx,
                    exact_order=1)
    for g, o in zip(got, ref):
        np.testing.assert_array_equal(g, o)
