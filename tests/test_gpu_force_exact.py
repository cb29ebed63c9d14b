"""FP64 force with ascending-j sums at the edges of its work split: bodies
per block (one block per SM holds up to 7 with overlapped sums, 152 SMs;
beyond 1064 active bodies up to 32 in two blocks per SM, beyond 9728 a block
takes several groups) and tiles of j (96 or 32). Bit-identical to the
oracle, as every sequential evaluation is."""
import numpy as np
import pytest

from paper_1205_2288_gb300 import inputs, tsbts
from test_gpu_force import gpu_force, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,n_act", [(2, 2), (31, 31), (96, 5), (97, 97),
                                     (193, 153), (1064, 1064), (1065, 1065),
                                     (4100, 2433), (10000, 10000)])
def test_work_split_edges_are_bit_identical(torch_cuda, orc, n,  # noqa: F811
                                            n_act):
    m, r, v = inputs.plummer(n, n)
    idx = inputs.active_subset(n, n_act, n_act)
    orc.set_threads(8)
    ref = orc.forces(m, r, v, 0.01, idx)
    got = gpu_force(torch_cuda, tsbts.TSBTS_FP64, m, r, v, 0.01, idx,
                    exact_order=1)
    for g, o in zip(got, ref):
        np.testing.assert_array_equal(g, o)
