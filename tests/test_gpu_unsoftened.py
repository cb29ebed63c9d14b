"""Mixed path with eps^2 that is no normal float (eps = 0, or below 1e-19),
where the reciprocal square root must take any s^2 >= 0: force calls of every
tiled width, with whole and ragged tiles and at a size that would be put in
spatial order with softening; a large system, an ensemble whose clusters
differ in eps, and the adjoint.

Force tolerances as in test_gpu_force.py (a 1e-6 of the pair magnitudes,
phi 1e-6, q 2e-6). Integrations against their FP64 run over spans of at most
2^-9 time units: forces that agree to 1e-6 move v by at most 1e-6 of the
closest pair's a t (a < 1e3: 2e-6 t ... 1e-6) and r by t times that (1e-8);
a step estimate this close to a power of two may fall on the other side of
it for a body or two. Gradients as in the other mixed adjoint tests: 1e-4 of
the largest."""
import numpy as np
import pytest

from paper_1205_2288_gb300 import inputs, tsbts
from test_gpu_adjoint import oracle_schedule, rel
from test_gpu_force import (gpu_force, pair_magnitude_sum,  # noqa: F401
                            torch_cuda)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,n_act,eps", [
    (511, 511, 0.0), (513, 300, 1e-20), (1025, 1025, 0.0), (5000, 4097, 0.0),
    (20000, 9, 0.0), (20000, 700, 1e-20), (47000, 47000, 0.0),
    (33000, 33000, 1e-20)])
def test_forces(torch_cuda, orc, n, n_act, eps):  # noqa: F811
    m, r, v = inputs.plummer(n, n)
    idx = inputs.active_subset(n, n_act, 3)
    a, phi, q = gpu_force(torch_cuda, tsbts.TSBTS_MIXED, m, r, v, eps, idx)
    pick = np.unique(np.linspace(0, n_act - 1, 500).astype(int))
    orc.set_threads(8)
    ao, phio, qo = orc.forces(m, r, v, eps, idx[pick])
    with np.errstate(divide="ignore"):
        scale = pair_magnitude_sum(m, r, eps, idx[pick])
    assert (np.abs(a[pick] - ao).max(1) / scale).max() < 1e-6
    np.testing.assert_allclose(phi[pick], phio, rtol=1e-6)
    np.testing.assert_allclose(q[pick], qo, rtol=2e-6)
    assert np.isfinite(a).all() and (q > 0).all()


def _near(s0, s1):
    assert np.abs(s0["r"] - s1["r"]).max() < 1e-8
    assert np.abs(s0["v"] - s1["v"]).max() < 1e-6
    assert (s0["dt"] != s1["dt"]).sum() <= 2


def test_large_system(torch_cuda):  # noqa: F811
    m, r, v = inputs.plummer(33000, 9)
    out = []
    for prec in (tsbts.TSBTS_FP64, tsbts.TSBTS_MIXED):
        with tsbts.Simulation(m, r, v, eps=0.0, eta=0.01, dt_max=1 / 8,
                              era_log2=3, precision=prec) as sim:
            sim.step_era(2.0 ** -13)
            out.append(sim.state())
    _near(*out)


def test_ensemble(torch_cuda):  # noqa: F811
    sizes, eps = [700, 300, 1500, 513], [0.0, 0.01, 1e-20, 0.0]
    off = np.concatenate([[0], np.cumsum(sizes)])
    sys = [inputs.plummer(n, 20 + n) for n in sizes]
    kw = dict(eta=0.01, dt_max=1 / 8, era_log2=3)
    with tsbts.Ensemble(off, *(np.concatenate([x[k] for x in sys])
                               for k in range(3)),
                        eps=np.array(eps), precision=tsbts.TSBTS_MIXED,
                        **kw) as ens:
        ens.step_era(2.0 ** -9)
        got = ens.state()
    for c in range(len(sizes)):
        with tsbts.Simulation(*sys[c], eps=eps[c], **kw) as sim:
            sim.step_era(2.0 ** -9)
            _near(sim.state(), {k: got[k][off[c]:off[c + 1]]
                                for k in ("r", "v", "dt")})


@pytest.mark.parametrize("n", [300, 1100])
def test_adjoint(torch_cuda, n):  # noqa: F811
    m, r, v = inputs.plummer(n, 40)
    sched = oracle_schedule(m, r, v, eps=0.01, t_end=2.0 ** -6, era_log2=6)
    out = []
    for prec in (tsbts.TSBTS_FP64, tsbts.TSBTS_MIXED):
        with tsbts.Adjoint(n, 0.0, sched, precision=prec) as adj:
            out.append(adj.loss_grad(m, r, v))
    assert abs(out[1][0] / out[0][0] - 1) < 1e-6
    for a, b in zip(out[1][1:], out[0][1:]):
        assert rel(a, b) < 1e-4
