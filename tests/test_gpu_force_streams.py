"""tsbts_force from several streams: calls share the scratch memory of their
device (j records, spatial order, partial sums), so each has to wait for the
one before it whatever stream that was on. Interleaved calls on two streams,
and two branches of one captured graph, give the bits of the same calls made
one after the other (every plan is fixed once its body count was tuned, and
results are deterministic)."""
import numpy as np
import pytest

from paper_1205_2288_gb300 import inputs, tsbts
from test_gpu_force import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu

# in spatial order, not, few active, FP64 in any order and in ascending j
CALLS = [(tsbts.TSBTS_MIXED, 70001, 70001), (tsbts.TSBTS_MIXED, 40000, 33),
         (tsbts.TSBTS_MIXED, 20000, 20000), (tsbts.TSBTS_FP64, 20000, 500),
         (tsbts.TSBTS_FP64, 4099, 129), (tsbts.TSBTS_MIXED, 66000, 66000)]


class Call:
    def __init__(self, torch, precision, n, n_act):
        m, r, v = inputs.plummer(n, n)
        idx = inputs.active_subset(n, n_act, 1)
        self.precision = precision
        self.args = [torch.from_numpy(np.ascontiguousarray(x)).to("cuda:0")
                     for x in (m, r, v, idx)]
        self.out = [torch.empty(n_act * k, dtype=torch.float64,
                                device="cuda:0") for k in (3, 1, 1)]

    def run(self):
        m, r, v, idx = self.args
        a, phi, q = self.out
        tsbts.tsbts_force(self.precision, m, r, v, 1 / 512, idx,
                          a.view(-1, 3), phi, q)

    def take(self, torch):
        torch.cuda.synchronize()
        got = [x.cpu().numpy().copy() for x in self.out]
        for x in self.out:
            x.fill_(float("nan"))
        torch.cuda.synchronize()
        return got


@pytest.fixture(scope="module")
def serial(torch_cuda):  # noqa: F811
    calls = [Call(torch_cuda, *c) for c in CALLS]
    for c in calls:  # buffers and plans
        c.run()
        c.take(torch_cuda)
    want = []
    for c in calls:
        c.run()
        want.append(c.take(torch_cuda))
    return calls, want


def _check(torch, calls, want):
    for c, w in zip(calls, want):
        for g, x in zip(c.take(torch), w):
            np.testing.assert_array_equal(g, x)


def test_two_streams(torch_cuda, serial):  # noqa: F811
    torch = torch_cuda
    calls, want = serial
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for k in range(4):
        for i, c in enumerate(calls):
            with torch.cuda.stream(streams[(i + k) % 2]):
                c.run()
        _check(torch, calls, want)


def test_branches_of_a_captured_graph(torch_cuda, serial):  # noqa: F811
    torch = torch_cuda
    calls, want = serial
    side = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        main = torch.cuda.current_stream()
        side.wait_stream(main)
        for i, c in enumerate(calls):
            with torch.cuda.stream(side if i % 2 else main):
                c.run()
        main.wait_stream(side)
    for _ in range(2):
        graph.replay()
        _check(torch, calls, want)
    # calls outside a capture still run, and a second capture starts afresh
    calls[0].run()
    _check(torch, calls[:1], want[:1])
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        calls[2].run()
        calls[3].run()
    graph.replay()
    _check(torch, calls[2:4], want[2:4])
