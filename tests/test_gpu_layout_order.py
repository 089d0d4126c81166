"""Copies at other strides, and other numbers of copies and of slices side by
side, between calls on a stream that is still busy: the tables of a call are
written after the calls before it have read theirs.  The stream is held up by
a bounded spin, so that all calls are made before the first one runs; every
table keeps every read inside the leaves."""
import numpy as np
import pytest

from paper_2002_01935_gb300 import inputs, planner

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    if not _t.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2002_01935_gb300 import build
    build.build()
    return _t


def setup(torch, q):
    edges = inputs.random_regular_graph(10, 3, 4)
    labels = [[int(u), int(v)] for u, v in edges]
    dims = {v: q for v in range(10)}
    g = torch.Generator(device="cuda").manual_seed(1)
    ts = [torch.rand(9, q, q, device="cuda", generator=g) + 0.1 for _ in edges]
    return labels, dims, planner.greedy_tree(labels, dims, []), ts


@pytest.mark.parametrize("q", [2, 3])
def test_copies(torch, q):
    from paper_2002_01935_gb300 import binding
    labels, dims, pairs, ts = setup(torch, q)
    calls = [(3, 1), (3, 4), (3, 2), (1, 1), (3, 0)]  # copies, leaves between them

    def run(h, c, step):
        return h.contract_instances(pairs, "fp32", c, [step * q * q] * len(ts))

    h = binding.TensorNetwork(labels, dims, [], ts, complex_=False)
    stream = torch.cuda.Stream()
    try:
        want = []
        for c in calls:
            m, e = run(h, *c)
            torch.cuda.synchronize()
            want.append((m.cpu().numpy().tobytes(), e.cpu().tolist()))
        with torch.cuda.stream(stream):
            torch.cuda._sleep(100_000_000)
            got = [run(h, *c) for c in calls]
        torch.cuda.synchronize()
        got = [(m.cpu().numpy().tobytes(), e.cpu().tolist()) for m, e in got]
    finally:
        h.close()
    assert got == want


@pytest.mark.parametrize("q", [2, 3])
def test_slices_side_by_side(torch, q):
    from paper_2002_01935_gb300 import binding
    labels, dims, pairs, ts = setup(torch, q)
    h = binding.TensorNetwork(labels, dims, [], [t[0].contiguous() for t in ts], complex_=False)
    stream = torch.cuda.Stream()
    try:
        first = h.contract(pairs, [0, 5], "fp32", slice_batch=4)
        torch.cuda.synchronize()
        want = (float(first[0].cpu()), int(first[1].cpu()))
        with torch.cuda.stream(stream):
            torch.cuda._sleep(100_000_000)
            got = [h.contract(pairs, [0, 5], "fp32", slice_batch=b) for b in (4, 1, 3, 2)]
        torch.cuda.synchronize()
        got = [(float(m.cpu()), int(e.cpu())) for m, e in got]
    finally:
        h.close()
    assert got == [want] * 4
