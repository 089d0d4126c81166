"""A contraction captured in the caller's CUDA graph keeps the leaves that it
was captured with: its replay gives their value after other leaves were
attached and contracted, and direct calls after a replay read the attached
ones.  Networks of two- and three-valued labels, with subtree regions."""
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


@pytest.mark.parametrize("q", [2, 3])
def test_replay_keeps_its_leaves(torch, q):
    from paper_2002_01935_gb300 import binding
    edges = inputs.random_regular_graph(12, 3, 4)
    labels = [[int(u), int(v)] for u, v in edges]
    dims = {v: q for v in range(12)}
    pairs = planner.greedy_tree(labels, dims, [])
    g = torch.Generator(device="cuda").manual_seed(1)
    sets = [list((torch.rand(len(edges), q, q, device="cuda", generator=g) + 0.1).unbind(0)) for _ in range(3)]
    sets = [[t.clone() for t in s] for s in sets]

    def value(m, e):
        return float(m.cpu()) * 2.0 ** int(e.cpu())

    def fresh(s):
        h = binding.TensorNetwork(labels, dims, [], s, complex_=False)
        try:
            return value(*h.contract(pairs, [], "fp32"))
        finally:
            h.close()

    want = [fresh(s) for s in sets]
    assert len(set(want)) == 3
    h = binding.TensorNetwork(labels, dims, [], sets[0], complex_=False)
    try:
        h.contract(pairs, [], "fp32")
        out = torch.empty((), dtype=torch.float64, device="cuda")
        ex = torch.empty((), dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            h.contract(pairs, [], "fp32", out=out, out_exp=ex)
        graph.replay()
        torch.cuda.synchronize()
        assert value(out, ex) == want[0]
        for j in (1, 2):
            h.set_tensors(sets[j])
            assert value(*h.contract(pairs, [], "fp32")) == want[j]
            graph.replay()
            torch.cuda.synchronize()
            assert value(out, ex) == want[0]
            assert value(*h.contract(pairs, [], "fp32")) == want[j]  # leaves not attached anew
    finally:
        h.close()
