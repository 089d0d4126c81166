"""NaN and infinities in a leaf stay where they belong.

One entry of a leaf with an open label is NaN or infinite, so that only the
outputs of that index are touched.  The node maxima leave NaN out in every
kernel (the largest number decides the scale), so subtree regions give the
same values as one launch per level (TN_NO_FLOW=1): the untouched outputs as
they are, the touched ones not finite.
"""
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


def circuit(r, c, depth, opened):
    circ = inputs.random_circuit(r, c, depth, seed=2)
    return inputs.circuit_network(circ, inputs.random_bitstrings(r * c, 1, seed=7)[0], open_qubits=range(opened))


def ising(n, opened):
    """Spin network whose first copies tensors get one more, open label."""
    edges = inputs.random_regular_graph(n, 3, 5)
    net = inputs.ising_network(n, edges, inputs.ising_couplings(len(edges), 5), 0.3)
    tensors, labels, dims = [np.array(t) for t in net.tensors], [list(l) for l in net.labels], dict(net.dims)
    new = max(dims) + 1
    for v in range(opened):
        tensors[v] = np.multiply.outer(np.array([1.0, 0.5 + v]), tensors[v])
        labels[v] = [new + v] + labels[v]
        dims[new + v] = 2
    return inputs.Network(tensors, labels, dims, list(range(new, new + opened)))


NETS = {
    "circuit_2x2": lambda: circuit(2, 2, 4, 2),
    "circuit_3x3": lambda: circuit(3, 3, 8, 3),
    "circuit_4x3": lambda: circuit(4, 3, 8, 6),
    "ising_20": lambda: ising(20, 3),
}


@pytest.mark.parametrize("name", list(NETS))
@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("sliced,slice_batch", [(0, 0), (2, 0), (3, 3)])
def test_untouched_outputs_stay(torch, monkeypatch, name, bad, sliced, slice_batch):
    from paper_2002_01935_gb300 import binding
    net = NETS[name]()
    dt = torch.complex64 if net.is_complex else torch.float32
    ts = [torch.from_numpy(np.array(t, order="C")).to(dt) for t in net.tensors]
    v = next(v for v, ls in enumerate(net.labels) if net.open[0] in ls)
    at = net.labels[v].index(net.open[0])
    ts[v][tuple(1 if j == at else 0 for j in range(ts[v].dim()))] = bad
    pairs = planner.greedy_tree(net.labels, net.dims, net.open)
    rng = np.random.default_rng(3)
    summed = [l for l in sorted(net.dims) if l not in net.open]
    sl = [int(x) for x in rng.choice(summed, size=sliced, replace=False)]
    res = []
    for flow in ("0", "1"):
        monkeypatch.setenv("TN_NO_FLOW", flow)
        h = binding.TensorNetwork(net.labels, net.dims, net.open, [t.cuda() for t in ts], complex_=net.is_complex)
        try:
            several = [s for s in h.plan_steps(pairs, sl, "fp32") if not s["wave"] and len(s["nodes"]) > 1]
            assert bool(several) == (flow == "0")
            m, e = h.contract(pairs, sl, "fp32", slice_batch=slice_batch)
            torch.cuda.synchronize()
            res.append((m.cpu().numpy(), int(e.cpu())))
        finally:
            h.close()
    (region, e_region), (level, e_level) = res
    assert np.isfinite(level[0]).all() and np.abs(level[0]).max() > 0  # outputs of the other index
    assert not np.isfinite(level[1]).all()
    assert e_region == e_level
    assert np.array_equal(np.isfinite(region), np.isfinite(level))
    assert np.array_equal(np.isnan(region), np.isnan(level))
    assert np.array_equal(region[np.isfinite(region)], level[np.isfinite(level)])
