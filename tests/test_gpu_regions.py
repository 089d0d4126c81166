"""Subtree regions (small connected pieces of the tree, one block each).

Networks of two-valued labels: a region adds up every output in the order of
the per-node launches (TN_NO_FLOW=1), so amplitudes, copies, slices and
gradients are the same bits.  Networks of other label sizes take another
kernel there: against the nested sum instead, with the bound of the other
any-size tests (1e-5 of the sum of |products|).
"""
import numpy as np
import pytest

from oracle import brute, tree
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


def handle(torch, net, copies=1):
    """Handle on stacked copies of the leaves (copy i: the leaf times 1 + i),
    and their strides."""
    from paper_2002_01935_gb300 import binding
    dt = torch.complex64 if net.is_complex else torch.float32
    ts = [torch.from_numpy(np.array(t, order="C")).to(dt).cuda() for t in net.tensors]
    strides = [t.numel() for t in ts]
    if copies > 1:
        ts = [torch.stack([t * (1 + i) for i in range(copies)]) for t in ts]
    return binding.TensorNetwork(net.labels, net.dims, net.open, ts, complex_=net.is_complex), strides


def circuit(r, c, depth, opened=0):
    circ = inputs.random_circuit(r, c, depth, seed=2)
    return inputs.circuit_network(circ, inputs.random_bitstrings(r * c, 1, seed=7)[0], open_qubits=range(opened))


NETS = {
    "circuit_2x2": lambda: circuit(2, 2, 4),
    "circuit_3x3_open": lambda: circuit(3, 3, 8, 3),
    "circuit_4x4": lambda: circuit(4, 4, 8),
    "ising_20": lambda: inputs.random_ising(20, seed=1),
    "ising_100": lambda: inputs.random_ising(100, seed=1),
}


def labels_to_slice(net, k):
    rng = np.random.default_rng(3)
    summed = [l for l in sorted(net.dims) if l not in net.open]
    return [int(x) for x in rng.choice(summed, size=k, replace=False)]


def regions(h, pairs, sliced=()):
    """Multi-node steps that are no waves."""
    return [s for s in h.plan_steps(pairs, list(sliced), "fp32") if not s["wave"] and len(s["nodes"]) > 1]


@pytest.mark.parametrize("name", list(NETS))
@pytest.mark.parametrize("sliced,slice_batch", [(0, 1), (2, 1), (3, 3)])
def test_same_bits_as_single_launches(torch, monkeypatch, name, sliced, slice_batch):
    net = NETS[name]()
    pairs = planner.greedy_tree(net.labels, net.dims, net.open)
    sl = labels_to_slice(net, sliced)
    res = []
    for flow in ("0", "1"):
        monkeypatch.setenv("TN_NO_FLOW", flow)
        h, strides = handle(torch, net)
        try:
            assert bool(regions(h, pairs, sl)) == (flow == "0")
            for _ in range(2):  # capture, then replay
                m, e = h.contract(pairs, sl, "fp32", slice_batch=slice_batch)
                torch.cuda.synchronize()
                res.append((m.cpu().numpy().tobytes(), int(e.cpu())))
        finally:
            h.close()
    assert res[1:] == res[:-1]


@pytest.mark.parametrize("name,n_inst", [("circuit_2x2", 2), ("circuit_4x4", 5), ("ising_20", 33)])
def test_same_bits_with_copies(torch, monkeypatch, name, n_inst):
    net = NETS[name]()
    pairs = planner.greedy_tree(net.labels, net.dims, net.open)
    res = []
    for flow in ("0", "1"):
        monkeypatch.setenv("TN_NO_FLOW", flow)
        h, strides = handle(torch, net, n_inst)
        try:
            m, e = h.contract_instances(pairs, "fp32", n_inst, strides)
            torch.cuda.synchronize()
            res.append((m.cpu().numpy().tobytes(), e.cpu().tolist()))
        finally:
            h.close()
    assert res[0] == res[1]


@pytest.mark.parametrize("name,n_inst,sliced", [("circuit_2x2", 1, 0), ("circuit_4x4", 1, 0), ("circuit_4x4", 1, 2),
                                                ("circuit_4x4", 3, 0), ("circuit_3x3_open", 1, 1),
                                                ("ising_20", 2, 0), ("ising_100", 1, 0)])
def test_gradients_have_the_same_bits(torch, monkeypatch, name, n_inst, sliced):
    """Both halves of the reverse sweep, and the sweep over kept values."""
    net = NETS[name]()
    pairs = planner.greedy_tree(net.labels, net.dims, net.open)
    sl = labels_to_slice(net, sliced)
    rng = np.random.default_rng(1)
    adj = rng.standard_normal((n_inst,) + tuple(net.dims[l] for l in net.open))
    adj = adj + 1j * rng.standard_normal(adj.shape) if net.is_complex else adj
    res = []
    for flow in ("0", "1"):
        monkeypatch.setenv("TN_NO_FLOW", flow)
        h, strides = handle(torch, net, n_inst)
        try:
            for _ in range(2):
                g = h.grad_instances(pairs, sl, "fp32", n_inst, strides, adj)
                torch.cuda.synchronize()
                res.append([x.cpu().numpy().tobytes() for x in g])
            if not sliced and not net.open:
                m, e, token = h.contract_instances_keep(pairs, "fp32", n_inst, strides)
                g = h.grad_instances(pairs, sl, "fp32", n_inst, strides, adj, kept_forward=token)
                torch.cuda.synchronize()
                res.append([x.cpu().numpy().tobytes() for x in g])
        finally:
            h.close()
    assert res[1:] == res[:-1]


@pytest.mark.parametrize("seed", range(24))
def test_any_label_sizes(torch, seed):
    net = inputs.random_network(5 + seed % 8, 7 + seed % 7, 400 + seed, n_open=seed % 3, max_dim=2 + seed % 4,
                                complex_=seed % 2 == 0)
    pairs = planner.greedy_tree(net.labels, net.dims, net.open)
    sl = labels_to_slice(net, min(seed % 4, len(net.dims) - len(net.open)))
    h, strides = handle(torch, net)
    try:
        m, e = h.contract(pairs, sl, "fp32", slice_batch=1 + seed % 3)
        torch.cuda.synchronize()
        got = m.cpu().numpy() * 2.0 ** int(e.cpu())
    finally:
        h.close()
    ref = brute.nested_sum(net.tensors, net.labels, net.dims, net.open)
    scale = brute.nested_sum([np.abs(t) for t in net.tensors], net.labels, net.dims, net.open)
    assert np.all(np.abs(got - ref) <= 1e-5 * np.abs(scale) + 1e-30)


def batch_nets():
    nets = [circuit(2, 2, 4), circuit(3, 3, 8), circuit(4, 4, 8)]
    nets += [inputs.random_ising(n, seed=n) for n in (8, 20, 60, 100)]
    return nets + nets[:4]  # more networks than concurrent groups


def test_batch_members(torch, monkeypatch):
    """Complex and real members of one to a few regions, roots inside a
    region (their completion time too), against the oracle with the bound of
    the other batch tests (a forest sums its waves' outputs in another order
    than a single network); capture and replay are the same bits."""
    from paper_2002_01935_gb300 import binding
    nets = batch_nets()
    trees = [planner.greedy_tree(n.labels, n.dims, n.open) for n in nets]
    ref = [tree.contract_net(n, t) for n, t in zip(nets, trees)]
    for flow in ("0", "1"):
        monkeypatch.setenv("TN_NO_FLOW", flow)
        hs = [handle(torch, n)[0] for n in nets]
        b = binding.Batch(hs, trees, "fp32")
        try:
            res = []
            for _ in range(2):
                m, e, lat = b.contract()
                torch.cuda.synchronize()
                assert bool((lat > 0).all()) and bool((lat < 10**9).all())
                res.append((m.cpu().numpy(), e.cpu().numpy()))
        finally:
            b.close()
            for h in hs:
                h.close()
        assert np.array_equal(res[0][0], res[1][0]) and np.array_equal(res[0][1], res[1][1])
        for i, (mo, eo) in enumerate(ref):
            got = complex(*res[0][0][i]) * 2.0 ** (int(res[0][1][i]) - eo)
            assert abs(got - complex(mo)) <= 1e-5 * abs(complex(mo)), (flow, i)
