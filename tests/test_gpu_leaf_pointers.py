"""Re-attached leaves: a captured launch sequence is kept when only leaves
that waves read move, and captured anew when a node with its own launch reads
the leaf, after autotuning and with other copy strides.  Every result is bit
for bit that of a fresh handle on the same leaves."""
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


def same(torch, x, y):
    assert torch.equal(torch.view_as_real(x[0]), torch.view_as_real(y[0])) and torch.equal(x[1], y[1])


def test_small_leaves_move(torch):
    from paper_2002_01935_gb300 import binding
    circ = inputs.random_circuit(4, 3, 8, seed=2)
    net = inputs.circuit_network(circ, [0] * 12, open_qubits=[9, 10, 11])
    pairs = planner.greedy_tree(net.labels, net.dims, net.open)
    base = [torch.from_numpy(np.array(t, order="C")).to(torch.complex64).cuda() for t in net.tensors]
    keep = binding.TensorNetwork(net.labels, net.dims, net.open, base)
    first = net.n_tensors - 9
    basis = torch.eye(2, dtype=torch.complex64, device="cuda")
    for bits in inputs.random_bitstrings(9, 6, seed=4):
        leaves = base[:first] + [basis[int(b)] for b in bits]
        keep.set_tensors(leaves)
        got = keep.contract(pairs, [], "fp32")
        fresh = binding.TensorNetwork(net.labels, net.dims, net.open, leaves)
        same(torch, got, fresh.contract(pairs, [], "fp32"))
        assert got[0].abs().max() > 0
        fresh.close()
    keep.close()


@pytest.mark.parametrize("mode", ["fp32", "fp16_split"])
def test_large_leaves_move(torch, mode):
    from paper_2002_01935_gb300 import binding
    g = torch.Generator(device="cuda").manual_seed(1)
    labels, dims = [[0, 1], [1, 2]], {0: 256, 1: 64, 2: 512}
    ts = [torch.randn([dims[l] for l in ls], dtype=torch.complex64, device="cuda", generator=g)
          for ls in labels for _ in range(2)]
    keep = binding.TensorNetwork(labels, dims, [0, 2], [ts[0], ts[2]])
    for a, b in ((0, 2), (1, 2), (1, 3), (0, 2)):
        keep.set_tensors([ts[a], ts[b]])
        fresh = binding.TensorNetwork(labels, dims, [0, 2], [ts[a], ts[b]])
        same(torch, keep.contract([(0, 1)], [], mode), fresh.contract([(0, 1)], [], mode))
        fresh.close()
    # after tuning, the kernels chosen then run (same value within rounding)
    before = keep.contract([(0, 1)], [], mode)
    keep.autotune([(0, 1)], [], mode, reps=1)
    after = keep.contract([(0, 1)], [], mode)
    assert (before[0] - after[0]).abs().max() <= 1e-5 * before[0].abs().max()
    keep.close()


def test_copy_strides_change(torch):
    from paper_2002_01935_gb300 import binding
    g = torch.Generator(device="cuda").manual_seed(2)
    a = torch.randn(6, 64, 64, dtype=torch.complex64, device="cuda", generator=g)
    b = torch.randn(64, 64, dtype=torch.complex64, device="cuda", generator=g)
    tnw = binding.TensorNetwork([[0, 1], [0, 1]], {0: 64, 1: 64}, [], [a, b])
    for step in (1, 2, 1):  # the same pointer, every copy or every other one
        m, e = tnw.contract_instances([(0, 1)], "fp32", 3, [step * 4096, 0])
        got = torch.view_as_complex(m).cpu() * 2.0 ** e.cpu()
        ref = (a[:3 * step:step].to(torch.complex128) * b).sum((1, 2)).cpu()
        assert (got - ref).abs().max() <= 1e-5 * (a.abs() * b.abs()).sum((1, 2)).max().cpu()
    tnw.close()


def test_tree_lists_that_change_are_seen():
    from paper_2002_01935_gb300 import binding
    pairs = [(0, 1), (2, 4), (3, 5)]
    first = binding._tree(pairs).tolist()
    assert binding._tree(pairs).tolist() == first
    pairs[1] = (3, 4)
    pairs[2] = (2, 5)
    assert binding._tree(pairs).tolist() == [0, 1, 3, 4, 2, 5]
    lists = [[0, 1], [2, 3]]
    assert binding._tree(lists).tolist() == [0, 1, 2, 3]
    lists[1][0] = 1
    assert binding._tree(lists).tolist() == [0, 1, 1, 3]
