"""tn_plan_info's workspace covers the workspace part of what tn_contract_noalloc
needs (host only: a tree beyond its 8 MiB is refused with the bytes needed,
before any device call), and exceeds it by no more than the order of
tn_contract's own launch sequence costs."""
import re

import numpy as np
import pytest

pytest.importorskip("torch")

from paper_2002_01935_gb300 import binding, inputs, planner  # noqa: E402


def hyper(n, q, seed):
    rng = np.random.default_rng(seed)
    edges = inputs.random_regular_graph(n, 3, seed)
    return inputs.Network([rng.random((q, q)) for _ in edges], [[int(u), int(v)] for u, v in edges],
                          {v: q for v in range(n)}, [])


def circuit(r, c, depth):
    return inputs.circuit_network(inputs.random_circuit(r, c, depth, seed=2), [0] * (r * c))


NETS = {"circuit_5x5": lambda: circuit(5, 5, 12), "circuit_6x5": lambda: circuit(6, 5, 10),
        "ising_150": lambda: inputs.random_ising(150, seed=3), "hyper_56": lambda: hyper(56, 5, 2)}


@pytest.mark.parametrize("name", list(NETS))
def test_no_allocation_call(name):
    net = NETS[name]()
    pairs = planner.greedy_tree(net.labels, net.dims, net.open)
    h = binding.TensorNetwork(net.labels, net.dims, net.open, None, complex_=net.is_complex)
    try:
        ws = int(h.plan_info(pairs, [], "fp32")["ws_bytes"])
        assert ws > 8 << 20
        entry = np.zeros(1)  # never read: the call is refused first
        for v in range(net.n_tensors):
            binding.tn_set_tensor(h.h, v, entry.ctypes.data, binding.TN_MEM_DEVICE)
        with pytest.raises(binding.TNError) as e:
            binding.tn_contract_noalloc(h.h, pairs, [], entry.ctypes.data, binding.TN_MEM_DEVICE, entry.ctypes.data)
        assert e.value.status == binding.TN_EUNSUPPORTED
        need = int(re.search(r"needs (\d+) bytes", str(e.value)).group(1))
    finally:
        h.close()
    # maxima and exponents per node, maxima, pointers and sizes per leaf,
    # control block, unit and accumulator, in 256-byte sections
    n = net.n_tensors
    sections = [0, 16, 4 * (n - 1), 8 * (n - 1), 4 * n, 8 * n, 8 * n, 16]
    part = need - sum((s + 255) // 256 * 256 for s in sections)
    assert part - 512 <= (ws + 255) // 256 * 256 <= 1.05 * part  # (512: the control block)
