"""The launch schedule counts what runs (host plan only, no GPU): a node of any
label sizes on the tile kernel reports its tile configuration, and its K parts
add the launch that sums them."""
import pytest

pytest.importorskip("torch")

from paper_2002_01935_gb300 import binding  # noqa: E402


def step(m, n, k, b=(), cplx=False):
    """The one step of a node with these label sizes."""
    ids, at = [], 0
    for g in (m, n, k, b):
        ids.append(list(range(at, at + len(g))))
        at += len(g)
    m_, n_, k_, b_ = ids
    dims = dict(enumerate([*m, *n, *k, *b]))
    h = binding.TensorNetwork([b_ + k_ + m_, n_ + k_ + b_], dims, b_ + m_ + n_, None, complex_=cplx)
    try:
        steps = h.plan_steps([(0, 1)], [], "fp32")
    finally:
        h.close()
    assert len(steps) == 1 and not steps[0]["wave"]
    return steps[0]


@pytest.mark.parametrize("cplx", [False, True])
def test_any_sizes(cplx):
    s = step([3] * 3, [3] * 3, [3] * 7, cplx=cplx)  # one tile over K = 2187: K parts and their sum
    assert (s["kind"], s["launches"]) == (0, 2) and s["cfg"] > 0
    s = step([5] * 5, [5] * 5, [5], cplx=cplx)  # 2401 tiles: no K parts
    assert (s["kind"], s["launches"]) == (0, 1) and s["cfg"] > 0
    s = step([3], [3], [3] * 4, cplx=cplx)  # one thread per output
    assert (s["kind"], s["cfg"], s["launches"]) == (0, 0, 1)


def test_power_of_two():
    s = step([2] * 6, [2] * 6, [2] * 14)
    assert (s["kind"], s["launches"]) == (1, 2) and s["cfg"] > 0


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("m,n,k,b,tiled", [
    (0, 0, 0, 10, False),  # products of single entries
    (1, 1, 1, 6, False), (1, 1, 1, 9, False), (2, 1, 1, 7, False), (0, 0, 2, 8, False), (0, 3, 1, 7, False),
    (2, 2, 2, 6, False), (0, 9, 0, 0, False),  # nearly empty tiles, few products
    (1, 1, 8, 0, True), (0, 0, 10, 0, True), (0, 0, 8, 3, True), (0, 1, 5, 5, True),  # long sums
    (5, 5, 5, 0, True), (3, 3, 4, 2, True),
])
def test_tiles_that_would_run_empty(m, n, k, b, tiled, cplx):
    """Nodes of three-valued labels: the tile kernel where its tiles are filled
    or the sums long, one thread per output elsewhere."""
    s = step([3] * m, [3] * n, [3] * k, [3] * b, cplx)
    assert s["kind"] == 0 and (s["cfg"] > 0) == tiled


@pytest.mark.parametrize("seed", range(24))
def test_small_networks_are_subtrees(seed):
    """The networks of any label sizes that the GPU tests contract in regions
    do have one: a step of several nodes that is no wave."""
    from paper_2002_01935_gb300 import inputs, planner
    net = inputs.random_network(5 + seed % 8, 7 + seed % 7, 400 + seed, n_open=seed % 3, max_dim=2 + seed % 4,
                                complex_=seed % 2 == 0)
    pairs = planner.greedy_tree(net.labels, net.dims, net.open)
    h = binding.TensorNetwork(net.labels, net.dims, net.open, None, complex_=net.is_complex)
    try:
        steps = h.plan_steps(pairs, [], "fp32")
    finally:
        h.close()
    assert any(not s["wave"] and len(s["nodes"]) > 1 and s["cfg"] == 0 and s["launches"] == 1 for s in steps)
