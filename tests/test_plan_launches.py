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
