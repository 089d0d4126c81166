"""Leaf maxima of small and large leaves beside one another: leaves below, at
and above one and many parts, unaligned ones, more large leaves than one launch
lists, with the maximum at either end -- seen through the result's exponent,
which is the sum of the leaves' own."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    if not _t.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2002_01935_gb300 import build
    build.build()
    return _t


def check(torch, sizes, place, shift):
    """A product of vectors, each zero but for one power of two."""
    from paper_2002_01935_gb300 import binding
    n = len(sizes)
    ts, total = [], 0
    for i, k in enumerate(sizes):
        buf = torch.zeros(k + 4, device="cuda")
        t = buf[shift:shift + k]
        e = (7 * i) % 41 - 20
        t[{"first": 0, "last": k - 1, "middle": k // 2}[place]] = 2.0 ** e
        total += e
        ts.append(t)
    pairs, last = [(0, 1)], n
    for i in range(2, n):
        pairs.append((last, i))
        last += 1
    h = binding.TensorNetwork([[i] for i in range(n)], {i: k for i, k in enumerate(sizes)}, [], ts, complex_=False)
    try:
        m, e = h.contract(pairs, [], "fp32")
        m2, e2 = h.contract(pairs, [], "fp32")  # the slots of the call before are not in the way
    finally:
        h.close()
    frac, x = np.frexp(float(m.cpu()))
    assert frac == 0.5 and x - 1 + int(e.cpu()) == total
    # every vertex is divided by its own largest entry: nothing is left over or flushed
    assert torch.equal(m, m2) and torch.equal(e, e2)


@pytest.mark.parametrize("place", ["first", "middle", "last"])
@pytest.mark.parametrize("shift", [0, 1, 2])
def test_mixed_sizes(torch, place, shift):
    check(torch, [2, 3, 4095, 4097, 16383, 16384, 16385, 2, 32768, 40001, 1 << 20, 5, (1 << 24) + 3, 2], place, shift)


@pytest.mark.parametrize("n", [127, 128, 129, 300])
def test_many_large_leaves(torch, n):
    check(torch, [16385 + 16384 * (i % 3) if i % 5 else 3 for i in range(n + n // 4 + 2)], "last", 0)
