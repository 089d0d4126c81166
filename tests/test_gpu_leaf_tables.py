"""Leaves re-attached between calls on a stream that is still busy: every call
reads the leaves that it was made with (the pointer table is written in stream
order, from memory that is the call's own).  The stream is held up by a
bounded spin, so that all calls are made before the first one runs."""
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


def spin_chain(n):
    """A ring of n matrices: more leaves than one table launch holds."""
    rng = np.random.default_rng(2)
    return inputs.Network([rng.random((2, 2)) + 0.2 for _ in range(n)], [[i, (i + 1) % n] for i in range(n)],
                          {i: 2 for i in range(n)}, [])


@pytest.mark.parametrize("n", [3, 500, 501, 1100])
def test_table_follows_the_calls(torch, n):
    from paper_2002_01935_gb300 import binding
    net = spin_chain(n)
    pairs, last = [(0, 1)], n
    for i in range(2, n):
        pairs.append((last, i))
        last += 1
    base = np.array([np.asarray(t) for t in net.tensors], dtype=np.float32)
    sets = [torch.from_numpy(base * np.float32(2.0) ** (j - 2)).cuda() for j in range(5)]  # exact factors
    h = binding.TensorNetwork(net.labels, net.dims, net.open, [t for t in sets[0]], complex_=False)
    stream = torch.cuda.Stream()
    try:
        h.contract(pairs, [], "fp32")
        torch.cuda.synchronize()
        got = []
        with torch.cuda.stream(stream):
            torch.cuda._sleep(100_000_000)
            for s in sets:
                h.set_tensors([t for t in s])
                got.append(h.contract(pairs, [], "fp32"))
        torch.cuda.synchronize()
        m = [float(x.cpu()) for x, _ in got]
        e = [int(x.cpu()) for _, x in got]
    finally:
        h.close()
    # copy j is 2^((j - 2) n) of the third: the same mantissa bits up to its own power of two
    frac = [np.frexp(x) for x in m]
    assert all(f[0] == frac[2][0] and f[0] > 0 for f in frac)
    assert [f[1] + x - (frac[2][1] + e[2]) for f, x in zip(frac, e)] == [(j - 2) * n for j in range(5)]
