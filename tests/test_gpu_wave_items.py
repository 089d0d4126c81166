"""Wave items of fewer, exactly and more outputs than threads, alone in their
launch (their offsets entered per output) and as part of a dataflow (offsets
from tables): a node as its own network, and the same bits from a two-node
network run level by level and as one dataflow.

Tolerance: a sum of K products in FP32, (8 sqrt(2 K) + 8) 2^-24 of the sum of
|products|.
"""
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


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("m,n,k,b", [(0, 1, 1, 0), (2, 2, 2, 10), (1, 1, 1, 10), (4, 4, 8, 0), (3, 5, 2, 0), (5, 4, 1, 0),
                                     (5, 5, 0, 0), (0, 0, 3, 12), (4, 4, 12, 0), (0, 8, 8, 2), (7, 7, 3, 0)])
def test_one_node(torch, monkeypatch, cplx, m, n, k, b):
    from paper_2002_01935_gb300 import binding
    ids, at = [], 0
    for q in (m, n, k, b):
        ids.append(list(range(at, at + q)))
        at += q
    m_, n_, k_, b_ = ids
    la, lb, lo = b_ + k_[::2] + m_ + k_[1::2], n_[:2] + k_ + b_ + n_[2:], b_ + m_ + n_
    dt = torch.complex64 if cplx else torch.float32
    g = torch.Generator(device="cuda").manual_seed(at)
    ts = [torch.randn([2] * len(ls), dtype=dt, device="cuda", generator=g) for ls in (la, lb)]
    wide = [t.to(torch.complex128 if cplx else torch.float64) for t in ts]
    ref = torch.einsum(wide[0], la, wide[1], lb, lo).cpu().numpy()
    scale = torch.einsum(wide[0].abs(), la, wide[1].abs(), lb, lo).cpu().numpy()
    dims = {l: 2 for l in range(at)}
    h = binding.TensorNetwork([la, lb], dims, lo, ts, complex_=cplx)
    try:
        assert h.plan_steps([(0, 1)], [], "fp32")[0]["wave"]
        mant, e = h.contract([(0, 1)], [], "fp32")
        got = (mant * 2.0 ** e.double()).cpu().numpy()
    finally:
        h.close()
    assert np.all(np.abs(got - ref) <= (8.0 * np.sqrt(2.0 * 2 ** k) + 8.0) * 2.0 ** -24 * scale)
    # and a sign for every output: two levels
    sign = torch.tensor([1.0, -1.0], dtype=dt, device="cuda")
    bits = []
    for flow in ("0", "1"):
        monkeypatch.setenv("TN_NO_FLOW", flow)
        h = binding.TensorNetwork([la, lb, [lo[0]]], dims, lo, ts + [sign], complex_=cplx)
        try:
            mant, e = h.contract([(0, 1), (3, 2)], [], "fp32")
            bits.append((mant.cpu().numpy().tobytes(), int(e.cpu())))
        finally:
            h.close()
    assert bits[0] == bits[1]
