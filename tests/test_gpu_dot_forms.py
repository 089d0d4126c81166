"""Inner-product nodes around the line between one block per output and one
block for all outputs (two tiles of 1024 products per SM; one row of 8192 tiles
or more, contiguous along K or not), with batch labels slowest and fastest, in
one and in several copies, against an FP64 einsum.

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


ORDERS = {"k_fastest": ("bmk", "bnk"), "batch_fastest": ("mkb", "nkb"), "rows_fastest": ("bkm", "kbn")}


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("order", list(ORDERS))
@pytest.mark.parametrize("m,n,k,b", [(8, 8, 9, 0), (8, 8, 12, 0), (8, 8, 13, 0), (1, 2, 17, 0), (1, 2, 18, 0),
                                     (1, 64, 16, 0), (1, 64, 17, 0), (1, 4, 14, 8), (4, 2, 10, 5), (4, 2, 10, 6),
                                     (1, 1, 11, 4)])
def test_forms(torch, cplx, order, m, n, k, b):
    from paper_2002_01935_gb300 import binding
    size = {"m": m, "n": n, "k": 2 ** k, "b": 2 ** b}
    ids = {c: i for i, c in enumerate("mnkb")}
    la, lb = ORDERS[order]
    g = torch.Generator(device="cuda").manual_seed(k)
    dt = torch.complex64 if cplx else torch.float32
    ts = [torch.randn([size[c] for c in ls], dtype=dt, device="cuda", generator=g) for ls in (la, lb)]
    h = binding.TensorNetwork([[ids[c] for c in la], [ids[c] for c in lb]], {ids[c]: size[c] for c in "mnkb"},
                              [ids["b"], ids["m"], ids["n"]], ts, complex_=cplx)
    try:
        step, = h.plan_steps([(0, 1)], [], "fp32")
        assert step["cfg"] == 5
        mant, e = h.contract([(0, 1)], [], "fp32")
        got = (mant * 2.0 ** e.double()).cpu().numpy()
    finally:
        h.close()
    wide = [t.to(torch.complex128 if cplx else torch.float64) for t in ts]
    ref = torch.einsum(f"{la},{lb}->bmn", *wide).cpu().numpy()
    scale = torch.einsum(f"{la},{lb}->bmn", *(t.abs() for t in wide)).cpu().numpy()
    assert np.all(np.abs(got - ref) <= (8.0 * np.sqrt(2.0 * 2 ** k) + 8.0) * 2.0 ** -24 * scale)


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("k,copies", [(12, 3), (12, 40), (18, 5), (18, 40)])
def test_copies(torch, cplx, k, copies):
    """Scalar networks of a row times a matrix times a column: the inner
    products of every copy."""
    from paper_2002_01935_gb300 import binding
    g = torch.Generator(device="cuda").manual_seed(k)
    dt = torch.complex64 if cplx else torch.float32
    ts = [torch.randn(copies, *s, dtype=dt, device="cuda", generator=g) for s in ((2 ** k,), (2 ** k, 2), (2,))]
    h = binding.TensorNetwork([[0], [0, 1], [1]], {0: 2 ** k, 1: 2}, [], ts, complex_=cplx)
    try:
        m, e = h.contract_instances([(0, 1), (3, 2)], "fp32", copies, [2 ** k, 2 ** (k + 1), 2])
        got = (m * 2.0 ** e.double()[:, None]).cpu().numpy()
    finally:
        h.close()
    got = got[:, 0] + 1j * got[:, 1]
    wide = [t.to(torch.complex128) for t in ts]
    ref = torch.einsum("ck,ckn,cn->c", *wide).cpu().numpy()
    scale = torch.einsum("ck,ckn,cn->c", *(t.abs() for t in wide)).cpu().numpy()
    assert np.all(np.abs(got - ref) <= (8.0 * np.sqrt(4.0 * 2 ** k) + 16.0) * 2.0 ** -24 * scale)
