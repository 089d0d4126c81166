"""A slice whose result is smaller than the others' by more than FP64 can
hold counts as zero in the sum, but a NaN or an infinity in it does not: the
fold gives the same with any number of slices side by side."""
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
@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("n_open", [1, 11])  # the plain and the permuted fold
def test_underflowing_slice(torch, cplx, bad, n_open):
    """Slice s of 32 vectors [2^20, 2^-20] and a matrix [s, open]: the second
    slice is 2^-1280 of the first."""
    from paper_2002_01935_gb300 import binding
    dt = torch.complex64 if cplx else torch.float32
    n, s = 32, 100
    opened = list(range(n_open))
    mat = torch.ones([2] * (n_open + 1), dtype=dt)
    mat[(1,) + (0,) * n_open] = bad
    labels = [[s]] * n + [[s] + opened]
    ts = [torch.tensor([2.0 ** 20, 2.0 ** -20], dtype=dt, device="cuda")] * n + [mat.cuda()]
    pairs, last = [(0, 1)], n + 1
    for i in range(2, n + 1):
        pairs.append((last, i))
        last += 1
    dims = {l: 2 for l in opened + [s]}
    res = []
    for batch in (1, 2):
        h = binding.TensorNetwork(labels, dims, opened[::-1], ts, complex_=cplx)
        try:
            m, e = h.contract(pairs, [s], "fp32", slice_batch=batch)
            torch.cuda.synchronize()
            res.append((m.cpu().numpy().reshape(-1), int(e.cpu())))
        finally:
            h.close()
    (one, e_one), (two, e_two) = res
    assert not np.isfinite(one[0]) and np.isfinite(one[1:]).all() and (one[1:] != 0).all()
    assert e_one == e_two
    assert np.array_equal(np.isnan(one), np.isnan(two))
    assert np.array_equal(one[1:], two[1:])
