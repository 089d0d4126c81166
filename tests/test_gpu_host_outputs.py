"""Host outputs below, at and above the size that comes back in one copy with
its exponent: the bits of device outputs, sliced and not, in pageable and
page-locked memory."""
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
@pytest.mark.parametrize("lg,pinned", [(0, False), (11, False), (12, False), (12, True), (13, False), (14, False),
                                       (18, True)])
@pytest.mark.parametrize("sliced", [0, 1])
def test_same_bits(torch, cplx, lg, pinned, sliced):
    from paper_2002_01935_gb300 import binding
    m = list(range(lg // 2))
    n = list(range(lg // 2, lg))
    k = [lg, lg + 1, lg + 2]
    dims = {l: 2 for l in range(lg + 3)}
    dt = torch.complex64 if cplx else torch.float32
    g = torch.Generator(device="cuda").manual_seed(lg)
    ts = [torch.randn([2] * len(ls), dtype=dt, device="cuda", generator=g) for ls in (m + k, k + n)]
    h = binding.TensorNetwork([m + k, k + n], dims, n + m, ts, complex_=cplx)
    try:
        dev, e_dev = h.contract([(0, 1)], k[:sliced], "fp32")
        out = torch.zeros(h.out_shape, dtype=dev.dtype)
        out = out.pin_memory() if pinned else out
        ex = torch.zeros((), dtype=torch.int64)
        h.contract([(0, 1)], k[:sliced], "fp32", out=out, out_exp=ex)
        assert torch.equal(out, dev.cpu()) and int(ex) == int(e_dev.cpu())
        assert bool((out != 0).any())
    finally:
        h.close()
