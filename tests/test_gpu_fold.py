"""The fold of the root into the result: outputs in the root's order and in
other orders (a transposed root, interleaved labels), few and many outputs,
label sizes that are not powers of two, one group or several (slices, slices
side by side), against an FP64 einsum.

Tolerance: K <= 16 products of standard normals per output in FP32, summed
over at most 8 slices in FP64: each output is off by at most (K + 2) 2^-24 of
the sum of its |products|; the bound below is 32 * 2^-24 of that sum.
"""
import numpy as np
import pytest

from paper_2002_01935_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL = 32 * 2.0 ** -24


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    if not _t.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2002_01935_gb300 import build
    build.build()
    return _t


def order(kind, m, n, rng):
    if kind == "mn":
        return m + n
    if kind == "nm":
        return n + m
    return [int(x) for x in rng.permutation(m + n)]


@pytest.mark.parametrize("cplx", [True, False])
@pytest.mark.parametrize("kind", ["mn", "nm", "mixed"])
@pytest.mark.parametrize("dims", [([2] * 5, [2] * 4, [2] * 3), ([2] * 5, [2] * 6, [2] * 4), ([4, 2, 8], [2] * 7, [2, 4]),
                                  ([2] * 9, [2] * 8, [2] * 3), ([3, 5, 2], [7, 2, 3], [2, 3]), ([33], [70], [5]),
                                  ([], [2] * 11, [2] * 4)])
def test_output_orders(torch, dims, kind, cplx):
    from paper_2002_01935_gb300 import binding
    rng = np.random.default_rng(sum(map(sum, dims)) + 10 * len(kind) + cplx)
    md, nd, kd = dims
    m = list(range(len(md)))
    n = list(range(len(md), len(md) + len(nd)))
    k = list(range(len(md) + len(nd), len(md) + len(nd) + len(kd)))
    size = dict(zip(m + n + k, md + nd + kd))
    la, lb, lo = k[::2] + m + k[1::2], n[:2] + k + n[2:], order(kind, m, n, rng)

    def t(ls):
        x = rng.standard_normal([size[l] for l in ls])
        return x + 1j * rng.standard_normal(x.shape) if cplx else x
    net = inputs.Network([t(la), t(lb)], [la, lb], size, lo).as_stored()
    dt = torch.complex64 if cplx else torch.float32
    ts = [torch.from_numpy(np.array(x, order="C")).to(dt).cuda() for x in net.tensors]
    tnw = binding.TensorNetwork(net.labels, net.dims, net.open, ts, complex_=cplx)
    ref = np.einsum(net.tensors[0], la, net.tensors[1], lb, lo)
    scale = np.einsum(np.abs(net.tensors[0]), la, np.abs(net.tensors[1]), lb, lo)
    try:
        for sliced, batch, host in (([], 0, False), ([], 0, True), (k[:1], 0, False), (k[:1], 2, False),
                                    (k[:2], 3, False)):
            out = ex = None
            if host:
                out = torch.empty(tnw.out_shape, dtype=torch.complex128 if cplx else torch.float64)
                ex = torch.empty((), dtype=torch.int64)
            for _ in range(2):  # the second call finds the first one's accumulator
                mant, e = tnw.contract([(0, 1)], sliced, "fp32", out=out, out_exp=ex, slice_batch=batch)
            got = mant.cpu().numpy() * 2.0 ** int(e)
            assert np.max(np.abs(got - ref) / scale) <= TOL, (sliced, batch, host)
        # a slice of zeros only, alone and as the last of the call's groups
        ts[0].zero_()
        mant, e = tnw.contract([(0, 1)], k[:1], "fp32")
        assert int(e) == 0 and not mant.abs().any()
    finally:
        tnw.close()


def test_zero_slices_keep_the_sum(torch):
    """Slices that are exactly zero, first or last, leave the others' sum."""
    from paper_2002_01935_gb300 import binding
    rng = np.random.default_rng(3)
    for zero in (0, 1, 2):
        a = rng.standard_normal((3, 40)).astype(np.float32)
        a[zero] = 0
        b = rng.standard_normal((3, 50)).astype(np.float32)
        tnw = binding.TensorNetwork([[0, 1], [0, 2]], {0: 3, 1: 40, 2: 50}, [2, 1],
                                    [torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()], complex_=False)
        for batch in (0, 2):
            m, e = tnw.contract([(0, 1)], [0], "fp32", slice_batch=batch)
            got = m.cpu().numpy() * 2.0 ** int(e)
            ref = b.T.astype(np.float64) @ a.astype(np.float64)
            assert np.max(np.abs(got - ref)) <= 8 * 2.0 ** -24 * np.max(np.abs(b).T @ np.abs(a))
        tnw.close()


def test_output_with_the_alignment_of_a_double(torch):
    """The C-ABI's output pointer need not be 16-byte aligned."""
    from paper_2002_01935_gb300 import binding
    g = torch.Generator(device="cuda").manual_seed(5)
    a = torch.randn(64, 8, dtype=torch.complex64, device="cuda", generator=g)
    b = torch.randn(8, 96, dtype=torch.complex64, device="cuda", generator=g)
    tnw = binding.TensorNetwork([[0, 1], [1, 2]], {0: 64, 1: 8, 2: 96}, [0, 2], [a, b])
    m, e = tnw.contract([(0, 1)], [], "fp32")
    buf = torch.empty(2 * 64 * 96 + 1, dtype=torch.float64, device="cuda")
    binding.tn_contract(tnw.h, [(0, 1)], [], 0, buf.data_ptr() + 8, 0, e.data_ptr(),
                        torch.cuda.current_stream().cuda_stream)
    assert torch.equal(buf[1:].view(64, 96, 2), torch.view_as_real(m))
    tnw.close()


@pytest.mark.parametrize("n", [1, 4095, 4096, 16385, 300007])
@pytest.mark.parametrize("shift", [0, 1])
def test_leaf_maximum_of_any_size_and_alignment(torch, n, shift):
    """A leaf's renormalisation exponent shows in the result's exponent: the
    largest entry wherever it stands, in leaves that start on 16 bytes or not."""
    from paper_2002_01935_gb300 import binding
    for at in {0, n // 2, n - 1}:
        buf = torch.full((n + shift,), 0.75, device="cuda")
        leaf = buf[shift:]
        leaf[at] = 3.0 * 2.0 ** 20
        one = torch.ones(1, device="cuda")
        tnw = binding.TensorNetwork([[0], [1]], {0: n, 1: 1}, [0, 1], [leaf, one], complex_=False)
        m, e = tnw.contract([(0, 1)], [], "fp32")
        assert int(e) == 22 + 1
        assert torch.equal(m.view(-1) * 2.0 ** 23, leaf.double())
        tnw.close()
