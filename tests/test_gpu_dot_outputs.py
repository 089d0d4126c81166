"""Inner-product nodes with several outputs: one CTA computes all of them from
one pass over either operand, so every split of 64 outputs into rows and
columns has its own thread layout and tile size.  Rows, columns and K labels
stand in seeded orders in both operands (rows below, between and above the K
strides), K from the shortest (2^9) to several tiles per part, batch labels,
labels summed in one operand only and slices side by side, against an FP64
einsum.  Tolerance: sums of K products in FP32 by at most 32 lanes, parts and
tiles each; (8 sqrt(2 K) + 8) 2^-24 of the sum of |products| covers a single
sequential sum as a random walk.
"""
import numpy as np
import pytest

from paper_2002_01935_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    if not _t.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2002_01935_gb300 import build
    build.build()
    return _t


@pytest.mark.parametrize("cplx", [True, False])
@pytest.mark.parametrize("shape", [(0, 0, 14, 0), (6, 0, 9, 0), (0, 6, 10, 0), (5, 1, 11, 0), (1, 5, 9, 1), (3, 3, 14, 0),
                                   (2, 2, 16, 0), (4, 2, 10, 2), (2, 0, 13, 0), (0, 1, 12, 1), (1, 1, 9, 0)])
def test_outputs(torch, shape, cplx):
    from paper_2002_01935_gb300 import binding
    mb, nb, kb, bb = shape
    for seed in range(3):
        rng = np.random.default_rng(100 * seed + sum(shape) + cplx)
        n_lab = mb + nb + kb + bb + 1
        ids = list(range(n_lab))
        m, n, k, b, one = ids[:mb], ids[mb:mb + nb], ids[mb + nb:mb + nb + kb], ids[mb + nb + kb:-1], ids[-1:]
        la = [int(x) for x in rng.permutation(m + k + b + (one if seed == 1 else []))]
        lb = [int(x) for x in rng.permutation(n + k + b + (one if seed != 1 else []))]
        lo = b + m + n

        def t(ls):
            x = rng.standard_normal([2] * len(ls))
            return x + 1j * rng.standard_normal(x.shape) if cplx else x
        net = inputs.Network([t(la), t(lb)], [la, lb], {l: 2 for l in ids}, lo).as_stored()
        ref = np.einsum(net.tensors[0], la, net.tensors[1], lb, lo, optimize=True)
        scale = np.einsum(np.abs(net.tensors[0]), la, np.abs(net.tensors[1]), lb, lo, optimize=True)
        dt = torch.complex64 if cplx else torch.float32
        ts = [torch.from_numpy(np.array(x, order="C")).to(dt).cuda() for x in net.tensors]
        tnw = binding.TensorNetwork(net.labels, net.dims, net.open, ts, complex_=cplx)
        tol = (8.0 * np.sqrt(2.0 * 2 ** (kb + 1)) + 8.0) * 2.0 ** -24
        try:
            for sliced, batch in (([], 0), (k[2:4] if kb > 11 else one, 2)):
                if not sliced:
                    assert [s["cfg"] for s in tnw.plan_steps([(0, 1)], [], "fp32")] == [5]
                mant, e = tnw.contract([(0, 1)], sliced, "fp32", slice_batch=batch)
                got = mant.cpu().numpy() * 2.0 ** int(e)
                assert np.max(np.abs(got - ref) / scale) <= tol
        finally:
            tnw.close()
