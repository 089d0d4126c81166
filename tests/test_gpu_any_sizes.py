"""The tile kernel on nodes of any label sizes and on the edges of its tiles,
against an FP64 einsum of the stored leaves.

Shapes: every tile shape (up to 4 rows, up to 32 rows or columns, square, the
128 x 128 tiles of large real nodes) one entry below, at and above its edges,
one row or column, K of one, beyond the 1024-entry offset table, K splits,
batch labels, labels summed in one operand only, sliced leaves, operands
contiguous along either side, the reverse sweep (conjugated operands) and
copies.

Tolerance: every output is a sum of K products in FP32 (2 K real ones for a
complex part) of which each addition rounds by 2^-24 of the partial sum; as a
random walk that stays below (8 sqrt(2 K) + 8) 2^-24 of the sum of |products|.
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


def tol(k):
    return (8.0 * np.sqrt(2.0 * k) + 8.0) * 2.0 ** -24


def network(groups, cplx, seed, one_sided=()):
    """m, n, k, b label sizes -> network whose operands hold their labels in a
    seeded order; one_sided: sizes of labels summed in one operand only."""
    rng = np.random.default_rng(seed)
    size, ids = {}, []
    for g in list(groups) + [list(one_sided)]:
        ids.append(list(range(len(size), len(size) + len(g))))
        size.update(zip(ids[-1], g))
    m, n, k, b, s = ids
    la = [int(x) for x in rng.permutation(m + k + b + s[::2])]
    lb = [int(x) for x in rng.permutation(n + k + b + s[1::2])]
    lo = [int(x) for x in rng.permutation(b + m + n)]

    def t(ls):
        x = rng.standard_normal([size[l] for l in ls])
        return x + 1j * rng.standard_normal(x.shape) if cplx else x
    return inputs.Network([t(la), t(lb)], [la, lb], size, lo).as_stored(), k


def handle(torch, net):
    from paper_2002_01935_gb300 import binding
    dt = torch.complex64 if net.is_complex else torch.float32
    ts = [torch.from_numpy(np.array(x, order="C")).to(dt).cuda() for x in net.tensors]
    return binding.TensorNetwork(net.labels, net.dims, net.open, ts, complex_=net.is_complex)


def check(torch, net, kk, sliced=(), mode="fp32", **kw):
    ref = np.einsum(net.tensors[0], net.labels[0], net.tensors[1], net.labels[1], net.open, optimize=True)
    scale = np.einsum(np.abs(net.tensors[0]), net.labels[0], np.abs(net.tensors[1]), net.labels[1], net.open,
                      optimize=True)
    tnw = handle(torch, net)
    try:
        m, e = tnw.contract([(0, 1)], list(sliced), mode, **kw)
        got = m.cpu().numpy() * 2.0 ** int(e)
    finally:
        tnw.close()
    assert np.max(np.abs(got - ref) / np.maximum(scale, 1e-30)) <= tol(kk)


SHAPES = [  # m, n, k, b
    ([63], [65], [7], []), ([64], [64], [8], []), ([3, 5, 6], [7, 3, 5], [3, 6], [3]), ([1], [4100], [5], []),
    ([4], [1023], [9], []), ([4], [1025], [3], []), ([5], [255], [17], []), ([17], [300], [16], [2]),
    ([300], [17], [24], []), ([257], [32], [5, 3], []), ([33], [129], [1], []), ([70], [90], [3] * 7, []),
    ([7], [5], [3] * 8, []), ([1], [1], [11, 997], []), ([6], [10], [1025], []), ([129], [127], [33], [5]),
    ([3] * 6, [3] * 6, [3], []), ([1300], [1700], [9], []), ([2] * 7, [2] * 7, [2] * 3, [2]), ([2] * 3, [2] * 11, [2] * 2, []),
    ([2] * 11, [2] * 11, [2] * 4, []), ([2] * 9, [2] * 4, [2] * 7, []), ([2], [2] * 12, [2] * 5, [2])]


@pytest.mark.parametrize("cplx", [True, False])
@pytest.mark.parametrize("seed", range(2))
@pytest.mark.parametrize("shape", SHAPES)
def test_node_shapes(torch, shape, seed, cplx):
    net, _ = network(shape, cplx, 17 * seed + sum(map(len, shape)))
    check(torch, net, int(np.prod(shape[2])))


@pytest.mark.parametrize("cplx", [True, False])
def test_one_sided_sums_slices_and_modes(torch, cplx):
    shape = ([5, 9], [7, 11], [3, 4, 5], [3])
    net, k = network(shape, cplx, 3, one_sided=[3, 2])
    kk = 60 * 6
    for sliced, batch in ((), 0), (k[:1], 0), (k[1:], 4):
        for mode in ("fp32", "fp16_split"):  # sizes of this kind run in FP32 in every mode
            check(torch, net, kk, sliced, mode, slice_batch=batch)


@pytest.mark.parametrize("cplx", [True, False])
def test_tile_and_per_output_kernels_agree(torch, cplx, monkeypatch):
    net, _ = network(([6, 7], [5, 9], [3, 5, 7], [3]), cplx, 8)
    check(torch, net, 105)
    monkeypatch.setenv("TN_FORCE_GENERIC", "1")
    check(torch, net, 105)


@pytest.mark.parametrize("cplx", [True, False])
def test_reverse_sweep(torch, cplx):
    """Gradients of sum(w * (A B) C) by A, B and C: the adjoint nodes read
    conjugated operands on the tile kernel."""
    rng = np.random.default_rng(5)
    size = {0: 30, 1: 45, 2: 27, 3: 50}
    labels = [[0, 1], [2, 1], [3, 2]]

    def t(ls):
        x = rng.standard_normal([size[l] for l in ls])
        return x + 1j * rng.standard_normal(x.shape) if cplx else x
    net = inputs.Network([t(ls) for ls in labels], labels, size, [0, 3]).as_stored()
    w = t([0, 3])
    tnw = handle(torch, net)
    try:
        for sliced in ([], [1]):
            grads = tnw.grad([(0, 1), (2, 3)], sliced, "fp32", w)
            a, b, c = (np.conj(x) for x in net.tensors)
            ref = [np.einsum("ad,cb,dc->ab", w, b, c), np.einsum("ad,ab,dc->cb", w, a, c),
                   np.einsum("ad,ab,cb->dc", w, a, b)]
            mag = [np.einsum("ad,cb,dc->ab", abs(w), abs(b), abs(c)), np.einsum("ad,ab,dc->cb", abs(w), abs(a), abs(c)),
                   np.einsum("ad,ab,cb->dc", abs(w), abs(a), abs(b))]
            for g, r, s in zip(grads, ref, mag):  # two contractions one after the other
                assert np.max(np.abs(g.cpu().numpy() - r) / s) <= 2 * tol(45)
    finally:
        tnw.close()


def test_copies(torch):
    """contract_instances: every copy's K parts in its own part buffer."""
    rng = np.random.default_rng(9)
    a = rng.standard_normal((3, 3 ** 7, 5)).astype(np.float32)
    b = rng.standard_normal((3 ** 7, 5)).astype(np.float32)
    from paper_2002_01935_gb300 import binding
    dims = {l: 3 for l in range(7)} | {7: 5}
    tnw = binding.TensorNetwork([list(range(8)), list(range(8))], dims, [],
                                [torch.from_numpy(a.reshape(-1)).cuda(), torch.from_numpy(b).cuda()], complex_=False)
    m, e = tnw.contract_instances([(0, 1)], "fp32", 3, [3 ** 7 * 5, 0])
    got = m[:, 0].cpu().numpy() * 2.0 ** e.cpu().numpy()
    ref = np.einsum("ikj,kj->i", a.astype(np.float64), b)
    assert np.max(np.abs(got - ref) / np.einsum("ikj,kj->i", np.abs(a), np.abs(b))) <= tol(3 ** 7 * 5)
    tnw.close()
