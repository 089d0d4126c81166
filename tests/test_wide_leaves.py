"""Slices of leaves that spread over 2^31 entries or more.

A sliced label leaves the node's label lists, but the remaining ones keep the
strides of the whole leaf.  The planner then takes kernels with 64-bit operand
offsets (tile configuration + 16; one thread per output for other sizes than
powers of two), which is checked on host plans, and the results on the GPU
against torch in 64 bits on a 16 GiB leaf.

Tolerance: a sum of K products in FP32, (8 sqrt(2 K) + 8) 2^-24 of the sum of
|products|; on the tensor cores 1e-5 of it.
"""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2002_01935_gb300 import binding  # noqa: E402

# labels m, n, k, x (summed in the large leaf only), s (sliced): the large
# leaf's label order, the other's, their sizes, and the configuration expected
CASES = {
    "tile": ("msk", "kn", dict(m=256, s=2 ** 16, k=256, n=256), (1, 1)),
    "tile_k_outside": ("ksm", "nk", dict(m=256, s=2 ** 16, k=256, n=256), (1, 1)),
    "tile_slices_fastest": ("mks", "kn", dict(m=256, s=2 ** 18, k=64, n=512), (1, 1)),
    "rows_4": ("nsk", "mk", dict(n=2 ** 14, s=2 ** 11, k=128, m=4), (1, 3)),
    "rows_16": ("nsk", "mk", dict(n=2 ** 12, s=2 ** 13, k=128, m=16), (1, 2)),
    "columns_16": ("nxsk", "mk", dict(n=16, x=64, s=2 ** 18, k=16, m=512), (1, 4)),
    "inner_product": ("ks", "k", dict(k=1024, s=2 ** 22), (1, 5)),
    "inner_products": ("msk", "kn", dict(m=8, s=2 ** 19, k=1024, n=4), (1, 5)),
    "inner_products_outside": ("ksm", "nk", dict(m=8, s=2 ** 17, k=4096, n=2), (1, 5)),
    "any_size": ("msk", "kn", dict(m=27, s=1900001, k=81, n=25), (0, None)),
}


def network(case, tensors=None):
    big, other, dims, _ = CASES[case]
    ids = {c: i for i, c in enumerate("mnkxs")}
    out = [c for c in "mn" if c in dims]
    return binding.TensorNetwork([[ids[c] for c in big], [ids[c] for c in other]],
                                 {ids[c]: n for c, n in dims.items()}, [ids[c] for c in out], tensors,
                                 complex_=False), [ids["s"]], out


@pytest.mark.parametrize("case", list(CASES))
def test_plan(case):
    h, sliced, _ = network(case)
    try:
        step, = h.plan_steps([(0, 1)], sliced, "fp32")
    finally:
        h.close()
    kind, cfg = CASES[case][3]
    assert step["kind"] == kind
    assert step["cfg"] == (cfg + 16 if kind else 0)


@pytest.mark.parametrize("order", ["mks", "msk", "smk"])
def test_just_below_the_limit(order):
    """2^31 entries in all: every offset is below."""
    size = dict(m=2 ** 10, k=2 ** 10, s=2 ** 11)  # nodes above the waves' sizes
    ids = {c: i for i, c in enumerate("mnks")}
    h = binding.TensorNetwork([[ids[c] for c in order], [ids["k"], ids["n"]]],
                              {ids["m"]: size["m"], ids["k"]: size["k"], ids["s"]: size["s"], ids["n"]: 64},
                              [ids["m"], ids["n"]], None, complex_=False)
    try:
        step, = h.plan_steps([(0, 1)], [ids["s"]], "fp32")
    finally:
        h.close()
    assert step["kind"] == 1 and step["cfg"] < 16


@pytest.fixture(scope="module")
def large():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2002_01935_gb300 import build
    build.build()
    t = torch.empty(2 ** 32, device="cuda").uniform_(-1.0, 1.0, generator=torch.Generator(device="cuda").manual_seed(3))
    yield t
    del t
    torch.cuda.empty_cache()


@pytest.mark.gpu
@pytest.mark.parametrize("case,mode", [(c, "fp32") for c in CASES] + [("tile", "fp16_split")])
def test_result(large, case, mode):
    big, other, dims, _ = CASES[case]
    a = large[:math.prod(dims[c] for c in big)].view([dims[c] for c in big])
    g = torch.Generator(device="cuda").manual_seed(4)
    b = torch.empty([dims[c] for c in other], device="cuda").uniform_(-1.0, 1.0, generator=g)
    h, sliced, out = network(case, [a, b])
    try:
        for begin in (0, dims["s"] - 3):
            m, e = h.contract([(0, 1)], sliced, mode, slice_begin=begin, slice_count=3, slice_batch=2)
            got = (m * 2.0 ** e.double()).cpu().numpy()
            part = a.narrow(big.index("s"), begin, 3).double()
            eq = f"{big},{other}->{''.join(out)}"
            ref = torch.einsum(eq, part, b.double()).cpu().numpy()
            scale = torch.einsum(eq, part.abs(), b.double().abs()).cpu().numpy()
            k = 3 * dims["k"] * dims.get("x", 1)
            tol = 1e-5 if mode != "fp32" else (8.0 * np.sqrt(2.0 * k) + 8.0) * 2.0 ** -24
            assert np.all(np.abs(got - ref) <= tol * scale)
    finally:
        h.close()
