"""A batch on a device whose memory is nearly taken: it runs with fewer
concurrent groups (each has a packing buffer of its own) rather than not at
all, and gives the same bits."""
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


def test_little_memory(torch):
    """Eight networks of 64 MiB workspace and 64 MiB packing buffer each, with
    960 MiB free: one buffer for all fits, one for each does not."""
    from paper_2002_01935_gb300 import binding
    m, n, k = 2 ** 12, 2 ** 12, 2 ** 11
    g = torch.Generator(device="cuda").manual_seed(1)
    ts = [torch.randn(*s, device="cuda", generator=g) for s in ((m, k), (k, n), (m, n))]
    pairs = [(0, 1), (3, 2)]
    nets = [binding.TensorNetwork([[0, 1], [1, 2], [0, 2]], {0: m, 1: k, 2: n}, [], ts, complex_=False)
            for _ in range(8)]

    def run():
        b = binding.Batch(nets, [pairs] * 8, "fp16_split")
        try:
            mant, e, _ = b.contract()
            torch.cuda.synchronize()
            return mant.cpu(), e.cpu()
        finally:
            b.close()

    want = run()
    torch.cuda.empty_cache()
    fill = []
    try:
        while True:  # in blocks: no single range need be free
            free, _ = torch.cuda.mem_get_info()
            over = free - (960 << 20)
            if over < (4 << 20):
                break
            fill.append(torch.empty(min(over // (2 << 20) * (2 << 20), 8 << 30), dtype=torch.uint8, device="cuda"))
        got = run()
    finally:
        fill.clear()
        torch.cuda.empty_cache()
        for h in nets:
            h.close()
    assert torch.equal(want[0], got[0]) and torch.equal(want[1], got[1]) and bool((want[0][:, 0] != 0).all())
