"""Calls on another stream than the current one: their scratch and outputs are
not given to the current stream's work while they run, and the numbers that they
return have arrived."""
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

BUSY = 200_000_000       # cycles: about 0.1 s before the call's kernels start


@pytest.fixture(scope="module")
def cms():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1108_1320_gb300 import build as b
    b.build()
    import paper_1108_1320_gb300 as m
    m.lib()
    return m


def operands(m, n):
    x = torch.from_numpy(W.gaussian(m, n, 3)).to("cuda", torch.float32)
    x[:, 5] = x[:, 9]
    torch.cuda.synchronize()
    return x


@pytest.mark.parametrize("n2", [40, 700])      # transform route, direct route
def test_scratch_is_not_reused_while_the_call_runs(cms, n2):
    x = operands(n2, 900)
    h = cms.make_hashes(1, 900, 14400, 3)
    want = cms.sketch_product(x.T, x, h)
    size = cms.workspace_size(h, 900, n2, 900)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        torch.cuda._sleep(BUSY)
    got = cms.sketch_product(x.T, x, h, stream=s)
    other = [torch.full((size,), 0x7F, dtype=torch.uint8, device="cuda") for _ in range(4)]   # of the same size
    torch.cuda.synchronize()
    assert torch.equal(got, want) and all(int(o[-1]) == 0x7F and int(o[0]) == 0x7F for o in other)
    h.free()


def test_counts_have_arrived(cms):
    n, m, b, d = 300, 2000, 1 << 16, 5
    x = operands(m, n)
    h = cms.make_hashes(1, n, b, d)
    s = torch.cuda.Stream()
    c = cms.remove_diagonal(x.T, x, h, cms.sketch_product(x.T, x, h))
    ij, val, count = cms.decode_threshold(c, h, n, n, 0.7 * m)
    at, found = cms.find_significant(x.T, x, h, 0.7 * m, 3)
    est, bound = cms.frobenius_estimate(x.T, x, 3, 5)
    torch.cuda.synchronize()
    assert count == 2 and found >= 2
    for f in (lambda: cms.decode_threshold(c, h, n, n, 0.7 * m, stream=s),
              lambda: cms.find_significant(x.T, x, h, 0.7 * m, 3, stream=s),
              lambda: cms.frobenius_estimate(x.T, x, 3, 5, stream=s)):
        with torch.cuda.stream(s):
            torch.cuda._sleep(BUSY)
        out = f()
        if len(out) == 3:
            assert out[2] == count and torch.equal(out[0], ij) and torch.equal(out[1], val)
        elif torch.is_tensor(out[1]) or isinstance(out[1], int):
            assert out[1] == found and torch.equal(out[0], at)
        else:
            assert out[1] == bound and torch.equal(out[0], est)
    h.free()
