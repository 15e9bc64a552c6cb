"""The removed diagonal at the lower end of FP32's range, where the products of
its entries underflow (the sums do not: additions into a bucket flush subnormals),
and of a column without any.

Tolerance: relative L2 1e-7, the rounding of a bucket to FP32 (6e-8 at most)."""
import pytest
import torch

from oracle import cms_oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cms():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1108_1320_gb300 import build as b
    b.build()
    import paper_1108_1320_gb300 as m
    m.lib()
    return m


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("e", [-40, -58, -66, -68])
def test_diagonal_of_small_values(cms, dtype, e):
    n, m, b = 200, 4096, 1 << 16
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    x = ((1 + torch.rand((m, n), generator=g, device="cuda", dtype=torch.float64)) * 2.0 ** e).to(dtype)
    x[:, 7] = 0
    h = cms.make_hashes(5, n, b, 1)
    c = cms.remove_diagonal(x.T, x, h, torch.zeros((1, b), device="cuda"))
    cms.check_async()
    tab = O.make_tables(5, n, b, 1)
    want = torch.zeros(b, dtype=torch.float64)
    z = torch.from_numpy((tab.h1[0] + tab.h2[0]).astype("int64") % b)
    s = torch.from_numpy((tab.s1[0] * tab.s2[0]).astype("float64"))
    want.index_add_(0, z, -(x.double() ** 2).sum(0).cpu() * s)
    assert O.rel_l2(c[0].cpu().numpy(), want.numpy()) < 1e-7
    h.free()
