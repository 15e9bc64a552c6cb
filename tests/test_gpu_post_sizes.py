"""Sizes at which the post-steps can go wrong.  The removed diagonal: one or
several blocks of a cluster per 32 positions, few inner indices, products
beyond FP32's range that cancel; relative to 64 bits the sums are exact to
2^-40 or better and each is rounded once to FP32, 2^-24, as is the sum of those
that share a bucket: tolerance 2^-22.  The listed estimates: rows of one
column to more than 15 segments of 32 columns, no hits, every entry a hit, and
a buffer that ends inside a row; positions and estimates are equal to the dense
decode's."""
import numpy as np
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


@pytest.mark.parametrize("m,n2", [(1, 1), (31, 255), (33, 256), (64, 511), (200, 512), (700, 1024), (2500, 4100),
                                  (5000, 300)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16, torch.float64])
def test_removed_diagonal(cms, m, n2, dtype):
    g = torch.Generator().manual_seed(m + n2)
    A = torch.randn(n2, m, generator=g, dtype=torch.float64).to(dtype)
    B = torch.randn(n2, m + 3, generator=g, dtype=torch.float64).to(dtype)
    h = cms.make_hashes(m, m + 3, 4096, 3)
    tab = O.make_tables(m, m + 3, 4096, 3)
    c = torch.zeros(3, 4096, device="cuda")
    cms.remove_diagonal(A.cuda().T, B.cuda(), h, c)
    diag = (A.double() * B.double()[:, :m]).sum(0).numpy()
    ref = O.remove_diagonal(np.zeros((3, 4096)), diag, tab)
    assert max(O.rel_l2(c[t].cpu().numpy(), ref[t]) for t in range(3)) < 2.0 ** -22
    h.free()


def test_removed_diagonal_beyond_fp32_on_the_way(cms):
    m, n2 = 40, 100
    A, B = torch.zeros(n2, m), torch.zeros(n2, m)
    A[1:32], B[1:32] = 2.0, 3.0
    A[0], B[0] = 2.0 ** 90, 2.0 ** 60
    A[32], B[32] = 2.0 ** 90, -2.0 ** 60
    h = cms.make_hashes(4, m, 1024, 2)
    c = torch.zeros(2, 1024, device="cuda")
    cms.remove_diagonal(A.cuda().T, B.cuda(), h, c)
    ref = O.remove_diagonal(np.zeros((2, 1024)), np.full(m, 186.0), O.make_tables(4, m, 1024, 2))
    np.testing.assert_array_equal(c.cpu().numpy(), ref.astype(np.float32))
    h.free()


@pytest.mark.parametrize("n1,n3", [(1, 1), (3, 31), (40, 33), (17, 480), (9, 481), (300, 257), (5, 2000)])
@pytest.mark.parametrize("quantile", [0.0, 0.5, 0.97, 1.0])
def test_listed_estimates(cms, n1, n3, quantile):
    n = max(n1, n3)
    g = torch.Generator().manual_seed(n1 * n3)
    h = cms.make_hashes(n1 + n3, n, 5000, 3)
    c = torch.randn(3, 5000, generator=g).cuda()
    dense = cms.decode_dense(c, h, n1, n3).cpu().numpy()
    tau = float(np.quantile(np.abs(dense), quantile)) if quantile else 0.0
    want = np.argwhere(np.abs(dense) > np.float32(tau))
    for capacity in (n1 * n3, max(1, len(want) // 2)):
        ij, val, count = cms.decode_threshold(c, h, n1, n3, tau, skip_diagonal=False, capacity=capacity)
        assert count == len(want)
        keep = want[:capacity]
        np.testing.assert_array_equal(ij.cpu().numpy()[:len(keep)], keep)
        np.testing.assert_array_equal(val.cpu().numpy()[:len(keep)], dense[keep[:, 0], keep[:, 1]])
    h.free()
