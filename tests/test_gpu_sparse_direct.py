"""Sparse outer products sketched term by term: long against short, heavy ones
shared by all blocks, beside light ones, against the FP64 oracle.

Tolerance: relative L2 1e-6 per repetition.  Terms are rounded once, to 2^-62
of the sum of all of them (or kept in FP64), and the buckets once to FP32: 6e-8,
with room for the FFT route's share (2.6e-7)."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import cms_oracle as O

pytestmark = pytest.mark.gpu

TOL = 1e-6


@pytest.fixture(scope="module")
def cms():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1108_1320_gb300 import build as b
    b.build()
    import paper_1108_1320_gb300 as m
    m.lib()
    return m


def sparse(na, nb, n, seed, dtype=np.float32):
    """CSC A and CSR B with na[k], nb[k] nonzeros of inner index k."""
    rng = W.rng(seed)

    def side(cnt):
        ptr = np.concatenate([[0], np.cumsum(cnt)]).astype(np.int64)
        idx = np.concatenate([np.sort(rng.choice(n, c, replace=False)) for c in cnt])
        return ptr, idx.astype(np.int32), rng.standard_normal(ptr[-1]).astype(dtype)
    return side(na) + side(nb)


def definition(data, tab, d, b):
    """The sketch in FP64, term by term."""
    c = np.zeros((d, b))
    ap, ai, av, bp, bi, bv = data
    for k in range(len(ap) - 1):
        i, x = ai[ap[k]:ap[k + 1]], av[ap[k]:ap[k + 1]].astype(np.float64)
        j, y = bi[bp[k]:bp[k + 1]], bv[bp[k]:bp[k + 1]].astype(np.float64)
        for t in range(d):
            z = (tab.h1[t][i][:, None] + tab.h2[t][j][None, :]) % b
            np.add.at(c[t], z, (tab.s1[t][i] * x)[:, None] * (tab.s2[t][j] * y)[None, :])
    return c


# terms: at the line between light and heavy (16384), pieces of every shape, more
# than 256 heavy inner indices
LISTS = {
    "thin columns": ([5000, 511, 512, 1, 1024], [1, 1, 1, 3000, 2]),
    "thin rows": ([1, 2, 7, 8, 9], [5000, 511, 505, 504, 600]),
    "heavy": ([128, 129, 300, 4000, 33, 1], [128, 128, 211, 5, 501, 6000]),
    "heavy and light": ([200, 3, 0, 40, 6, 150, 20] * 2, [300, 9, 5, 0, 6000, 150, 30] * 2),
    "many heavy": ([130] * 300, [130] * 300),
}


@pytest.mark.parametrize("name", LISTS)
@pytest.mark.parametrize("d,pairs", [(2, None), (9, None), (2, 1 << 20)])
def test_outer_products_of_every_shape(cms, name, d, pairs):
    na, nb = LISTS[name]
    if name == "many heavy" and d > 2:
        pytest.skip("covered with two repetitions")
    n, b = 8192, 1 << 16 if pairs else 1 << 18
    data = sparse(na, nb, n, 7)
    assert max(x * y for x, y in zip(na, nb)) <= (pairs or b * 18 // 50)       # none on the FFT route
    h = cms.make_hashes(5, n, b, d)
    args = [torch.from_numpy(x).to("cuda") for x in data]
    c = cms.sketch_product_csr(*args, n, n, h, direct_max_pairs=pairs)
    again = cms.sketch_product_csr(*args, n, n, h, direct_max_pairs=pairs)
    cms.check_async()
    ref = definition(data, O.make_tables(5, n, b, d), d, b)
    assert max(O.rel_l2(c[t].cpu().numpy(), ref[t]) for t in range(d)) < TOL
    if pairs is None:
        assert torch.equal(c, again)
    h.free()


def milliseconds(cms, data, n, h, pairs):
    args = [torch.from_numpy(x).to("cuda") for x in data]
    ws = cms.alloc_workspace(cms.sparse_workspace_size(h, n, len(data[0]) - 1, n))
    out = []
    for q in range(8):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        e[0].record()
        cms.sketch_product_csr(*args, n, n, h, ws=ws, direct_max_pairs=pairs)
        e[1].record()
        e[1].synchronize()
        out.append(e[0].elapsed_time(e[1]))
    return min(out[2:])


def test_time_follows_the_terms_not_their_shape(cms):
    # 100000 terms: one block per inner index took 15 times as long for a column
    # against one element, and 16 for one product as for 16 of the same terms
    n, b, d = 1 << 17, 1 << 20, 3
    h = cms.make_hashes(5, n, b, d)
    even = milliseconds(cms, sparse([79] * 16, [79] * 16, n, 1), n, h, -1)
    for na, nb in (([316], [316]), ([100000], [1]), ([1], [100000])):
        assert milliseconds(cms, sparse(na, nb, n, 2), n, h, -1) < 4 * even
    h.free()


@pytest.mark.parametrize("count", [1, 3, 13, 250])
def test_fft_route_with_several_tasks_per_block(cms, monkeypatch, count):
    # every inner index on the FFT route: more (repetition, row, chunk) tasks than
    # blocks, most chunks of a short list empty; both scatter forms, the same bits
    n, b, d = 900, 16384, 3
    rng = W.rng(count)
    data = sparse(rng.integers(1, 60, count), rng.integers(1, 60, count), n, 9)
    h = cms.make_hashes(3, n, b, d)
    args = [torch.from_numpy(x).to("cuda") for x in data]
    out = []
    for env in (None, None, "1"):
        if env:
            monkeypatch.setenv("CMS_SPARSE_INPLACE_Y", env)
        cms.profile_enable(True)
        out.append(cms.sketch_product_csr(*args, n, n, h, direct_max_pairs=0))
        torch.cuda.synchronize()
        assert "k_sketch_sparse" in cms.profile_summary()
        cms.profile_enable(False)
    monkeypatch.delenv("CMS_SPARSE_INPLACE_Y")
    cms.check_async()
    assert torch.equal(out[0], out[1]) and torch.equal(out[0], out[2])
    ref = definition(data, O.make_tables(3, n, b, d), d, b)
    assert max(O.rel_l2(out[0][t].cpu().numpy(), ref[t]) for t in range(d)) < 1e-5
    h.free()


def test_short_lists_do_not_crowd_into_a_few_blocks(cms):
    # one inner index on the FFT route fills one chunk of each row; with the
    # blocks' turns over the chunks first, every fourth block had all of them
    n, b, d = 1 << 20, 1 << 20, 7
    h = cms.make_hashes(5, n, b, d)
    light = milliseconds(cms, sparse([1], [1], n, 3), n, h, 0)
    heavy = milliseconds(cms, sparse([2000], [2000], n, 3), n, h, 0)
    assert heavy < 1.95 * light      # 3.60 of 1.70 ms with the chunks first, 2.81 of 1.59 with the rows first
    h.free()
