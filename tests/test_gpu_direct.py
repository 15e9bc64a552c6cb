"""The direct route (tensor-core tiles of AB added to the buckets) against the
FP64 oracle, at the sizes where it can go wrong: edges of the 128 x 128 tiles
and of the 32, 64 and 128 inner indices of a stage and a superblock, every
storage type, aliased and separate operands, unaligned rows, split and folded
inner dimensions, values far apart in magnitude, infinities and NaN.

Tolerance: relative L2 1e-6 per repetition.  The products of a drain (64 with
FP16 terms, 128 with BF16) are summed with a relative error of a few 2^-24,
at most 64 drains follow each other in one FP32 sum (1/sqrt(3) 2^-24 sqrt(32)
of it in the mean) and the rest is added exactly: about 2.5e-7, with room for
a factor of four."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import cms_oracle as O

pytestmark = pytest.mark.gpu

TOL = 1e-6
DT = {"f32": torch.float32, "bf16": torch.bfloat16, "f64": torch.float64}


@pytest.fixture(scope="module")
def cms():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1108_1320_gb300 import build as b
    b.build()
    import paper_1108_1320_gb300 as m
    m.lib()
    return m


def dev():
    return torch.device("cuda", torch.cuda.current_device())


def operands(n1, n2, n3, dts, alias, pad, seed, scale=None):
    """Device A, B and the FP64 values they hold."""
    def stored(x):
        return W.bf16_round(x.astype(np.float32))[0] if dts == "bf16" else x.astype(np.float32 if dts == "f32" else np.float64)

    def put(x):
        buf = torch.zeros((x.shape[0], x.shape[1] + pad), dtype=DT[dts], device=dev())
        buf[:, :x.shape[1]] = torch.from_numpy(x).to(dev(), DT[dts])
        return buf[:, :x.shape[1]]

    At = W.gaussian(n2, n1, seed)
    if scale is not None:
        At = At * scale(n2, n1)
    At = stored(At)
    at = put(At)
    if alias:
        return at.T, at, At.astype(np.float64).T, At.astype(np.float64)
    B = stored(W.gaussian(n2, n3, seed + 1))
    return at.T, put(B), At.astype(np.float64).T, B.astype(np.float64)


def run(cms, A, B, h, **kw):
    cms.profile_enable(True)
    c = cms.sketch_product(A, B, h, **kw)
    torch.cuda.synchronize()
    kernels = cms.profile_summary()
    cms.profile_enable(False)
    cms.check_async()
    return c, kernels


def worst(c, ref):
    return max(O.rel_l2(c[t].cpu().numpy(), ref[t]) for t in range(ref.shape[0]))


@pytest.mark.parametrize("n1,n2,n3,b,d,dts,alias,pad", [
    (128, 128, 128, 1 << 17, 3, "f32", True, 0),       # one tile, one superblock
    (127, 127, 129, 64800, 3, "f32", False, 1),      # one short of and one past a tile
    (129, 129, 127, 1 << 15, 3, "bf16", False, 1),
    (257, 95, 257, 1 << 17, 2, "f32", True, 3),       # 3 stages of 32: an odd number in the last drain
    (300, 65, 300, 1 << 18, 2, "bf16", True, 0),      # one inner index in the second stage of 64
    (200, 385, 333, 20000, 2, "f64", False, 0),     # FP64 storage
    (640, 1000, 640, 10240, 3, "f32", True, 0),     # upper triangle of 5 x 5 tiles, split inner dimension
    (512, 9000, 384, 8192, 1, "bf16", False, 0),
])
def test_direct_route_matches_oracle(cms, n1, n2, n3, b, d, dts, alias, pad):
    n = max(n1, n3)
    seed = n1 + n2
    A, B, Ad, Bd = operands(n1, n2, n3, dts, alias, pad, seed)
    h = cms.make_hashes(seed, n, b, d)
    c, kernels = run(cms, A, B, h)
    assert "k_direct_tile" in kernels
    ref = O.sketch_definition(Ad, Bd, O.make_tables(seed, n, b, d))
    assert worst(c, ref) < TOL
    c2, _ = run(cms, A, B, h)
    assert torch.equal(c, c2)                       # the order of the integer sums does not matter
    h.free()


@pytest.mark.parametrize("n,m,dts", [(1920, 4500, "f32"), (1920, 8500, "bf16")])
def test_direct_route_folds_long_sums(cms, n, m, dts):
    # enough tiles that the inner dimension is not split, and more than 64
    # drains: the register sums are folded
    A, B, Ad, Bd = operands(n, m, n, dts, True, 0, 7)
    h = cms.make_hashes(8, n, 16 * n, 1)
    c, kernels = run(cms, A, B, h)
    assert "k_direct_tile" in kernels
    ref = O.sketch_definition(Ad, Bd, O.make_tables(8, n, 16 * n, 1))
    assert worst(c, ref) < TOL
    h.free()


@pytest.mark.parametrize("dts", ["f32", "bf16"])
@pytest.mark.parametrize("case", ["rows", "tiny", "huge", "outlier"])
def test_direct_route_over_magnitudes(cms, dts, case):
    # inner indices 2^-40 .. 2^40 apart, values near either end of FP32's
    # range, and one entry that dwarfs the others
    def scale(n2, n1):
        if case == "rows":
            return np.exp2(np.linspace(-40, 40, n2))[:, None]
        s = np.ones((n2, n1))
        if case == "outlier":
            s[n2 // 2, n1 // 3] = 1e6
            return s
        return s * (1e-17 if case == "tiny" else 1e16)
    A, B, Ad, Bd = operands(200, 300, 200, dts, True, 0, 5, scale)
    h = cms.make_hashes(6, 200, 1 << 16, 2)
    c, kernels = run(cms, A, B, h)
    assert "k_direct_tile" in kernels
    assert worst(c, O.sketch_definition(Ad, Bd, O.make_tables(6, 200, 1 << 16, 2))) < TOL
    h.free()


@pytest.mark.parametrize("n2", [40, 200])            # transform route, direct route
@pytest.mark.parametrize("value", [float("inf"), float("nan")])
def test_non_finite_operands_give_nan_on_both_routes(cms, n2, value):
    A, B, _, _ = operands(200, n2, 200, "f32", False, 0, 9)
    A[3, n2 // 2] = value
    h = cms.make_hashes(6, 200, 1 << 16, 2)
    c, kernels = run(cms, A, B, h)
    assert ("k_direct_tile" in kernels) == (n2 >= 64)
    assert torch.isnan(c).all()
    A.zero_()
    c, _ = run(cms, A, B, h)
    assert torch.count_nonzero(c).item() == 0
    h.free()


@pytest.mark.parametrize("n1,n2,n3,b,d,dts,alias", [
    (1100, 200, 1000, 20000, 3, "f32", False), (1025, 700, 1025, 27000, 3, "f32", True),
    (1001, 64, 1025, 28800, 4, "f32", False), (1500, 130, 1500, 65536, 5, "bf16", True),
    (1153, 300, 1153, 5000, 3, "bf16", True), (1024, 100, 1153, 40000, 7, "f64", False)])
def test_stored_entries_with_a_window_of_the_buckets(cms, n1, n2, n3, b, d, dts, alias):
    # all buckets in shared memory, or the first 28672 and the rest in L2
    A, B, Ad, Bd = operands(n1, n2, n3, dts, alias, 0, n1 + b)
    h = cms.make_hashes(b, max(n1, n3), b, d)
    c, kernels = run(cms, A, B, h)
    again, _ = run(cms, A, B, h)
    assert "k_direct_window" in kernels
    assert worst(c, O.sketch_definition(Ad, Bd, O.make_tables(b, max(n1, n3), b, d))) < TOL
    assert torch.equal(c, again)
    h.free()


def test_workspace_of_the_transform_route_still_serves(cms):
    # a workspace smaller than the direct route's layout: the transform route
    A, B, Ad, Bd = operands(400, 4000, 400, "f32", True, 0, 11)
    h = cms.make_hashes(12, 400, 4096, 1)
    full = cms.workspace_size(h, 400, 4000, 400)
    c, kernels = run(cms, A, B, h, ws=cms.alloc_workspace(full))
    assert "k_direct_tile" in kernels
    c2, kernels = run(cms, A, B, h, ws=cms.alloc_workspace(6 << 20))
    assert (6 << 20) < full and "k_direct_tile" not in kernels
    ref = O.sketch_definition(Ad, Bd, O.make_tables(12, 400, 4096, 1))
    assert worst(c, ref) < TOL and worst(c2, ref) < 1e-5
    h.free()


def test_batch_of_both_routes(cms):
    # instances on the direct route beside instances on the transform route
    # (few inner indices), twice: the sums are left zero for the next run
    items, refs = [], []
    for q, (n, m, dts) in enumerate([(300, 700, "f32"), (600, 40, "f32"), (500, 900, "bf16"), (450, 30, "bf16")]):
        A, B, Ad, Bd = operands(n, m, n, dts, True, 0, 20 + q)
        items.append((A, B, cms.make_hashes(30 + q, n, 16 * n, 2)))
        refs.append(O.sketch_definition(Ad, Bd, O.make_tables(30 + q, n, 16 * n, 2)))
    batch = cms.Batch(items)
    for _ in range(2):
        cms.profile_enable(True)
        batch.run()
        torch.cuda.synchronize()
        kernels = cms.profile_summary()
        cms.profile_enable(False)
        cms.check_async()
        assert kernels["k_direct_tile_batched"]["launches"] == 1 and kernels["k_sketch_batched"]["launches"] == 1
        for c, ref in zip(batch.c, refs):
            assert worst(c, ref) < 1e-5
            c.zero_()
    batch.free()


def sparse_pair(rng, n1, n2, n3, na, nb):
    """CSC A (n1 x n2) and CSR B (n2 x n3) with na[k], nb[k] nonzeros."""
    def side(n, cnt):
        ptr = np.concatenate([[0], np.cumsum(cnt)]).astype(np.int64)
        idx = np.concatenate([np.sort(rng.choice(n, c, replace=False)) for c in cnt] + [np.zeros(0, np.int64)])
        return ptr, idx.astype(np.int32), rng.standard_normal(ptr[-1]).astype(np.float32)
    return side(n1, na) + side(n3, nb)


@pytest.mark.parametrize("d", [2, 9])
def test_sparse_default_split(cms, d):
    # outer products of every kind: empty, one term, more rows and columns
    # than a block holds at a time (32 x 128), and some past the split
    # (b log2(b) / 50 = 2129 terms), which take the FFT route; the same bits twice
    rng = W.rng(3)
    n, b = 700, 8192
    na = np.array([0, 1, 33, 70, 5, 40, 0, 200, 31, 64] * 4)
    nb = np.array([4, 1, 7, 20, 129, 300, 0, 9, 60, 150] * 4)
    data = sparse_pair(rng, n, na.size, n, na, nb)
    import scipy.sparse as sp
    A = sp.csc_matrix((data[2], data[1], data[0]), shape=(n, na.size)).toarray().astype(np.float64)
    B = sp.csr_matrix((data[5], data[4], data[3]), shape=(na.size, n)).toarray().astype(np.float64)
    assert ((na * nb > 0) & (na * nb <= 2129)).any() and (na * nb > 2129).any()
    h = cms.make_hashes(5, n, b, d)
    args = [torch.from_numpy(x).to(dev()) for x in data]
    c = cms.sketch_product_csr(*args, n, n, h)
    c2 = cms.sketch_product_csr(*args, n, n, h)
    cms.check_async()
    assert torch.equal(c, c2)
    assert worst(c, O.sketch_definition(A, B, O.make_tables(5, n, b, d))) < TOL
    # indices outside the matrix are skipped, an infinity makes c NaN
    small = [torch.from_numpy(x).to(dev()) for x in sparse_pair(rng, n, 6, n, np.full(6, 9), np.full(6, 11))]
    want = cms.sketch_product_csr(*small, n, n, h)
    drop = small[1].clone()
    drop[4] = n + 5
    zero = small[2].clone()
    zero[4] = 0
    got = cms.sketch_product_csr(small[0], drop, small[2], *small[3:], n, n, h)
    ref = cms.sketch_product_csr(small[0], small[1], zero, *small[3:], n, n, h)
    assert worst(got, ref.cpu().numpy()) < TOL and not torch.equal(got, want)
    zero[7] = float("inf")
    assert torch.isnan(cms.sketch_product_csr(small[0], small[1], zero, *small[3:], n, n, h)).all()
    h.free()


@pytest.mark.parametrize("n1,n2,n3,b,d", [(64, 300, 64, 12, 2), (200, 130, 150, 1, 3), (140, 64, 140, 96, 7)])
def test_direct_route_short_sketches(cms, n1, n2, n3, b, d):
    # few buckets: blocks add to copies of the sums (and the finish adds
    # those up); the direct route where the rule picks it
    A, B, Ad, Bd = operands(n1, n2, n3, "f32", False, 0, n1)
    h = cms.make_hashes(n1, max(n1, n3), b, d)
    c, _ = run(cms, A, B, h)
    ref = O.sketch_definition(Ad, Bd, O.make_tables(n1, max(n1, n3), b, d))
    assert worst(c, ref) < 1e-5
    h.free()


@pytest.mark.parametrize("n1,n2,n3,rho,alias", [(300, 80, 280, 1, False), (257, 200, 257, 3, True), (90, 64, 1, 2, False)])
def test_find_significant_on_the_direct_route(cms, n1, n2, n3, rho, alias):
    # planted entries far above the noise: exactly these positions, from the
    # masked sums of one pass over the entries of AB
    b, d = 16384, 5
    g = W.rng(50 + n1)
    At = (0.01 * g.standard_normal((n2, n1))).astype(np.float32)
    B = At if alias else (0.01 * g.standard_normal((n2, n3))).astype(np.float32)
    big = [(3, 5), (min(117, n1 - 1), 230), (n1 - 1, 0), (21, 21)]
    for q, (i, j) in enumerate(big):
        At[q, i] += 10.0
        B[q, j % n3] += 10.0 + q
    AB = At.astype(np.float64).T @ B.astype(np.float64)
    want = sorted((int(i), int(j)) for i, j in zip(*np.nonzero(np.abs(AB) > 50.0)))
    h = cms.make_hashes(151, max(n1, n3), b, d)
    at = torch.from_numpy(At).to(dev())
    bt = at if alias else torch.from_numpy(B).to(dev())
    cms.profile_enable(True)
    got, count = cms.find_significant(at.T, bt, h, 50.0, rho)
    kernels = cms.profile_summary()
    cms.profile_enable(False)
    cms.check_async()
    assert "k_direct_sig_decode" in kernels and "k_mask_copy" not in kernels
    assert [tuple(p) for p in got.cpu().numpy().tolist()] == want and count == len(want)
    h.free()


@pytest.mark.parametrize("n1,n2,n3,b,d,dts,alias,pad", [
    (3000, 500, 2500, 600, 3, "f32", False, 1),    # R = 1, a last superblock of 116 inner indices
    (5000, 300, 5000, 1500, 2, "bf16", True, 0),   # R = 2, C = 750: the last tile is not full
    (8000, 513, 8000, 1944, 3, "f32", True, 0),    # R = 2, C = 972: the last tile is not full; one inner index in the last stage
    (6000, 400, 6000, 2187, 3, "f64", True, 3),    # R = 3: rows without a bucket in every tile
])
def test_pre_sketched_operands_match_oracle(cms, n1, n2, n3, b, d, dts, alias, pad):
    n = max(n1, n3)
    A, B, Ad, Bd = operands(n1, n2, n3, dts, alias, pad, n1)
    h = cms.make_hashes(n1, n, b, d)
    c, kernels = run(cms, A, B, h)
    assert "k_pre_pack" in kernels
    tab = O.make_tables(n1, n, b, d)
    ref = O.sketch_definition(Ad, Bd, tab)
    assert worst(c, ref) < TOL
    c2, _ = run(cms, A, B, h)
    assert torch.equal(c, c2)
    A[7, n2 // 2] = float("nan")
    c, _ = run(cms, A, B, h)
    assert torch.isnan(c).all()
    h.free()


def test_pre_sketched_operands_skewed_tables(cms):
    # every row of A in two buckets (lists of 2000 entries), columns of B spread
    n, m, b = 4000, 200, 512
    g = W.rng(5)
    h1 = (np.arange(n) % 2 * 300)[None, :].astype(np.uint32)
    h2 = g.integers(0, b, size=(1, n)).astype(np.uint32)
    s1 = g.choice([-1, 1], size=(1, n)).astype(np.int8)
    s2 = g.choice([-1, 1], size=(1, n)).astype(np.int8)
    h = cms.Hashes.from_tables(h1, s1, h2, s2, b)
    A, B, Ad, Bd = operands(n, m, n, "f32", True, 0, 6)
    c, kernels = run(cms, A, B, h)
    assert "k_pre_pack" in kernels
    tab = O.Tables(h1.astype(np.int64), s1.astype(np.int64), h2.astype(np.int64), s2.astype(np.int64), b)
    assert worst(c, O.sketch_definition(Ad, Bd, tab)) < TOL
    h.free()
