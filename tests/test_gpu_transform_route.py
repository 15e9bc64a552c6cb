"""The transform route's kernels where the direct route would take the call: with
a workspace of the transform route's size, against the FP64 oracle.

Tolerance: relative L2 1e-5 per repetition, as for these kernels elsewhere."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import cms_oracle as O

pytestmark = pytest.mark.gpu

TOL = 1e-5
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


def operands(n1, n2, n3, dts, alias, pad, seed):
    """Device A, B and the FP64 values they hold."""
    def put(x):
        buf = torch.zeros((x.shape[0], x.shape[1] + pad), dtype=DT[dts], device="cuda")
        buf[:, :x.shape[1]] = torch.from_numpy(x).to("cuda").to(DT[dts])
        v = buf[:, :x.shape[1]]
        return v, v.double().cpu().numpy()
    a, Ad = put(W.gaussian(n2, n1, seed))
    if alias:
        return a.T, a, Ad.T, Ad
    b, Bd = put(W.gaussian(n2, n3, seed + 1))
    return a.T, b, Ad.T, Bd


def by_spectra(cms, A, B, h):
    """The sketch by the transform route, and the kernels that ran."""
    least = cms.workspace_size(h, A.shape[0], A.shape[1], B.shape[1], A.dtype, smallest=True)
    cms.profile_enable(True)
    c = cms.sketch_product(A, B, h, ws=cms.alloc_workspace(least))
    torch.cuda.synchronize()
    kernels = cms.profile_summary()
    cms.profile_enable(False)
    cms.check_async()
    assert "k_direct_tile" not in kernels
    return c, kernels


def worst(c, ref):
    return max(O.rel_l2(c[t].cpu().numpy(), ref[t]) for t in range(ref.shape[0]))


def test_staging_rows_that_fill_shared_memory(cms):
    # two staged operands and their records come to within 128 bytes of what a
    # block can ask for: the kernel's static variables no longer fit beside them
    A, B, Ad, Bd = operands(2044, 112, 1470, "f32", False, 4, 3)
    h = cms.make_hashes(1, 2044, 20736, 3)
    c, kernels = by_spectra(cms, A, B, h)
    assert "k_sketch_fast" in kernels
    assert worst(c, O.sketch_definition(Ad, Bd, O.make_tables(1, 2044, 20736, 3))) < TOL
    h.free()


# kernel, n1, inner indices (several Kahan folds: 32 groups of two or three in the
# register kernels), n3, b, d, storage, aliased, row padding
CASES = [
    ("k_sketch_ws", "warp_specialised", 1500, 3001, 1500, 16384, 2, "f32", True, 0),
    ("k_sketch_ws", "warp_specialised", 700, 2500, 640, 8192, 2, "f32", False, 4),
    ("k_sketch_fast", "lockstep", 1000, 3000, 1000, 16000, 2, "f32", True, 0),
    ("k_sketch_fast", "lockstep", 1280, 2777, 900, 20480, 2, "bf16", False, 0),
    ("k_sketch_fast", "lockstep", 675, 2000, 675, 10800, 2, "f32", True, 1),     # rows not aligned
    ("k_sketch_fused", "shared_memory", 600, 1500, 500, 9600, 2, "f64", False, 0),
    ("k_sketch_fused", "shared_memory", 300, 2000, 300, 128, 3, "f32", True, 0),
]


@pytest.mark.parametrize("kernel,plan,n1,n2,n3,b,d,dts,alias,pad", CASES)
def test_long_inner_dimensions_by_the_spectra(cms, kernel, plan, n1, n2, n3, b, d, dts, alias, pad):
    n, seed = max(n1, n3), n1 + n2
    A, B, Ad, Bd = operands(n1, n2, n3, dts, alias, pad, seed)
    h = cms.make_hashes(seed, n, b, d)
    assert cms.plan_kernel(A, B, h) == plan
    c, kernels = by_spectra(cms, A, B, h)
    again, _ = by_spectra(cms, A, B, h)
    assert kernel in kernels and torch.equal(c, again)
    assert worst(c, O.sketch_definition(Ad, Bd, O.make_tables(seed, n, b, d))) < TOL
    h.free()


def test_both_spectrum_swaps_of_the_warp_specialised_kernel(cms, monkeypatch):
    n, m, b, d = 2048, 4096, 65536, 2
    A, B, Ad, Bd = operands(n, m, n, "f32", True, 0, 17)
    h = cms.make_hashes(23, n, b, d)
    ref = O.sketch_definition(Ad, Bd, O.make_tables(23, n, b, d))
    for swap in (None, "1"):
        if swap:
            monkeypatch.setenv("CMS_WS_SMEM_SWAP", swap)
        c, kernels = by_spectra(cms, A, B, h)
        assert "k_sketch_ws" in kernels and worst(c, ref) < TOL
    monkeypatch.delenv("CMS_WS_SMEM_SWAP")
    h.free()


@pytest.mark.parametrize("plan,kernel,n,m,b,dts", [
    ("lockstep_tmem", "k_sketch_fast", 7776, 1500, 16 * 7776, "f32"),
    ("lockstep_tmem", "k_sketch_fast", 8192, 1200, 16 * 8192, "bf16"),
    ("cluster", "k_sketch_wide", 16384, 3000, 1 << 18, "bf16"),
    ("cluster", "k_sketch_wide", 9000, 2000, 1 << 18, "f32"),
])
def test_large_hash_domains_by_the_spectra(cms, plan, kernel, n, m, b, dts):
    # sampled buckets of X^T X
    A, B, Ad, Bd = operands(n, m, n, dts, True, 0, n)
    h = cms.make_hashes(7, n, b, 1)
    assert cms.plan_kernel(A, B, h) == plan
    c, kernels = by_spectra(cms, A, B, h)
    assert kernel in kernels
    zs = W.rng(n).choice(b, 64, replace=False)
    want = O.sketch_bucket_values(Ad, Bd, O.make_tables(7, n, b, 1), 0, zs)
    got = c[0].cpu().numpy().astype(np.float64)[zs]
    assert np.linalg.norm(got - want) / np.linalg.norm(want) < TOL
    h.free()


def test_batch_by_the_spectra(cms, tmp_path):
    # 2 n inner indices each, every storage type and body of the persistent kernel;
    # the route is set in a tuning cache (a count of chunks: the spectra)
    items, refs = [], []
    for q, (n, dts, alias) in enumerate([(512, "f32", True), (1000, "f32", False), (768, "bf16", True),
                                         (675, "f32", True), (625, "bf16", False), (600, "f64", True)]):
        A, B, Ad, Bd = operands(n, 2 * n, n, dts, alias, 0, 40 + q)
        items.append((A, B, cms.make_hashes(60 + q, n, 16 * n, 2)))
        refs.append(O.sketch_definition(Ad, Bd, O.make_tables(60 + q, n, 16 * n, 2)))
    cache = tmp_path / "tune.txt"
    cms.Batch(items, autotune=True, tune_cache=str(cache)).free()
    lines = [ln.split() for ln in cache.read_text().splitlines()]
    assert sum("kernel=direct" in ln[0] for ln in lines) == len(items)
    cache.write_text("".join(f"{ln[0]} {max(int(ln[1]), 1)} {ln[2]} {ln[3]}\n" for ln in lines))
    batch = cms.Batch(items, tune_cache=str(cache))
    outs = []
    for _ in range(2):
        cms.profile_enable(True)
        outs.append([c.clone() for c in batch.run()])
        torch.cuda.synchronize()
        kernels = cms.profile_summary()
        cms.profile_enable(False)
        cms.check_async()
        assert "k_sketch_batched" in kernels and "k_direct_tile_batched" not in kernels
    for c, again, ref in zip(outs[0], outs[1], refs):
        assert torch.equal(c, again) and worst(c, ref) < TOL
    s = torch.cuda.Stream()
    batch.run_graph(s)
    s.synchronize()
    for c, w in zip(batch.c, outs[0]):
        assert torch.equal(c, w)
    batch.free()


def test_reseeded_hashes_reach_the_front_end_tables(cms):
    n, m, b, d = 1000, 600, 16000, 2
    A, B, Ad, Bd = operands(n, m, n, "f32", True, 0, 3)
    h = cms.make_hashes(1, n, b, d)
    by_spectra(cms, A, B, h)
    h.reseed(2)
    c, kernels = by_spectra(cms, A, B, h)
    assert "k_sketch_fast" in kernels
    assert worst(c, O.sketch_definition(Ad, Bd, O.make_tables(2, n, b, d))) < TOL
    h.free()


# few buckets: blocks of the direct route add to copies of the sums, which its
# conversion adds up
@pytest.mark.parametrize("n1,n2,n3,b,d,alias", [(64, 20000, 64, 12, 2, True), (150, 9000, 200, 96, 3, False),
                                                (300, 3000, 300, 1000, 1, True)])
def test_copies_of_the_sums_of_short_sketches(cms, n1, n2, n3, b, d, alias):
    A, B, Ad, Bd = operands(n1, n2, n3, "f32", alias, 0, n1)
    h = cms.make_hashes(n1, max(n1, n3), b, d)
    cms.profile_enable(True)
    c = cms.sketch_product(A, B, h)
    torch.cuda.synchronize()
    kernels = cms.profile_summary()
    cms.profile_enable(False)
    cms.check_async()
    assert "k_direct_tile" in kernels and "k_pre_pack" not in kernels
    assert worst(c, O.sketch_definition(Ad, Bd, O.make_tables(n1, max(n1, n3), b, d))) < 1e-6
    h.free()
