"""Which calls the direct route takes, where the other route was measured to be
the better one or memory is short."""
import pytest
import torch

pytestmark = pytest.mark.gpu

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


def kernels_of(cms, f):
    cms.profile_enable(True)
    out = f()
    torch.cuda.synchronize()
    kernels = cms.profile_summary()
    cms.profile_enable(False)
    cms.check_async()
    return out, kernels


# long inner dimensions, packed operands beyond L2 (ms by the tiles, by the
# pre-sketched operands' tiles, by the spectra)
@pytest.mark.parametrize("n1,n2,n3,b,d,dts,alias,route", [
    (2904, 20698, 2802, 3200, 1, "f32", False, "transform"),    # 1.54, 2.61, 0.94
    (5022, 19702, 5022, 3125, 1, "f32", True, "transform"),     # 1.76, 2.21, 1.01
    (4556, 33925, 5628, 4500, 1, "bf16", False, "transform"),   # 2.49, -, 1.71
    (3919, 19732, 3919, 675, 2, "f32", True, "k_pre_pack"),     # 1.24, 0.67, 1.17
    (2147, 88447, 847, 4096, 3, "f32", False, "k_direct_grid"),  # about 2, -, 6
])
def test_long_inner_dimensions_take_the_faster_route(cms, n1, n2, n3, b, d, dts, alias, route):
    x = torch.randn((n2, n1), device="cuda").to(DT[dts])
    y = x if alias else torch.randn((n2, n3), device="cuda").to(DT[dts])
    h = cms.make_hashes(1, max(n1, n3), b, d)
    _, kernels = kernels_of(cms, lambda: cms.sketch_product(x.T, y, h))
    if route == "transform":
        assert "k_direct_tile" not in kernels
    else:
        assert route in kernels or (route == "k_direct_grid" and "k_direct_window" in kernels)
    h.free()


GIB = 1 << 30


def test_workspace_of_large_operands_stays_bounded(cms):
    # packed copies of the operands would take 305 GB, 215 GB and 34 GB
    for n, m, b, d in [(9000, 1 << 22, 65536, 1), (3072, 8400000, 128, 1), (256, 1 << 24, 4096, 3)]:
        h = cms.make_hashes(1, n, b, d)
        full, least = cms.workspace_size(h, n, m, n), cms.workspace_size(h, n, m, n, smallest=True)
        assert least <= full <= 16 * GIB and least < 64 << 20
        h.free()


def test_least_workspace_is_taken_and_used_when_memory_is_short(cms, monkeypatch):
    n, m, b, d = 700, 5000, 12000, 3
    x = torch.randn((m, n), device="cuda")
    h = cms.make_hashes(2, n, b, d)
    full, least = cms.workspace_size(h, n, m, n), cms.workspace_size(h, n, m, n, smallest=True)
    want, kernels = kernels_of(cms, lambda: cms.sketch_product(x.T, x, h))
    assert "k_direct_tile" in kernels and least < full
    got, kernels = kernels_of(cms, lambda: cms.sketch_product(x.T, x, h, ws=cms.alloc_workspace(least)))
    assert "k_direct_tile" not in kernels
    assert ((got - want).norm() / want.norm()).item() < 1e-5
    from paper_1108_1320_gb300 import cms as binding
    with pytest.raises(binding.CmsError):
        cms.sketch_product(x.T, x, h, ws=cms.alloc_workspace(least)[:least - 256])
    real, asked = binding.alloc_workspace, []

    def short(nbytes, device=None):
        asked.append(nbytes)
        if nbytes >= full:
            raise torch.cuda.OutOfMemoryError("no room")
        return real(nbytes, device)
    monkeypatch.setattr(binding, "alloc_workspace", short)
    again, kernels = kernels_of(cms, lambda: cms.sketch_product(x.T, x, h))
    assert asked == [full, least] and torch.equal(again, got)
    h.free()


def test_batch_of_large_operands_stays_bounded(cms):
    # 24 products of one 1 GiB operand: packed copies of all would take 26 GB
    n, m, b = 8192, 1 << 15, 1 << 16
    x = torch.randn((m, n), device="cuda")
    hs = [cms.make_hashes(q, n, b, 1) for q in range(24)]
    batch = cms.Batch([(x.T, x, h) for h in hs])
    assert batch.info()["ws_bytes"] <= 17 * GIB
    out, kernels = kernels_of(cms, batch.run)
    assert "k_direct_tile_batched" in kernels and "k_sketch_batched" in kernels
    for c, h in zip(out, hs):                      # both routes against the single call
        want = cms.sketch_product(x.T, x, h)
        assert ((c - want).norm() / want.norm()).item() < 1e-5
    batch.free()
    for h in hs:
        h.free()


def planted(n1, n3, m, big, alias, seed):
    """Operands whose product has the entries `big` far above the others."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    x = 0.01 * torch.randn((m, n1), generator=g, device="cuda")
    y = x if alias else 0.01 * torch.randn((m, n3), generator=g, device="cuda")
    for q, (i, j) in enumerate(big):
        x[q, i] += 10.0
        y[q, j] += 10.0 + q
    return x, y


# 71 x 71 and 40 x 110 tiles: stored entries in bands of 48 and 36 tile rows (two
# parts each where the units are single tiles), the last band shorter
@pytest.mark.parametrize("n1,n3,alias", [(9000, 9000, True), (8970, 8973, False), (5100, 14000, False)])
def test_significant_entries_in_bands_of_rows(cms, n1, n3, alias):
    m, b, d = 1000, 16384, 5
    big = [(3, 5), (n1 - 1, 0), (n1 // 2, n3 - 1), (6143, 7001), (6144, 21)] if n1 > 6144 else \
        [(3, 5), (n1 - 1, 0), (n1 // 2, n3 - 1), (1535, 13999), (1536, 21), (4607, 4608), (4608, 4607)]
    x, y = planted(n1, n3, m, big, alias, n1)
    ab = x.double().T @ y.double()
    want = torch.nonzero(ab.abs() > 50.0).cpu().tolist()
    del ab
    h = cms.make_hashes(15, max(n1, n3), b, d)
    (ij, count), kernels = kernels_of(cms, lambda: cms.find_significant(x.T, y, h, 50.0, 3))
    assert kernels["k_direct_tile"]["launches"] > 1 and kernels["k_direct_grid"]["launches"] > 1
    assert count == len(want) and ij.cpu().tolist() == want
    h.free()


def test_significant_workspace_stays_bounded(cms, monkeypatch):
    # the entries of AB would take 1.07 GB
    import ctypes
    h = cms.make_hashes(1, 16384, 1 << 16, 5)
    full, least = ctypes.c_size_t(), ctypes.c_size_t()
    for query, out in ((cms.lib().cms_significant_workspace_size, full),
                       (cms.lib().cms_significant_workspace_size_min, least)):
        assert query(h.handle, 16384, 2000, 16384, 0, 3, ctypes.byref(out)) == 0
    assert least.value < 430e6 and least.value <= full.value < 760e6
    h.free()
    # the least is used when memory is short, with the same positions
    big = [(3, 5), (117, 230), (299, 0)]
    x, y = planted(300, 280, 5000, big, False, 3)
    h = cms.make_hashes(4, 300, 16384, 5)
    (want, count), kernels = kernels_of(cms, lambda: cms.find_significant(x.T, y, h, 50.0, 1))
    assert "k_direct_sig_decode" in kernels and count == 3
    from paper_1108_1320_gb300 import cms as binding
    real, asked = binding.alloc_workspace, []

    def short(nbytes, device=None):
        asked.append(nbytes)
        if len(asked) == 1:
            raise torch.cuda.OutOfMemoryError("no room")
        return real(nbytes, device)
    monkeypatch.setattr(binding, "alloc_workspace", short)
    (got, again), kernels = kernels_of(cms, lambda: cms.find_significant(x.T, y, h, 50.0, 1))
    assert "k_mask_copy" in kernels and "k_direct_tile" not in kernels and asked[1] < asked[0]
    assert again == count and torch.equal(got, want)
    h.free()


def test_tuned_route_of_a_batch_knows_aliased_operands(cms, tmp_path):
    # FP64 storage: X^T X packs one operand and skips half of the tiles, so that its
    # tuned route is not that of two operands of the same shape
    n, m, b, d = 640, 1280, 10240, 2
    x = torch.randn((m, n), device="cuda", dtype=torch.float64)
    y = torch.randn((m, n), device="cuda", dtype=torch.float64)
    hs = [cms.make_hashes(q, n, b, d) for q in range(2)]
    items = [(x.T, x, hs[0]), (x.T, y, hs[1])]
    cache = tmp_path / "tune.txt"
    batch = cms.Batch(items, autotune=True, tune_cache=str(cache))
    want, _ = kernels_of(cms, batch.run)
    want = [c.clone() for c in want]
    lines = [ln for ln in cache.read_text().splitlines() if "kernel=direct" in ln]
    assert sorted(ln.split()[0].endswith("-alias") for ln in lines) == [False, True]
    # each key decides for its own instance (a count of chunks: the transform route)
    tuned = [ln.split()[0] + (" 3 0 1.0" if "-alias" in ln else " 0 0 1.0") for ln in lines]
    cache.write_text("\n".join(tuned) + "\n")
    again = cms.Batch(items, tune_cache=str(cache))
    out, kernels = kernels_of(cms, again.run)
    assert "k_direct_tile_batched" in kernels and "k_sketch_batched" in kernels
    assert kernels["k_direct_balance_batched"]["launches"] == 1      # the two operands, by the tiles
    for c, w in zip(out, want):
        assert ((c - w).norm() / w.norm()).item() < 1e-5
    batch.free()
    again.free()
    for h in hs:
        h.free()


# long inner dimensions in a batch, packed operands beyond L2 (ms an instance by the
# tiles, by the spectra)
@pytest.mark.parametrize("n,m,b,d,dts,direct", [
    (8975, 30000, 2592, 2, "bf16", True),       # 3.74, 5.79
    (2001, 28282, 1350, 2, "bf16", True),       # 0.30, 0.91
    (5022, 19702, 3125, 1, "f32", False),       # 1.69, 1.03
    (4096, 8192, 4096, 1, "f32", False),        # 0.46, 0.34
])
def test_long_inner_dimensions_of_a_batch(cms, n, m, b, d, dts, direct):
    x = torch.randn((m, n), device="cuda").to(DT[dts])
    hs = [cms.make_hashes(q, n, b, d) for q in range(2)]
    batch = cms.Batch([(x.T, x, h) for h in hs])
    _, kernels = kernels_of(cms, batch.run)
    assert ("k_direct_tile_batched" in kernels) == direct
    batch.free()
    for h in hs:
        h.free()


def test_short_sketches_of_a_batch_split_little(cms, tmp_path):
    # additions to few buckets queue up: with the inner dimension split for the full
    # rate the tiles took 89 us an instance where the spectra take 42, now 12
    n, m, b = 242, 6456, 64
    xs = [torch.randn((m, n), device="cuda").bfloat16() for _ in range(8)]
    hs = [cms.make_hashes(q, n, b, 1) for q in range(8)]
    items = [(x.T, x, h) for x, h in zip(xs, hs)]
    cache = tmp_path / "tune.txt"
    cms.Batch(items, autotune=True, tune_cache=str(cache)).free()
    key = [ln.split()[0] for ln in cache.read_text().splitlines() if "kernel=direct" in ln][0]
    best, outs = [], []
    for chunks in (0, 64):                  # the tiles, the spectra
        cache.write_text(f"{key} {chunks} 0 1.0\n")
        batch = cms.Batch(items, tune_cache=str(cache))
        out, kernels = kernels_of(cms, batch.run)
        assert ("k_direct_tile_batched" in kernels) == (chunks == 0)
        outs.append([c.clone() for c in out])
        times = []
        for _ in range(8):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            batch.run()
            e[1].record()
            e[1].synchronize()
            times.append(e[0].elapsed_time(e[1]))
        best.append(min(times))
        batch.free()
    assert best[0] < best[1]
    for c, w in zip(*outs):
        assert ((c - w).norm() / w.norm()).item() < 1e-5
    for h in hs:
        h.free()


# few buckets or few inner indices: pre-sketched operands have few blocks to sum them
# in, or tiles with few rows (ms by them, by the spectra)
@pytest.mark.parametrize("n1,n2,n3,b,d,dts,alias", [
    (10847, 947, 5263, 128, 1, "bf16", False),      # 0.33, 0.18
    (11552, 535, 11552, 144, 1, "bf16", True),      # 0.21, 0.16
    (5120, 415, 5120, 27, 3, "f64", True),          # 0.32, 0.18
])
def test_pre_sketched_operands_need_blocks_to_sum_in(cms, n1, n2, n3, b, d, dts, alias):
    x = torch.randn((n2, n1), device="cuda").to(DT[dts])
    y = x if alias else torch.randn((n2, n3), device="cuda").to(DT[dts])
    h = cms.make_hashes(1, max(n1, n3), b, d)
    _, kernels = kernels_of(cms, lambda: cms.sketch_product(x.T, y, h))
    assert "k_pre_pack" not in kernels and "k_direct_tile" not in kernels
    h.free()


def test_shortest_sketches_split_little(cms):
    # three buckets: 64 parts of the inner dimension would each add their own share
    # to them (0.52 ms, 0.33 by the spectra)
    n1, n2, n3, b = 362, 35456, 209, 3
    x, y = torch.randn((n2, n1), device="cuda"), torch.randn((n2, n3), device="cuda")
    h = cms.make_hashes(1, n1, b, 1)
    least = cms.alloc_workspace(cms.workspace_size(h, n1, n2, n3, smallest=True))
    room = cms.alloc_workspace(cms.workspace_size(h, n1, n2, n3))
    want, kernels = kernels_of(cms, lambda: cms.sketch_product(x.T, y, h, ws=least))
    assert "k_direct_tile" not in kernels
    got, kernels = kernels_of(cms, lambda: cms.sketch_product(x.T, y, h, ws=room))
    assert ((got - want).norm() / want.norm()).item() < 1e-5
    best = []
    for ws in (room, least):
        times = []
        for _ in range(10):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            cms.sketch_product(x.T, y, h, ws=ws)
            e[1].record()
            e[1].synchronize()
            times.append(e[0].elapsed_time(e[1]))
        best.append(min(times))
    assert best[0] < 1.15 * best[1]
    h.free()
