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
