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
