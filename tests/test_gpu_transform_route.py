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
