"""The direct route over the magnitudes that FP32 holds, against the FP64
oracle: a large a_k beside a small b_k and the other way round.

Tolerance: relative L2 1e-6 per repetition, as for operands of one magnitude
(about 2.5e-7 expected, with room for a factor of four): scaling a_k and b_k by
inverse powers of two changes no term of AB."""
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


def put(x, dts, pad=0):
    """x (rows in double) on the device in its storage type, and the values held."""
    buf = torch.zeros((x.shape[0], x.shape[1] + pad), dtype=DT[dts], device="cuda")
    buf[:, :x.shape[1]] = torch.from_numpy(np.ascontiguousarray(x)).to("cuda").to(DT[dts])
    v = buf[:, :x.shape[1]]
    return v, v.double().cpu().numpy()


def scaled(n1, n2, n3, dts, span, seed, pad=0):
    """Columns of A times 2^e, rows of B times 2^-e, e in -span .. span."""
    s = np.exp2(W.rng(seed).integers(-span, span + 1, size=(n2, 1)).astype(np.float64))
    at, At = put(W.gaussian(n2, n1, seed) * s, dts, pad)
    b, B = put(W.gaussian(n2, n3, seed + 1) / s, dts, pad)
    return at.T, b, At.T, B


def run(cms, A, B, h):
    cms.profile_enable(True)
    c = cms.sketch_product(A, B, h)
    torch.cuda.synchronize()
    kernels = cms.profile_summary()
    cms.profile_enable(False)
    cms.check_async()
    return c, kernels


def worst(c, ref):
    return max(O.rel_l2(c[t].cpu().numpy(), ref[t]) for t in range(ref.shape[0]))


@pytest.mark.parametrize("dts", ["f32", "bf16", "f64"])
@pytest.mark.parametrize("n1,n2,n3,b,kernel,pad", [
    (300, 512, 260, 16384, "k_direct_grid", 0),
    (257, 333, 300, 64800, "k_direct_grid", 1),        # a last superblock of 77 inner indices, rows not aligned
    (1100, 129, 1200, 20000, "k_direct_grid", 0),      # one inner index in the second superblock
    (1400, 200, 1200, 20000, "k_direct_window", 0),
    (6000, 400, 5000, 1536, "k_pre_pack", 0),
])
def test_inner_indices_of_opposite_scales(cms, dts, n1, n2, n3, b, kernel, pad):
    A, B, Ad, Bd = scaled(n1, n2, n3, dts, 30, n1 + n2, pad)
    h = cms.make_hashes(5, max(n1, n3), b, 2)
    c, kernels = run(cms, A, B, h)
    assert kernel in kernels
    assert worst(c, O.sketch_definition(Ad, Bd, O.make_tables(5, max(n1, n3), b, 2))) < TOL
    h.free()


def test_inner_indices_of_opposite_scales_in_a_batch(cms):
    # beside an instance X^T X, which needs no balance
    items, refs = [], []
    for q, (n1, n2, n3, dts) in enumerate([(300, 700, 280, "f32"), (500, 900, 500, "bf16"), (400, 200, 400, "f64")]):
        A, B, Ad, Bd = scaled(n1, n2, n3, dts, 30, q)
        items.append((A, B, cms.make_hashes(q, max(n1, n3), 8192, 2)))
        refs.append(O.sketch_definition(Ad, Bd, O.make_tables(q, max(n1, n3), 8192, 2)))
    x, X = put(W.gaussian(600, 350, 9), "f32")
    items.append((x.T, x, cms.make_hashes(9, 350, 8192, 2)))
    refs.append(O.sketch_definition(X.T, X, O.make_tables(9, 350, 8192, 2)))
    batch = cms.Batch(items)
    for _ in range(2):
        cms.profile_enable(True)
        batch.run()
        torch.cuda.synchronize()
        kernels = cms.profile_summary()
        cms.profile_enable(False)
        cms.check_async()
        assert "k_direct_tile_batched" in kernels and "k_sketch_batched" not in kernels
        assert sum(k["launches"] for k in kernels.values()) <= batch.info()["launches"]
        for c, ref in zip(batch.c, refs):
            assert worst(c, ref) < TOL
            c.zero_()
    batch.free()


def test_significant_entries_of_opposite_scales(cms):
    # one entry far above the others, from inner indices of very different size
    n, m = 200, 300
    s = np.exp2(W.rng(1).integers(-25, 26, size=(m, 1)).astype(np.float64))
    At, B = 0.01 * W.gaussian(m, n, 2) * s, 0.01 * W.gaussian(m, n, 3) / s
    At[:, 17] += 3.0 * s[:, 0]
    B[:, 121] += 3.0 / s[:, 0]
    a, b = put(At, "f32")[0], put(B, "f32")[0]
    h = cms.make_hashes(4, n, 16384, 5)
    ij, count = cms.find_significant(a.T, b, h, 1000.0, 2)
    assert count == 1 and ij.cpu().numpy().tolist() == [[17, 121]]
    h.free()


@pytest.mark.parametrize("n1,n2,n3,b", [(300, 512, 260, 16384), (6000, 400, 5000, 1536)])
@pytest.mark.parametrize("e", [-118, -126])
def test_smallest_normal_values_times_large_ones(cms, e, n1, n2, n3, b):
    # AB is of ordinary size although A is at the end of FP32's range
    at, At = put(np.exp2(e) * (1 + W.rng(3).random((n2, n1))), "f32")
    bd, B = put(np.exp2(100) * W.gaussian(n2, n3, 4), "f32")
    for A, X, Ad, Xd in [(at.T, bd, At.T, B), (bd.T, at, B.T, At)]:
        h = cms.make_hashes(5, max(n1, n3), b, 2)
        c, kernels = run(cms, A, X, h)
        assert "k_direct_tile" in kernels
        assert worst(c, O.sketch_definition(Ad, Xd, O.make_tables(5, max(n1, n3), b, 2))) < TOL
        h.free()


@pytest.mark.parametrize("n1,n2,n3,b,kernel", [(300, 500, 260, 16384, "k_direct_grid"), (1400, 200, 1200, 20000, "k_direct_window"),
                                               (6000, 400, 5000, 1536, "k_pre_pack")])
def test_two_operands_replayed_from_a_graph(cms, n1, n2, n3, b, kernel):
    # the balance, the packing and what follows them overlap at their ends; a graph
    # keeps that, on new values in the same buffers
    A, B, Ad, Bd = scaled(n1, n2, n3, "f32", 20, 5)
    h = cms.make_hashes(5, max(n1, n3), b, 2)
    ws = cms.alloc_workspace(cms.workspace_size(h, n1, n2, n3))
    c = torch.empty((2, b), device="cuda")
    cms.profile_enable(True)
    cms.sketch_product(A, B, h, c=c, ws=ws)
    torch.cuda.synchronize()
    assert kernel in cms.profile_summary()
    cms.profile_enable(False)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        cms.sketch_product(A, B, h, c=c, ws=ws, stream=torch.cuda.current_stream())
    C, D, Cd, Dd = scaled(n1, n2, n3, "f32", 20, 6)
    ref = O.sketch_definition(Cd, Dd, O.make_tables(5, max(n1, n3), b, 2))
    A.copy_(C)
    B.copy_(D)
    for _ in range(3):
        c.zero_()
        ws.fill_(0x7F)
        graph.replay()
        torch.cuda.synchronize()
        assert worst(c, ref) < TOL
    cms.check_async()
    h.free()
