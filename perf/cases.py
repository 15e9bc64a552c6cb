"""The work that users of the compressed product have it do, as timed cases.

Each case is one pass through the public entry points of the package: a
sketch of a product (dense, sparse or a batch of products), with the decoding
that belongs to it.  Sizes are those of the repository's workloads, tests and
benchmark, or generic ones between them.

    listed()            the fixed cases
    draw(rng)           one more case of the same ranges
    prepare(case, seed) inputs and handles on the GPU
    run(state)          one pass, its outputs
    work(case)          bytes and operations that a pass cannot do without
    exact(case, seed)   the outputs in 64 bits, in plain torch
"""
import math

import numpy as np
import torch

import paper_1108_1320_gb300 as cms

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f64": torch.float64}


def _product(name, n1, n2, n3, b, d, dtype, alias, pad=0, then="", reseed=False):
    return {"name": name, "kind": "product", "n1": n1, "n2": n2, "n3": n3, "b": b, "d": d, "dtype": dtype,
            "alias": alias, "pad": pad, "then": then, "reseed": reseed}


def listed():
    return [
        # the smallest use: one product of two 256 x 256 FP64 matrices, one
        # short sketch (the plain-method configuration)
        _product("plain_256", 256, 256, 256, 1024, 1, "f64", False),
        # two different operands, every size odd or ragged, rows not aligned,
        # b not a power of two
        _product("ragged_ab", 1777, 1203, 1003, 20000, 3, "f32", False, pad=1),
        # the benchmarked step: a fresh hash draw, the sketch of X^T X for a
        # sample covariance, every estimate decoded
        _product("cov_step", 2048, 4096, 2048, 65536, 5, "f32", True, then="dense", reseed=True),
        # a mid-size covariance of BF16 samples (one member of the batch)
        _product("cov_bf16", 4096, 8192, 4096, 65536, 3, "bf16", True),
        # a sketch much shorter than the number of variables: many columns
        # summarised in little space
        _product("short_sketch", 16384, 2048, 16384, 2048, 5, "f32", True),
        # the large covariance configuration
        _product("large", 32768, 16384, 32768, 1 << 20, 7, "bf16", True),
        # correlated pairs found without a dense output: sketch, diagonal
        # removed, estimates above a threshold listed (Fig. 2)
        _product("cov_pairs", 1500, 3000, 1500, 30000, 5, "f32", True, then="pairs"),
        # 64 covariances of uneven size in one persistent launch, replayed
        # from a CUDA graph
        {"name": "batch_64", "kind": "batch", "count": 64, "n_lo": 512, "n_hi": 8192, "d": 3},
        # sparse factors with a sparse integer product (Theorem 5), FFT route
        {"name": "sparse_fft", "kind": "sparse", "n": 1 << 20, "blocks": 256, "inner": 8, "rows": 32, "cols": 32,
         "b": 1 << 20, "d": 3, "dtype": "f32", "hybrid": False},
        # the same, small outer products sketched directly
        {"name": "sparse_hybrid", "kind": "sparse", "n": 1 << 20, "blocks": 256, "inner": 8, "rows": 32, "cols": 32,
         "b": 1 << 20, "d": 3, "dtype": "f32", "hybrid": True},
        # chosen entries decoded from a long sketch
        {"name": "decode_pairs", "kind": "decode", "n": 32768, "b": 1 << 20, "d": 7, "q": 100000},
        # positions of the significant entries (Sec. 4)
        {"name": "significant", "kind": "significant", "n": 256, "m": 2000, "b": 1 << 16, "d": 5, "rho": 3},
    ]


def _smooth(x):
    """The largest 5-smooth integer <= x."""
    best, p2 = 1, 1
    while p2 <= x:
        p3 = p2
        while p3 <= x:
            p5 = p3
            while p5 * 5 <= x:
                p5 *= 5
            best = max(best, p5)
            p3 *= 3
        p2 *= 2
    return best


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _fft_flops(b):
    return 5.0 * b * math.log2(max(b, 2)) + 4.0 * b


def draw(rng):
    kind = rng.choices(["product", "batch", "sparse", "decode", "significant"], [12, 2, 3, 1, 1])[0]
    d = rng.randint(1, 7)
    if kind == "product":
        dtype = rng.choices(["f32", "bf16", "f64"], [10, 7, 3])[0]
        alias = rng.random() < 0.6
        n1 = _log_uniform(rng, 96, 1200 if dtype == "f64" else 12288)
        n3 = n1 if alias else max(64, min(2 * n1, _log_uniform(rng, n1 / 3, 2 * n1)))
        n = max(n1, n3)
        b = _smooth(min(1 << 20, max(64, _log_uniform(rng, n / 8, 32 * n))))
        n2 = _log_uniform(rng, 16, 8192)
        n2 = max(16, min(n2, int(4e12 / (d * _fft_flops(b)))))
        if dtype == "f64":
            n2 = min(n2, 1024)
        then = rng.choices(["", "dense", "pairs"], [6, 3, 2])[0]
        if then == "pairs" and not (alias and dtype == "f32" and b >= 8 * n and n >= 700 and n2 >= 256 and d % 2):
            then = ""
        c = _product("", n1, n2, n3, b, d, dtype, alias, pad=rng.choice([0, 0, 0, 1, 3]), then=then,
                     reseed=rng.random() < 0.3)
        del c["name"]
        return c
    if kind == "batch":
        lo = _log_uniform(rng, 128, 1024)
        return {"kind": "batch", "count": rng.randint(3, 24), "n_lo": lo,
                "n_hi": min(8192, lo * rng.choice([2, 4, 8])), "d": rng.randint(1, 4)}
    if kind == "sparse":
        n = _log_uniform(rng, 1 << 13, 1 << 20)
        rows, cols, inner = rng.randint(5, 48), rng.randint(5, 48), rng.randint(2, 12)
        blocks = max(1, min(256, n // (2 * max(rows, cols, inner))))
        # the sparse entry point takes multiples of 1024
        b = 1024 * _smooth(min(1 << 10, max(1, int(blocks * rows * cols * rng.uniform(0.5, 8)) // 1024)))
        return {"kind": "sparse", "n": n, "blocks": blocks, "inner": inner, "rows": rows, "cols": cols, "b": b,
                "d": rng.randint(1, 3), "dtype": rng.choice(["f32", "bf16"]), "hybrid": rng.random() < 0.5}
    if kind == "decode":
        n = _log_uniform(rng, 300, 32768)
        return {"kind": "decode", "n": n, "b": _smooth(min(1 << 20, 16 * n)), "d": d,
                "q": _log_uniform(rng, 20000, 2000000)}
    return {"kind": "significant", "n": rng.randint(100, 300), "m": _log_uniform(rng, 1000, 3000), "b": 1 << 16,
            "d": 5, "rho": 3}


# ------------------------------------------------------------------ inputs --
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _covariance(m, n, pairs, rho, g, dtype, pad=0):
    """m samples of n N(0, 1) variables, `pairs` disjoint planted pairs."""
    buf = torch.empty((m, n + pad), dtype=dtype, device="cuda")
    perm = torch.randperm(n, generator=g, device="cuda")
    u, v = perm[:pairs], perm[pairs:2 * pairs]
    rows = max(1, (1 << 26) // max(n, 1))
    for r in range(0, m, rows):
        k = min(rows, m - r)
        x = torch.randn((k, n), generator=g, device="cuda", dtype=torch.float32)
        if pairs:
            x[:, v] = rho * x[:, u] + math.sqrt(1 - rho * rho) * torch.randn((k, pairs), generator=g, device="cuda")
        buf[r:r + k, :n] = x.to(dtype)
        if pad:
            buf[r:r + k, n:] = 0
    return buf[:, :n]


def _gaussian(rows, cols, g, dtype, pad=0):
    buf = torch.zeros((rows, cols + pad), dtype=dtype, device="cuda")
    buf[:, :cols] = torch.randn((rows, cols), generator=g, device="cuda", dtype=torch.float32).to(dtype)
    return buf[:, :cols]


def _operands(case, seed):
    """(A, B): A column-major n1 x n2, B row-major n2 x n3."""
    g = _gen(seed)
    dt = DTYPES[case["dtype"]]
    if case["alias"]:
        n = case["n1"]
        pairs = max(1, n // 64)
        X = _covariance(case["n2"], n, pairs, 0.3 if n >= 16384 else 0.5, g, dt, case["pad"])
        return X.T, X
    At = _gaussian(case["n2"], case["n1"], g, dt, case["pad"])
    return At.T, _gaussian(case["n2"], case["n3"], g, dt, case["pad"])


def _batch_sizes(case):
    """(n, m, dtype) of each instance: n log-uniform and 5-smooth, m = 2 n, the first half FP32, the rest BF16."""
    r = np.random.RandomState(case["count"] * 7919 + case["n_hi"])
    ns = np.exp(r.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]), case["count"]))
    half = (case["count"] + 1) // 2
    return [(_smooth(int(n)), 2 * _smooth(int(n)), "f32" if q < half else "bf16") for q, n in enumerate(ns)]


def _batch_data(case, seed):
    g = _gen(seed)
    return [_covariance(m, n, n // 100, 0.5, g, DTYPES[dt]) for n, m, dt in _batch_sizes(case)]


def _sparse_data(case, seed):
    """Disjoint blocks of inner indices x rows of A x columns of B, integers in [-8, 8] without 0."""
    g = _gen(seed)
    n, nb, inner, rows, cols = (case[k] for k in ("n", "blocks", "inner", "rows", "cols"))
    pick = lambda k: torch.randperm(n, generator=g, device="cuda")[:nb * k]  # noqa: E731
    ks, order = torch.sort(pick(inner))
    block = order // inner

    def side(width):
        ids = torch.sort(pick(width).reshape(nb, width), dim=1).values
        idx = ids[block]
        val = torch.randint(1, 9, idx.shape, generator=g, device="cuda")
        val = val * (2 * torch.randint(0, 2, idx.shape, generator=g, device="cuda") - 1)
        cnt = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
        cnt[ks + 1] = width
        return torch.cumsum(cnt, 0), idx.reshape(-1).to(torch.int32), val.reshape(-1).to(DTYPES[case["dtype"]])

    return side(rows) + side(cols)


def _hash_seed(seed):
    return 1000 + int(seed)


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "kind": kind}
    if kind == "product":
        A, B = _operands(case, seed)
        h = cms.make_hashes(_hash_seed(seed), max(case["n1"], case["n3"]), case["b"], case["d"])
        st.update(A=A, B=B, h=h, seed=_hash_seed(seed),
                  c=torch.empty((case["d"], case["b"]), dtype=torch.float32, device="cuda"),
                  ws=cms.alloc_workspace(cms.workspace_size(h, case["n1"], case["n2"], case["n3"], A.dtype)))
        if case["then"] == "dense":
            st["est"] = torch.empty((case["n1"], case["n3"]), dtype=torch.float32, device="cuda")
    elif kind == "batch":
        xs = _batch_data(case, seed)
        items = [(X.T, X, cms.make_hashes(_hash_seed(seed) + q, X.shape[1], 16 * X.shape[1], case["d"]))
                 for q, X in enumerate(xs)]
        st["batch"] = cms.Batch(items)
        st["stream"] = torch.cuda.Stream()
        torch.cuda.synchronize()
    elif kind == "sparse":
        st["data"] = _sparse_data(case, seed)
        st["h"] = cms.make_hashes(_hash_seed(seed), case["n"], case["b"], case["d"])
        st["c"] = torch.empty((case["d"], case["b"]), dtype=torch.float32, device="cuda")
        st["ws"] = cms.alloc_workspace(cms.sparse_workspace_size(st["h"], case["n"], case["n"], case["n"]))
    elif kind == "decode":
        g = _gen(seed)
        st["c"] = torch.randn((case["d"], case["b"]), generator=g, device="cuda")
        st["ij"] = torch.randint(0, case["n"], (case["q"], 2), generator=g, device="cuda", dtype=torch.int64)
        st["out"] = torch.empty(case["q"], dtype=torch.float32, device="cuda")
        st["h"] = cms.make_hashes(_hash_seed(seed), case["n"], case["b"], case["d"])
    else:
        X = _covariance(case["m"], case["n"], 8, 0.8, _gen(seed), torch.float32)
        st.update(X=X, h=cms.make_hashes(_hash_seed(seed), case["n"], case["b"], case["d"]))
    return st


PAIRS = 256   # buffer of the thresholded decode: the first hits in row-major order, and the count of all


def _tau(case):
    """Three standard deviations of the estimates of uncorrelated pairs."""
    sd = math.sqrt(case["n2"] * case["n1"] * case["n3"] / case["b"])
    return 3.0 * sd * {1: 1.0, 3: 0.67, 5: 0.54, 7: 0.46}[case["d"]]


def run(st):
    case, kind = st["case"], st["kind"]
    if kind == "product":
        if case["reseed"]:
            st["h"].reseed(st["seed"])
        c = cms.sketch_product(st["A"], st["B"], st["h"], c=st["c"], ws=st["ws"])
        if case["then"] == "dense":
            return c, cms.decode_dense(c, st["h"], case["n1"], case["n3"], out=st["est"])
        if case["then"] == "pairs":
            cms.remove_diagonal(st["A"], st["B"], st["h"], c)
            ij, val, count = cms.decode_threshold(c, st["h"], case["n1"], case["n3"], _tau(case), capacity=PAIRS)
            return c, ij, val, count
        return c
    if kind == "batch":
        s = st["stream"]
        s.wait_stream(torch.cuda.current_stream())
        out = st["batch"].run_graph(s)
        torch.cuda.current_stream().wait_stream(s)
        return list(out)
    if kind == "sparse":
        n = case["n"]
        return cms.sketch_product_csr(*st["data"], n, n, st["h"], c=st["c"], ws=st["ws"],
                                      direct_max_pairs=-1 if case["hybrid"] else None)
    if kind == "decode":
        return cms.decode(st["c"], st["h"], st["ij"], out=st["out"])
    ij, count = cms.find_significant(st["X"].T, st["X"], st["h"], 0.4 * case["m"], case["rho"])
    return ij, count


# -------------------------------------------------------------------- work --
def _product_work(n1, n2, n3, b, d, esz, alias, then=""):
    """A pass reads the operands once and writes the sketch once; its
    operations are those of the transform route or, where that is fewer, of
    the product's entries and their sketch."""
    by = esz * n2 * (n1 if alias else n1 + n3) + 4.0 * d * b
    fl = min(d * n2 * _fft_flops(b), (1.0 if alias else 2.0) * n1 * n2 * n3 + float(d) * n1 * n3)
    if then == "dense":
        by += 4.0 * n1 * n3
    if then:
        fl += float(d) * n1 * n3
    return by, fl


def work(case):
    kind = case["kind"]
    if kind == "product":
        by, fl = _product_work(case["n1"], case["n2"], case["n3"], case["b"], case["d"],
                               DTYPES[case["dtype"]].itemsize, case["alias"], case["then"])
    elif kind == "batch":
        by = fl = 0.0
        for n, m, dt in _batch_sizes(case):
            x, y = _product_work(n, m, n, 16 * n, case["d"], DTYPES[dt].itemsize, True)
            by, fl = by + x, fl + y
    elif kind == "sparse":
        k = case["blocks"] * case["inner"]
        esz = DTYPES[case["dtype"]].itemsize
        by = 16.0 * case["n"] + k * (case["rows"] + case["cols"]) * (4.0 + esz) + 4.0 * case["d"] * case["b"]
        fl = 2.0 * case["d"] * k * case["rows"] * case["cols"]
    elif kind == "decode":
        by, fl = case["q"] * (16.0 + 4.0 + 4.0 * case["d"]), float(case["q"] * case["d"])
    else:
        bits = 2 * case["rho"] * math.ceil(math.log2(case["n"]))
        by = 4.0 * case["n"] * case["m"]
        fl = 1.0 * case["n"] ** 2 * case["m"] + 2.0 * bits * case["d"] * case["n"] ** 2
    return {"bytes": by, "flops": fl}


# ----------------------------------------------------------- 64-bit values --
def _tables(seed, n, b, d):
    """h1, s1, h2, s2 (each d x n, on the GPU) of the polynomial family drawn by splitmix64."""
    p, state, mask = (1 << 31) - 1, int(seed), (1 << 64) - 1
    x = torch.arange(n, dtype=torch.int64, device="cuda")
    out = [[], [], [], []]
    for _ in range(d):
        for q in range(4):
            ac = []
            for _ in range(2):
                state = (state + 0x9E3779B97F4A7C15) & mask
                z = state
                z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
                z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
                ac.append(z ^ (z >> 31))
            v = ((1 + ac[0] % (p - 1)) * x + ac[1] % p) % p
            out[q].append(v % b if q % 2 == 0 else 1 - 2 * (v % 2))
    return [torch.stack(t) for t in out]


def _scatter(c, G, h1, s1, h2, s2, b):
    """Adds the entries of G (rows of h1, columns of h2) to the sketches c."""
    for t in range(c.shape[0]):
        z = (h1[t][:, None] + h2[t][None, :]) % b
        c[t].index_add_(0, z.reshape(-1), (G * (s1[t][:, None] * s2[t][None, :])).reshape(-1))


def _exact_sketch(A, B, alias, tab, b, d):
    """(sketch, diagonal of AB) in 64 bits; X^T X by its upper panels."""
    n1, n3 = A.shape[0], B.shape[1]
    c = torch.zeros((d, b), dtype=torch.float64, device="cuda")
    diag = torch.zeros(min(n1, n3), dtype=torch.float64, device="cuda")
    h1, s1, h2, s2 = tab
    Bd = B.double()
    step = max(1, min(n1, (1 << 26) // max(n3, 1)))
    for i in range(0, n1, step):
        j = min(n1, i + step)
        j0 = i if alias else 0
        G = A[i:j].double() @ Bd[:, j0:]
        k = min(j, n3)
        if k > i:
            diag[i:k] = torch.diagonal(G[:, i - j0:k - j0])
        _scatter(c, G, h1[:, i:j], s1[:, i:j], h2[:, j0:n3], s2[:, j0:n3], b)
        if alias and j < n1:
            _scatter(c, G[:, j - j0:].T, h1[:, j:n1], s1[:, j:n1], h2[:, i:j], s2[:, i:j], b)
    return c, diag


def _estimates(c, tab, n1, n3, b):
    """Median over the repetitions of s1 s2 c[(h1 + h2) mod b], n1 x n3."""
    h1, s1, h2, s2 = tab
    out = torch.empty((n1, n3), dtype=torch.float64, device="cuda")
    step = max(1, (1 << 25) // max(n3, 1))
    d = c.shape[0]
    for i in range(0, n1, step):
        j = min(n1, i + step)
        e = torch.stack([c[t][(h1[t, i:j, None] + h2[t, None, :n3]) % b] * (s1[t, i:j, None] * s2[t, None, :n3])
                         for t in range(d)]).sort(dim=0).values
        out[i:j] = e[d // 2] if d % 2 else 0.5 * (e[d // 2 - 1] + e[d // 2])
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "product":
        A, B = _operands(case, seed)
        n1, n3, b, d = case["n1"], case["n3"], case["b"], case["d"]
        tab = _tables(_hash_seed(seed), max(n1, n3), b, d)
        c, diag = _exact_sketch(A, B, case["alias"], tab, b, d)
        if case["then"] == "dense":
            return c, _estimates(c, tab, n1, n3, b)
        if case["then"] == "pairs":
            h1, s1, h2, s2 = tab
            k = diag.numel()
            for t in range(d):
                c[t].index_add_(0, (h1[t, :k] + h2[t, :k]) % b, -diag * (s1[t, :k] * s2[t, :k]))
            e = _estimates(c, tab, n1, n3, b)
            hit = e.abs() > _tau(case)
            hit.fill_diagonal_(False)
            return c, None, e[hit][:PAIRS], None
        return c
    if kind == "batch":
        out = []
        for q, X in enumerate(_batch_data(case, seed)):
            n = X.shape[1]
            tab = _tables(_hash_seed(seed) + q, n, 16 * n, case["d"])
            out.append(_exact_sketch(X.T, X, True, tab, 16 * n, case["d"])[0])
        return out
    if kind == "sparse":
        ap, ai, av, bp, bi, bv = _sparse_data(case, seed)
        n, b, d, rows, cols = case["n"], case["b"], case["d"], case["rows"], case["cols"]
        h1, s1, h2, s2 = _tables(_hash_seed(seed), n, b, d)
        c = torch.zeros((d, b), dtype=torch.float64, device="cuda")
        i, j = ai.long().reshape(-1, rows, 1), bi.long().reshape(-1, 1, cols)
        v = av.double().reshape(-1, rows, 1) * bv.double().reshape(-1, 1, cols)
        for t in range(d):
            c[t].index_add_(0, ((h1[t][i] + h2[t][j]) % b).reshape(-1), (v * (s1[t][i] * s2[t][j])).reshape(-1))
        return c
    if kind == "decode":
        g = _gen(seed)
        c = torch.randn((case["d"], case["b"]), generator=g, device="cuda").double()
        ij = torch.randint(0, case["n"], (case["q"], 2), generator=g, device="cuda", dtype=torch.int64)
        h1, s1, h2, s2 = _tables(_hash_seed(seed), case["n"], case["b"], case["d"])
        i, j, d = ij[:, 0], ij[:, 1], case["d"]
        e = torch.stack([c[t][(h1[t][i] + h2[t][j]) % case["b"]] * (s1[t][i] * s2[t][j])
                         for t in range(d)]).sort(dim=0).values
        return e[d // 2] if d % 2 else 0.5 * (e[d // 2 - 1] + e[d // 2])
    return None
