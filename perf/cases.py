"""The work this library is measured on: CSR x dense products, their gradients, semiring products and batches,
each through the package's public entry points, over the ranges of sizes that its users run.

A case is a dict of plain values:
  form    "product" (C = A B), "train" (forward and backward of a layer Y = A X on a pattern that stays), "sampled"
          (the same on a pattern that is new at every step), "semiring" (a (min, +) relaxation), "batched"
  rows    row lengths of A: "uniform", "poisson", "mesh" (1 + Poisson), "power_law" (density exponent 2, 1 % of the
          rows empty), "graph" (symmetric-normalised adjacency of a Chung-Lu graph, exponent 2.2, hub columns too)
  m, k    shape of A;  mean: stored entries per row;  cap: longest row of "power_law"
  n       columns of B
  types   storage of A's values, B and C
  entry   "matrix" (CSRMatrix, which knows its longest row) or "plain" (the spmm function and its default choice)
"""
import math

import torch

import paper_1803_08601_gb300 as pkg

_TYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
_BATCH_WIDTHS = (32, 64, 128)
_MOST_PRODUCTS = 2_000_000_000  # stored entries x columns of a drawn case: below the largest listed ones


def _product(name, rows, m, k, mean, n, types="f32/f32/f32", cap=100_000, entry="matrix"):
    return dict(name=name, form="product", rows=rows, m=m, k=k, mean=float(mean), n=n, types=types, cap=cap, entry=entry)


def listed():
    return [
        # one small layer, called on its own: launch and host time count as much as the kernel
        _product("small_layer_n64", "uniform", 4096, 4096, 16, 64, entry="plain"),
        # y = A x on a skewed matrix: an iterative solver or a ranking step
        _product("vector_power_law", "power_law", 1_000_000, 1_000_000, 16, 1),
        # tall-skinny products on the skewed matrix: a block of vectors, a hidden layer, a wide one
        _product("block_power_law_n8", "power_law", 1_000_000, 1_000_000, 16, 8),
        _product("block_power_law_n32", "power_law", 1_000_000, 1_000_000, 16, 32),
        _product("block_power_law_n128", "power_law", 1_000_000, 1_000_000, 16, 128),
        # short uneven rows and a feature width that is no power of two
        _product("short_rows_n100", "poisson", 600_000, 400_001, 3, 100),
        # the last layer of a node classifier: as many columns as classes, an odd number
        _product("classes_graph_n47", "graph", 250_000, 250_000, 20, 47),
        # inference with 16-bit weights and features
        _product("inference_bf16_n128", "uniform", 1_000_000, 1_000_000, 32, 128, types="bf16/bf16/bf16"),
        # one full-graph training step of a graph layer: Y = A X, dX, dvals
        dict(name="train_graph_n256", form="train", rows="graph", m=500_000, k=500_000, mean=20.0, n=256),
        # one step on a freshly sampled neighbourhood: the pattern (its longest row, its transpose) is new every time
        dict(name="sampled_step_n128", form="sampled", rows="poisson", m=60_000, k=200_003, mean=15.0, n=128),
        # sixteen sources of shortest paths relaxed at once over a road-like network
        dict(name="paths_min_plus_n16", form="semiring", rows="mesh", m=1_000_000, k=1_000_000, mean=4.0, n=16),
        # many independent products of uneven size, replayed as a graph
        dict(name="batch_of_256", form="batched", count=256, m_lo=64, m_hi=65536, mean_lo=4.0, mean_hi=64.0),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng):
    """Columns of B: the usual powers of two, other even widths, and odd ones, from 1 to 256."""
    kind = rng.random()
    if kind < 0.4:
        return 2 ** rng.randint(0, 8)
    if kind < 0.75:
        return 4 * _log_uniform(rng, 1, 64)
    return _log_uniform(rng, 1, 256)


def draw(rng):
    form = rng.choice(["product"] * 6 + ["train", "sampled", "semiring", "batched"])
    if form == "batched":
        return dict(form=form, count=_log_uniform(rng, 8, 256), m_lo=_log_uniform(rng, 64, 1000),
                    m_hi=_log_uniform(rng, 4000, 65536), mean_lo=rng.uniform(2.0, 10.0), mean_hi=rng.uniform(12.0, 64.0))
    n = _width(rng)
    mean = rng.uniform(2.0, 40.0)
    m = _log_uniform(rng, 1500, 1_000_000)
    m = max(1500, min(m, int(16_000_000 / mean), int(_MOST_PRODUCTS / (mean * n))))
    k = max(256, int(m * rng.choice([1.0, 1.0, rng.uniform(0.4, 2.5)])))
    if form == "semiring":
        return dict(form=form, rows="mesh", m=m, k=m, mean=min(mean, 12.0), n=min(n, 64))
    if form == "sampled":
        return dict(form=form, rows="poisson", m=min(m, 100_000), k=min(k, 250_000), mean=mean, n=n)
    if form == "train":
        m = min(m, 500_000)
        return dict(form=form, rows="graph", m=m, k=m, mean=max(mean, 4.0), n=n)
    rows = rng.choice(["uniform", "poisson", "power_law", "graph"])
    if rows == "graph":
        k = m
    if rows == "power_law":  # smaller caps cannot reach a mean below about ln(cap)
        mean = max(mean, 14.0)
        m = max(1500, min(m, int(16_000_000 / mean), int(_MOST_PRODUCTS / (mean * n))))
        k = max(k, m)
    types = rng.choice(["f32/f32/f32"] * 4 + ["bf16/bf16/bf16", "bf16/bf16/f32", "f16/f16/f16", "f16/f16/f32"])
    entry = "matrix" if rows in ("power_law", "graph") else rng.choice(["matrix", "plain"])
    c = _product("", rows, m, k, mean, n, types=types, cap=min(100_000, m // 10), entry=entry)
    del c["name"]
    return c


# ----------------------------------------------------------------------------- inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 1803)


def _lengths(rows, m, mean, cap, g):
    if rows == "uniform":
        return torch.full((m,), int(round(mean)), dtype=torch.int64, device="cuda")
    if rows == "poisson":  # with exactly the expected total, so that gradients of A's values keep their length
        lens = torch.poisson(torch.full((m,), mean, device="cuda"), generator=g).long()
        off = int(m * mean) - int(lens.sum())
        room = torch.nonzero(lens > 0).flatten() if off < 0 else torch.arange(m, device="cuda")
        pick = room[torch.randperm(room.numel(), device="cuda", generator=g)[:abs(off)]]
        lens[pick] += 1 if off > 0 else -1
        return lens
    if rows == "mesh":
        return 1 + torch.poisson(torch.full((m,), mean - 1.0, device="cuda"), generator=g).long()
    tail = 1.0 / (1.0 - torch.rand(m, dtype=torch.float64, device="cuda", generator=g))
    lo, hi = 0.5, float(mean)
    for _ in range(24):
        mid = 0.5 * (lo + hi)
        if float((mid * tail).floor().clamp(1, cap).mean()) < mean:
            lo = mid
        else:
            hi = mid
    lens = (lo * tail).floor().clamp(1, cap).long()
    lens[torch.randperm(m, device="cuda", generator=g)[: m // 100]] = 0
    return lens


def _row_ptr(lens):
    rp = torch.zeros(lens.numel() + 1, dtype=torch.int32, device="cuda")
    rp[1:] = torch.cumsum(lens, 0)
    return rp


def _columns(lens, k, g):
    """Uniform columns, increasing inside each row (a column may repeat, as in an assembled matrix; entries add up)."""
    nnz = int(lens.sum())
    base = torch.repeat_interleave(torch.arange(lens.numel(), device="cuda"), lens, output_size=nnz) * k
    key = base + torch.randint(k, (nnz,), device="cuda", generator=g)
    return (torch.sort(key)[0] - base).int()


def _graph(m, mean, g):
    """D^-1/2 (S + I) D^-1/2 of a Chung-Lu graph with m (mean - 1) / 2 edges: row_ptr, col_ind, float32 values.
    Twice as many pairs are drawn, since self-loops and repeated pairs are dropped."""
    edges = int((mean - 1.0) * m / 2)
    w = (1.0 - torch.rand(m, dtype=torch.float64, device="cuda", generator=g)) ** (-1.0 / 1.2)
    cdf = torch.cumsum(w, 0)
    cdf /= cdf[-1].clone()
    ends = torch.rand(2, 2 * edges, dtype=torch.float64, device="cuda", generator=g)
    ends = torch.searchsorted(cdf, ends).clamp_(max=m - 1)
    a, b = ends.min(0)[0], ends.max(0)[0]
    pairs = torch.unique((a * m + b)[a != b])
    pairs = pairs[torch.randperm(pairs.numel(), device="cuda", generator=g)[:edges]]
    a, b = pairs // m, pairs % m
    i = torch.arange(m, device="cuda")
    key = torch.sort(torch.cat([a * m + b, b * m + a, i * m + i]))[0]
    r, c = key // m, key % m
    deg = torch.bincount(r, minlength=m)
    return _row_ptr(deg), c.int(), (deg[r].double() * deg[c].double()).rsqrt().float()


def _matrix(case, g):
    """row_ptr, col_ind, float32 values of A."""
    if case["rows"] == "graph":
        return _graph(case["m"], case["mean"], g)
    lens = _lengths(case["rows"], case["m"], case["mean"], case.get("cap", 0), g)
    ci = _columns(lens, case["k"], g)
    return _row_ptr(lens), ci, torch.rand(ci.numel(), device="cuda", generator=g) * 2 - 1


def _normal(rows, cols, g):
    return torch.randn(rows, cols, device="cuda", generator=g)


def _batch_shapes(case):
    """Sizes spread evenly over the logarithm of m; mean lengths and widths in a fixed, unrelated order."""
    out = []
    for i in range(case["count"]):
        m = int(round(case["m_lo"] * (case["m_hi"] / case["m_lo"]) ** ((i + 0.5) / case["count"])))
        lam = case["mean_lo"] + (case["mean_hi"] - case["mean_lo"]) * ((i * 0.6180339887) % 1.0)
        out.append((m, lam, _BATCH_WIDTHS[i % 3]))
    return out


def _batch(case, seed):
    g = _gen(seed)
    out = []
    for m, lam, n in _batch_shapes(case):
        lens = torch.poisson(torch.full((m,), lam, device="cuda"), generator=g).long().clamp_(max=m)
        ci = _columns(lens, m, g)
        out.append((_row_ptr(lens), ci, torch.rand(ci.numel(), device="cuda", generator=g) * 2 - 1, _normal(m, n, g)))
    return out


def _inputs(case, seed):
    """Everything a case computes from, in storage types."""
    g = _gen(seed)
    rp, ci, v = _matrix(case, g)
    if case["form"] == "product":
        tv, tb, _ = (_TYPES[t] for t in case["types"].split("/"))
        return rp, ci, v.to(tv), _normal(case["k"], case["n"], g).to(tb)
    if case["form"] == "semiring":  # edge lengths and the distances known so far
        B = torch.rand(case["k"], case["n"], device="cuda", generator=g) * 100
        return rp, ci, v.abs() + 0.01, B
    return rp, ci, v, _normal(case["k"], case["n"], g), _normal(case["m"], case["n"], g)


def prepare(case, seed):
    form = case["form"]
    if form == "batched":
        mats = _batch(case, seed)
        rps, cis, vs, Bs = (list(x) for x in zip(*mats))
        C = torch.empty(sum(B.numel() for B in Bs), device="cuda")  # the results one after the other
        Cs = [c.view_as(B) for c, B in zip(C.split([B.numel() for B in Bs]), Bs)]
        plan = pkg.BatchedPlan(rps, cis, vs, Bs, Cs)
        plan.capture_graph()
        return dict(form=form, plan=plan, C=C)
    x = _inputs(case, seed)
    s = dict(form=form, rp=x[0], ci=x[1], v=x[2], B=x[3], nnz=x[1].numel(), shape=(case["m"], case["k"]))
    if form == "product":
        s["entry"], s["out"] = case["entry"], _TYPES[case["types"].split("/")[2]]
    if form in ("train", "sampled"):
        s["dY"] = x[4]
        s["v"].requires_grad_(True)
        s["B"].requires_grad_(True)
    if form == "train" or s.get("entry") == "matrix":
        s["A"] = pkg.CSRMatrix(s["rp"], s["ci"], s["shape"])
        s["A"].max_row  # measured once for a pattern that stays
        if form == "train":
            s["A"].transpose_pattern()
    return s


def _step(A, s):
    Y = pkg.spmm_autograd(A, s["v"], s["B"])
    dv, dB = torch.autograd.grad(Y, (s["v"], s["B"]), s["dY"])
    return [Y.detach(), dv, dB]


def run(s):
    form = s["form"]
    if form == "product":
        if s["entry"] == "plain":
            return pkg.spmm(s["rp"], s["ci"], s["v"], s["B"], out_dtype=s["out"], nnz=s["nnz"])
        return s["A"].spmm(s["v"], s["B"], out_dtype=s["out"])
    if form == "train":
        return _step(s["A"], s)
    if form == "sampled":
        return _step(pkg.CSRMatrix(s["rp"], s["ci"], s["shape"]), s)
    if form == "semiring":
        return pkg.semiring_spmm(s["rp"], s["ci"], s["v"], s["B"], "min_plus", nnz=s["nnz"])
    s["plan"].launch_graph()
    return s["C"]


# ----------------------------------------------------------------------------- what a pass cannot do without

def _bytes_flops(m, k, nnz, n, sv=4, sb=4, sc=4):
    return 4 * (m + 1) + nnz * (4 + sv) + min(k, nnz) * n * sb + m * n * sc, 2 * nnz * n


def work(case):
    if case["form"] == "batched":
        parts = [_bytes_flops(m, m, int(m * min(lam, m)), n) for m, lam, n in _batch_shapes(case)]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    m, k, n = case["m"], case["k"], case["n"]
    nnz = int(m * case["mean"])
    if case["form"] == "product":
        b, f = _bytes_flops(m, k, nnz, n, *(4 if t == "f32" else 2 for t in case["types"].split("/")))
        return {"bytes": b, "flops": f}
    b, f = _bytes_flops(m, k, nnz, n)
    if case["form"] in ("train", "sampled"):  # dY read, dvals and dB written as well; three products' worth of arithmetic
        b, f = b + 4 * m * n + 4 * nnz + 4 * k * n, 3 * f
    return {"bytes": b, "flops": f}


# ----------------------------------------------------------------------------- the same in 64 bits

def _csr64(rp, ci, v, shape):
    return torch.sparse_csr_tensor(rp, ci, v.double(), size=shape)


def _rows_of(rp):
    rp = rp.long()
    return torch.repeat_interleave(torch.arange(rp.numel() - 1, device="cuda"), rp[1:] - rp[:-1])


def exact(case, seed):
    with torch.no_grad():
        if case["form"] == "batched":
            return torch.cat([(_csr64(rp, ci, v, (B.shape[0],) * 2) @ B.double()).flatten()
                              for rp, ci, v, B in _batch(case, seed)])
        x = _inputs(case, seed)
        rp, ci, v, B = x[:4]
        m, k, n = case["m"], case["k"], case["n"]
        if case["form"] == "product":
            return _csr64(rp, ci, v, (m, k)) @ B.double()
        rows = _rows_of(rp)
        chunk = max(1, (1 << 26) // n)
        if case["form"] == "semiring":
            out = torch.full((m, n), math.inf, dtype=torch.float64, device="cuda")
            for p in range(0, ci.numel(), chunk):
                t = v[p:p + chunk, None].double() + B[ci[p:p + chunk].long()].double()
                out.scatter_reduce_(0, rows[p:p + chunk, None].expand_as(t), t, "amin")
            return out
        dY = x[4]
        Y = _csr64(rp, ci, v, (m, k)) @ B.double()
        by_column = torch.sort(ci.long() * m + rows)[1]
        rpt = _row_ptr(torch.bincount(ci.long(), minlength=k))
        dB = _csr64(rpt, rows[by_column].int(), v[by_column], (k, m)) @ dY.double()
        dv = torch.cat([(dY[rows[p:p + chunk]].double() * B[ci[p:p + chunk].long()].double()).sum(1)
                        for p in range(0, ci.numel(), chunk)])
        return [Y, dv, dB]
