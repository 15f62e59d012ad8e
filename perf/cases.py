"""Performance cases of the library's public entry points.

``listed()`` names the cases, ``draw(rng)`` gives further ones of the same
ranges, ``prepare(case, seed)`` makes what a program holds before the call
(pattern, plan, operands, all on the GPU and from the seed alone),
``run(state)`` is one pass through the public calls, ``work(case)`` the bytes
and operations the pass cannot do without, and ``exact(case, seed)`` the same
outputs in float64 by plain torch.

A case is a flat dict:
  op       what is called (see ``run``)
  pattern  er (exactly ``deg`` distinct columns per row), rmat (power-law
           graph, ``deg`` edge draws per vertex), zipf (Zipf(1.2) row lengths
           of mean ``deg``), ragged (a fifth of the rows empty, exponential
           row lengths, a few hub rows, unsorted and repeated columns)
  m, n     rows and columns of S        deg   mean nonzeros per row
  r        dense width                  dtype f32 or bf16 (dense operands)
  vals     whether S has values (else every value is 1)
and, per op, heads (gat), iters (als), transpose (train), count, rows_lo,
rows_hi and specs (batch: how many matrices, their row range, and which
draw of the sizes).
"""
import math

import torch

from paper_2203_07673_gb300 import als, autograd, fmm
from paper_2203_07673_gb300 import workloads as wl

DEV = "cuda"
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}
ALS_LAMBDA = 0.1
GAT_SLOPE = 0.2


def _case(name, op, pattern, m, n, deg, r, dtype, vals=True, **more):
    c = dict(op=op, pattern=pattern, m=m, n=n, deg=deg, r=r, dtype=dtype, vals=vals, **more)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one small FusedMMA call (the smallest configuration of the
        # benchmark): what a caller pays per call
        _case("small forward", "forward", "er", 4096, 4096, 32, 32, "f32"),
        # a training step on one small sampled subgraph, rectangular and of odd
        # sizes: launches and host time of forward and backward together
        _case("small training", "train", "er", 3001, 2003, 16, 64, "bf16", transpose=False),
        # a training step on a mid-size graph, float32
        _case("mid training", "train", "rmat", 1 << 17, 1 << 17, 16, 128, "f32",
              transpose=False),
        # Erdos-Renyi with both products (the benchmark's default step)
        _case("large both products", "both", "er", 1 << 20, 1 << 20, 32, 128, "f32"),
        # power-law graph, bfloat16 training step (s = 1)
        _case("large training", "train", "rmat", 1 << 22, 1 << 22, 16, 64, "bf16", False,
              transpose=False),
        # rectangular ratings-shaped matrix, both products in bfloat16
        _case("ratings both products", "both", "zipf", 1 << 21, 1 << 19, 38, 64, "bf16"),
        # an ALS sweep on a ratings-shaped matrix
        _case("als sweep", "als", "zipf", 1 << 19, 1 << 17, 38, 64, "f32", iters=5),
        # graph attention over a power-law graph, 4 heads of 32
        _case("attention", "gat", "rmat", 1 << 20, 1 << 20, 16, 128, "f32", False, heads=4),
        # a width that is no power of two, irregular rows, odd sizes: training
        _case("ragged width training", "train", "ragged", 60013, 41999, 20, 100, "f32",
              transpose=False),
        # SDDMM, SpMM and its transpose as separate calls
        _case("separate calls", "unfused", "er", 1 << 17, 1 << 17, 16, 256, "f32"),
        # FusedMMA without a plan, for callers that may not allocate
        _case("without a plan", "noalloc", "zipf", 200003, 100003, 24, 128, "bf16"),
        # many uneven matrices in one launch per phase, forward and backward
        _case("batch", "batch", "mixed", 0, 0, 0, 0, "bf16", count=64, rows_lo=1000,
              rows_hi=200000, specs=5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["forward", "both", "train", "train", "unfused", "noalloc", "als", "gat",
                     "batch"])
    dtype = rng.choice(["f32", "bf16"])
    if op == "batch":
        return _case(None, op, "mixed", 0, 0, 0, 0, dtype, count=_log_int(rng, 4, 48),
                     rows_lo=1000, rows_hi=_log_int(rng, 4000, 60000),
                     specs=rng.randrange(6, 1000))
    # widths: the benchmark's powers of two, or any other
    r = rng.choice([32, 64, 128, 256]) if rng.random() < 0.7 else _log_int(rng, 8, 300)
    more = {}
    if op == "als":
        dtype, more = "f32", dict(iters=rng.randrange(2, 6))
    elif op == "gat":
        more = dict(heads=rng.choice([h for h in (1, 2, 4, 8) if r % h == 0]))
    elif op == "train":
        more = dict(transpose=rng.random() < 0.25)
    pattern = rng.choice(["er", "rmat", "zipf", "ragged"])
    if op == "als":
        pattern = rng.choice(["er", "zipf"])
    m = _log_int(rng, 300, 1 << 20)
    n = {"er": m, "rmat": m, "zipf": max(75, m // 4)}.get(pattern) or _log_int(rng, 300, 1 << 19)
    if pattern == "er" and rng.random() < 0.3:
        n = _log_int(rng, 300, 1 << 20)
    deg = _log_int(rng, 4, 64)
    deg = max(2, min(deg, int(math.sqrt(2 * n)) if pattern == "er" else n // 16))
    # the cost of a drawn case stays below that of the largest listed ones
    most = {"als": 1.2e8}.get(op, 1e9) / (1 if r in (32, 64, 128, 256) else 6)
    while m * deg * r > most and m > 300:
        m = m * 2 // 3
        if pattern == "rmat":
            n = m
    return _case(None, op, pattern, m, n, deg, r, dtype, op == "als" or rng.random() < 0.7, **more)


# ------------------------------------------------------------------ inputs

def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1000003 + stream)
    return g


def _ragged(m, n, deg, g):
    u = torch.rand(m, generator=g, device=DEV)
    d = torch.round(-torch.log1p(-u) * (deg / 0.8)).long()
    d[torch.rand(m, generator=g, device=DEV) < 0.2] = 0
    hubs = torch.randint(0, m, (max(1, m // 10000),), generator=g, device=DEV)
    d[hubs] = min(60 * deg, n)
    row_ptr = torch.zeros(m + 1, dtype=torch.int64, device=DEV)
    row_ptr[1:] = torch.cumsum(d, 0)
    cols = torch.randint(0, n, (int(row_ptr[-1]),), generator=g, device=DEV)
    return row_ptr.int(), cols.int()


def _relabel(rp, ci, n, g, ordered):
    """The pattern under a random relabeling of its rows and columns: other
    positions, as many nonzeros.  Columns stay sorted within rows if they
    were (``ordered``)."""
    m = rp.numel() - 1
    rows = torch.randperm(m, generator=g, device=DEV)[_rows_of(rp)]
    cols = torch.randperm(n, generator=g, device=DEV)[ci.long()]
    if ordered:
        keys = torch.sort(rows * n + cols).values
        rows, cols = keys // n, keys % n
    else:
        rows, order = torch.sort(rows, stable=True)
        cols = cols[order]
    row_ptr = torch.zeros(m + 1, dtype=torch.int64, device=DEV)
    row_ptr[1:] = torch.cumsum(torch.bincount(rows, minlength=m), 0)
    return row_ptr.int(), cols.int()


def _pattern(kind, m, n, deg, seed, t=0):
    """Pattern t of a seed (row_ptr, col_idx).  Patterns whose number of
    nonzeros is random are drawn once and relabeled by the seed, so that all
    seeds have it alike."""
    if kind == "er":
        return wl.er_exact_degree_torch(m, n, deg, _gen(seed, 64 * t), DEV)
    g = _gen(7, 64 * t)
    if kind == "rmat":
        scale = max(1, math.ceil(math.log2(m)))
        rp, ci = wl.rmat_torch(scale, m * deg, 0.57, 0.19, 0.19, g, DEV, m)
    elif kind == "zipf":
        rp, ci = wl.zipf_rows_torch(m, n, m * deg, 1.2, min(4096, max(2, n // 8)), g, DEV)
    else:
        rp, ci = _ragged(m, n, deg, g)
    return _relabel(rp, ci, n, _gen(seed, 64 * t), kind != "ragged")


def _normal(rows, r, variance, seed, stream):
    return torch.randn(rows, r, generator=_gen(seed, stream), device=DEV) * math.sqrt(variance)


def _inputs(c, seed):
    """Pattern and operands of a single-matrix case (A, B in the case's
    dtype; variance 1/r, as in the benchmark's float32 workloads)."""
    m, n, r, dt, op = c["m"], c["n"], c["r"], DTYPES[c["dtype"]], c["op"]
    rp, ci = _pattern(c["pattern"], m, n, c["deg"], seed)
    x = dict(rp=rp, ci=ci)
    if c["vals"]:
        x["vals"] = torch.rand(ci.numel(), generator=_gen(seed, 1), device=DEV)
    if op == "als":
        # ratings 1, 1.5, ..., 5
        x["vals"] = torch.round((x["vals"] * 4 + 1) * 2) / 2
    if op == "gat":
        x["H"] = _normal(n, r, 1.0, seed, 2)
        x["X"] = x["H"] if m == n else _normal(m, r, 1.0, seed, 3)
        x["a_l"] = _normal(1, r, 1.0 / r, seed, 4).reshape(r)
        x["a_r"] = _normal(1, r, 1.0 / r, seed, 5).reshape(r)
        x["Hp"] = x["H"].to(dt)
        return x
    var = 0.1 if op == "als" else 1.0 / r
    x["A"], x["B"] = _normal(m, r, var, seed, 2).to(dt), _normal(n, r, var, seed, 3).to(dt)
    if op == "train":
        x["G"] = _normal(n if c["transpose"] else m, r, 1.0, seed, 4)
    return x


def _batch_inputs(c, seed):
    specs = wl.batched_specs(c["count"], c["specs"], c["rows_lo"], c["rows_hi"])
    items, dt = [], DTYPES[c["dtype"]]
    for t, sp in enumerate(specs):
        m, r, k = sp["rows"], sp["r"], 64 * t
        rp, ci = _pattern(sp["kind"], m, m, sp["deg"], seed, t)
        items.append(dict(rp=rp, ci=ci, m=m, n=m, r=r,
                          vals=torch.rand(ci.numel(), generator=_gen(seed, k + 1), device=DEV),
                          A=_normal(m, r, 1.0 / r, seed, k + 2).to(dt),
                          B=_normal(m, r, 1.0 / r, seed, k + 3).to(dt),
                          G=_normal(m, r, 1.0, seed, k + 4)))
    return items


def prepare(case, seed):
    c = case
    st = dict(case=c)
    if c["op"] == "batch":
        xs = _batch_inputs(c, seed)
        # the outputs of all matrices end to end in one buffer each
        size = dict(out=[x["m"] * x["r"] for x in xs], dA=[x["m"] * x["r"] for x in xs],
                    dB=[x["n"] * x["r"] for x in xs], ds=[x["ci"].numel() for x in xs])
        st["outputs"] = {k: torch.empty(sum(v), device=DEV) for k, v in size.items()}
        part = {k: torch.split(st["outputs"][k], v) for k, v in size.items()}
        items = []
        for t, x in enumerate(xs):
            plan = fmm.Plan(x["rp"], x["ci"], x["n"], x["r"], DTYPES[c["dtype"]],
                            split_nnz=1 << 30)
            items.append(dict(plan=plan, vals=x["vals"], A=x["A"], B=x["B"], G=x["G"],
                              out=part["out"][t].view(x["m"], x["r"]),
                              dA=part["dA"][t].view(x["m"], x["r"]),
                              dB=part["dB"][t].view(x["n"], x["r"]), ds=part["ds"][t]))
        st["batch"] = fmm.Batch(items)
        return st
    x = _inputs(c, seed)
    st.update(x)
    st.setdefault("vals", None)
    if c["op"] != "noalloc":
        st["plan"] = fmm.Plan(x["rp"], x["ci"], c["n"], c["r"], DTYPES[c["dtype"]])
    if c["op"] == "als":
        st["solver"] = als.ALS(st["plan"], st["vals"], x["A"], x["B"], ALS_LAMBDA)
    if c["op"] == "train":
        st["leaves"] = [st[k].requires_grad_(True) for k in ("vals", "A", "B")
                        if st[k] is not None]
    return st


# --------------------------------------------------------------------- run

def run(state):
    s, c = state, state["case"]
    op = c["op"]
    if op == "batch":
        s["batch"].forward()
        s["batch"].backward()
        return s["outputs"]
    if op == "forward":
        return fmm.fusedmm(s["plan"], s["vals"], s["A"], s["B"])
    if op == "both":
        return (fmm.fusedmm(s["plan"], s["vals"], s["A"], s["B"]),
                fmm.fusedmm_t(s["plan"], s["vals"], s["A"], s["B"]))
    if op == "train":
        out = autograd.fusedmm(s["plan"], s["vals"], s["A"], s["B"], transpose=c["transpose"])
        return [out.detach(), *torch.autograd.grad(out, s["leaves"], s["G"])]
    if op == "unfused":
        v = fmm.sddmm(s["plan"], s["vals"], s["A"], s["B"])
        return v, fmm.spmm(s["plan"], v, s["B"]), fmm.spmm_t(s["plan"], v, s["A"])
    if op == "noalloc":
        return fmm.fusedmm_noalloc(s["rp"], s["ci"], c["n"], s["vals"], s["A"], s["B"])
    if op == "als":
        s["solver"].sweep(c["iters"])
        return s["solver"].A, s["solver"].B
    f = fmm.gat_project(s["X"], s["a_l"], c["heads"])
    g = fmm.gat_project(s["H"], s["a_r"], c["heads"])
    return f, g, fmm.gat_forward(s["plan"], c["heads"], s["vals"], f, g, s["Hp"], GAT_SLOPE)


# -------------------------------------------------------------------- work

def _work_one(op, m, n, nnz, r, e, vals, heads=1, iters=0, transpose=False):
    pat = 4 * (m + 1) + 4 * nnz + (4 * nnz if vals else 0)
    ab = (m + n) * r * e
    if op in ("forward", "noalloc"):
        return pat + ab + 4 * m * r, 4 * nnz * r
    if op == "both":
        return pat + ab + 4 * (m + n) * r, 8 * nnz * r
    if op == "train":
        k = n if transpose else m
        return pat + ab + 8 * k * r + ab + (4 * nnz if vals else 0), 14 * nnz * r
    if op == "unfused":
        return pat + ab + 4 * nnz + 4 * (m + n) * r, 6 * nnz * r
    if op == "gat":
        return (pat + 4 * n * r + (4 * m * r if m != n else 0) + (n * r * e if e == 2 else 0)
                + 4 * (m + n) * heads + 4 * m * r), 2 * nnz * r + 2 * (m + n) * r
    # als: both factors read and written once
    return pat + 2 * ab, (iters + 2) * 2 * 4 * nnz * r


def work(case):
    c = case
    e = 4 if c["dtype"] == "f32" else 2
    if c["op"] == "batch":
        b = f = 0
        for sp in wl.batched_specs(c["count"], c["specs"], c["rows_lo"], c["rows_hi"]):
            m, nnz, r = sp["rows"], sp["rows"] * sp["deg"], sp["r"]
            b += 4 * (m + 1) + 8 * nnz + 2 * m * r * e + 4 * m * r + 12 * m * r + 4 * nnz
            f += 14 * nnz * r
        return {"bytes": b, "flops": f}
    b, f = _work_one(c["op"], c["m"], c["n"], c["m"] * c["deg"], c["r"], e, c["vals"],
                     c.get("heads", 1), c.get("iters", 0), c.get("transpose", False))
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------- exact

def _rows_of(rp):
    d = (rp[1:] - rp[:-1]).long()
    return torch.repeat_interleave(torch.arange(d.numel(), device=DEV), d)


def _blocks(nnz, r):
    step = max(1, (1 << 27) // max(1, r))
    for p in range(0, nnz, step):
        yield slice(p, min(nnz, p + step))


def _dots(i, j, A, B, s):
    """s * <A_i, B_j> of every nonzero, float64."""
    v = torch.empty(i.numel(), dtype=torch.float64, device=DEV)
    for b in _blocks(i.numel(), A.shape[1]):
        v[b] = (A[i[b]].double() * B[j[b]].double()).sum(1)
    return v if s is None else v * s.double()


def _gather_sum(rows, to, frm, w, X):
    """out[to] += w X[frm], float64."""
    out = torch.zeros(rows, X.shape[1], dtype=torch.float64, device=DEV)
    for b in _blocks(to.numel(), X.shape[1]):
        out.index_add_(0, to[b], X[frm[b]].double() * w[b, None])
    return out


def _train_exact(i, j, m, n, s, A, B, G, transpose):
    if transpose:   # FusedMMB is FusedMMA with the roles of A and B exchanged
        *first, dB, dA = _train_exact(j, i, n, m, s, B, A, G, False)
        return [*first, dA, dB]
    d, w = _dots(i, j, A, B, None), _dots(i, j, G, B, None)
    sd, sw = (d, w) if s is None else (d * s.double(), w * s.double())
    out = _gather_sum(m, i, j, sd, B)
    dA = _gather_sum(m, i, j, sw, B)
    dB = _gather_sum(n, j, i, sd, G) + _gather_sum(n, j, i, sw, A)
    return [out] + ([d * w] if s is not None else []) + [dA, dB]


def _als_exact(i, j, c, A, B, lam, iters):
    A, B = A.double(), B.double()

    def side(X, Y, to, frm):
        b = _gather_sum(X.shape[0], to, frm, c.double(), Y)

        def query(P):
            return _gather_sum(X.shape[0], to, frm, _dots(to, frm, P, Y, None), Y) + lam * P
        res = b - query(X)
        p, rs = res.clone(), (res * res).sum(1)
        for _ in range(iters):
            t = query(p)
            pt = (p * t).sum(1)
            alpha = torch.where(pt > 0, rs / pt, torch.zeros_like(pt))
            X = X + alpha[:, None] * p
            res = res - alpha[:, None] * t
            new = (res * res).sum(1)
            beta = torch.where(rs > 0, new / rs, torch.zeros_like(rs))
            p, rs = res + beta[:, None] * p, new
        return X
    A = side(A, B, i, j)
    return A, side(B, A, j, i)


def _gat_exact(i, j, m, x, heads):
    r = x["H"].shape[1]
    rh = r // heads
    f = (x["X"].double() * x["a_l"].double()).reshape(-1, heads, rh).sum(2)
    g = (x["H"].double() * x["a_r"].double()).reshape(-1, heads, rh).sum(2)
    e = f[i] + g[j]
    if x.get("vals") is not None:
        e = e * x["vals"].double()[:, None]
    e = torch.where(e > 0, e, GAT_SLOPE * e)
    at = i[:, None].expand(-1, heads)
    top = torch.full((m, heads), -math.inf, dtype=torch.float64, device=DEV)
    top.scatter_reduce_(0, at, e, "amax")
    w = torch.exp(e - top[i])
    total = torch.zeros(m, heads, dtype=torch.float64, device=DEV).index_add_(0, i, w)
    w = w / total[i]
    out = torch.cat([_gather_sum(m, i, j, w[:, h].contiguous(),
                                 x["Hp"][:, h * rh:(h + 1) * rh].contiguous())
                     for h in range(heads)], 1)
    return f, g, out


def exact(case, seed):
    c = case
    if c["op"] == "batch":
        parts = []
        for x in _batch_inputs(c, seed):
            i, j = _rows_of(x["rp"]), x["ci"].long()
            parts.append(_train_exact(i, j, x["m"], x["n"], x["vals"], x["A"], x["B"], x["G"],
                                      False))
        return {k: torch.cat([p[q].reshape(-1) for p in parts])
                for k, q in (("out", 0), ("ds", 1), ("dA", 2), ("dB", 3))}
    x = _inputs(c, seed)
    m, n, s, op = c["m"], c["n"], x.get("vals"), c["op"]
    i, j = _rows_of(x["rp"]), x["ci"].long()
    if op == "gat":
        return _gat_exact(i, j, m, x, c["heads"])
    if op == "als":
        return _als_exact(i, j, s, x["A"], x["B"], ALS_LAMBDA, c["iters"])
    A, B = x["A"], x["B"]
    if op == "train":
        return _train_exact(i, j, m, n, s, A, B, x["G"], c["transpose"])
    v = _dots(i, j, A, B, s)
    out = _gather_sum(m, i, j, v, B)
    if op in ("forward", "noalloc"):
        return out
    out_t = _gather_sum(n, j, i, v, A)
    return (out, out_t) if op == "both" else (v, out, out_t)
