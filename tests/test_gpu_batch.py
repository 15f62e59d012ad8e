"""Batched persistent launch: every item against its own per-matrix calls
(bitwise, same kernel variants) and against the FP64 oracle; forward and
backward replayed from a CUDA graph."""
import numpy as np
import pytest
import torch

import oracle
from parity_utils import U32, relF
from paper_2203_07673_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def batch_codes(r, dtype):
    """Variant codes the batch kernels run in every role at width r (the
    rule of fmm_batch.cu: at most 32 floats live per lane in the forward
    phase, 48 in the backward phase)."""
    es = 4 if dtype == torch.float32 else 2
    vecs = r * es // 16
    base = max(1, vecs // 32)
    ok = []
    for code in (112, 114, 122, 212, 214, 221):
        V, N, U = (code // 100) * base, (code // 10) % 10, code % 10
        if vecs % V:
            continue
        g = vecs // V
        E = V * (16 // es)
        if g & (g - 1) or g * N > 32 or 32 % (g * N):
            continue
        if E * (U + 2) <= 32 and E * (2 * U + 2) <= 48 and E * (U + 3) <= 48:
            ok.append(code)
    return ok


def make_items(dtype, seed=0, count=10, variants=None):
    from paper_2203_07673_gb300 import fmm
    rng = np.random.default_rng(seed)
    specs = wl.batched_specs(count, seed_index=50 + seed, rows_lo=60, rows_hi=3000)
    items, host = [], []
    for t, sp in enumerate(specs):
        m = wl.batched_matrix(sp, t, seed_index=50 + seed)
        S, r = m["S"], m["r"]
        rp = torch.from_numpy(S.row_ptr).cuda()
        ci = torch.from_numpy(S.col_idx).cuda()
        plan = fmm.Plan(rp, ci, S.n, r, dtype, split_nnz=1 << 30)
        if variants is not None:
            codes = [c for c in variants if c in batch_codes(r, dtype)]
            plan.set_variant(codes[t % len(codes)], codes[(t + 1) % len(codes)])
        vals = torch.from_numpy(m["vals"]).cuda()
        A = torch.from_numpy(m["A"]).cuda().to(dtype).contiguous()
        B = torch.from_numpy(m["B"]).cuda().to(dtype).contiguous()
        G = torch.from_numpy(rng.standard_normal((S.m, r)).astype(np.float32)).cuda()
        items.append(dict(plan=plan, vals=vals, A=A, B=B, G=G,
                          out=torch.full((S.m, r), np.nan, device="cuda"),
                          dA=torch.full((S.m, r), np.nan, device="cuda"),
                          dB=torch.full((S.n, r), np.nan, device="cuda"),
                          ds=torch.full((S.nnz,), np.nan, device="cuda"),
                          rp=rp, ci=ci))
        host.append(m)
    return items, host


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
def test_batch_matches_per_matrix_calls_and_oracle(dtype):
    from paper_2203_07673_gb300 import fmm
    items, host = make_items(dtype, seed=1, variants=[112, 114, 122, 212, 214, 221])
    batch = fmm.Batch([{k: it[k] for k in ("plan", "vals", "A", "B", "out", "G", "dA", "dB", "ds")}
                       for it in items])
    batch.forward()
    batch.backward()
    torch.cuda.synchronize()
    for it, m in zip(items, host):
        p = it["plan"]
        # per-matrix calls with the same variants give the same bits
        # (only variants the batch kernels have were selected above)
        ref_out = fmm.fusedmm(p, it["vals"], it["A"], it["B"])
        dA, dB, ds = fmm.fusedmm_bwd(p, it["vals"], it["A"], it["B"], it["G"])
        torch.cuda.synchronize()
        assert torch.equal(it["out"], ref_out)
        assert torch.equal(it["dA"], dA) and torch.equal(it["dB"], dB) and torch.equal(it["ds"], ds)
        # and the oracle agrees
        S = m["S"]
        A64 = it["A"].double().cpu().numpy(); B64 = it["B"].double().cpu().numpy()
        G64 = it["G"].double().cpu().numpy(); s64 = m["vals"].astype(np.float64)
        exp = oracle.fusedmm(S.row_ptr, S.col_idx, s64, A64, B64, S.n)
        mag = oracle.fusedmm(S.row_ptr, S.col_idx, s64, np.abs(A64), np.abs(B64), S.n)
        deg = max(int(S.degrees().max()), int(np.bincount(S.col_idx, minlength=S.n).max()))
        got = it["out"].double().cpu().numpy()
        assert np.all(np.abs(got - exp) <= 2 * (m["r"] + deg + 4) * U32 * mag + 1e-30)
        assert relF(got, exp) <= 1e-5
        g = oracle.fusedmm_grad(S.row_ptr, S.col_idx, s64, A64, B64, G64, S.n)
        gm = oracle.fusedmm_grad(S.row_ptr, S.col_idx, s64, np.abs(A64), np.abs(B64),
                                 np.abs(G64), S.n)
        for name, x, e, mg in (("dA", it["dA"], g[0], gm[0]), ("dB", it["dB"], g[1], gm[1]),
                               ("ds", it["ds"], g[2], gm[2])):
            xx = x.double().cpu().numpy()
            assert np.all(np.abs(xx - e) <= 2 * (2 * m["r"] + deg + 4) * U32 * mg + 1e-30), name
            assert relF(xx, e) <= 1e-5, name
    batch.close()


def test_batch_cuda_graph_replay():
    from paper_2203_07673_gb300 import fmm
    items, _ = make_items(torch.bfloat16, seed=2, count=8)
    batch = fmm.Batch([{k: it[k] for k in ("plan", "vals", "A", "B", "out", "G", "dA", "dB", "ds")}
                       for it in items])
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        batch.forward(); batch.backward()          # warm-up outside the graph
    torch.cuda.current_stream().wait_stream(s)
    torch.cuda.synchronize()
    eager = [(it["out"].clone(), it["dA"].clone(), it["dB"].clone(), it["ds"].clone())
             for it in items]
    for it in items:
        for k in ("out", "dA", "dB", "ds"):
            it[k].fill_(float("nan"))
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        batch.forward()
        batch.backward()
    for _ in range(2):
        g.replay()
        torch.cuda.synchronize()
        for it, e in zip(items, eager):
            for k, x in zip(("out", "dA", "dB", "ds"), e):
                assert torch.equal(it[k], x), k
    batch.close()


def test_batch_rejects_split_rows_and_mixed_dtypes():
    from paper_2203_07673_gb300 import fmm
    rng = np.random.default_rng(0)
    S = wl.random_csr(50, 40, rng, mean_deg=3, hubs=((0, 600),))
    rp = torch.from_numpy(S.row_ptr).cuda(); ci = torch.from_numpy(S.col_idx).cuda()
    A = torch.randn(50, 32, device="cuda"); B = torch.randn(40, 32, device="cuda")
    out = torch.empty(50, 32, device="cuda")
    split = fmm.Plan(rp, ci, 40, 32, split_nnz=64)
    with pytest.raises(fmm.FmmError) as ei:
        fmm.Batch([dict(plan=split, A=A, B=B, out=out)])
    assert ei.value.status == fmm.FMM_EUNSUPPORTED
    p32 = fmm.Plan(rp, ci, 40, 32, split_nnz=1 << 30)
    p16 = fmm.Plan(rp, ci, 40, 32, torch.bfloat16, split_nnz=1 << 30)
    with pytest.raises(fmm.FmmError):
        fmm.Batch([dict(plan=p32, A=A, B=B, out=out),
                   dict(plan=p16, A=A.bfloat16(), B=B.bfloat16(), out=out)])
    # forward-only batch: backward is refused
    b = fmm.Batch([dict(plan=p32, A=A, B=B, out=out)])
    b.forward()
    with pytest.raises(fmm.FmmError):
        b.backward()
    torch.cuda.synchronize()
    assert relF(out.double().cpu().numpy(),
                oracle.fusedmm(S.row_ptr, S.col_idx, None, A.double().cpu().numpy(),
                               B.double().cpu().numpy(), 40)) <= 1e-5


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
@pytest.mark.parametrize("hub", [256, 257, 700, 5000])
def test_batch_cuts_long_rows(hub, dtype):
    """Rows and columns around and far above the default split size in a
    batch: plans that count as unsplit, chunks summed in the batch's own
    memory, one plan used by two items with different operands, each item
    bitwise its per-matrix call and within the rounding bound of the oracle."""
    from paper_2203_07673_gb300 import fmm
    rng = np.random.default_rng(hub)
    r = 64
    S = wl.random_csr(400, 300, rng, mean_deg=6, hubs=((0, hub), (399, hub), (7, 300)))
    S.col_idx[::3] = 11   # a hub column
    rp, ci = torch.from_numpy(S.row_ptr).cuda(), torch.from_numpy(S.col_idx).cuda()
    plan = fmm.Plan(rp, ci, S.n, r, dtype, split_nnz=1 << 30, variant=112)
    assert plan.info()["split_rows"] == 0 and plan.info()["split_cols"] == 0
    items = []
    for _ in range(2):
        f = lambda *s: torch.from_numpy(rng.standard_normal(s).astype(np.float32)).cuda()
        items.append(dict(plan=plan, vals=f(S.nnz).abs(), A=f(S.m, r).to(dtype),
                          B=f(S.n, r).to(dtype), G=f(S.m, r),
                          out=torch.full((S.m, r), np.nan, device="cuda"),
                          dA=torch.full((S.m, r), np.nan, device="cuda"),
                          dB=torch.full((S.n, r), np.nan, device="cuda"),
                          ds=torch.full((S.nnz,), np.nan, device="cuda")))
    batch = fmm.Batch(items)
    batch.forward()
    batch.backward()
    deg = max(int(S.degrees().max()), int(np.bincount(S.col_idx, minlength=S.n).max()))
    for it in items:
        assert torch.equal(it["out"], fmm.fusedmm(plan, it["vals"], it["A"], it["B"]))
        g = fmm.fusedmm_bwd(plan, it["vals"], it["A"], it["B"], it["G"])
        for k, x in zip(("dA", "dB", "ds"), g):
            assert torch.equal(it[k], x), k
        a, b, s, gg = (it[k].double().cpu().numpy() for k in ("A", "B", "vals", "G"))
        ref = [oracle.fusedmm(S.row_ptr, S.col_idx, s, a, b, S.n),
               *oracle.fusedmm_grad(S.row_ptr, S.col_idx, s, a, b, gg, S.n)]
        mag = [oracle.fusedmm(S.row_ptr, S.col_idx, s, abs(a), abs(b), S.n),
               *oracle.fusedmm_grad(S.row_ptr, S.col_idx, s, abs(a), abs(b), abs(gg), S.n)]
        for k, x, m in zip(("out", "dA", "dB", "ds"), ref, mag):
            err = np.abs(it[k].double().cpu().numpy() - x)
            assert np.all(err <= 2 * (2 * r + deg + 4) * U32 * m + 1e-30), k
    batch.close()


@pytest.mark.parametrize("offset", [0, 8])
@pytest.mark.parametrize("r", [32, 64, 128, 256])
def test_batch_of_default_bfloat16_plans(r, offset):
    """bfloat16 plans left to their own choice run the register-ring layouts in
    the batch: bitwise the per-matrix calls with those layouts set (the call
    of a plan left to its own choice may run its long rows a warp each)
    where every operand is 32-byte aligned; operands 16 bytes further on
    (offset 8) take the team kernel.
    Either way within the rounding bound of the oracle; forward and backward
    twice, a matrix without nonzeros and one of a single row among them."""
    from paper_2203_07673_gb300 import fmm
    rng = np.random.default_rng(r + offset)
    items, host = [], []
    for m, n, deg in ((300, 250, 9.0), (1, 40, 30.0), (50, 60, 0.0), (700, 90, 3.0)):
        S = wl.random_csr(m, n, rng, mean_deg=deg, hubs=((0, 400),) if m == 700 else ())
        f = lambda *s: torch.from_numpy(rng.standard_normal(s).astype(np.float32)).cuda()

        def rows(k):
            buf = torch.empty(k * r + offset, dtype=torch.bfloat16, device="cuda")
            buf[offset:] = f(k * r).bfloat16()
            return buf[offset:].view(k, r)
        plan = fmm.Plan(torch.from_numpy(S.row_ptr).cuda(), torch.from_numpy(S.col_idx).cuda(), n, r,
                        torch.bfloat16, split_nnz=1 << 30)
        items.append(dict(plan=plan, vals=f(S.nnz), A=rows(m), B=rows(n), G=f(m, r),
                          out=torch.empty(m, r, device="cuda"), dA=torch.empty(m, r, device="cuda"),
                          dB=torch.empty(n, r, device="cuda"), ds=torch.empty(S.nnz, device="cuda")))
        host.append(S)
    batch = fmm.Batch(items)
    for _ in range(2):
        for it in items:
            for k in ("out", "dA", "dB", "ds"):
                it[k].fill_(float("nan"))
        batch.forward()
        batch.backward()
    for it, S in zip(items, host):
        p = it["plan"]
        p.set_variant(32412, 112 if r == 32 else 0)
        want = (fmm.fusedmm(p, it["vals"], it["A"], it["B"]),
                *fmm.fusedmm_bwd(p, it["vals"], it["A"], it["B"], it["G"]))
        a, b, s, g = (it[k].double().cpu().numpy() for k in ("A", "B", "vals", "G"))
        ref = [oracle.fusedmm(S.row_ptr, S.col_idx, s, a, b, S.n),
               *oracle.fusedmm_grad(S.row_ptr, S.col_idx, s, a, b, g, S.n)]
        mag = [oracle.fusedmm(S.row_ptr, S.col_idx, abs(s), abs(a), abs(b), S.n),
               *oracle.fusedmm_grad(S.row_ptr, S.col_idx, abs(s), abs(a), abs(b), abs(g), S.n)]
        deg = max(int(S.degrees().max()), int(np.bincount(S.col_idx, minlength=S.n).max()))
        for k, w, x, m in zip(("out", "dA", "dB", "ds"), want, ref, mag):
            if offset == 0:
                assert torch.equal(it[k], w), k
            err = np.abs(it[k].double().cpu().numpy() - x)
            assert np.all(err <= 2 * (2 * r + deg + 4) * U32 * m + 1e-30), k
    batch.close()


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
def test_split_nnz_and_what_the_info_says(dtype):
    """split_nnz up to nnz is the caller's: rows whole from the longest on, cut
    below it, whatever the default; above nnz it sets no limit, and the info
    tells the chunks and their size."""
    from paper_2203_07673_gb300 import fmm
    rng = np.random.default_rng(5)
    S = wl.random_csr(300, 250, rng, mean_deg=5, hubs=((0, 900), (5, 400)))
    longest = max(int(S.degrees().max()), int(np.bincount(S.col_idx, minlength=S.n).max()))
    deg, cdeg = S.degrees(), np.bincount(S.col_idx, minlength=S.n)
    rp, ci = torch.from_numpy(S.row_ptr).cuda(), torch.from_numpy(S.col_idx).cuda()
    f = lambda *s: torch.from_numpy(rng.standard_normal(s).astype(np.float32)).cuda()
    A, B, out = f(S.m, 64).to(dtype), f(S.n, 64).to(dtype), torch.empty(S.m, 64, device="cuda")
    chunks = lambda d, k: int(np.ceil(d[d > k] / k).sum())
    for split, size in ((longest - 1, longest - 1), (longest, None), (S.nnz, None),
                        (S.nnz + 1, 256), (1 << 30, 256)):
        plan = fmm.Plan(rp, ci, S.n, 64, dtype, split_nnz=split)
        i = plan.info()
        if size is None:
            assert i["split_rows"] == i["split_cols"] == i["row_chunks"] == i["col_chunks"] == 0
        else:
            assert i["split_nnz"] == size
            assert (i["row_chunks"], i["col_chunks"]) == (chunks(deg, size), chunks(cdeg, size))
            assert i["split_rows"] == ((deg > size).sum() if split <= S.nnz else 0)
        item = dict(plan=plan, A=A, B=B, out=out)
        if split == longest - 1:
            with pytest.raises(fmm.FmmError):
                fmm.Batch([item])
            continue
        batch = fmm.Batch([item])
        batch.forward()
        assert relF(out.double().cpu().numpy(),
                    oracle.fusedmm(S.row_ptr, S.col_idx, None, A.double().cpu().numpy(),
                                   B.double().cpu().numpy(), S.n)) <= 1e-5
        batch.close()


@pytest.mark.parametrize("dtype,offset", [(torch.float32, 0), (torch.float32, 4), (torch.bfloat16, 0),
                                          (torch.bfloat16, 8)])
@pytest.mark.parametrize("r", [32, 64, 128, 256])
def test_batch_of_untouched_plans(r, dtype, offset):
    """Plans left to their own choice: a batch gives the bits of their own
    calls, which take other passes where the pattern asks for them (rows of
    their own warp, rows in chunks), also with operands that are 16-byte but not
    32-byte aligned (offset)."""
    from paper_2203_07673_gb300 import fmm
    rng = np.random.default_rng(r + offset)
    f = lambda *s: torch.from_numpy(rng.standard_normal(s).astype(np.float32)).cuda()

    def rows(k):
        buf = torch.zeros(k * r + offset, dtype=dtype, device="cuda")
        buf[offset:] = f(k * r).to(dtype)
        return buf[offset:].view(k, r)
    items = []
    for m, n, deg, hubs in ((300, 250, 9.0, ()), (1, 40, 30.0, ()), (700, 90, 3.0, ((0, 400), (9, 47))),
                            (9000, 5000, 12.0, ((3, 255), (4000, 48))), (40, 3000, 20.0, ((7, 3000),))):
        S = wl.random_csr(m, n, rng, mean_deg=deg, empty_frac=0.1, hubs=hubs)
        for split in (1 << 30, max(1, int(S.degrees().max()), int(np.bincount(S.col_idx, minlength=n).max()))):
            plan = fmm.Plan(torch.from_numpy(S.row_ptr).cuda(), torch.from_numpy(S.col_idx).cuda(), n,
                            r, dtype, split_nnz=split)
            items.append(dict(plan=plan, vals=f(S.nnz), A=rows(m), B=rows(n), G=f(m, r),
                              out=torch.empty(m, r, device="cuda"), dA=torch.empty(m, r, device="cuda"),
                              dB=torch.empty(n, r, device="cuda"), ds=torch.empty(S.nnz, device="cuda")))
    batch = fmm.Batch(items)
    batch.forward()
    batch.backward()
    for k, it in enumerate(items):
        p = it["plan"]
        want = (fmm.fusedmm(p, it["vals"], it["A"], it["B"]),
                *fmm.fusedmm_bwd(p, it["vals"], it["A"], it["B"], it["G"]))
        for name, w in zip(("out", "dA", "dB", "ds"), want):
            assert torch.equal(it[name], w), (k, name)
    batch.close()


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
def test_batch_with_empty_matrices(dtype):
    """Matrices without rows, without columns and without either beside others:
    their outputs are zeros or nothing, the others those of their own calls, and
    a matrix without columns whose dB is given has an adjoint."""
    import ctypes
    from paper_2203_07673_gb300 import fmm
    rng = np.random.default_rng(2)
    r = 32
    f = lambda *s: torch.from_numpy(rng.standard_normal(s).astype(np.float32)).cuda()
    items = []
    for m, n, deg in ((0, 50, 0.0), (40, 30, 4.0), (30, 0, 0.0), (0, 0, 0.0)):
        S = wl.random_csr(m, n, rng, mean_deg=deg) if deg else wl.CSR(
            m, n, np.zeros(m + 1, np.int32), np.zeros(0, np.int32))
        plan = fmm.Plan(torch.from_numpy(S.row_ptr).cuda(), torch.from_numpy(S.col_idx).cuda(), n, r,
                        dtype, split_nnz=1 << 30)
        items.append(dict(plan=plan, vals=f(S.nnz), A=f(m, r).to(dtype), B=f(n, r).to(dtype), G=f(m, r),
                          out=torch.full((m, r), np.nan, device="cuda"),
                          dA=torch.full((m, r), np.nan, device="cuda")))
    batch = fmm.Batch(items)
    batch.forward()
    for it in items:
        assert torch.equal(it["out"], fmm.fusedmm(it["plan"], it["vals"], it["A"], it["B"]))
    batch.close()
    it, spare = items[2], torch.zeros(4 * r, device="cuda")
    ptr = lambda t: t.data_ptr()
    arr = (fmm._BatchItem * 1)(fmm._BatchItem(it["plan"].handle, None, ptr(it["A"]), None, ptr(it["out"]),
                                              ptr(it["G"]), ptr(it["dA"]), ptr(spare), None))
    out = ctypes.c_void_p()
    assert fmm.lib().fmm_batch_create(arr, 1, fmm._stream(), ctypes.byref(out)) == fmm.FMM_OK
    it["out"].fill_(float("nan"))
    for call in (fmm.lib().fmm_batch_forward, fmm.lib().fmm_batch_backward):
        assert call(out, fmm._stream()) == fmm.FMM_OK
    torch.cuda.synchronize()
    assert not it["out"].any() and not it["dA"].any() and not spare.any()
    assert fmm.lib().fmm_batch_destroy(out) == fmm.FMM_OK
