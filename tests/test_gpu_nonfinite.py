"""Infinities and NaN in the operands: every pass, by every kind of kernel,
gives them where the float64 oracle does and nowhere else.  Rows of every length
around the index blocks of the passes (8 and 16 nonzeros), so that positions
past the end of a row run beside longer rows, with the non-finite elements in
the pass's local rows (A and the gradient rows over S, B over S^T).  The rows
beside them keep their bits."""
import numpy as np
import pytest
import torch

import oracle
from parity_utils import U32, deg_max, oracle_all
from paper_2203_07673_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

LENGTHS = tuple(range(0, 19)) + (31, 32, 33, 70)


def pattern():
    rng = np.random.default_rng(3)
    m = 7 * len(LENGTHS)
    deg = np.array([LENGTHS[i % len(LENGTHS)] for i in range(m)])
    rp = np.zeros(m + 1, np.int32)
    rp[1:] = np.cumsum(deg)
    return wl.CSR(m, 120, rp, rng.integers(0, 120, int(rp[-1])).astype(np.int32))


def spoil(x, rng):
    """A third of the rows get an infinity or a NaN."""
    x = x.copy()
    for i in rng.choice(len(x), len(x) // 3, replace=False):
        x[i, rng.integers(x.shape[1])] = rng.choice([np.inf, -np.inf, np.nan])
    return x


def check(name, got, ref, clean, terms):
    got = got.double().cpu().numpy()
    for kind in (np.isnan, np.isposinf, np.isneginf):
        assert np.array_equal(kind(got), kind(ref)), (name, kind.__name__)
    fin = np.isfinite(ref)
    assert np.all(np.abs(got[fin] - ref[fin]) <= (2 * terms * U32 * clean + 1e-30)[fin]), name


@pytest.mark.parametrize("side", ["rows", "columns"])
@pytest.mark.parametrize("r,dtype,variant", [
    *((r, d, 0) for r in (32, 64, 128, 256, 20, 520) for d in ("f32", "bf16")),
    *((64, d, v) for d in ("f32", "bf16") for v in (112, 122, 1041, 22212, 32212, 24221, 44041, 52212))])
def test_non_finite_operands(r, dtype, variant, side):
    from paper_2203_07673_gb300 import fmm
    rng = np.random.default_rng(r)
    S = pattern()
    n32 = lambda *s: rng.standard_normal(s).astype(np.float32)
    vals = rng.uniform(0.5, 1.5, S.nnz).astype(np.float32)
    A, B, G, Gn = n32(S.m, r), n32(S.n, r), n32(S.m, r), n32(S.n, r)
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    cu = lambda x: torch.from_numpy(x).cuda()
    plan = fmm.Plan(cu(S.row_ptr), cu(S.col_idx), S.n, r, dt, variant=variant)
    vt = cu(vals)

    def local_passes():
        """The output rows of the passes whose local rows are spoiled."""
        a, b = cu(A).to(dt), cu(B).to(dt)
        if side == "rows":
            return fmm.fusedmm(plan, vt, a, b), fmm.fusedmm_bwd(plan, vt, a, b, cu(G))[0]
        return fmm.fusedmm_t(plan, vt, a, b), fmm.fusedmm_t_bwd(plan, vt, a, b, cu(Gn))[1]
    before = local_passes()
    if side == "rows":
        A, G = spoil(A, rng), spoil(G, rng)
        same = np.isfinite(A).all(1) & np.isfinite(G).all(1)
    else:
        B, Gn = spoil(B, rng), spoil(Gn, rng)
        same = np.isfinite(B).all(1) & np.isfinite(Gn).all(1)
    assert same.sum() > 20
    for x, y in zip(local_passes(), before):
        assert torch.equal(x[cu(same)], y[cu(same)])
    At, Bt, Gt, Gnt = cu(A).to(dt), cu(B).to(dt), cu(G), cu(Gn)
    got = dict(fusedmm=fmm.fusedmm(plan, vt, At, Bt), fusedmm_t=fmm.fusedmm_t(plan, vt, At, Bt),
               sddmm=fmm.sddmm(plan, vt, At, Bt), bwd=fmm.fusedmm_bwd(plan, vt, At, Bt, Gt),
               t_bwd=fmm.fusedmm_t_bwd(plan, vt, At, Bt, Gnt))
    if variant == 0:
        got["noalloc"] = fmm.fusedmm_noalloc(plan.row_ptr, plan.col_idx, S.n, vt, At, Bt)
    if variant == 0 and r in (32, 64, 128, 256):
        it = dict(plan=plan, vals=vt, A=At, B=Bt, G=Gt, out=torch.empty(S.m, r, device="cuda"),
                  dA=torch.empty(S.m, r, device="cuda"), dB=torch.empty(S.n, r, device="cuda"),
                  ds=torch.empty(S.nnz, device="cuda"))
        batch = fmm.Batch([it])
        batch.forward()
        batch.backward()
        got["batch"], got["batch_bwd"] = it["out"], (it["dA"], it["dB"], it["ds"])
    A64, B64 = At.double().cpu().numpy(), Bt.double().cpu().numpy()
    size = lambda x: np.abs(np.where(np.isfinite(x), x, 0.0))
    with np.errstate(all="ignore"):
        ref = oracle_all(S, vals.astype(np.float64), A64, B64, G, Gn)
        mag = oracle_all(S, vals.astype(np.float64), size(A64), size(B64), size(G), size(Gn))
    for x in (ref, mag):
        x["noalloc"], x["batch"], x["batch_bwd"] = x["fusedmm"], x["fusedmm"], x["bwd"]
    terms = 2 * r + deg_max(S) + 4
    for name, x in got.items():
        pairs = zip(x, ref[name], mag[name]) if isinstance(x, tuple) else [(x, ref[name], mag[name])]
        for g, e, c in pairs:
            check(name, g, e, c, terms)
    assert np.isfinite(ref["fusedmm" if side == "rows" else "fusedmm_t"]).any(axis=1).mean() > 0.5
    plan.close()
