"""The pass with a warp per long row, at the edges of its choices: rows of
every length around its steps (8 nonzeros), its two lines (8 and 48) and a
chunk, few rows and many, both dtypes and every role, each within the float32
rounding bound of the FP64 oracle; float32 FusedMM and SpMM bit for bit the
team pass, accumulating calls among them."""
import numpy as np
import pytest
import torch

from paper_2203_07673_gb300 import workloads as wl
from test_gpu_parity import run_all

pytestmark = pytest.mark.gpu

LENGTHS = (0, 1, 2, 7, 8, 9, 15, 16, 17, 47, 48, 49, 63, 64, 65, 127, 255, 256, 257, 600)


def ladder(m, n, seed):
    """Rows of LENGTHS at odd places among m rows of 3 on average."""
    rng = np.random.default_rng(seed)
    hubs = tuple((i * (m // len(LENGTHS)), d) for i, d in enumerate(LENGTHS))
    return wl.random_csr(m, n, rng, mean_deg=3, empty_frac=0.1, dup_frac=0.05, hubs=hubs)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
@pytest.mark.parametrize("r", [32, 64, 128, 256])
@pytest.mark.parametrize("m", [20, 3000, 9000])
def test_rows_by_warps(m, r, dtype):
    run_all(ladder(m, 700, m + r), {}, r, dtype, seed=r)


@pytest.mark.parametrize("r,code", [(32, 212), (64, 212), (128, 212), (128, 1042), (256, 112)])
@pytest.mark.parametrize("m", [20, 3000, 9000])
def test_float32_order(m, r, code):
    from paper_2203_07673_gb300 import fmm
    S = ladder(m, 700, m + 1)
    rng = np.random.default_rng(r)
    f = lambda *s: torch.from_numpy(rng.standard_normal(s).astype(np.float32)).cuda()
    rp, ci = torch.from_numpy(S.row_ptr).cuda(), torch.from_numpy(S.col_idx).cuda()
    own = fmm.Plan(rp, ci, S.n, r, torch.float32)
    team = fmm.Plan(rp, ci, S.n, r, torch.float32, variant=code)
    vals, A, B = f(S.nnz), f(S.m, r), f(S.n, r)
    for acc in (False, True):
        for name, x in (("fusedmm", (A, B)), ("fusedmm_t", (A, B)), ("spmm", (B,)),
                        ("spmm_t", (A,))):
            rows = S.n if name.endswith("_t") else S.m
            base = f(rows, r)
            got, want = base.clone(), base.clone()
            call = getattr(fmm, name + ("_acc" if acc else ""))
            call(own, vals, *x, out=got)
            call(team, vals, *x, out=want)
            assert torch.equal(got, want), (name, acc)


@pytest.mark.parametrize("dtype,r", [(torch.float32, 128), (torch.float32, 256), (torch.bfloat16, 32)])
@pytest.mark.parametrize("k", [1, 4, 5, 13, 14, 17, 18, 40])
def test_rows_alike(k, dtype, r):
    """Patterns of k nonzeros in every row, on both sides of the averages at which
    SDDMM and the adjoints of a plan left to its own choice change their layout,
    and with one long row, which changes it back."""
    rng = np.random.default_rng(k)
    run_all(wl.er_exact_degree(700, 300, k, rng), {}, r, dtype, seed=k)
    run_all(wl.random_csr(700, 300, rng, mean_deg=k, hubs=((5, 250),)), {}, r, dtype, seed=k)
