"""The flexible-width row pass at the edges of its layouts: widths around its
powers of two and its largest (512; wider rows take the generic kernel),
vector widths from two to sixteen bytes, operands aligned to less than a
vector, several lane groups per row (few rows) and long rows in chunks, each
role against the FP64 oracle within the float32 rounding bound."""
import numpy as np
import pytest
import torch

import oracle
from parity_utils import assert_close, host64
from paper_2203_07673_gb300 import workloads as wl
from test_gpu_parity import pattern, run_all

pytestmark = pytest.mark.gpu

DTYPES = pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])


@DTYPES
@pytest.mark.parametrize("r", [1, 2, 7, 9, 33, 130, 255, 258, 504, 511, 513])
@pytest.mark.parametrize("kind", ["irregular", "hubs"])
def test_widths(kind, r, dtype):
    S, opts = pattern(kind, 60 + r)
    run_all(S, opts, r, dtype, seed=r)


@DTYPES
@pytest.mark.parametrize("shift", [1, 2, 4])
@pytest.mark.parametrize("r", [64, 36])
def test_operands_off_a_vector_boundary(r, shift, dtype):
    """A, B and the output start `shift` elements past an aligned address."""
    from paper_2203_07673_gb300 import fmm
    S, _ = pattern("irregular", 5)
    rng = np.random.default_rng(r + shift)

    def off(x, dt):
        buf = torch.zeros(x.size + shift, dtype=dt, device="cuda")
        buf[shift:] = torch.from_numpy(x.reshape(-1)).cuda().to(dt)
        return buf[shift:].view(*x.shape)
    A = off(rng.standard_normal((S.m, r)).astype(np.float32), dtype)
    B = off(rng.standard_normal((S.n, r)).astype(np.float32), dtype)
    out = off(np.zeros((S.m, r), np.float32), torch.float32)
    vals = rng.uniform(0, 1, S.nnz).astype(np.float32)
    rp, ci = torch.from_numpy(S.row_ptr).cuda(), torch.from_numpy(S.col_idx).cuda()
    plan = fmm.Plan(rp, ci, S.n, r, dtype)
    fmm.fusedmm(plan, torch.from_numpy(vals).cuda(), A, B, out=out)
    A64, B64 = host64(A), host64(B)
    ref = oracle.fusedmm(S.row_ptr, S.col_idx, vals, A64, B64, S.n)
    mag = oracle.fusedmm(S.row_ptr, S.col_idx, vals, np.abs(A64), np.abs(B64), S.n)
    assert_close("out", out, ref, mag, r, int(S.degrees().max()))


@pytest.mark.parametrize("m", [1, 3, 17])
def test_few_rows(m):
    """Fewer rows than one block of groups: every lane group of a team works."""
    S = wl.random_csr(m, 90, np.random.default_rng(m), mean_deg=40, empty_frac=0.0)
    run_all(S, {}, 12, torch.float32, seed=m)


@pytest.mark.parametrize("r", [32, 12, 13, 132])
@pytest.mark.parametrize("hub", [64, 65, 512, 513, 3000])
def test_sums_of_partial_rows(hub, r):
    """Rows of 1 to 47 chunks of 64: summed by one warp up to eight chunks,
    by a block above, several of both kinds in one block."""
    S = wl.random_csr(300, 280, np.random.default_rng(hub + r), mean_deg=6,
                      hubs=((0, hub), (1, 700), (2, 100), (299, 600)))
    run_all(S, {"split_nnz": 64}, r, torch.float32, seed=hub)


@DTYPES
@pytest.mark.parametrize("r", [12, 31, 65, 96, 128 + 4, 257, 300, 384, 385, 545, 1030])
def test_long_rows_beside_short_ones(r, dtype):
    """Rows around the length that gets a warp each, unsplit and in chunks, at
    the edges of the elements per lane and past the widest row."""
    hubs = tuple((i * 9, d) for i, d in enumerate((0, 1, 62, 63, 64, 65, 66, 127, 128, 255, 256, 257,
                                                   600)))
    S = wl.random_csr(400, 500, np.random.default_rng(r), mean_deg=4, empty_frac=0.1, hubs=hubs)
    run_all(S, {}, r, dtype, seed=r)


@DTYPES
@pytest.mark.parametrize("r", [25, 300, 513, 545, 1030])
def test_accumulating_call(r, dtype):
    from paper_2203_07673_gb300 import fmm
    S, opts = pattern("hubs", r)
    rng = np.random.default_rng(r)
    f = lambda *s: torch.from_numpy(rng.standard_normal(s).astype(np.float32)).cuda()
    plan = fmm.Plan(torch.from_numpy(S.row_ptr).cuda(), torch.from_numpy(S.col_idx).cuda(), S.n, r,
                    dtype, **opts)
    vals, A, B, base = f(S.nnz), f(S.m, r).to(dtype), f(S.n, r).to(dtype), f(S.m, r)
    out = base.clone()
    fmm.fusedmm_acc(plan, vals, A, B, out=out)
    v, A64, B64, b = vals.cpu().numpy(), host64(A), host64(B), host64(base)
    ref = b + oracle.fusedmm(S.row_ptr, S.col_idx, v, A64, B64, S.n)
    mag = np.abs(b) + oracle.fusedmm(S.row_ptr, S.col_idx, np.abs(v), np.abs(A64), np.abs(B64), S.n)
    assert_close("out", out, ref, mag, r, int(S.degrees().max()) + 1)
