"""fmm_fusedmm_noalloc beyond one slab of 2^20 rows and at the widths of its
row passes: long rows in every slab, rows of one chunk and of one nonzero
more, widths on the flexible and the generic pass; against the FP64 oracle
within the float32 rounding bound, and the same bits on a repeated call."""
import numpy as np
import pytest
import torch

import oracle
from parity_utils import assert_close, host64, upload
from paper_2203_07673_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def check(S, r, dtype, seed):
    from paper_2203_07673_gb300 import fmm
    rng = np.random.default_rng(seed)
    vals = rng.uniform(0, 1, S.nnz).astype(np.float32)
    A = rng.standard_normal((S.m, r)).astype(np.float32)
    B = rng.standard_normal((S.n, r)).astype(np.float32)
    rp, ci, vt, At, Bt = upload(S, vals, A, B, dtype)
    out = torch.full((S.m, r), float("nan"), device="cuda")
    fmm.fusedmm_noalloc(rp, ci, S.n, vt, At, Bt, out=out)
    assert torch.equal(out, fmm.fusedmm_noalloc(rp, ci, S.n, vt, At, Bt))
    A64, B64 = host64(At), host64(Bt)
    ref = oracle.fusedmm(S.row_ptr, S.col_idx, vals, A64, B64, S.n)
    mag = oracle.fusedmm(S.row_ptr, S.col_idx, vals, np.abs(A64), np.abs(B64), S.n)
    assert_close("out", out, ref, mag, r, int(S.degrees().max()))


def csr(deg, n, rng):
    rp = np.zeros(deg.size + 1, np.int64)
    np.cumsum(deg, out=rp[1:])
    return wl.CSR(deg.size, n, rp.astype(np.int32),
                  rng.integers(0, n, int(rp[-1])).astype(np.int32))


@pytest.mark.parametrize("extra", [0, 1, 5000])
def test_slabs_of_rows(extra):
    rng = np.random.default_rng(extra)
    deg = rng.integers(0, 3, (1 << 20) + extra)
    deg[[0, 777, (1 << 20) - 1, -1]] = (300, 5000, 129, 128 + extra)
    check(csr(deg, 999, rng), 8, torch.float32, extra)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
@pytest.mark.parametrize("r", [1, 31, 32, 64, 100, 128, 256, 300, 600])
def test_widths_and_chunk_edges(r, dtype):
    rng = np.random.default_rng(r)
    deg = rng.integers(0, 40, 700)
    deg[[1, 2, 3, 4, 699]] = (127, 128, 129, 256, 1500)
    check(csr(deg, 333, rng), r, dtype, r)


def test_no_nonzeros():
    check(csr(np.zeros(1500, np.int64), 7, np.random.default_rng(0)), 64, torch.float32, 0)


@pytest.mark.parametrize("m,hub", [(1, 5000), (31, 129), (4095, 700), (4096, 128), (4097, 700),
                                   (4096, 262000), (4096, 262200), (4000, 300000)])
def test_few_rows(m, hub):
    """The order of the rows by one block, up to 4096 rows and 4096 chunk slots (2
    nnz / 128), and by the kernels above either."""
    rng = np.random.default_rng(m + hub)
    deg = np.zeros(m, np.int64) if hub > 200000 else rng.integers(0, 300, m) * (rng.random(m) < 0.3)
    deg[m // 2] = hub
    check(csr(deg, 211, rng), 32, torch.float32, m)
    check(csr(deg, 211, rng), 20, torch.bfloat16, m)


def test_rows_of_one_length():
    check(csr(np.full(3000, 17, np.int64), 211, np.random.default_rng(1)), 128, torch.float32, 3)
