"""The value permutation through shared memory (plans of more than 2^24
nonzeros): integer values make every sum exact, so S^T times a matrix of ones
must equal the column sums exactly.  Patterns without structure (short runs),
diagonal and reversed ones (a run per tile), a few hub columns (one S^T tile
for many S tiles), ragged last tiles, and values off a 16-byte boundary;
registered values take the same path."""
import pytest
import torch

pytestmark = pytest.mark.gpu

TILE = 49152


def columns(kind, nnz, n, g):
    if kind == "random":
        return torch.randint(0, n, (nnz,), generator=g, device="cuda")
    if kind == "hubs":
        return torch.randint(0, n, (nnz,), generator=g, device="cuda") // 64 * 64
    i = torch.arange(nnz, device="cuda")
    return (i if kind == "diagonal" else nnz - 1 - i) % n


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("kind", ["random", "hubs", "diagonal", "reversed"])
@pytest.mark.parametrize("nnz", [(1 << 24) + 1, 342 * TILE, 342 * TILE + 33])
def test_values_reach_their_columns(nnz, kind, shift):
    from paper_2203_07673_gb300 import fmm
    g = torch.Generator(device="cuda").manual_seed(nnz + shift)
    m, n = 1000, 1 << 20
    cols = columns(kind, nnz, n, g)
    row_ptr = torch.div(torch.arange(m + 1, device="cuda") * nnz, m, rounding_mode="floor")
    buf = torch.randint(0, 8, (nnz + shift,), generator=g, device="cuda").float()
    v = buf[shift:]
    plan = fmm.Plan(row_ptr.int(), cols.int(), n, 4)
    got = fmm.spmm_t(plan, v, torch.ones(m, 4, device="cuda"))
    want = torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, cols, v.double())
    assert want.max() < 2 ** 24
    assert torch.equal(got.double(), want[:, None].expand(n, 4))
    plan.set_values(v)
    assert torch.equal(fmm.spmm_t(plan, v, torch.ones(m, 4, device="cuda")), got)
    plan.close()


@pytest.mark.parametrize("side", [3000, 4200, 16400])
def test_every_value_keeps_its_row(side):
    """All three ways to the order of S^T: a single gather (9.0M nonzeros),
    through shared memory (17.6M) and in windows (269M, above 2^28).  A full
    pattern with the columns of each row in an order of its own, and operand
    rows that differ, so that two values changed about show even inside a
    column; integers small enough for every sum to be exact."""
    from paper_2203_07673_gb300 import fmm
    g = torch.Generator(device="cuda").manual_seed(side)
    i = torch.arange(side, device="cuda")
    cols = torch.cat([(i * 1009 + 37 * r) % side for r in range(side)]).int()
    assert side % 1009 != 0
    plan = fmm.Plan((torch.arange(side + 1, device="cuda") * side).int(), cols, side, 32)
    v = torch.randint(0, 8, (side * side,), generator=g, device="cuda").float()
    A = torch.randint(0, 64, (side, 32), generator=g, device="cuda").float()
    dense = torch.empty(side, side, device="cuda")
    dense.scatter_(1, cols.view(side, side).long(), v.view(side, side))
    want = dense.double().t() @ A.double()
    assert want.max() < 2 ** 24
    del dense
    assert torch.equal(fmm.spmm_t(plan, v, A).double(), want)
    plan.set_values(v)
    assert torch.equal(fmm.spmm_t(plan, v, A).double(), want)
    plan.close()
