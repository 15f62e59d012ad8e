"""The native call path (csrc/torch_calls.cpp) against the Python one: the same
bits in every call and gradient, and the same answer where it declines
(wrong arguments, modes, transforms, forward-mode differentiation, a closed
plan)."""
import gc
import threading
import weakref

import numpy as np
import pytest
import torch

from paper_2203_07673_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def make(dtype=torch.float32, r=24, with_vals=True, seed=0):
    from paper_2203_07673_gb300 import fmm
    rng = np.random.default_rng(seed)
    S = wl.random_csr(120, 90, rng, mean_deg=5)
    f = lambda *s: torch.from_numpy(rng.standard_normal(s).astype(np.float32)).cuda()
    plan = fmm.Plan(torch.from_numpy(S.row_ptr).cuda(), torch.from_numpy(S.col_idx).cuda(), S.n, r,
                    dtype)
    assert plan.fast is not None
    return (plan, f(S.nnz) if with_vals else None, f(S.m, r).to(dtype), f(S.n, r).to(dtype),
            f(S.m, r), f(S.n, r))


def slow(plan, fn, *args):
    """fn on the Python path."""
    fast, plan.fast = plan.fast, None
    try:
        return fn(*args)
    finally:
        plan.fast = fast


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
@pytest.mark.parametrize("with_vals", [True, False])
def test_calls_give_the_same_bits(dtype, with_vals):
    from paper_2203_07673_gb300 import fmm
    plan, v, A, B, _, _ = make(dtype, with_vals=with_vals)
    w = torch.randn(plan.nnz, device="cuda")
    for fn, args in ((fmm.fusedmm, (v, A, B)), (fmm.fusedmm_t, (v, A, B)), (fmm.sddmm, (v, A, B)),
                     (fmm.spmm, (w, B)), (fmm.spmm_t, (w, A))):
        want = slow(plan, fn, plan, *args)
        got = fn(plan, *args)
        assert torch.equal(got, want) and got.dtype == torch.float32
        out = torch.full_like(want, float("nan"))
        assert fn(plan, *args, out=out) is out and torch.equal(out, want)
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            assert torch.equal(fn(plan, *args), want)
        torch.cuda.current_stream().wait_stream(side)


def test_cg_update_gives_the_same_bits(monkeypatch):
    from paper_2203_07673_gb300 import fmm
    x, res, p, q = (torch.randn(70, 20, device="cuda") for _ in range(4))
    rs = (res * res).sum(1)
    a = [t.clone() for t in (x, res, p, q, rs)]
    b = [t.clone() for t in (x, res, p, q, rs)]
    fmm.cg_update(0.5, *a)
    monkeypatch.setattr(fmm, "_calls", None)
    fmm.cg_update(0.5, *b)
    assert all(torch.equal(s, t) for s, t in zip(a, b))
    monkeypatch.undo()
    with pytest.raises(ValueError):
        fmm.cg_update(0.5, x, res, p, q, rs[:-1])


@pytest.mark.parametrize("transpose", [False, True], ids=["A", "B"])
@pytest.mark.parametrize("dtype,r", [(torch.float32, 24), (torch.bfloat16, 64), (torch.bfloat16, 520)])
@pytest.mark.parametrize("needs", [(1, 1, 1), (0, 1, 0), (0, 0, 1), (1, 0, 0)])
def test_gradients_are_the_same(needs, dtype, r, transpose):
    from paper_2203_07673_gb300 import autograd
    plan, v, A, B, Gm, Gn = make(dtype, r)
    G = (Gn if transpose else Gm).t().contiguous().t()   # not contiguous
    leaves = [t.requires_grad_(bool(k)) for t, k in zip((v, A, B), needs)]
    wanted = [t for t, k in zip(leaves, needs) if k]

    def step():
        out = autograd.fusedmm(plan, v, A, B, transpose=transpose)
        return [out.detach(), *torch.autograd.grad(out, wanted, G)]
    for x, y in zip(step(), slow(plan, step)):
        assert x.dtype == y.dtype and torch.equal(x, y)
    out = autograd.fusedmm(plan, v, A, B, transpose=transpose)
    out.backward(G)
    assert all((t.grad is not None) == bool(k) for t, k in zip(leaves, needs))
    with pytest.raises(RuntimeError):
        out.backward(G)   # the graph is freed
    with torch.no_grad():
        assert not autograd.fusedmm(plan, v, A, B, transpose=transpose).requires_grad


def test_no_values_and_no_gradients():
    from paper_2203_07673_gb300 import autograd
    plan, _, A, B, G, _ = make(with_vals=False)
    assert not autograd.fusedmm(plan, None, A, B).requires_grad
    A.requires_grad_(True)
    out = autograd.fusedmm(plan, None, A, B)
    assert torch.equal(torch.autograd.grad(out, A, G)[0],
                       slow(plan, lambda: torch.autograd.grad(autograd.fusedmm(plan, None, A, B), A, G)[0]))


def test_saved_tensors():
    from paper_2203_07673_gb300 import autograd
    plan, v, A, B, G, _ = make()
    for t in (v, A, B):
        t.requires_grad_(True)
    want = torch.autograd.grad(autograd.fusedmm(plan, v, A, B), (v, A, B), G)
    packed = []
    with torch.autograd.graph.saved_tensors_hooks(lambda t: packed.append(t) or t.cpu(),
                                                  lambda t: t.cuda()):
        out = autograd.fusedmm(plan, v, A, B)
    assert len(packed) == 3
    assert all(torch.equal(x, y) for x, y in zip(torch.autograd.grad(out, (v, A, B), G), want))
    out = autograd.fusedmm(plan, v, A, B)
    with torch.no_grad():
        A.mul_(2)
    with pytest.raises(RuntimeError, match="inplace"):
        torch.autograd.grad(out, B, G)


@pytest.mark.parametrize("which", ["vals", "A", "B"])
@pytest.mark.parametrize("unpack", ["strides", "expanded", "narrower", "dtype", "host"])
@pytest.mark.parametrize("transpose", [False, True], ids=["A", "B"])
def test_unpacked_tensors_are_checked(transpose, unpack, which):
    """A saved-tensor hook may give back any tensor: operands that the call
    would refuse are refused in the adjoint too, with the same error, and the
    same values in the right layout are taken."""
    from paper_2203_07673_gb300 import autograd
    plan, v, A, B, Gm, Gn = make()
    G = Gn if transpose else Gm
    leaves = dict(vals=v, A=A, B=B)
    for t in leaves.values():
        t.requires_grad_(True)
    bad = leaves[which].detach()
    bad = {"strides": lambda t: t.repeat_interleave(2, -1)[..., ::2],
           "expanded": lambda t: t[:1].expand(t.shape), "narrower": lambda t: t[:-1].contiguous(),
           "dtype": lambda t: t.double(), "host": lambda t: t.cpu()}[unpack](bad)

    def step(swap):
        packed = []
        with torch.autograd.graph.saved_tensors_hooks(
                lambda t: packed.append(t) or len(packed) - 1,
                lambda i: bad if swap and packed[i].shape == leaves[which].shape
                and packed[i].data_ptr() == leaves[which].data_ptr() else packed[i]):
            out = autograd.fusedmm(plan, v, A, B, transpose=transpose)
        assert len(packed) == 3
        return torch.autograd.grad(out, (v, A, B), G)
    with pytest.raises((TypeError, ValueError)) as want:
        slow(plan, step, True)
    with pytest.raises(type(want.value)) as got:
        step(True)
    assert str(got.value) == str(want.value)
    assert all(torch.equal(x, y) for x, y in zip(step(False), slow(plan, step, False)))


def test_other_ways_to_differentiate():
    from paper_2203_07673_gb300 import autograd
    plan, v, A, B, G, _ = make()
    A.requires_grad_(True)
    # a second derivative is not provided: the first one does not require grad
    out = autograd.fusedmm(plan, v, A, B)
    g, = torch.autograd.grad(out, A, G, create_graph=True)
    assert g.requires_grad == slow(
        plan, lambda: torch.autograd.grad(autograd.fusedmm(plan, v, A, B), A, G, create_graph=True)[0]
    ).requires_grad
    import torch.autograd.forward_ad as fwad
    with fwad.dual_level():
        dual = fwad.make_dual(A.detach(), torch.ones_like(A))
        with pytest.raises(Exception):
            autograd.fusedmm(plan, v, dual, B)
    with pytest.raises(Exception):
        torch.func.vmap(lambda a: autograd.fusedmm(plan, v, a, B))(torch.stack([A.detach()] * 2))
    with pytest.raises(Exception):
        torch.func.grad(lambda a: autograd.fusedmm(plan, v, a, B).sum())(A.detach())


def test_wrong_arguments_raise_as_before():
    from paper_2203_07673_gb300 import autograd, fmm
    plan, v, A, B, _, _ = make()
    bad = [(TypeError, (v, A.double(), B)), (ValueError, (v[:-1], A, B)), (ValueError, (v, A[:-1], B)),
           (ValueError, (v, A.cpu(), B)), (ValueError, (v, A.t().contiguous().t(), B)),
           (TypeError, (v, A.tolist(), B))]
    for err, args in bad:
        with pytest.raises(err):
            fmm.fusedmm(plan, *args)
        if not isinstance(args[1], list):
            with pytest.raises(err):
                autograd.fusedmm(plan, *args)
    with pytest.raises(TypeError):
        fmm.fusedmm(plan, v, A, B, out=torch.empty_like(A, dtype=torch.float64))
    with pytest.raises(fmm.FmmError):
        fmm.spmm(plan, None, B)


def test_closed_plans():
    from paper_2203_07673_gb300 import autograd, fmm
    plan, v, A, B, G, _ = make()
    A.requires_grad_(True)
    out = autograd.fusedmm(plan, v, A, B)
    plan.close()
    with pytest.raises(fmm.FmmError):
        torch.autograd.grad(out, A, G)
    with pytest.raises(fmm.FmmError):
        fmm.fusedmm(plan, v, A.detach(), B)


def test_a_graph_keeps_its_plan():
    from paper_2203_07673_gb300 import autograd
    plan, v, A, B, G, _ = make()
    A.requires_grad_(True)
    want, = torch.autograd.grad(autograd.fusedmm(plan, v, A, B), A, G)
    out = autograd.fusedmm(plan, v, A, B)
    alive = weakref.ref(plan)
    del plan
    gc.collect()
    assert alive() is not None
    assert torch.equal(torch.autograd.grad(out, A, G)[0], want)
    del out
    gc.collect()
    assert alive() is None


def test_threads():
    from paper_2203_07673_gb300 import autograd
    failed = []

    def work(k):
        try:
            plan, v, A, B, G, _ = make(seed=k)
            A.requires_grad_(True)
            with torch.cuda.stream(torch.cuda.Stream()):
                torch.cuda.synchronize()
                for _ in range(50):
                    g, = torch.autograd.grad(autograd.fusedmm(plan, v, A, B), A, G)
                w, = slow(plan, lambda: torch.autograd.grad(autograd.fusedmm(plan, v, A, B), A, G))
                assert torch.equal(g, w)
        except Exception as e:
            failed.append(e)
    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed


@pytest.mark.parametrize("dtype,r,own,other", [(torch.bfloat16, 64, 32212, 112), (torch.float32, 256, 112, 122)])
def test_default_code_gives_a_side_its_own_choice_back(dtype, r, own, other):
    """fmm_plan_set_variant with the code of a plan's default on one side: that
    side runs what an untouched plan runs (another layout than the code's in one
    of the adjoints, which shows in its bits), whatever the other side has."""
    from paper_2203_07673_gb300 import fmm
    rng = np.random.default_rng(r)
    S = wl.random_csr(500, 400, rng, mean_deg=12, hubs=((3, 200),))
    f = lambda *s: torch.from_numpy(rng.standard_normal(s).astype(np.float32)).cuda()
    v, A, B, G = f(S.nnz), f(S.m, r).to(dtype), f(S.n, r).to(dtype), f(S.m, r)

    def grads(*codes, **kw):
        plan = fmm.Plan(torch.from_numpy(S.row_ptr).cuda(), torch.from_numpy(S.col_idx).cuda(), S.n, r,
                        dtype, **kw)
        assert kw or plan.info()["variant"] == plan.info()["variant_t"] == own
        for c in codes:
            plan.set_variant(*c)
        out = fmm.fusedmm_bwd(plan, v, A, B, G)
        plan.close()
        return out
    side = 1 if dtype == torch.bfloat16 else 0   # dB by the columns, dA by the rows
    want, plain = grads()[side], grads(variant=own)[side]
    assert not torch.equal(want, plain)
    pair = lambda mine, theirs: (theirs, mine) if side else (mine, theirs)
    for codes in ([pair(own, other)], [pair(own, 0)], [(own, own)], [pair(other, other), pair(own, 0)]):
        assert torch.equal(grads(*codes)[side], want), codes
    assert not torch.equal(grads(pair(other, own))[side], want)
