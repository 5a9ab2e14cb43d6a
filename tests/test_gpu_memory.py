"""Short device memory: buffers that the allocator refuses, when they are asked for again, and what feti_stats says
about it.  Bars: the FP64 parity bar 1e-12 between two assemblies of the same problem, twice for both sides."""
import numpy as np
import pytest
import torch

from paper_2502_08382_gb300 import feti
from paper_2502_08382_gb300.problems import make_problem, make_W

pytestmark = pytest.mark.gpu


class Refuser:
    """torch's allocator, refusing the requests that `rule(nbytes)` picks while it is armed; counts them."""

    def __init__(self, monkeypatch):
        self.rule, self.refused, self.real = None, 0, torch.cuda.caching_allocator_alloc
        monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", self)

    def __call__(self, nbytes, *a, **k):
        if self.rule and self.rule(nbytes):
            self.refused += 1
            raise torch.cuda.OutOfMemoryError("refused by the test")
        return self.real(nbytes, *a, **k)


@pytest.fixture
def ref():
    P = make_problem(dim=3, physics="elasticity", cuts=[[6, 5]] * 3, material="lognormal", sigma=0.5)
    op = feti.FetiOperator(P, prec="fp64")
    op.assemble()
    F = [op.get_F(i) for i in range(P.nsub)]
    op.close()
    return P, F


def check(op, F):
    for i, f in enumerate(F):
        assert np.linalg.norm(op.get_F(i) - f) <= 2e-12 * np.linalg.norm(f)


def test_syrk_refused(monkeypatch, ref):
    """A refused digit buffer is not asked for again while no more memory is free; the FP64-pipe kernel does the SYRK."""
    P, F = ref
    r = Refuser(monkeypatch)
    op = feti.FetiOperator(P, prec="fp64")
    r.rule = lambda n: n > 1 << 20
    for _ in range(4):
        op.assemble()
        check(op, F)
    assert r.refused == 2  # all subdomains, then one at a time, in the first assembly only
    assert op.stats()["digit_kernels"] == 0
    op.close()


def test_syrk_passing_shortage(monkeypatch, ref):
    """With recompute_X the buffer is asked for at every assembly, so a passing shortage passes."""
    P, F = ref
    r = Refuser(monkeypatch)
    op = feti.FetiOperator(P, prec="fp64", recompute_X=True)
    x = 8 * op.stats()["X_elems"]
    for short in (False, True, False):
        r.rule = (lambda n: n > x + 256) if short else None  # X itself is granted
        op.assemble()
        r.rule = None
        check(op, F)
        # one subdomain at a time fits
        assert op.stats()["digit_kernels"] == 1
    r.rule = lambda n: n != (x + 255) // 256 * 256 and n > 1 << 20
    op.assemble()
    r.rule = None
    check(op, F)
    assert op.stats()["digit_kernels"] == 0
    op.assemble()
    check(op, F)
    assert op.stats()["digit_kernels"] == 1
    op.close()


@pytest.mark.parametrize("recompute", [False, True])
def test_trsm_refused_once(monkeypatch, ref, recompute):
    """The digits of L are refused for all subdomains together and granted one subdomain at a time."""
    P, F = ref
    r = Refuser(monkeypatch)
    op = feti.FetiOperator(P, prec="fp64", chol_tc_front=128, recompute_X=recompute)
    r.rule = lambda n: n > 1 << 20 and r.refused == 0
    for _ in range(3):
        op.assemble()
        check(op, F)
        assert op.stats()["digit_kernels"] == 3
    assert r.refused == 1
    op.close()


def test_trsm_passing_shortage(monkeypatch, ref):
    """With recompute_X a shortage at one assembly does not keep the next ones from the digits."""
    P, F = ref
    r = Refuser(monkeypatch)
    op = feti.FetiOperator(P, prec="fp64", chol_tc_front=128, recompute_X=True)
    x = (8 * op.stats()["X_elems"] + 255) // 256 * 256
    for short in (True, False, True, False):
        r.rule = (lambda n: n != x and n > 1 << 20) if short else None  # X itself is granted
        op.assemble()
        r.rule = None
        check(op, F)
        assert op.stats()["digit_kernels"] == (0 if short else 3)
    op.close()


def test_trsm_refused(monkeypatch, ref):
    """Refused for good, the digits are not asked for again while no more memory is free."""
    P, F = ref
    r = Refuser(monkeypatch)
    op = feti.FetiOperator(P, prec="fp64", chol_tc_front=128)
    r.rule = lambda n: n > 1 << 20
    op.assemble()
    first = r.refused
    for _ in range(3):
        op.assemble()
        check(op, F)
    assert first == 4 and r.refused == first  # L and X, all subdomains and then one at a time
    assert op.stats()["digit_kernels"] == 0
    op.close()


def elast(axis=2, elems=6):
    return make_problem(dim=3, physics="elasticity", cuts=[[elems] * axis] * 3, material="density", seed=3)


@pytest.mark.parametrize("recompute", [False, True])
def test_adjoint_dense_refused(monkeypatch, recompute):
    """The dense product's digits refused, Y comes from X W, with the assembly's X or with X_u solved for again: the same
    gradient at the parity bar 1e-10."""
    P = elast()
    Ws = make_W(P, seed=0)
    op = feti.FetiOperator(P, prec="fp64", with_elements=True)
    op.assemble()
    g = op.adjoint(Ws).cpu().numpy()
    op.close()
    r = Refuser(monkeypatch)
    op = feti.FetiOperator(P, prec="fp64", with_elements=True, recompute_X=recompute)
    op.assemble()
    W = op._W_dev(Ws)
    x = (8 * op.stats()["X_elems"] + 255) // 256 * 256
    r.rule = lambda n: n != x and n > 4096 and r.refused == 0
    h = op.adjoint(W).cpu().numpy()
    op.close()
    assert r.refused == 1
    assert np.linalg.norm(h - g) <= 1e-10 * np.linalg.norm(g)


def test_adjoint_budget():
    """adjoint_work_bytes caps what feti_adjoint takes, its digits included, besides the fixed scratch."""
    P = elast()
    Ws = make_W(P, seed=0)
    op = feti.FetiOperator(P, prec="fp64", with_elements=True)
    op.assemble()
    g = op.adjoint(Ws).cpu().numpy()
    op.close()
    cap = 60 << 20
    op = feti.FetiOperator(P, prec="fp64", with_elements=True, adjoint_work_bytes=cap)
    op.assemble()
    before = torch.cuda.memory_allocated()
    assert np.array_equal(op.adjoint(Ws).cpu().numpy(), g)
    scratch = torch.cuda.get_device_properties(0).multi_processor_count * 128 * (2048 + 4)
    assert torch.cuda.memory_allocated() - before <= cap + scratch + (1 << 20)  # and a few small lists
    op.close()


def test_adjoint_short_memory():
    """Later calls do as many subdomains at a time as the first, whose buffers they take over (700 MB are left free)."""
    P = elast(axis=3)
    Ws = make_W(P, seed=0)
    op = feti.FetiOperator(P, prec="fp64", with_elements=True, torch_alloc=False)
    op.assemble()
    W = op._W_dev(Ws)
    torch.cuda.empty_cache()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - (700 << 20), dtype=torch.uint8, device="cuda")
    counts, grads = [], []
    for _ in range(3):
        n = op.stats()["launches"]
        grads.append(op.adjoint(W))
        counts.append(op.stats()["launches"] - n)
    del hog
    torch.cuda.empty_cache()
    op.close()
    assert torch.equal(grads[0], grads[1]) and torch.equal(grads[0], grads[2])
    assert max(counts) <= 1.5 * counts[0], counts


def test_adjoint_refused(monkeypatch):
    """Where nothing large is granted beyond the work array, the FP64-pipe kernels do the adjoint (the parity bar 1e-10)."""
    P = elast()
    Ws = make_W(P, seed=0)
    r = Refuser(monkeypatch)
    op = feti.FetiOperator(P, prec="fp64", with_elements=True)
    op.assemble()
    g = op.adjoint(Ws).cpu().numpy()
    op.close()
    op = feti.FetiOperator(P, prec="fp64", with_elements=True)
    op.assemble()
    W = op._W_dev(Ws)
    # digits and work array, with and without the assembly's digits held; then the work array is granted
    r.rule = lambda n: n > 4096 and r.refused < 4
    h = op.adjoint(W).cpu().numpy()
    r.rule = None
    assert r.refused == 4
    assert np.linalg.norm(h - g) <= 1e-10 * np.linalg.norm(g)
    op.assemble()
    assert op.stats()["digit_kernels"] & 1
    assert np.linalg.norm(op.adjoint(W).cpu().numpy() - g) <= 1e-10 * np.linalg.norm(g)
    op.close()


def test_adjoint_backward_refused(monkeypatch):
    """The digits of L^T refused, the FP64-pipe kernel does the whole backward solve."""
    P = elast()
    Ws = make_W(P, seed=0)
    op = feti.FetiOperator(P, prec="fp64", with_elements=True)
    op.assemble()
    g = op.adjoint(Ws).cpu().numpy()
    op.close()
    r, big = Refuser(monkeypatch), [0]
    op = feti.FetiOperator(P, prec="fp64", with_elements=True)
    op.assemble()
    W = op._W_dev(Ws)

    def third(n):  # after the dense digits and the work array
        big[0] += n > 4096
        return big[0] == 3 and n > 4096

    r.rule = third
    h = op.adjoint(W).cpu().numpy()
    op.close()
    assert r.refused == 1
    assert np.linalg.norm(h - g) <= 1e-10 * np.linalg.norm(g)


def test_adjoint_frees_idle_buffers(monkeypatch):
    """A buffer goes back to dev_free only when no launch uses it any more (a caller's allocator may hand it on)."""
    P = make_problem(dim=3, physics="elasticity", cuts=[[7, 4, 6]] * 3, material="density", seed=3)
    Ws = make_W(P, seed=0)
    idle, real = [], torch.cuda.caching_allocator_delete

    def delete(p):
        idle.append(torch.cuda.current_stream().query())
        real(p)

    for cap in (20, 40, 60, 100):
        op = feti.FetiOperator(P, prec="fp64", with_elements=True, adjoint_work_bytes=cap << 20)
        op.assemble()
        W = op._W_dev(Ws)
        with monkeypatch.context() as mp:
            mp.setattr(torch.cuda, "caching_allocator_delete", delete)
            op.adjoint(W)
        op.close()
    assert len(idle) > 0 and all(idle), (len(idle), sum(idle))


@pytest.mark.parametrize("prec", ["fp64", "split_bf16"])
def test_allocator_alignment(monkeypatch, prec):
    """An allocator that aligns to 16 bytes only: every buffer is aligned by the library, and goes back as it came."""
    P = elast(elems=4)
    Ws = make_W(P, seed=0)
    op = feti.FetiOperator(P, prec=prec, with_elements=True, chol_tc_front=128)
    op.assemble()
    g, F = op.adjoint(Ws).cpu().numpy(), op.get_F(0)
    op.close()
    alloc, delete, live = torch.cuda.caching_allocator_alloc, torch.cuda.caching_allocator_delete, set()

    def odd_alloc(nbytes, *a, **k):
        p = alloc(nbytes + 16, *a, **k) + 16
        live.add(p)
        return p

    def odd_delete(p):
        live.remove(p)
        delete(p - 16)

    monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", odd_alloc)
    monkeypatch.setattr(torch.cuda, "caching_allocator_delete", odd_delete)
    op = feti.FetiOperator(P, prec=prec, with_elements=True, chol_tc_front=128, recompute_X=True)
    op.assemble()
    assert np.linalg.norm(op.adjoint(Ws).cpu().numpy() - g) <= 1e-10 * np.linalg.norm(g)
    if prec == "fp64":
        assert np.linalg.norm(op.get_F(0) - F) <= 2e-12 * np.linalg.norm(F)
    op.close()
    assert not live


def test_workspace_size():
    """The workspace holds what the kernels use: with few multipliers the TRSM needs little, and no Cholesky kernel keeps a
    stack of whole fronts per CTA any more (chol_stack doubles, per CTA of the TRSM)."""
    P = make_problem(dim=3, physics="elasticity", cuts=[[8, 8]] * 3)
    op = feti.FetiOperator(P, prec="fp64", route="schur")
    st = op.stats()
    stack = max(feti.analyse(s, route="schur")["chol_stack"] for s in P.subs)
    op.assemble()
    ctas = op.stats()["trsm_grid"]
    op.close()
    assert st["workspace_bytes"] < 8 * ctas * stack


@pytest.mark.parametrize("cuts", [[[1], [1]], [[2], [2]], [[1, 1], [1, 1]], [[2, 2], [2, 2]]])
def test_trsm_path_holds_no_digits(monkeypatch, cuts):
    """Where the autotuner keeps the TRSM path, no digits of X and L are kept or asked for (on tiny problems the two routes
    take about the same time, so some of these keep it)."""
    P = make_problem(dim=2, physics="heat", cuts=cuts)
    op = feti.FetiOperator(P, prec="fp64", route="auto")
    op.assemble()
    r = Refuser(monkeypatch)
    r.rule = lambda n: True
    op.assemble()
    st = op.stats()
    op.close()
    if st["assembly_route"] == 2:
        assert st["digit_kernels"] == 0 and r.refused == 0
    else:
        assert st["digit_kernels"] == 1
