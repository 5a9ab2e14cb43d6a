"""FP64 forward solve of the large fronts on the tensor cores: fronts from 128 wide on (options.chol_tc_front), so that
partial 128-column blocks, fronts without rows below, columns on both sides of a 128-column tile and mixed children
occur in small problems.  Bars: the FP64 parity bar 1e-12 against the oracle; two assemblies of the same factorisation
problem may differ by twice that."""
import numpy as np
import pytest
import torch

from oracle import feti_oracle as O
from paper_2502_08382_gb300 import feti
from paper_2502_08382_gb300.problems import make_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,physics,cuts,route", [
    (3, "elasticity", [[6, 4]] * 3, "syrk"),
    (3, "elasticity", [[7]] * 3, "syrk"),        # one subdomain, Dirichlet rows only: few columns
    (3, "heat", [[9, 11]] * 3, "syrk"),
    (2, "heat", [[90, 94]] * 2, "syrk"),         # narrow separators just above the threshold
    (3, "elasticity", [[4, 5]] * 3, "schur"),    # one dense root
])
def test_against_oracle(dim, physics, cuts, route):
    P = make_problem(dim=dim, physics=physics, cuts=cuts, material="lognormal", sigma=0.5)
    op = feti.FetiOperator(P, prec="fp64", chol_tc_front=128, route=route)
    op.assemble()
    op.assemble()  # the captured launches
    for i, s in enumerate(P.subs):
        if s.n > 4000 and i > 1:
            continue
        Fo = O.local_F(s)
        assert np.linalg.norm(op.get_F(i) - Fo) <= 1e-12 * np.linalg.norm(Fo)
    op.close()


def test_released_and_refused(monkeypatch):
    """recompute_X gives the digits back after each assembly; a refused digit buffer leaves the FP64-pipe solve."""
    P = make_problem(dim=3, physics="elasticity", cuts=[[6, 5]] * 3, material="lognormal", sigma=0.5)
    ref = feti.FetiOperator(P, prec="fp64")
    ref.assemble()
    Fr = [ref.get_F(i) for i in range(P.nsub)]
    ref.close()
    op = feti.FetiOperator(P, prec="fp64", recompute_X=True, chol_tc_front=128)
    for _ in range(3):
        op.assemble()
        for i in range(P.nsub):
            assert np.linalg.norm(op.get_F(i) - Fr[i]) <= 2e-12 * np.linalg.norm(Fr[i])
    op.close()
    real, armed = torch.cuda.caching_allocator_alloc, [False]

    def alloc(nbytes, *a, **k):
        if armed[0]:
            raise torch.cuda.OutOfMemoryError("refused by the test")
        return real(nbytes, *a, **k)

    monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", alloc)
    op = feti.FetiOperator(P, prec="fp64", chol_tc_front=128)
    armed[0] = True  # neither the solve's nor the SYRK's digits
    op.assemble()
    armed[0] = False
    for i in range(P.nsub):
        assert np.linalg.norm(op.get_F(i) - Fr[i]) <= 2e-12 * np.linalg.norm(Fr[i])
    op.close()
