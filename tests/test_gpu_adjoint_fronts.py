"""The adjoint where the tree's top holds fronts of about 96 to 300 rows: the line between the FP64-pipe and the
tensor-core backward solve, supernodes narrower and wider than 64 columns, ragged multiplier counts.  Bar: that of the
adjoint's parity test."""
import numpy as np
import pytest

from oracle import feti_oracle as O
from paper_2502_08382_gb300 import feti
from paper_2502_08382_gb300.problems import make_problem, make_W

pytestmark = pytest.mark.gpu

CASES = [
    (3, "elasticity", [[5, 2]] * 3),
    (3, "elasticity", [[7, 4]] * 3),
    (3, "heat", [[9, 5]] * 3),
    (2, "heat", [[45, 7], [40, 12]]),
]


@pytest.mark.parametrize("dim,physics,cuts", CASES)
def test_gradient(dim, physics, cuts):
    P = make_problem(dim=dim, physics=physics, cuts=cuts, material="lognormal", sigma=0.3, seed=5)
    Ws = make_W(P, seed=0)
    op = feti.FetiOperator(P, prec="fp64", with_elements=True)
    op.assemble()
    g = op.adjoint(Ws).cpu().numpy()
    again = op.adjoint(Ws).cpu().numpy()
    op.close()
    off = 0
    for i, s in enumerate(P.subs):
        ne = s.elem_dofs.shape[0]
        go = O.gradient_sub(s, Ws[i], P.K_ref)
        assert np.linalg.norm(g[off:off + ne] - go) <= 1e-10 * np.linalg.norm(go)
        off += ne
    assert np.array_equal(g, again)
