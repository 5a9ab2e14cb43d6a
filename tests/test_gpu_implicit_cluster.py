"""The implicit solves shared by the CTAs of a cluster (as many per subdomain as the plans' estimates ask for): the
operator B K_reg^{-1} B^T and the solve's two other uses of the factor, on uneven subdomains, one subdomain, few large
ones and as many as need one CTA each.

Bar of the operator: the substitutions are backward stable, so subdomain i's part of q is off by a small multiple of
u kappa_1(K_reg,i) |q_i|; 8 of them, with the largest condition number, cover both sides' solves.  The solution's bar is
that of the other parity tests (1e-10 against the monolithic solve)."""
import numpy as np
import pytest
import torch

from oracle import feti_oracle as O
from paper_2502_08382_gb300 import feti
from paper_2502_08382_gb300.problems import make_problem, seeded_vector

pytestmark = pytest.mark.gpu

CASES = [
    (2, "heat", [[1], [1]]),
    (2, "heat", [[40, 3], [40, 3]]),
    (2, "heat", [[48, 24, 40, 8]] * 2),
    (3, "heat", [[14, 3]] * 3),
    (3, "heat", [[9, 2, 7]] * 3),
    (3, "heat", [[4, 3, 2, 5]] * 3),
    (3, "elasticity", [[8, 5]] * 3),
]


@pytest.mark.parametrize("dim,physics,cuts", CASES)
def test_operator(dim, physics, cuts):
    P = make_problem(dim=dim, physics=physics, cuts=cuts, material="lognormal", sigma=0.5, seed=4)
    op = feti.FetiOperator(P, prec="fp64")
    op.assemble()
    if P.n_lambda == 0:
        op.close()
        return
    p = seeded_vector(P.n_lambda, 6)
    q = op.apply_implicit(torch.from_numpy(p).cuda()).cpu().numpy()
    again = op.apply_implicit(torch.from_numpy(p).cuda()).cpu().numpy()
    op.close()
    ref, size, kappa = np.zeros_like(q), 0.0, 0.0
    for s in P.subs:
        l = np.asarray(s.B_lambda, dtype=np.int64)
        K = O.K_reg(s)
        part = O.local_F(s, K) @ p[l]
        ref[l] += part
        size += np.linalg.norm(part)
        kappa = max(kappa, np.linalg.cond(K, 1))
    assert np.linalg.norm(q - ref) <= 8 * 2.0 ** -53 * kappa * size
    assert np.array_equal(q, again)


@pytest.mark.parametrize("cuts", [[[9, 2]] * 3, [[4, 3, 5]] * 3])
def test_solution(cuts):
    P = make_problem(dim=3, physics="heat", cuts=cuts, material="lognormal", sigma=0.5, seed=4)
    um = O.monolithic_solve(P)
    op = feti.FetiOperator(P, prec="split_bf16", tol=1e-12, maxit=3000, refine_every=10)
    op.assemble()
    lam, alpha, u, info = op.solve()
    u = u.cpu().numpy()
    op.close()
    assert info["converged"], info
    off = 0
    for s in P.subs:
        assert np.abs(u[off:off + s.n] - um[s.l2g]).max() <= 1e-10 * np.abs(um).max()
        off += s.n
