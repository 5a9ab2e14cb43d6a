"""Unknowns of very different stiffness: K -> S K S with S a diagonal of powers of two (exponents -20 .. 20, so entries of
K over 24 decades).  FP64 arithmetic commutes with such a scaling: every result, its scaling undone, is that of the
unscaled problem to the last bit.  The products by digits cut whole vectors at one exponent, so they have to follow the
unknowns' scales to be as accurate; each test here holds the scaled problem, its scaling undone (exactly), to the bar of
the unscaled one.

The subdomains are made regular (K_reg in place of K, no kernel), because the penalty rho = max diag K does not scale.
chol_tc_front = 128 brings the tensor-core kernels to these small problems."""
import dataclasses

import numpy as np
import pytest
import torch

from oracle import feti_oracle as O
from paper_2502_08382_gb300 import feti
from paper_2502_08382_gb300.problems import make_problem, make_W, seeded_vector

pytestmark = pytest.mark.gpu

CASES = [
    (3, "elasticity", [[6, 5]] * 3),
    (3, "heat", [[11, 9]] * 3),
    (2, "heat", [[60, 50]] * 2),
]


def scaled(P, seed, reach=20):
    """P with regular subdomains, the same scaled by S, S per global DOF and per multiplier."""
    g = np.exp2(np.random.default_rng([seed, 9]).integers(-reach, reach + 1, size=P.n_global_dofs).astype(np.float64))
    lam = np.ones(P.n_lambda)
    plain, scal = [], []
    for s in P.subs:
        K = O.K_reg(s)
        S = g[s.l2g]
        rows = np.repeat(np.arange(s.n), np.diff(s.K_rowptr))
        val = K[rows, s.K_col]
        none = dict(R=np.zeros((s.n, 0)), fix_dofs=np.zeros(0, np.int32))
        plain.append(dataclasses.replace(s, K_val=val, **none))
        scal.append(dataclasses.replace(s, K_val=val * S[rows] * S[s.K_col], f=s.f * S, **none))
        lam[s.B_lambda] = S[s.B_dof]
    return dataclasses.replace(P, subs=plain), dataclasses.replace(P, subs=scal), g, lam


def problem(dim, physics, cuts, seed=1):
    return scaled(make_problem(dim=dim, physics=physics, cuts=cuts, material="lognormal", sigma=0.5, seed=seed), seed)


@pytest.mark.parametrize("dim,physics,cuts", CASES)
def test_factor(dim, physics, cuts):
    """The Cholesky, seen through the implicit operator (FP64 substitutions); the bar is that of its own test."""
    P, Q, _, lam = problem(dim, physics, cuts)
    p = seeded_vector(P.n_lambda, 6)
    op = feti.FetiOperator(Q, prec="fp64", chol_tc_front=128)
    op.assemble()
    q = op.apply_implicit(torch.from_numpy(p * lam).cuda()).cpu().numpy() * lam
    op.close()
    ref, size, kappa = np.zeros_like(q), 0.0, 0.0
    for s in P.subs:
        l = np.asarray(s.B_lambda, dtype=np.int64)
        K = O.K_dense(s)
        part = O.local_F(s, K) @ p[l]
        ref[l] += part
        size += np.linalg.norm(part)
        kappa = max(kappa, np.linalg.cond(K, 1))
    assert np.linalg.norm(q - ref) <= 8 * 2.0 ** -53 * kappa * size


@pytest.mark.parametrize("dim,physics,cuts", CASES)
def test_F(dim, physics, cuts):
    """The forward solve and the SYRK, at the FP64 parity bar."""
    P, Q, _, lam = problem(dim, physics, cuts)
    op = feti.FetiOperator(Q, prec="fp64", chol_tc_front=128)
    op.assemble()
    for i, s in enumerate(P.subs):
        l = lam[s.B_lambda]
        F = op.get_F(i) * l[:, None] * l[None, :]
        Fo = O.local_F(s, O.K_dense(s))
        assert np.linalg.norm(F - Fo) <= 1e-12 * np.linalg.norm(Fo)
    op.close()


@pytest.mark.parametrize("dim,physics,cuts", CASES)
def test_backward(dim, physics, cuts):
    """The backward solve: F_i of the TRSM-path assembly, at the FP64 parity bar."""
    P, Q, _, lam = problem(dim, physics, cuts)
    op = feti.FetiOperator(Q, prec="fp64", chol_tc_front=128, route="trsm")
    op.assemble()
    for i, s in enumerate(P.subs):
        l = lam[s.B_lambda]
        F = op.get_F(i) * l[:, None] * l[None, :]
        Fo = O.local_F(s, O.K_dense(s))
        assert np.linalg.norm(F - Fo) <= 1e-12 * np.linalg.norm(Fo)
    op.close()


@pytest.mark.parametrize("physics,elems", [("elasticity", 7), ("heat", 13)])
def test_adjoint(physics, elems):
    """One subdomain with element matrices and weights scaled along, at the adjoint's parity bar (the gradient does not
    change under the scaling)."""
    P, Q, g, lam = problem(3, physics, [[elems]] * 3)
    s, S = P.subs[0], g[P.subs[0].l2g]
    W = make_W(P, seed=0)[0]
    Se = S[s.elem_dofs]
    Q = dataclasses.replace(Q, K_ref=np.asarray(P.K_ref)[None] * Se[:, :, None] * Se[:, None, :])
    op = feti.FetiOperator(Q, prec="fp64", chol_tc_front=128, with_elements=True, per_element=True)
    op.assemble()
    l = lam[s.B_lambda]
    grad = op.adjoint([W * l[:, None] * l[None, :]]).cpu().numpy()
    op.close()
    go = O.gradient_sub(s, W, P.K_ref, Kr=O.K_dense(s))
    assert np.linalg.norm(grad - go) <= 1e-10 * np.linalg.norm(go)


@pytest.mark.parametrize("kernel", [0, 6])
@pytest.mark.parametrize("dim,physics,cuts", CASES + [(2, "heat", [[31, 34], [34, 31]])])
def test_apply(dim, physics, cuts, kernel):
    """The explicit apply against its own F_i.  Bar: n 2^-52 (|F| |p|)_l for FP64 sums in any order; the tile kernel by
    digits has F_ij / (s_i s_j) below 4 and p_j s_j below sqrt(F_jj) |p_j| (s_j = 2^floor(log2 F_jj / 2)), each cut to
    within 2^-62 of the next power of two above its largest and multiplied without the pairs p + q >= 8 (7.1 2^-62 at
    most): below 2^-55 sqrt(F_ll) max_j sqrt(F_jj) |p_j| a product."""
    P, Q, _, lam = problem(dim, physics, cuts)
    op = feti.FetiOperator(Q, prec="fp64", apply_kernel=kernel)
    op.assemble()
    Fs = [op.get_F(i) * lam[s.B_lambda][:, None] * lam[s.B_lambda] for i, s in enumerate(P.subs)]
    rng = np.random.default_rng(4)
    for k in range(3):
        p = rng.normal(size=P.n_lambda)
        if k == 1:
            p *= np.exp2(rng.integers(-30, 30, size=P.n_lambda))
        if k == 2:
            p[rng.random(P.n_lambda) < 0.95] = 0.0
        q = op.apply(torch.from_numpy(p * lam).cuda()).cpu().numpy() * lam
        ref, bar = np.zeros_like(q), np.zeros_like(q)
        for s, F in zip(P.subs, Fs):
            l = np.asarray(s.B_lambda, dtype=np.int64)
            ref[l] += F @ p[l]
            d = np.sqrt(np.diag(F))
            bar[l] += (s.m + 8) * (2.0 ** -52 * (np.abs(F) @ np.abs(p[l])) + 2.0 ** -55 * d * (d * np.abs(p[l])).max())
        assert np.all(np.abs(q - ref) <= bar)
    op.close()


def test_dirichlet_tiles():
    """The Dirichlet preconditioner's tiles by either tile kernel: the same solution at the solve's tolerance."""
    P = make_problem(dim=2, physics="heat", cuts=[[12, 9], [9, 12]], material="lognormal", sigma=1.0, seed=2)
    um = O.monolithic_solve(P)
    for kernel in (0, 6):
        op = feti.FetiOperator(P, prec="fp64", route="schur", precond="dirichlet", apply_kernel=kernel, tol=1e-12)
        op.assemble()
        u, info = op.solve()[2:]
        u = u.cpu().numpy()
        op.close()
        assert info["converged"]
        off = 0
        for s in P.subs:
            assert np.abs(u[off:off + s.n] - um[s.l2g]).max() <= 1e-10 * np.abs(um).max()
            off += s.n
