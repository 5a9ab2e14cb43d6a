"""Kernels that a rule or an autotuner picks, each forced through its option, so that none goes untested because another
was faster: every tile kernel of the explicit apply, and the implicit solves on one 256-thread CTA or a cluster of 1, 2, 4
or 8 wide ones per subdomain (whose results are the same bit for bit).

Bars.  Apply: q_l sums products F_ab p_b and the partials of at most nb + 1 tiles; FP64 summation in any order is off by
at most n 2^-52 (|F| |p|)_l for n terms, and a sliced tile by 64 2^-52 max |F| max |p| at most.  Implicit operator: as in
test_gpu_implicit_cluster.py, 8 u kappa_1(K_reg) |q_i| per subdomain."""
import numpy as np
import pytest
import torch

from oracle import feti_oracle as O
from paper_2502_08382_gb300 import feti
from paper_2502_08382_gb300.problems import make_problem, seeded_vector

pytestmark = pytest.mark.gpu

APPLY = [
    (2, "heat", [[2, 3], [3, 2]]),
    (2, "heat", [[31, 34], [34, 31]]),
    (3, "heat", [[4, 6, 5]] * 3),
]


@pytest.mark.parametrize("kernel", range(7))
@pytest.mark.parametrize("dim,physics,cuts", APPLY)
def test_apply_kernels(dim, physics, cuts, kernel):
    P = make_problem(dim=dim, physics=physics, cuts=cuts, material="lognormal", sigma=0.5)
    op = feti.FetiOperator(P, prec="fp64", apply_kernel=kernel)
    op.assemble()
    assert op.stats()["apply_variant"] == kernel
    Fs = [op.get_F(i) for i in range(P.nsub)]
    rng = np.random.default_rng(3)
    for k in range(4):
        p = rng.normal(size=P.n_lambda)
        if k == 1:
            p *= np.exp2(rng.integers(-40, 40, size=P.n_lambda))
        if k == 2:
            p[rng.random(P.n_lambda) < 0.9] = 0.0
        if k == 3:
            p *= 2.0 ** -900
        q = op.apply(torch.from_numpy(p).cuda()).cpu().numpy()
        ref, bar = np.zeros_like(q), np.zeros_like(q)
        for s, F in zip(P.subs, Fs):
            l = np.asarray(s.B_lambda, dtype=np.int64)
            ref[l] += F @ p[l]
            bar[l] += (s.m + 8) * 2.0 ** -52 * (np.abs(F) @ np.abs(p[l])) \
                + 64 * 2.0 ** -52 * np.abs(F).max() * np.abs(p[l]).max()
        assert np.all(np.abs(q - ref) <= bar)
    for bad in (np.nan, np.inf):
        p = rng.normal(size=P.n_lambda)
        p[P.n_lambda // 2] = bad
        q = op.apply(torch.from_numpy(p).cuda()).cpu().numpy()
        touched = np.zeros(P.n_lambda, dtype=bool)
        for s in P.subs:
            l = np.asarray(s.B_lambda, dtype=np.int64)
            if P.n_lambda // 2 in l:
                touched[l] = True
        assert not np.isfinite(q[touched]).any() and np.isfinite(q[~touched]).all()
    op.close()


@pytest.mark.parametrize("dim,physics,cuts", [
    (2, "heat", [[40, 3], [40, 3]]),
    (3, "heat", [[9, 2, 7]] * 3),
    (3, "elasticity", [[8, 5]] * 3),
])
def test_implicit_clusters(dim, physics, cuts):
    P = make_problem(dim=dim, physics=physics, cuts=cuts, material="lognormal", sigma=0.5, seed=4)
    p = seeded_vector(P.n_lambda, 6)
    ref, size, kappa = np.zeros(P.n_lambda), 0.0, 0.0
    for s in P.subs:
        l = np.asarray(s.B_lambda, dtype=np.int64)
        K = O.K_reg(s)
        part = O.local_F(s, K) @ p[l]
        ref[l] += part
        size += np.linalg.norm(part)
        kappa = max(kappa, np.linalg.cond(K, 1))
    wide = []
    for c in (-1, 1, 2, 4, 8):
        op = feti.FetiOperator(P, prec="fp64", implicit_cluster=c, tol=1e-11)
        op.assemble()
        assert op.stats()["implicit_cluster"] == c
        q = op.apply_implicit(torch.from_numpy(p).cuda()).cpu().numpy()
        u = op.solve()[2].cpu().numpy()
        op.close()
        assert np.linalg.norm(q - ref) <= 8 * 2.0 ** -53 * kappa * size
        if c > 0:
            wide.append((q, u))
    for q, u in wide[1:]:
        assert np.array_equal(q, wide[0][0]) and np.array_equal(u, wide[0][1])


def test_refused_options():
    P = make_problem(dim=2, physics="heat", cuts=[[4, 4], [4, 4]])
    for kw in ({"implicit_cluster": 3}, {"implicit_cluster": 16}, {"apply_kernel": 7}, {"apply_kernel": 6, "prec": "tf32"}):
        with pytest.raises(feti.FetiError):
            feti.FetiOperator(P, **kw)


@pytest.mark.parametrize("kernel", [0, 6])
def test_apply_top_binade(kernel):
    """Results between 2^1023 and the largest FP64 number are finite: column j of F, scaled by a power of two that takes
    its largest off-diagonal entry there (one product an entry: exact up to the tiles' cut, 2^-55 max |F|)."""
    P = make_problem(dim=2, physics="heat", cuts=[[30], [30]], material="lognormal", sigma=0.5)
    op = feti.FetiOperator(P, prec="fp64", apply_kernel=kernel)
    op.assemble()
    F, j = op.get_F(0), P.n_lambda // 2
    off = np.delete(F[:, j], j)
    k = 1023 - int(np.floor(np.log2(np.abs(off).max())))
    p = np.zeros(P.n_lambda)
    p[j] = 2.0 ** k if k < 1024 else 2.0 ** 1023
    q = np.delete(op.apply(torch.from_numpy(p).cuda()).cpu().numpy(), j)
    op.close()
    assert np.isfinite(q).all()
    assert np.abs(q / p[j] - off).max() <= 2.0 ** -55 * np.abs(F).max()
    if k < 1024:
        assert np.abs(q).max() >= 2.0 ** 1023


@pytest.mark.parametrize("kernel", range(7))
def test_apply_subnormal(kernel):
    """p of subnormal numbers (and one of a single smallest one): products and sums are multiples of 2^-1074, each rounded
    to within half of it, so m + 8 of them are off by as many at most."""
    P = make_problem(dim=2, physics="heat", cuts=[[30], [30]], material="lognormal", sigma=0.5)
    op = feti.FetiOperator(P, prec="fp64", apply_kernel=kernel)
    op.assemble()
    F = op.get_F(0)
    rng = np.random.default_rng(5)
    k = rng.integers(-2 ** 40, 2 ** 40, size=P.n_lambda)
    for ints in (k, np.eye(1, P.n_lambda, P.n_lambda // 2, dtype=np.int64)[0]):
        p = ints.astype(np.float64) * 2.0 ** -1074
        q = op.apply(torch.from_numpy(p).cuda()).cpu().numpy()
        ref = F @ ints  # in units of 2^-1074
        got = np.ldexp(q, 600) * 2.0 ** 474
        assert np.abs(got - ref).max() <= P.n_lambda + 8 + 2.0 ** -40 * np.abs(ref).max()
        assert np.abs(got).max() > 0
    op.close()
