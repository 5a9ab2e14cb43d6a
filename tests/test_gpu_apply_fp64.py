"""FP64 explicit apply against the assembled F_i, whichever tile kernel the autotuner keeps: subdomains with fewer than
64 multipliers, ragged last blocks, p over many binades, zeros, infinities and NaN.

Bar: q_l sums products F_ab p_b and the partials of at most nb + 1 tiles; FP64 summation in any order is off by at most
n 2^-52 (|F| |p|)_l for n terms, and the sliced tiles lie within 2^-60 of their strip's and vector block's largest
entries per product, which 64 2^-52 max |F| max |p| covers (the second term of the bar)."""
import numpy as np
import pytest
import torch

from paper_2502_08382_gb300 import feti
from paper_2502_08382_gb300.problems import make_problem

pytestmark = pytest.mark.gpu

CASES = [
    (2, "heat", [[2, 3], [3, 2]]),
    (2, "heat", [[16, 15], [15, 16]]),
    (2, "heat", [[31, 34], [34, 31]]),
    (3, "heat", [[4, 6, 5]] * 3),
    (3, "elasticity", [[5, 4]] * 3),
]


@pytest.mark.parametrize("dim,physics,cuts", CASES)
def test_apply_matches_F(dim, physics, cuts):
    P = make_problem(dim=dim, physics=physics, cuts=cuts, material="lognormal", sigma=0.5)
    op = feti.FetiOperator(P, prec="fp64")
    op.assemble()
    Fs = [op.get_F(i) for i in range(P.nsub)]
    rng = np.random.default_rng(3)
    for k in range(4):
        p = rng.normal(size=P.n_lambda)
        if k == 1:
            p *= np.exp2(rng.integers(-40, 40, size=P.n_lambda))
        if k == 2:
            p[rng.random(P.n_lambda) < 0.9] = 0.0
        if k == 3:
            p = np.zeros(P.n_lambda)
        q = op.apply(torch.from_numpy(p).cuda()).cpu().numpy()
        ref, bar, n = np.zeros_like(q), np.zeros_like(q), np.zeros_like(q)
        for s, F in zip(P.subs, Fs):
            l = np.asarray(s.B_lambda, dtype=np.int64)
            ref[l] += F @ p[l]
            bar[l] += (s.m + 8) * 2.0 ** -52 * (np.abs(F) @ np.abs(p[l])) \
                + 64 * 2.0 ** -52 * np.abs(F).max() * np.abs(p[l]).max()
            n[l] += 1
        assert np.all(np.abs(q - ref) <= bar)
        assert np.array_equal(q, op.apply(torch.from_numpy(p).cuda()).cpu().numpy())
    op.close()


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_special_values(bad):
    P = make_problem(dim=2, physics="heat", cuts=[[20, 17], [17, 20]], material="lognormal", sigma=0.5)
    op = feti.FetiOperator(P, prec="fp64")
    op.assemble()
    p = np.random.default_rng(1).normal(size=P.n_lambda)
    j = P.n_lambda // 2
    p[j] = bad
    q = op.apply(torch.from_numpy(p).cuda()).cpu().numpy()
    touched = np.zeros(P.n_lambda, dtype=bool)
    for i, s in enumerate(P.subs):
        l = np.asarray(s.B_lambda, dtype=np.int64)
        if j in l:
            touched[l] = True
    assert touched.any() and not touched.all()
    # F_i is dense: every multiplier of the subdomains that hold j is reached, no other one
    assert not np.isfinite(q[touched]).any() and np.isfinite(q[~touched]).all()
    op.close()
