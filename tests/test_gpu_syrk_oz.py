"""FP64 SYRK by exact slicing on the tensor cores, at the edges of its tiles, batches and memory limits.

Bars: each entry of X^T X is a sum of at most n products, so FP64 summation in any order is off by at most
n 2^-53 sqrt(F_aa F_bb), hence n 2^-53 tr(F) in the Frobenius norm; the sliced sum (62-bit digits, exact integer
accumulation, two final roundings) lies inside that.  Two assemblies from the same factor may differ by twice it.
Against the oracle (its own factorisation): the FP64 parity bar 1e-12."""
import numpy as np
import pytest
import torch

from oracle import feti_oracle as O
from paper_2502_08382_gb300 import feti
from paper_2502_08382_gb300.problems import make_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,physics,cuts", [
    (2, "heat", [[2, 3], [3, 2]]),          # m far below one 64-wide block
    (2, "heat", [[15, 17], [17, 15]]),      # m on both sides of 64
    (2, "heat", [[31, 33], [33, 31]]),      # m on both sides of 128
    (3, "heat", [[4, 6, 5]] * 3),           # ragged last block rows, many narrow supernodes
    (3, "elasticity", [[5, 4]] * 3),        # several 128-row tiles
])
def test_against_oracle(dim, physics, cuts):
    P = make_problem(dim=dim, physics=physics, cuts=cuts, material="lognormal", sigma=0.5)
    op = feti.FetiOperator(P, prec="fp64")
    op.assemble()
    for i, s in enumerate(P.subs):
        Fo = O.local_F(s)
        assert np.linalg.norm(op.get_F(i) - Fo) <= 1e-12 * np.linalg.norm(Fo)
    op.assemble()  # the captured launches
    Fo = O.local_F(P.subs[-1])
    assert np.linalg.norm(op.get_F(P.nsub - 1) - Fo) <= 1e-12 * np.linalg.norm(Fo)
    op.close()


@pytest.mark.parametrize("refuse", ["digits_once", "all_large"])
def test_small_memory(monkeypatch, refuse):
    """One subdomain per batch when the full digit buffer is refused; the FP64-pipe kernel when every one is."""
    P = make_problem(dim=3, physics="elasticity", cuts=[[6, 5]] * 3, material="lognormal", sigma=0.5)
    ref = feti.FetiOperator(P, prec="fp64")
    ref.assemble()
    real, armed, refused = torch.cuda.caching_allocator_alloc, [False], [0]

    def alloc(nbytes, *a, **k):
        if armed[0] and nbytes > 1 << 20 and (refuse == "all_large" or refused[0] == 0):
            refused[0] += 1
            raise torch.cuda.OutOfMemoryError("refused by the test")
        return real(nbytes, *a, **k)

    monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", alloc)
    op = feti.FetiOperator(P, prec="fp64")
    armed[0] = True
    op.assemble()
    armed[0] = False
    assert refused[0] == (2 if refuse == "all_large" else 1)
    for i, s in enumerate(P.subs):
        Fa, Fb = ref.get_F(i), op.get_F(i)
        assert np.linalg.norm(Fa - Fb) <= 2 * s.n * 2.0 ** -53 * np.trace(Fa)
    op.close()
    ref.close()
