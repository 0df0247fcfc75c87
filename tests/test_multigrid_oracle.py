"""The FP64 definition of the multigrid V-cycle: its fine operator is the oracle's, it is symmetric and positive, and as a
preconditioner it solves in a few iterations -- on grids whose periodic axes join positions of one colour too."""
import numpy as np
import pytest

import oracle
import workloads as W
from oracle.multigrid import VCycle

CASES = [((24, 20, 13), (1, 2, 3, 3, 3, 3)), ((22, 22, 22), (0,) * 6), ((25, 12, 9), (0, 0, 3, 3, 0, 0)), ((28, 12, 12), (1, 2, 0, 0, 0, 0))]


@pytest.mark.parametrize("body", [False, True])
@pytest.mark.parametrize("shape,bc", CASES)
def test_the_vcycle_is_a_symmetric_preconditioner(shape, bc, body):
    ref = oracle.Case(*shape, bc=bc)
    if body:
        ref.classify(W.random_soup(60, (0.5, 0.5, 0.5), tuple(n - 0.5 for n in shape), 4.0, seed=8))
    V = VCycle(shape, bc, ref.flags, target=60)
    L = V.lev[0]
    A = lambda x: L.W @ x - L.dg * x  # noqa: E731
    rng = np.random.default_rng(1)
    a, b = rng.standard_normal((2, L.n))
    assert np.allclose(A(a), ref.apply(a), rtol=0, atol=1e-12)
    # reciprocal diagonals are rounded to FP32 on the coarse levels
    assert abs(a @ V(b) - V(a) @ b) <= 2.0 ** -24 * np.linalg.norm(a) * np.linalg.norm(V(b))
    assert a @ V(a) < 0 and b @ V(b) < 0                       # A is negative definite, V approximates its inverse
    rhs = A(rng.standard_normal(L.n))
    x, r, p, rz = np.zeros(L.n), rhs, 0.0, 1.0
    for it in range(1, 61):
        z = V(r)
        n = r @ z
        p = z + (n / rz if it > 1 else 0.0) * p
        rz, q = n, A(p)
        x, r = x + rz / (p @ q) * p, r - rz / (p @ q) * q
        if np.linalg.norm(r) <= 1e-8 * np.linalg.norm(rhs):
            break
    assert it <= (40 if body else 12), it
