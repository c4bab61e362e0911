"""Factors of single subsystems at the edges of the precompute kernel (columns at
multiples of 32 and 64 and the largest, shared memory or global scratch, both
factor kinds, dependent rows): two FP64 iterations against the projection taken
from a dense pseudo-inverse.  Tolerance: the factors are orthonormal to a few
ulps times n (Gram-Schmidt applied twice), the iterates are of order 5, so
1e-16 * 256 * 40 ~ 1e-12 at the largest size; 1e-10 leaves the rest to the
condition of the random rows (at most some 1e2 here)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 63, 64, 65, 128, 255, 256])
@pytest.mark.parametrize("share", [0.3, 0.9])
def test_one_subsystem(n, share):
    from paper_2310_09410_gb300 import opf

    rng = np.random.default_rng(1000 * n + int(10 * share))
    m = max(1, int(share * n))
    A = rng.standard_normal((m, n))
    if m > 2:
        A[m // 2] = A[0] - 2.0 * A[1]                      # a dependent row, consistent with the point below
    point = rng.uniform(-1.0, 1.0, n)
    c = rng.standard_normal(n)
    lb, ub = -5.0 * np.ones(n), 5.0 * np.ones(n)
    solver = opf.Solver.from_generic(c, lb, ub, [dict(idx=np.arange(n), A=A, b=A @ point)])
    solver.precompute()
    solver.solve(rho=10.0, eps_rel=0.0, max_iter=2, check_every=2, precision=opf.PREC_FP64, engine=1)
    got, _ = solver.solution()
    solver.close()
    pinv = np.linalg.pinv(A, rcond=1e-9)
    x0 = np.clip(np.zeros(n), lb, ub)
    xs, lam, rho = None, np.zeros(n), 10.0
    # the start is the library's own (bounds' midpoints, 0 here): x_s = x0, lambda = 0
    xs = x0.copy()
    for _ in range(2):
        x = np.clip(xs - lam / rho - c / rho, lb, ub)
        v = x + lam / rho
        xs = v - pinv @ (A @ v) + pinv @ (A @ point)
        lam = lam + rho * (x - xs)
    assert np.max(np.abs(got - x)) <= 1e-10
