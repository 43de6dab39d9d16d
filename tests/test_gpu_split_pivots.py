"""Pivots of the split factor at the ends of the range: 1 / pivot is not a
normal number for pivots below 2^-1022 or above 2^1022, and the elimination
divides by them."""
import numpy as np
import pytest

import paper_1807_00370_gb300 as crs
from tests.gpu_helpers import rel_err, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [7, 8, 11, 16, 24, 40])
@pytest.mark.parametrize("N", [2, 150, 2500])
@pytest.mark.parametrize("e", [-1036, -1023, -1000, 990, 1019])
def test_scaled_matrix(cuda_ok, m, N, e):
    """2^e A x = 2^e y with tridiagonal A_j and B = 0, which 2^e scales exactly: x is
    that of e = 0.  Below 2^-1022 the elimination works on subnormal numbers
    (absolute rounding 2^-1074), m of which add up in a condition of 3."""
    k = 2
    A = np.zeros((N, m, m), complex)
    A[:] = 2.0 * np.eye(m)
    i = np.arange(m - 1)
    A[:, i + 1, i] = A[:, i, i + 1] = 0.5
    B = np.zeros((N - 1, m, m), complex)
    y = np.random.default_rng(m).integers(1, 9, (N, m, k)).astype(complex)
    s = np.ldexp(1.0, e)
    dA, dB, dy = to_dev(A * s, B, y * s)
    plan = crs.Plan(N, m, k)
    crs.crsolve_factor(plan, dA, dB)
    x = crs.crsolve_solve(plan, dy).cpu().numpy()
    assert crs.crsolve_info_get(plan)["status"] == 0
    ref = np.linalg.solve(A[0], y.transpose(1, 0, 2).reshape(m, N * k)).reshape(m, N, k).transpose(1, 0, 2)
    assert rel_err(x, ref) <= max(1e-12, 3 * m * 2.0 ** (-1074 - e))
