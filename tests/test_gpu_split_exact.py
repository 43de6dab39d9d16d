"""The split forms against exact values where the digits of many terms add up
in step: constant couplings, right-hand sides and cotangents (uniform
coupling, mean-field blocks), for which the result is a few rational
operations.  Every product is rounded once, on top of at most 2^-52 of the
sum of its terms' magnitudes (the operands' grid and the dropped digits)."""
from fractions import Fraction as F

import numpy as np
import pytest
import torch

import paper_1807_00370_gb300 as crs

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


def _constants(m, seed):
    """Couplings c (1 + i), m |c (1 + i)| <= 0.7."""
    return [0.007 * 64 / m] + list(np.random.default_rng(seed).uniform(0.1, 0.49, 24) / m)


@pytest.mark.parametrize("m", [11, 16, 24, 32, 40, 64])
def test_constant_coupling(cuda_ok, m):
    """A = I, B = c (1 + i) times the all-ones matrix, y constant in each block:
    the reduced block I - B B^H, and x in the span of the all-ones vectors."""
    k = 3
    A = torch.eye(m, dtype=torch.complex128, device="cuda").expand(2, m, m).contiguous()
    eye = np.eye(m)
    for c in _constants(m, m):
        B = torch.full((1, m, m), complex(c, c), dtype=torch.complex128, device="cuda")
        y = torch.ones(2, m, k, dtype=torch.complex128, device="cuda")
        y[1] = 0.3
        plan = crs.Plan(2, m, k)
        crs.crsolve_factor(plan, A, B)
        x = crs.crsolve_solve(plan, y).cpu().numpy()
        V = crs.crsolve_debug_level_system(plan, 1)[0].cpu().numpy().reshape(m, m)
        assert crs.crsolve_info_get(plan)["status"] == 0
        w = m * 2 * F(c) ** 2
        # Z is rounded once from B: three roundings and the product's 2^-52
        off = ~eye.astype(bool)
        assert np.abs(V[off] + float(w)).max() <= 8 * U * float(w), c
        assert np.abs(V[~off] - float(1 - w)).max() <= 8 * U, c
        # x_1 + conj(b) x_2 = 1, b x_1 + x_2 = 0.3 with b = m c (1 + i)
        bb, f = m * F(c), F(0.3)
        den = 1 - 2 * bb * bb
        x1 = complex(float((1 - bb * f) / den), float(bb * f / den))
        x2 = complex(float((f - bb) / den), float(-bb / den))
        # condition of the 2 x 2 system times the steps' roundings
        cond = (1 + 0.7) / (1 - 0.7)
        for got, ref in ((x[0], x1), (x[1], x2)):
            assert np.abs(got - ref).max() <= 16 * cond * U * max(abs(x1), abs(x2)), c


@pytest.mark.parametrize("m,k", [(8, 4), (12, 11), (16, 16), (16, 32), (33, 24), (64, 32)])
def test_constant_outer_products(cuda_ok, m, k):
    """A = I, B = 0 and constant x, g: every gradient entry is the same product."""
    N = 3
    A = torch.eye(m, dtype=torch.complex128, device="cuda").expand(N, m, m).contiguous()
    B = torch.zeros(N - 1, m, m, dtype=torch.complex128, device="cuda")
    plan = crs.Plan(N, m, k)
    crs.crsolve_factor(plan, A, B)
    rng = np.random.default_rng(k)
    for p, q in rng.uniform(0.5, 1.0, (24, 2)):
        x = torch.full((N, m, k), complex(p, 0.0), dtype=torch.complex128, device="cuda")
        g = torch.full((N, m, k), complex(q, 0.0), dtype=torch.complex128, device="cuda")
        gy, gA, gB = (t.cpu().numpy() for t in crs.crsolve_backward(plan, x, g))
        assert (gy == q).all()
        ref = float(k * F(p) * F(q))
        assert np.abs(gA + ref).max() <= 4 * U * ref, (p, q)
        assert np.abs(gB + 2 * ref).max() <= 8 * U * ref, (p, q)
