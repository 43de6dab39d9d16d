"""GPU parity of the tensor-core forms of the FP64 levels (m = 7, 8 and m >= 12)
where they can go wrong: blocks that do and do not fill their 8 x 8 tiles,
one to several column tiles, single blocks, badly scaled unknowns, and
entries outside the range of the splitting (tiny couplings, infinities,
NaN).  Every product is rounded about once, so the forward error is at most
that of the FP64 oracle: the bound is the parity tests' 1e-12."""
import numpy as np
import pytest
import torch

import oracle
import synthetic
import paper_1807_00370_gb300 as crs
from tests.gpu_helpers import rel_err, to_dev

pytestmark = pytest.mark.gpu

TOL = 1e-12


def _solve(A, B, y):
    N, m, k = y.shape
    dA, dB, dy = to_dev(A, B, y)
    plan = crs.Plan(N, m, k)
    crs.crsolve_factor(plan, dA, dB if N > 1 else None)
    return crs.crsolve_solve(plan, dy).cpu().numpy(), crs.crsolve_info_get(plan)


@pytest.mark.parametrize("m", [7, 8, 12, 15, 16, 17, 24, 31, 32, 33, 41, 57, 63, 64])
@pytest.mark.parametrize("N,k", [(1, 1), (2, 9), (3, 8), (37, 1), (130, 17)])
def test_block_sizes(cuda_ok, m, N, k):
    A, B, y = synthetic.gen_system(N, m, k, seed=m + N)
    x, info = _solve(A, B, y)
    xo, io = oracle.cr_solve(A, B, y)
    assert info == io
    assert rel_err(x, xo) <= TOL


@pytest.mark.parametrize("m", [8, 16, 40])
def test_scaled_unknowns(cuda_ok, m):
    """D A D, D B D, D y with D = powers of two over 2^-60 .. 2^60 inside a
    block: the solution D^-1 x in every component to the same relative error
    (FMAs and substitution keep it, exactly for powers of two)."""
    N, k = 33, 3
    A, B, y = synthetic.gen_system(N, m, k, seed=7 * m)
    d = 2.0 ** np.random.default_rng(m).integers(-60, 61, size=(N, m))
    As = A * d[:, :, None] * d[:, None, :]
    Bs = B * d[1:, :, None] * d[:-1, None, :]
    x, info = _solve(As, Bs, y * d[:, :, None])
    xo, _ = oracle.cr_solve(A, B, y)
    assert info["status"] == 0
    assert rel_err(x * d[:, :, None], xo) <= TOL


@pytest.mark.parametrize("m", [8, 16, 24])
@pytest.mark.parametrize("scale", [1e-300, 1e-160, 1e-40, 1e130])
def test_scaled_systems(cuda_ok, m, scale):
    """A right-hand side, or the couplings, scaled far down or up."""
    N, k = 40, 2
    A, B, y = synthetic.gen_system(N, m, k, seed=m)
    xo, _ = oracle.cr_solve(A, B, y)
    x, _ = _solve(A, B, y * scale)
    assert rel_err(x / scale, xo) <= TOL
    if scale < 1:
        x, info = _solve(A, B * scale, y)
        xo, _ = oracle.cr_solve(A, B * scale, y)
        assert info["status"] == 0 and rel_err(x, xo) <= TOL


@pytest.mark.parametrize("m", [8, 16, 24])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_nonfinite_right_hand_side_stays_in_its_column(cuda_ok, m, bad):
    N, k = 29, 11
    A, B, y = synthetic.gen_system(N, m, k, seed=m)
    xo, _ = oracle.cr_solve(A, B, y)
    y = y.copy()
    y[N // 2, m // 2, 4] = bad
    x, info = _solve(A, B, y)
    assert info["status"] == 0
    keep = [c for c in range(k) if c != 4]
    assert rel_err(x[:, :, keep], xo[:, :, keep]) <= TOL
    assert not np.isfinite(x[:, :, 4]).any()


@pytest.mark.parametrize("m", [8, 16, 24])
@pytest.mark.parametrize("where", ["A", "B"])
def test_nonfinite_matrix_is_a_breakdown_where_the_oracle_says(cuda_ok, m, where):
    N, k = 29, 2
    A, B, y = synthetic.gen_system(N, m, k, seed=m)
    if where == "A":
        A[7, m - 1, m - 1] = np.nan
    else:
        B[7, 0, m - 1] = np.nan
    x, info = _solve(A, B, y)
    _, io = oracle.cr_solve(A, B, y)
    assert io["status"] == 1 and info == io
    assert np.isnan(x).all()


@pytest.mark.parametrize("m,k", [(7, 4), (8, 2), (8, 9), (9, 16), (12, 5), (16, 8), (17, 32), (33, 3), (64, 17)])
def test_outer_products(cuda_ok, m, k):
    """The gradients' outer products by tiles against the formula in numpy
    from the call's own x and g_y, with columns of very different scale: each
    gradient entry sums 2k products, so both sides are within 4k ulp of the
    sum of the products' magnitudes."""
    N = 21
    A, B, y = synthetic.gen_system(N, m, k, seed=m + k)
    s = 2.0 ** np.random.default_rng(k).integers(-30, 31, size=k)
    dA, dB, dy, dg = to_dev(A, B, y * s, synthetic.gen_cotangent(N, m, k, seed=m) / s)
    plan = crs.Plan(N, m, k)
    crs.crsolve_factor(plan, dA, dB)
    x = crs.crsolve_solve(plan, dy)
    gy, gA, gB = (t.cpu().numpy() for t in crs.crsolve_backward(plan, x, dg))
    x = x.cpu().numpy()
    h = lambda t: np.conj(np.swapaxes(t, 1, 2))
    tol = 4 * k * 2.0 ** -53
    ref, mag = gy @ h(x), np.abs(gy) @ h(np.abs(x))
    assert (np.abs(gA + 0.5 * (ref + h(ref))) <= tol * (mag + h(mag))).all()
    ref = gy[1:] @ h(x[:-1]) + x[1:] @ h(gy[:-1])
    mag = np.abs(gy[1:]) @ h(np.abs(x[:-1])) + np.abs(x[1:]) @ h(np.abs(gy[:-1]))
    assert (np.abs(gB + ref) <= tol * mag).all()
