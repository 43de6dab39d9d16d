"""Results of the split forms that are much smaller than the largest operands
of their tile: a localised source in a diagonal or a banded block, rows of
other units, a tiny imaginary part.  FMAs keep each to its own terms'
magnitudes; so do the split forms, which form such results by FMAs.

Bounds (split_guard): over K real terms a result is within K 2^-45.3 of the
sum of its terms' moduli, and each part within K 2^-39.3 of the sum of its
own real products, where all errors of the terms add up."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import synthetic
import paper_1807_00370_gb300 as crs
from tests import split_device
from tests.gpu_helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib(tmp_path_factory, cuda_ok):
    return split_device.load(tmp_path_factory.mktemp("split"))


def _exact_sum(terms):
    """Correctly rounded sums of exact products (two-part) over the last axis."""
    from fractions import Fraction
    flat = terms.reshape(-1, *terms.shape[-2:])
    out = [float(sum(Fraction(p) * Fraction(q) for p, q in row if p and q)) for row in flat.tolist()]
    return np.array(out).reshape(terms.shape[:-2])


@pytest.mark.parametrize("kind", [0, 1, 2])
@pytest.mark.parametrize("ks", [1, 2, 4, 8, 16])
@pytest.mark.parametrize("spread", ["none", "entries", "rows", "imag", "sparse"])
def test_tile(lib, kind, ks, spread):
    K = 8 * ks
    rng = np.random.default_rng(1000 * ks + 10 * kind + len(spread))
    a, b = (rng.standard_normal((2, 8, K)) + 1j * rng.standard_normal((2, 8, K)))
    if spread == "entries":
        a *= 2.0 ** rng.integers(-70, 1, (8, K))
        b *= 2.0 ** rng.integers(-70, 1, (8, K))
    elif spread == "rows":
        a *= 2.0 ** rng.integers(-70, 71, (8, 1))
        b *= 2.0 ** rng.integers(-70, 71, (8, 1))
    elif spread == "imag":
        a = a.real + 1e-20j * a.imag
        b = b.real + 0j
    elif spread == "sparse":
        a *= rng.random((8, K)) < 0.2
        b *= (rng.random((8, K)) < 0.3) * 2.0 ** rng.integers(-40, 1, (8, K))
    da, db = to_dev(a, b)
    out = torch.empty(8, 8, dtype=torch.complex128, device="cuda")
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    torch.cuda.synchronize()
    assert lib.split_tile_device(kind, ks, p(da), p(db), p(out)) == 0
    x, y = (np.conj(a) if kind == 0 else a)[:, None, :], (np.conj(b) if kind == 2 else b)[None, :, :]
    x, y = np.broadcast_arrays(x, y)
    st = lambda u, v: np.stack([u, v], -1)
    re = np.concatenate([st(x.real, y.real), st(-x.imag, y.imag)], -2)
    im = np.concatenate([st(x.real, y.imag), st(x.imag, y.real)], -2)
    got = out.cpu().numpy()
    moduli = (np.abs(x) * np.abs(y)).sum(-1)
    for part, terms in ((got.real, re), (got.imag, im)):
        err = np.abs(part - _exact_sum(terms))
        own = np.abs(terms[..., 0] * terms[..., 1]).sum(-1)
        assert (err <= 2 * K * 2.0 ** -39.3 * own).all()
        assert (err <= 2 * K * 2.0 ** -45.3 * moduli + 2.0 ** -52 * own).all()


def _solve(A, B, y):
    N, m, k = y.shape
    dA, dB, dy = to_dev(A, B, y)
    plan = crs.Plan(N, m, k)
    crs.crsolve_factor(plan, dA, dB if N > 1 else None)
    return crs.crsolve_solve(plan, dy).cpu().numpy()


@pytest.mark.parametrize("m", [7, 8, 11, 16, 24, 40, 64])
def test_diagonal_blocks_keep_every_component(cuda_ok, m):
    """A and B diagonal: m independent chains, each component of x that of its own."""
    N, k = 21, 3
    rng = np.random.default_rng(m)
    d = rng.uniform(2.5, 3.0, (N, m))
    e = rng.uniform(-1.0, 1.0, (N - 1, m))
    y = rng.standard_normal((N, m, k)) * 10.0 ** rng.uniform(-40, 0, (1, m, 1))
    A = np.einsum("jr,rs->jrs", d, np.eye(m)).astype(complex)
    B = np.einsum("jr,rs->jrs", e, np.eye(m)).astype(complex)
    x = _solve(A, B, y.astype(complex))
    for r in range(m):
        T = np.diag(d[:, r]) + np.diag(e[:, r], -1) + np.diag(e[:, r], 1)
        ref = np.linalg.solve(T, y[:, r])
        assert np.abs(x[:, r] - ref).max() <= 1e-12 * np.abs(ref).max(), r


@pytest.mark.parametrize("m", [8, 16, 24, 48])
def test_far_field_of_a_localised_source(cuda_ok, m):
    """Tridiagonal A_j with decay 1e-1 to 1e-2 per row, diagonal B_j (an M-matrix):
    the solution of a point source is positive, and all of its components
    agree with the oracle's substitutions to a small relative error."""
    N = 9
    rng = np.random.default_rng(m)
    off = rng.uniform(0.5, 1.0, (N, m - 1))
    A = np.zeros((N, m, m), complex)
    i = np.arange(m)
    A[:, i, i] = rng.uniform(20.0, 30.0, (N, m))
    A[:, i[1:], i[:-1]] = A[:, i[:-1], i[1:]] = -off
    B = np.einsum("jr,rs->jrs", -rng.uniform(0.5, 1.0, (N - 1, m)), np.eye(m)).astype(complex)
    y = np.zeros((N, m, 1), complex)
    y[N // 2, 0, 0] = 1.0
    x = _solve(A, B, y)
    xo, _ = oracle.cr_solve(A, B, y)
    assert (xo.real > 0).all()
    assert (np.abs(x - xo) <= 1e-10 * np.abs(xo)).all()


@pytest.mark.parametrize("m", [8, 16, 24])
def test_complex_step(cuda_ok, m):
    """A real system and y + 1e-20 i dy: the imaginary part of x is 1e-20 times
    the solution for dy."""
    N, k = 40, 2
    A, B, y = synthetic.gen_system(N, m, k, seed=m)
    A, B = A.real.astype(complex), B.real.astype(complex)
    x = _solve(A, B, y.real + 1e-20j * y.imag)
    ref = _solve(A, B, y.imag.astype(complex))
    assert np.abs(x.imag * 1e20 - ref.real).max() <= 1e-12 * np.abs(ref.real).max()


@pytest.mark.parametrize("m,k", [(8, 4), (12, 5), (16, 8), (17, 32), (33, 24), (64, 17)])
def test_outer_products_of_scaled_rows(cuda_ok, m, k):
    """Gradients where the rows of x and g_y differ by powers of two over
    2^-60 .. 2^60 (unknowns in different units): every entry to the sum of its own
    products' moduli, 4k real ones for each of its two."""
    N = 11
    rng = np.random.default_rng(m + k)
    cn = lambda: rng.standard_normal((N, m, k)) + 1j * rng.standard_normal((N, m, k))
    d = 2.0 ** rng.integers(-60, 61, size=(N, m, 1))
    x, g = cn() * d, cn() / d
    A = np.broadcast_to(np.eye(m, dtype=complex), (N, m, m))
    B = np.zeros((N - 1, m, m), complex)
    dA, dB, dx, dg = to_dev(A, B, x, g)
    plan = crs.Plan(N, m, k)
    crs.crsolve_factor(plan, dA, dB)
    g, gA, gB = (t.cpu().numpy() for t in crs.crsolve_backward(plan, dx, dg))
    h = lambda t: np.conj(np.swapaxes(t, 1, 2))
    tol = 4 * k * 2.0 ** -45.3
    ref, mag = g @ h(x), np.abs(g) @ h(np.abs(x))
    assert (np.abs(gA + 0.5 * (ref + h(ref))) <= tol * (mag + h(mag))).all()
    ref = g[1:] @ h(x[:-1]) + x[1:] @ h(g[:-1])
    mag = np.abs(g[1:]) @ h(np.abs(x[:-1])) + np.abs(x[1:]) @ h(np.abs(g[:-1]))
    assert (np.abs(gB + ref) <= tol * mag).all()
