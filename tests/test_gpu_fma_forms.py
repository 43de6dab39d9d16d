"""The FMA forms of the FP64 levels (m <= 6 and m = 9, 10) in the level kernels:
N >= 8192 runs every level in a kernel of its own, at 1 to the most blocks per
CTA, wide forms and forms of a column per thread, full and narrowed
right-hand-side chunks.  x within the parity bound of the oracle and, bit for
bit, the batched form's; a breakdown on a coarse level where the oracle has
it.  And m = 11, the smallest block above them that takes the tensor-core
tiles, at the sizes of the other tile tests."""
import numpy as np
import pytest
import torch

import oracle
import synthetic
import paper_1807_00370_gb300 as crs
from tests.gpu_helpers import rel_err, to_dev

pytestmark = pytest.mark.gpu

TOL = 1e-12


def _plain(A, B, y):
    N, m, k = y.shape
    dA, dB, dy = to_dev(A, B if N > 1 else None, y)
    plan = crs.Plan(N, m, k)
    crs.crsolve_factor(plan, dA, dB)
    return crs.crsolve_solve(plan, dy).cpu().numpy(), crs.crsolve_info_get(plan)


@pytest.mark.parametrize("m,k", [(3, 2), (6, 1), (6, 17), (9, 1), (9, 4), (10, 16), (10, 33)])
def test_level_kernels(cuda_ok, m, k):
    N = 8200
    s = synthetic.gen_system(N, m, k, seed=10 * m + k)
    x, info = _plain(*s)
    xo, io = oracle.cr_solve(*s)
    assert info == io and io["status"] == 0
    assert rel_err(x, xo) <= TOL
    b = crs.Batch([N], [m], [k])
    A, B, y = b.pack([s])
    assert np.array_equal(crs.crsolve_batch_solve(b, A, B, y).cpu().numpy().reshape(x.shape), x)


@pytest.mark.parametrize("m", [4, 10])
def test_breakdown_in_a_level_kernel(cuda_ok, m):
    N = 8192
    for seed in range(40):
        A, B, y = synthetic.gen_system(N, m, 2, seed=seed)
        A = synthetic.make_indefinite(A)
        _, io = oracle.cr_solve(A, B, y)
        if io["status"] == 1 and io["level"] >= 4:
            break
    else:
        pytest.skip("no seed gave a coarse-level breakdown")
    x, info = _plain(A, B, y)
    assert info == io and np.isnan(x).all()


@pytest.mark.parametrize("N,k", [(1, 1), (2, 9), (37, 1), (130, 17), (8200, 3)])
def test_m_11(cuda_ok, N, k):
    s = synthetic.gen_system(N, 11, k, seed=N + k)
    x, info = _plain(*s)
    xo, io = oracle.cr_solve(*s)
    assert info == io and rel_err(x, xo) <= TOL
