"""The coarse levels of a short system in one launch per sweep direction
(N < 8192): the same numbers, bit for bit, as the batched form, which runs the
levels of a system in one CTA, and as the plan that re-factors its coarse
levels from a kept one; the oracle's breakdown location; x within the FP64
bound of the oracle.  The sizes put levels at one to the most blocks per CTA,
one to eight CTAs, and whole systems inside the launch."""
import numpy as np
import pytest
import torch

import oracle
import synthetic
import paper_1807_00370_gb300 as crs
from tests.gpu_helpers import rel_err, to_dev

pytestmark = pytest.mark.gpu

TOL = 1e-12


@pytest.mark.parametrize("m", [1, 4, 6, 8, 10, 13, 16, 24, 40, 64])
@pytest.mark.parametrize("k", [1, 9, 17])
def test_tail_equals_batched_form(cuda_ok, m, k):
    Ns = (1, 2, 3, 9, 17, 40, 65, 128, 130) if m <= 24 else (2, 9, 17, 40)
    systems = [synthetic.gen_system(N, m, k, seed=100 * m + N) for N in Ns]
    b = crs.Batch(Ns, [m] * len(Ns), [k] * len(Ns))
    A, B, y = b.pack(systems)
    xb = crs.crsolve_batch_solve(b, A, B, y)
    for i, (Ai, Bi, yi) in enumerate(systems):
        N = Ns[i]
        dA, dB, dy = to_dev(Ai, Bi, yi)
        plan = crs.Plan(N, m, k)
        for _ in range(2):
            crs.crsolve_factor(plan, dA, dB if N > 1 else None)
            x = crs.crsolve_solve(plan, dy).cpu().numpy()
            assert np.array_equal(x, b.system_view(i, A, B, xb)[2].cpu().numpy()), N
        xo, io = oracle.cr_solve(Ai, Bi, yi)
        assert crs.crsolve_info_get(plan) == io and rel_err(x, xo) <= TOL, N


@pytest.mark.parametrize("m", [3, 8, 24])
def test_tail_with_kept_levels_and_breakdown(cuda_ok, m):
    N, k = 100, 3
    A, B, y = synthetic.gen_system(N, m, k, seed=m)
    dA, dB, dy = to_dev(A, B, y)
    plain = crs.Plan(N, m, k)
    crs.crsolve_factor(plain, dA, dB)
    x = crs.crsolve_solve(plain, dy)
    for keep in (0, 1, 4):
        p = crs.Plan(N, m, k, keep_levels=keep)
        crs.crsolve_factor(p, dA, dB)
        p.release_scratch()
        assert torch.equal(crs.crsolve_solve(p, dy), x)
    Ai = synthetic.make_indefinite(A)
    crs.crsolve_factor(plain, to_dev(Ai)[0], dB)
    x = crs.crsolve_solve(plain, dy).cpu().numpy()
    _, io = oracle.cr_solve(Ai, B, y)
    assert crs.crsolve_info_get(plain) == io
    assert np.isnan(x).all() == (io["status"] == 1)
