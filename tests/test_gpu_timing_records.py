"""Timing records of short systems: one per level and kernel, as for long ones,
with the same numbers as the untimed calls, which run the coarse levels in
one launch."""
import pytest
import torch

import synthetic
import paper_1807_00370_gb300 as crs
from paper_1807_00370_gb300 import _native as nat
from tests.gpu_helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,m", [(64, 4), (100, 8), (1000, 24)])
def test_records_per_level(cuda_ok, N, m):
    dA, dB, dy = to_dev(*synthetic.gen_system(N, m, 2, seed=m))
    plan = crs.Plan(N, m, 2)
    crs.crsolve_factor(plan, dA, dB)
    x = crs.crsolve_solve(plan, dy)
    n0 = crs.crsolve_launch_count(plan)
    crs.crsolve_factor(plan, dA, dB)
    untimed = crs.crsolve_launch_count(plan) - n0
    crs.crsolve_timing_enable(plan, True)
    crs.crsolve_factor(plan, dA, dB)
    xt = crs.crsolve_solve(plan, dy)
    recs = crs.crsolve_timing_read(plan)
    crs.crsolve_timing_enable(plan, False)
    assert torch.equal(x, xt)
    levels = list(range(N.bit_length()))
    for kind in (nat.KERNEL_KINDS[i] for i in (0, 2, 4)):      # factor, solve down, solve up
        assert sorted(level for name, level, _, _ in recs if name == kind) == levels
    n0 = crs.crsolve_launch_count(plan)
    crs.crsolve_factor(plan, dA, dB)
    assert crs.crsolve_launch_count(plan) - n0 == untimed < len(levels)
    assert torch.equal(crs.crsolve_solve(plan, dy), x)
