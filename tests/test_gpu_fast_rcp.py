"""The pivots' reciprocal (fast_rcp) against 1 / d: within one ulp over the
exponents it takes, both ends included, and none taken outside them (zero,
negative, subnormal, infinite and NaN pivots, which take the division)."""
import ctypes

import numpy as np
import pytest
import torch

from tests import split_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib(tmp_path_factory, cuda_ok):
    return split_device.load(tmp_path_factory.mktemp("rcp"))


def _rcp(lib, d):
    x = torch.from_numpy(d).cuda()
    r = torch.empty_like(x)
    torch.cuda.synchronize()
    assert lib.fast_rcp_device(ctypes.c_void_p(x.data_ptr()), ctypes.c_void_p(r.data_ptr()), d.size) == 0
    return r.cpu().numpy()


def test_within_an_ulp(lib):
    rng = np.random.default_rng(0)
    mant = np.concatenate([[1.0, np.nextafter(1.0, 2.0), np.nextafter(2.0, 1.0), 1.5], rng.uniform(1.0, 2.0, 1000)])
    ends = np.ldexp(np.tile(mant, 2), np.repeat([-999, 985 - 1], mant.size))
    d = np.concatenate([ends, np.ldexp(rng.uniform(1.0, 2.0, 200000), rng.integers(-999, 985, 200000)),
                        rng.uniform(1.0, 2.0, 200000)])
    r, ref = _rcp(lib, d), 1.0 / d
    assert (np.abs(r - ref) <= np.spacing(ref)).all()


def test_outside_its_range(lib):
    d = np.array([0.0, -0.0, -1.0, -np.inf, np.inf, np.nan, 5e-324, 2.0 ** -1022, np.nextafter(2.0 ** -999, 0.0),
                  2.0 ** 985, 1.7e308])
    assert (_rcp(lib, d) == 0.0).all()
