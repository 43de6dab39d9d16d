"""The mixed form's handover rule prices a refinement step by what it takes on
the tensor-core paths: within a quarter of measured shares of the FP64
factor + solve (GB300; m, k, share)."""
import pytest

from tests import split_device

MEASURED = [(33, 1, 0.238), (33, 32, 0.226), (40, 1, 0.221), (40, 32, 0.221), (48, 1, 0.168), (48, 32, 0.171),
            (64, 1, 0.128), (64, 32, 0.140)]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return split_device.load(tmp_path_factory.mktemp("cost"))


@pytest.mark.parametrize("m,k,share", MEASURED)
def test_step_cost(lib, m, k, share):
    assert abs(lib.mixed_step_cost_host(m, k, 1) / share - 1) <= 0.25
