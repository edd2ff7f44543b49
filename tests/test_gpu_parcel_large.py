"""The parcel scheme's kernel for systems whose matrices do not fit in shared memory: the first size it
takes and the first on a block of 1,024 threads."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [113, 161])
def test_large_parcel_systems_match_oracle(S):
    """As the smaller systems: 10 x the oracle's own spread under perturbations of 1e-13 relative (at
    least 1e-9); step counts agree when the spread's do."""
    from tests.test_gpu_parcel_sizes import test_parcel_sizes_match_oracle
    test_parcel_sizes_match_oracle(S)
