"""One-pass matrices (n = 5, 6) whose X-masks have very different sizes: a class
of subnormal numbers beside classes of normal ones."""
import numpy as np
import pytest
import torch

import oracle
from _helpers import to_string_order

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [5, 6, 7])
def test_subnormal_class_beside_normal_ones(n):
    """Diagonal entries of size 1, all others multiples of 2^-1074: an exact
    case up to the subnormal results' own rounding, half a unit each."""
    import paper_2310_13421_gb300 as tpd
    rng = np.random.default_rng(n)
    N = 2 ** n
    A = (rng.integers(-2000, 2001, (N, N)) + 1j * rng.integers(-2000, 2001, (N, N))) * (2.0 ** -1060)
    A[np.diag_indices(N)] = rng.integers(-8, 9, N)
    got = to_string_order(tpd.decompose(torch.from_numpy(A).cuda(), precision="fixed").cpu().numpy(), n)
    assert np.max(np.abs(got - oracle.coeffs_fwht(A))) <= 2.0 ** -1074 * 2 ** n
