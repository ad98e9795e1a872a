"""The nonzero list at the sizes where its blocks and chunks begin and end
(n < 4: one partial block; n = 4: one block; n = 7: one chunk; above: several),
from empty to full matrices, against the same list made by indexing."""
import pytest
import torch

from _helpers import rc_positions


@pytest.mark.gpu
@pytest.mark.parametrize("n", [1, 2, 3, 4, 6, 7, 8, 9])
@pytest.mark.parametrize("dtype", [torch.complex128, torch.complex64])
@pytest.mark.parametrize("share", [0.0, 0.002, 0.5, 1.0])
def test_list_equals_indexing(n, dtype, share):
    import paper_2310_13421_gb300 as tpd
    g = torch.Generator(device="cuda").manual_seed(n)
    W = torch.randn(2 ** n, 2 ** n, dtype=torch.complex128, device="cuda", generator=g).to(dtype)
    W = torch.where(torch.rand(2 ** n, 2 ** n, device="cuda", generator=g) < share, W, torch.zeros((), dtype=dtype,
                                                                                                  device="cuda"))
    real = torch.view_as_real(W)
    real[..., 1] *= -1.0                                  # zeros of either sign
    if share == 0.5:
        real[-1, 0, 0] = float("nan")                     # kept
    order = torch.from_numpy(rc_positions(n)).cuda()
    flat = W.reshape(-1)[order]
    for tol in (0.0, 0.7):
        kept = ~((flat.real.abs() <= tol) & (flat.imag.abs() <= tol))
        want = kept.nonzero().reshape(-1)
        strings, weights = tpd.nonzero_list(W, tol=tol)
        assert torch.equal(strings, want)
        assert torch.equal(torch.view_as_real(weights).nan_to_num(5.0), torch.view_as_real(flat[want]).nan_to_num(5.0))
        cap = max(1, want.numel() // 2)
        strings, weights, count = tpd.nonzero_list(W, tol=tol, capacity=cap)
        assert int(count) == want.numel()
        assert torch.equal(strings[:min(cap, want.numel())], want[:cap])


def test_write_argument_errors():
    from paper_2310_13421_gb300 import _lib as L, buildlib
    buildlib.build()
    size = L.tpd_nonzero_workspace_size(4)
    assert L.tpd_nonzero_write(4096, 4, L.TPD_C128, 0.0, 0, 0, 5, 4096, size) == L.TPD_ERR_INVALID_ARG
    assert L.tpd_nonzero_write(4096, 4, L.TPD_C128, -1.0, 8192, 8192, 5, 4096, size) == L.TPD_ERR_INVALID_ARG
    assert L.tpd_nonzero_write(4096, 4, L.TPD_C128, 0.0, 8192, 8192, 5, 4096, size - 1) == L.TPD_ERR_WORKSPACE
    assert L.tpd_nonzero_write(4096, 4, L.TPD_C128, 0.0, 8192, 8200, 5, 4096, size) == L.TPD_ERR_MISALIGNED
    assert L.tpd_nonzero_write(4096, 4, L.TPD_C128, 0.0, 8192, 8192, 5, 4100, size) == L.TPD_ERR_MISALIGNED
