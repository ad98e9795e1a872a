"""The out-of-place calls (the first pass reads the caller's matrix and writes
the result's buffer) against the in-place calls on a copy: every output bit,
and the input untouched.  Sizes cover the whole-matrix kernel (n <= 4), one
pass, several passes and the two-CTA clusters (n = 11)."""
import numpy as np
import pytest
import torch

ARITH = [("c128", None), ("c128", "plain"), ("c64", None), ("c64", "compensated"), ("c64", "fixed")]


def _matrix(n, dtype, seed=3):
    g = torch.Generator().manual_seed(seed)
    A = torch.randn(2 ** n, 2 ** n, dtype=torch.complex128, generator=g)
    return A.to(torch.complex64 if dtype == "c64" else torch.complex128)


def _bits(t):
    t = torch.view_as_real(t)
    return t.view(torch.int32 if t.dtype == torch.float32 else torch.int64)


def _check(A, call):
    kept = A.clone()
    got = call(A, False)
    assert got.data_ptr() != A.data_ptr()
    assert torch.equal(_bits(A), _bits(kept))
    want = call(kept, True)
    assert torch.equal(_bits(got), _bits(want))


@pytest.mark.gpu
@pytest.mark.parametrize("n", [1, 3, 5, 7, 9, 11, 12])
@pytest.mark.parametrize("dtype,precision", ARITH)
def test_equals_the_call_on_a_copy(n, dtype, precision):
    import paper_2310_13421_gb300 as tpd
    A = _matrix(n, dtype).cuda()
    _check(A, lambda X, inplace: tpd.decompose(X, precision=precision, inplace=inplace))
    _check(A, lambda X, inplace: tpd.compose(X, scale=2.0 ** -n, precision=precision, inplace=inplace))


@pytest.mark.gpu
@pytest.mark.parametrize("variant", [1, 2, 3, 5])
@pytest.mark.parametrize("n", [10, 11])
def test_kernel_forms(n, variant):
    import paper_2310_13421_gb300 as tpd
    _check(_matrix(n, "c128").cuda(), lambda X, inplace: tpd.decompose(X, variant=variant, inplace=inplace))


@pytest.mark.gpu
@pytest.mark.parametrize("n", [3, 6, 8, 11])
@pytest.mark.parametrize("dtype,precision", ARITH)
def test_zero_skipping_and_nonfinite_tiles(n, dtype, precision):
    """All-zero tiles (of either sign) reach the output unchanged, tiles with
    Inf / NaN take the IEEE path, whatever the output's buffer held."""
    import paper_2310_13421_gb300 as tpd
    A = torch.zeros(2 ** n, 2 ** n, dtype=torch.complex64 if dtype == "c64" else torch.complex128)
    real = torch.view_as_real(A)
    real[::2, :, 0] = -0.0
    real[0, 1, 0] = 1.5
    real[-1, -1, 1] = float("inf")
    A = A.cuda()
    torch.full((4 ** n,), float("nan"), dtype=A.dtype, device="cuda")     # freed at once: memory to be handed on
    _check(A, lambda X, inplace: tpd.decompose(X, precision=precision, skip_zero=True, inplace=inplace))
    zero = torch.view_as_complex(torch.full((2 ** n, 2 ** n, 2), -0.0, dtype=real.dtype)).cuda()
    _check(zero, lambda X, inplace: tpd.decompose(X, precision=precision, skip_zero=True, inplace=inplace))


@pytest.mark.gpu
def test_inputs_that_need_a_copy():
    """Lazily conjugated views and tensors whose copy autograd follows give
    what they gave from a copy."""
    import paper_2310_13421_gb300 as tpd
    A = _matrix(6, "c128").cuda()
    assert torch.equal(tpd.decompose(A.conj()), tpd.decompose(A.conj().resolve_conj()))
    leaf = A.clone().requires_grad_()
    assert tpd.decompose(leaf).requires_grad
    assert torch.equal(tpd.decompose(leaf).detach(), tpd.decompose(A))


def test_which_inputs_are_read_in_place():
    """The rule itself, on host tensors."""
    from paper_2310_13421_gb300 import api
    A = torch.zeros(4, 4, dtype=torch.complex64)
    assert api._target(A, True) == (A, A)
    src, out = api._target(A, False)
    assert src is A and out.shape == A.shape and out.data_ptr() != A.data_ptr()
    raw = np.zeros(2 * 16 + 1, dtype=np.float32)
    skewed = torch.from_numpy(raw[1:].view(np.complex64).reshape(4, 4))       # one of the two views is
    even = torch.from_numpy(raw[:-1].view(np.complex64).reshape(4, 4))        # aligned to 4 bytes only
    for X in (skewed, even, A.conj(), torch._neg_view(A), A.clone().requires_grad_()):
        src, out = api._target(X, False)
        copied = X.is_conj() or X.is_neg() or X.requires_grad or X.data_ptr() % 8 != 0
        assert (src is not X) == copied and (src is out) == copied
        assert out.data_ptr() % 8 == 0 and not out.is_conj() and not out.is_neg()
    assert (skewed.data_ptr() % 8 != 0) != (even.data_ptr() % 8 != 0)
    with torch.autograd.forward_ad.dual_level():
        assert api._target(A, False)[0] is not A
    with torch.no_grad():
        X = A.clone().requires_grad_()
        assert api._target(X, False)[0] is X


def test_argument_errors():
    from paper_2310_13421_gb300 import _lib as L, buildlib
    buildlib.build()
    size = 16 * 4 ** 4
    for call in (lambda a, w: L.tpd_decompose_to(a, w, 4, L.TPD_C128),
                 lambda a, w: L.tpd_compose_to(a, w, 4, L.TPD_C128, 1.0)):
        assert call(0, 4096) == L.TPD_ERR_INVALID_ARG
        assert call(4096, 0) == L.TPD_ERR_INVALID_ARG
        assert call(4096, 4096 + size - 16) == L.TPD_ERR_INVALID_ARG          # overlap
        assert call(4096 + size - 16, 4096) == L.TPD_ERR_INVALID_ARG
        assert call(4096 + 8, 1 << 20) == L.TPD_ERR_MISALIGNED
        assert call(4096, (1 << 20) + 8) == L.TPD_ERR_MISALIGNED
