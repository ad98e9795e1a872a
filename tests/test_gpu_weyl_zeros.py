"""Weyl basis, complex128 block fixed point: what the level maps give exactly
comes out exactly.  Zeros stay zeros, a tensor product of cyclic shifts has one
nonzero weight, a real diagonal's weights are conjugate pairs, and a negated
input gives the negated result, bit for bit: every step of the arithmetic
(truncation toward zero, the 3-point DFT, the factor 3^-n, the rounding to
double) is an odd function that keeps zero."""
import pytest
import torch

pytestmark = pytest.mark.gpu

SIZES = [(3, 1), (3, 2), (3, 3), (3, 4), (3, 7), (2, 3), (2, 6), (4, 1), (4, 3)]


def _digits(x, d, n):
    return torch.stack([x // d ** k % d for k in range(n)])


def _number(v, d):
    return sum(v[k] * d ** k for k in range(len(v)))


@pytest.mark.parametrize("d,n", SIZES)
def test_zeros_stay_zeros(d, n):
    import paper_2310_13421_gb300 as tpd
    Z = torch.zeros(d ** n, d ** n, dtype=torch.complex128, device="cuda")
    assert not torch.view_as_real(tpd.weyl_decompose(Z, d)).any()
    for scale in (1.0, 0.3, 2.0 ** 900):
        assert not torch.view_as_real(tpd.weyl_compose(Z, d, scale=scale)).any()


@pytest.mark.parametrize("d,n", SIZES)
def test_shifts_have_one_weight(d, n):
    import paper_2310_13421_gb300 as tpd
    N = d ** n
    c = torch.arange(N, device="cuda")
    for a in sorted({0, 1, N // d, N - 1}):
        A = torch.zeros(N, N, dtype=torch.complex128, device="cuda")      # X^a: ones at (c + a, c)
        A[_number((_digits(c, d, n) + _digits(torch.tensor(a, device="cuda"), d, n)[:, None]) % d, d), c] = 1
        C = torch.zeros_like(A)                                           # weight (a, 0) at row 0, column a
        C[0, a] = 1
        assert torch.equal(tpd.weyl_decompose(A, d), C)
        assert torch.equal(tpd.weyl_compose(C, d), A)


@pytest.mark.parametrize("d,n", SIZES)
def test_real_diagonals_give_conjugate_pairs(d, n):
    import paper_2310_13421_gb300 as tpd
    N = d ** n
    g = torch.Generator(device="cuda").manual_seed(n)
    W = tpd.weyl_decompose(torch.diag(torch.randn(N, dtype=torch.float64, device="cuda", generator=g)).to(torch.complex128), d)
    w = W.diagonal().clone()                                              # shift 0: weight b at (b, b)
    minus = _number((d - _digits(torch.arange(N, device="cuda"), d, n)) % d, d)
    assert torch.equal(w[minus], w.conj()) and float(w[0].imag) == 0.0
    W.diagonal().zero_()
    assert not torch.view_as_real(W).any()


@pytest.mark.parametrize("d,n", SIZES)
def test_negated_inputs_give_negated_results(d, n):
    import paper_2310_13421_gb300 as tpd
    g = torch.Generator(device="cuda").manual_seed(10 + n)
    A = torch.randn(d ** n, d ** n, dtype=torch.complex128, device="cuda", generator=g)
    A[0] = torch.round(4 * A[0].real) + 0j                                # small integers and zeros among them
    for call in (lambda X: tpd.weyl_decompose(X, d), lambda X: tpd.weyl_compose(X, d, scale=0.3)):
        assert torch.equal(call(-A), -call(A))
