"""Weyl basis, complex128: weights of which one part is Inf or NaN and the other
finite.  The block fixed point and IEEE fp64 agree on which parts are
non-finite, and on the finite parts to rounding: 16 n u of their norm each
way, as in the other tests of this basis (each level rounds an output at most
16 times and does not increase the norm)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _matrix(d, n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(d ** n, d ** n, dtype=torch.complex128, device="cuda", generator=g)


@pytest.mark.parametrize("d,n", [(3, 3), (3, 4), (3, 5), (3, 6), (3, 7), (2, 6), (4, 3)])
@pytest.mark.parametrize("part", ["real", "imag"])
def test_finite_parts_beside_non_finite_ones(d, n, part):
    import paper_2310_13421_gb300 as tpd
    N = d ** n
    A = _matrix(d, n, n)
    for at, v in (((0, 0), float("inf")), ((N - 1, 1), float("-inf")), ((2, N // 2), float("nan"))):
        A[at] = complex(v, 0.25) if part == "real" else complex(0.25, v)
    for call in (lambda p: tpd.weyl_decompose(A, d, precision=p), lambda p: tpd.weyl_compose(A, d, precision=p),
                 lambda p: tpd.weyl_compose(A, d, scale=float(d) ** -n, precision=p)):
        fixed, ieee = (torch.view_as_real(call(p)) for p in ("fixed", "plain"))
        assert torch.equal(fixed.isnan(), ieee.isnan()) and torch.equal(fixed.isinf(), ieee.isinf())
        finite = ieee.isfinite()
        half = finite.any(-1) & ~finite.all(-1)               # one part of the two
        assert int(half.sum()) > 0
        for rows in (half, finite.all(-1)):
            x, y = fixed[rows][finite[rows]], ieee[rows][finite[rows]]
            assert float((x - y).norm()) <= 32 * n * 2.0 ** -53 * float(y.norm())


def test_one_infinite_diagonal_entry():
    import paper_2310_13421_gb300 as tpd
    A = _matrix(3, 4, 1)
    A[5, 5] = complex(float("inf"), 0.25)
    fixed, ieee = (tpd.weyl_decompose(A, 3, precision=p)[0, 0] for p in ("fixed", "plain"))
    assert float(fixed.real) == float("inf") == float(ieee.real)
    assert abs(float(fixed.imag - ieee.imag)) <= 16 * 4 * 2.0 ** -53 * float(A.diagonal().imag.abs().max())
