"""Split tiles on the GPU: runs whose 2^12-element tiles are halved against runs
of whole tiles (variant 1), every output bit -- decomposition, composition
and batches; dense, Hermitian (real weights) and partly zero matrices, classes
of subnormal numbers beside large ones.  A tile that meets Inf or NaN runs IEEE
fp64 as a whole, so there the halves are compared with the same halves read at
run time (variant 5)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _bits(t):
    return torch.view_as_real(t).view(torch.int64)


def _matrices(n):
    g = torch.Generator(device="cuda").manual_seed(n)
    A = torch.randn(2 ** n, 2 ** n, dtype=torch.complex128, device="cuda", generator=g)
    sparse = torch.where(torch.rand(A.shape, device="cuda", generator=g) < 0.01, A, torch.zeros_like(A))
    wide = A * torch.exp2(torch.randint(-1060, 900, A.shape, device="cuda", generator=g).double())
    return [A, (A + A.mH) * 0.5, sparse, wide, A * 2.0 ** -1070]


@pytest.mark.parametrize("n", [7, 9, 10, 12, 13])
def test_halves_equal_whole_tiles(n):
    import paper_2310_13421_gb300 as tpd
    for A in _matrices(n):
        assert torch.equal(_bits(tpd.decompose(A)), _bits(tpd.decompose(A, variant=1)))
        assert torch.equal(_bits(tpd.compose(A, scale=2.0 ** -n)), _bits(tpd.compose(A, scale=2.0 ** -n, variant=1)))
    A[1, 5] = float("inf")
    A[-3, 0] = float("nan")
    assert torch.equal(_bits(tpd.decompose(A)), _bits(tpd.decompose(A, variant=5)))
    assert torch.equal(_bits(tpd.compose(A)), _bits(tpd.compose(A, variant=5)))


def test_batches():
    import paper_2310_13421_gb300 as tpd
    g = torch.Generator(device="cuda").manual_seed(5)
    mats = [torch.randn(2 ** n, 2 ** n, dtype=torch.complex128, device="cuda", generator=g) for n in (9, 7, 10, 9, 12, 3)]
    for got, want in zip(tpd.decompose_batched(mats), tpd.decompose_batched(mats, variant=1)):
        assert torch.equal(_bits(got), _bits(want))
    for got, want in zip(tpd.compose_batched(mats, adjoint=True), tpd.compose_batched(mats, adjoint=True, variant=1)):
        assert torch.equal(_bits(got), _bits(want))
