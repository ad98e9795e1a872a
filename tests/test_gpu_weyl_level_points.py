"""Weyl basis, complex128 block fixed point: the d elements that one level's DFT
adds are on their own binary point at every level, so large elements that
cancel exactly at one level leave no trace in the weights of small ones that
only meet them at a later level: those weights are bit for bit what they are
without the large elements."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,n,level,mix", [(2, 2, 0, 1), (2, 4, 0, 3), (2, 4, 1, 2), (2, 4, 2, 3), (2, 9, 1, 4), (3, 2, 0, 1),
                                           (3, 3, 0, 1), (3, 3, 0, 2), (3, 3, 1, 2), (3, 6, 3, 5), (3, 6, 1, 4), (4, 2, 0, 1),
                                           (4, 4, 2, 3)])
@pytest.mark.parametrize("dec", [True, False])
@pytest.mark.parametrize("small", [1e-3, 1e-20, 1e-60])
def test_cancelled_elements_leave_no_trace(d, n, level, mix, dec, small):
    # Element (c, a) of a level map's class a: at (c + a, c) for the
    # decomposition, (c, c + a) for the composition.  Those whose digit `mix`
    # of c is 0 are large and constant over digit `level` of c: the outputs
    # with digit b_level != 0 take nothing from them.
    import paper_2310_13421_gb300 as tpd
    N = d ** n
    g = torch.Generator(device="cuda").manual_seed(100 * d + 10 * n + level)
    i = torch.arange(N * N, device="cuda")
    a, c = i // N, i % N
    ca = sum((a // d ** k + c // d ** k) % d * d ** k for k in range(n))
    v = small * torch.randn(N * N, dtype=torch.complex128, device="cuda", generator=g)
    large = c // d ** mix % d == 0
    flat = a * N + c - c // d ** level % d * d ** level                    # the same for every digit `level` of c
    big = torch.randn(N * N, dtype=torch.complex128, device="cuda", generator=g)[flat]
    with_big, without = (torch.zeros(N, N, dtype=torch.complex128, device="cuda") for _ in range(2))
    at = (ca, c) if dec else (c, ca)
    with_big[at] = torch.where(large, big, v)
    without[at] = torch.where(large, torch.zeros_like(v), v)
    call = tpd.weyl_decompose if dec else tpd.weyl_compose
    out = (c, ca) if dec else (ca, c)                                      # output (a, b = c)
    free = c // d ** level % d != 0
    got, want = call(with_big, d)[out][free], call(without, d)[out][free]
    assert bool((want != 0).any()) and torch.equal(got, want)


def test_small_weight_beside_a_cancelling_pair():
    import paper_2310_13421_gb300 as tpd
    A = torch.diag(torch.tensor([1.0, 1.0, 1e-20, 0.0], dtype=torch.complex128, device="cuda"))
    assert tpd.weyl_decompose(A, 2).diagonal().tolist() == [0.5, 2.5e-21, 0.5, -2.5e-21]
