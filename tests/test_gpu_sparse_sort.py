"""Sparse input whose lists need the merges of the final sort: from one chunk of
2048 entries to several, exact powers of two and one more or less, against the
dense decomposition; and levels that just fit or just exceed the capacity."""
import pytest
import torch

from _helpers import rc_positions

pytestmark = pytest.mark.gpu


def _random(n, masks, seed):
    """One integer entry per X-mask: its 2^n weights are all nonzero."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randperm(2 ** n, device="cuda", generator=g)[:masks]
    r = torch.randint(0, 2 ** n, (masks,), device="cuda", generator=g)
    v = torch.randint(1, 9, (masks,), device="cuda", generator=g).to(torch.complex128) * (1 - 2j)
    return r.to(torch.int32), (r ^ x).to(torch.int32), v


@pytest.mark.parametrize("n,masks", [(1, 1), (1, 2), (6, 32), (7, 16), (8, 8), (8, 9), (7, 33), (9, 40), (10, 64), (11, 65)])
def test_lists_across_the_sort_chunks(n, masks):
    import paper_2310_13421_gb300 as tpd
    r, c, v = _random(n, masks, 100 * n + masks)
    strings, weights = tpd.decompose_coo(r, c, v, n)
    H = torch.zeros(2 ** n, 2 ** n, dtype=torch.complex128, device="cuda")
    H[r.long(), c.long()] = v
    flat = tpd.decompose(H).reshape(-1)[torch.from_numpy(rc_positions(n)).cuda()]
    want = (flat != 0).nonzero().reshape(-1)
    assert want.numel() == masks * 2 ** n
    assert torch.equal(strings, want) and torch.equal(weights, flat[want])


def test_capacity_is_of_every_level():
    import paper_2310_13421_gb300 as tpd
    from paper_2310_13421_gb300 import _lib as L
    r, c, v = _random(8, 8, 3)                              # 8 entries, doubling to 2048
    strings, _ = tpd.decompose_coo(r, c, v, 8, max_entries=2048)
    assert strings.numel() == 2048
    for most in (2047, 1024, 7):
        with pytest.raises(L.TPDError):
            tpd.decompose_coo(r, c, v, 8, max_entries=most)
    d = torch.arange(2 ** 8, device="cuda", dtype=torch.int32)
    one = torch.ones(2 ** 8, dtype=torch.complex128, device="cuda")
    assert tpd.decompose_coo(d, d, one, 8, max_entries=256)[0].tolist() == [0]      # the identity
    with pytest.raises(L.TPDError):
        tpd.decompose_coo(d, d, one, 8, max_entries=255)                            # its entries do not fit
