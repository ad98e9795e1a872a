"""Sparse input past max_entries, through the C ABI: the status says so and the
list holds what fitted, sorted, in *count.  Where only the last level passed the
capacity, the entries that it kept are right."""
import pytest
import torch

from test_gpu_sparse_sort import _random

pytestmark = pytest.mark.gpu


def _call(r, c, v, n, most):
    from paper_2310_13421_gb300 import _lib as L
    meta = torch.zeros(2, dtype=torch.int64, device="cuda")
    ws = torch.empty(L.tpd_sparse_workspace_size(most), dtype=torch.uint8, device="cuda")
    strings = torch.full((most,), -1, dtype=torch.int64, device="cuda")
    weights = torch.empty(most, dtype=torch.complex128, device="cuda")
    st = L.tpd_decompose_coo(r.data_ptr(), c.data_ptr(), v.data_ptr(), v.numel(), n, L.TPD_C128, most,
                             strings.data_ptr(), weights.data_ptr(), most, meta.data_ptr(), meta.data_ptr() + 8,
                             ws.data_ptr(), ws.numel(), torch.cuda.current_stream().cuda_stream)
    assert st == L.TPD_OK
    count, status = meta.tolist()
    return strings[:count], weights[:count], status, strings[count:]


@pytest.mark.parametrize("n,masks,most", [(8, 8, 2048), (8, 8, 2047), (8, 8, 1300), (8, 8, 1024), (11, 40, 60000), (11, 40, 40960)])
def test_entries_that_fit_are_kept(n, masks, most):
    import paper_2310_13421_gb300 as tpd
    from paper_2310_13421_gb300 import _lib as L
    r, c, v = _random(n, masks, 7 * n)                       # doubling at every level, to masks 2^n
    full_s, full_w = tpd.decompose_coo(r, c, v, n)
    assert full_s.numel() == masks * 2 ** n and most >= full_s.numel() // 2
    s, w, status, rest = _call(r, c, v, n, most)
    assert status == (L.TPD_OK if most >= full_s.numel() else L.TPD_ERR_WORKSPACE)
    assert s.numel() == min(most, full_s.numel()) and bool((s[1:] > s[:-1]).all()) and bool((rest == -1).all())
    at = torch.searchsorted(full_s, s)
    assert torch.equal(full_s[at], s) and torch.equal(full_w[at], w)


@pytest.mark.parametrize("most", [1, 7, 100, 1023])
def test_levels_that_do_not_fit(most):
    from paper_2310_13421_gb300 import _lib as L
    r, c, v = _random(8, 8, 3)
    s, w, status, rest = _call(r, c, v, 8, most)
    assert status == L.TPD_ERR_WORKSPACE and 0 < s.numel() <= most and bool((rest == -1).all())
    assert bool((s[1:] > s[:-1]).all()) and int(s[0]) >= 0 and int(s[-1]) < 4 ** 8
    assert bool(torch.isfinite(torch.view_as_real(w)).all())
