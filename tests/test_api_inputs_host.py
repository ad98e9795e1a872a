"""CPU: which inputs an out-of-place call reads where they are, and which it copies
first."""
import pytest

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def api():
    from paper_2310_13421_gb300 import api as a
    return a


def _copied(api, A):
    src, out = api._target(A, False)
    assert out.data_ptr() not in (0, A.data_ptr()) and out.shape == A.shape and out.dtype == A.dtype
    assert src is A or src is out
    return src is out


def test_plain_inputs_are_read_in_place(api):
    A = torch.randn(8, 8, dtype=torch.complex128)
    assert not _copied(api, A) and not _copied(api, A.detach())
    assert api._target(A, True) == (A, A)


def test_lazy_and_followed_inputs_are_copied(api):
    A = torch.randn(8, 8, dtype=torch.complex128)
    assert _copied(api, A.conj()) and _copied(api, A.clone().requires_grad_())
    with torch.no_grad():
        assert not _copied(api, A.clone().requires_grad_())


def test_zeros_without_memory_are_copied(api):
    Z = torch._efficientzerotensor((8, 8), dtype=torch.complex128)
    assert Z.data_ptr() == 0 and _copied(api, Z)


def test_options_by_value(api):
    # anything that converts to a number, also what cannot be hashed or changes later
    import numpy as np
    t = torch.tensor(11)
    assert api._options("fixed", tile_bits=t).tile_bits == 11
    t += 1
    assert api._options("fixed", tile_bits=t).tile_bits == 12
    o = api._options(np.array(0), np.bool_(True), np.array(12), 3.0, variant=np.int64(1))
    assert (o.skip_zero, o.tile_bits, o.max_levels, o.variant) == (1, 12, 3, 1)
    assert api._options(None) is api._options("default")
    for bad in ("exact", "Fixed"):
        with pytest.raises(KeyError):
            api._options(bad)


def test_without_the_forward_mode_level_inputs_are_copied(api, monkeypatch):
    monkeypatch.delattr(torch.autograd.forward_ad, "_current_level")
    assert _copied(api, torch.randn(8, 8, dtype=torch.complex128))


def test_without_the_raw_stream_function_the_stream_is_entered(api, monkeypatch):
    class Stream:
        cuda_stream = 77

    class Entered:
        def __init__(self, what):
            self.what = what

        def __enter__(self):
            entered.append(self.what)

        def __exit__(self, *exc):
            left.append(self.what)

    entered, left, s, dev = [], [], Stream(), torch.device("cuda", 0)
    monkeypatch.setattr(api, "_raw_stream", None)
    for name, f in (("current_device", lambda: 0), ("current_stream", lambda: s), ("device", Entered), ("stream", Entered)):
        monkeypatch.setattr(torch.cuda, name, f)
    with api._enqueue(dev, None) as handle:
        assert handle == 77 and entered == [dev, s] and left == []
    assert left == [s, dev]
