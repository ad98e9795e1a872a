"""CPU: device memory of the sparse input per entry that a level may hold -- two
hash tables of 2.5 20-byte slots an entry, which the final list and its sort
buffers share -- beside a fixed part (counters, one exponent per X-mask)."""
import pytest

from paper_2310_13421_gb300 import _lib as L
from paper_2310_13421_gb300 import buildlib


@pytest.mark.parametrize("entries", [2, 1000, 4096, 4097, 122880 * 4 + 1024, 1 << 20, (1 << 20) + 1, 1 << 29, 3 << 28])
def test_bytes_per_entry(entries):
    buildlib.build()
    size = L.tpd_sparse_workspace_size(entries)
    assert 99 * entries <= size <= 100 * entries + (1 << 18)
