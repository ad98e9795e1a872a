"""Split tiles on the CPU: the pass descriptors a default run really uses (the
plan's, with the halves of split tiles in their place) emulated level by level
like the plan itself, and which plans split."""
import re

import numpy as np
import pytest

from paper_2310_13421_gb300 import synth
from test_abi_host import _emulate, _parse


@pytest.fixture(scope="module")
def L():
    from paper_2310_13421_gb300 import buildlib, _lib
    buildlib.build()
    _lib.load()
    return _lib


def _run_passes(desc):
    """Plan passes with the halves of split tiles in their place, and how many there are."""
    lines = desc.strip().splitlines()
    split = {re.match(r"split pass (\d+)", x).group(1): x[len("split "):] for x in lines if x.startswith("split ")}
    run = [split.get(re.match(r"pass (\d+)", x).group(1), x) for x in lines if x.startswith("pass ")]
    return _parse("\n".join(run)), len(split)


@pytest.mark.parametrize("n", [7, 9])
@pytest.mark.parametrize("max_levels", [0, 4])
def test_split_plans_compute_the_decomposition(L, n, max_levels):
    passes, count = _run_passes(L.tpd_plan_describe(n, 0, L.options(max_levels=max_levels))[1])
    assert count > 0 and all(p["D"] == 11 for p in passes if p["K"] >= 4)
    A = synth.int_general(n, seed=n)
    assert np.array_equal(_emulate(A, passes, n), _emulate(A, _parse(L.tpd_plan_describe(
        n, 0, L.options(max_levels=max_levels))[1]), n))


@pytest.mark.parametrize("n", range(7, 17))
def test_what_is_split(L, n):
    """Halves are 2^11-element tiles with a compiled layout, of passes planned
    on 2^12; zero skipping, IEEE arithmetic, complex64 and explicit tiles keep
    the plan's tiles or have none to split."""
    desc = L.tpd_plan_describe(n, 0, L.options())[1]
    plan, (run, count) = _parse(desc), _run_passes(desc)
    assert count == sum(1 for p, q in zip(plan, run) if p["D"] != q["D"])
    for p, q in zip(plan, run):
        assert (q["K"], q["b"]) == (p["K"], p["b"]) and (p["D"], q["D"]) in ((p["D"], p["D"]), (12, 11))
    for line in desc.splitlines():
        if line.startswith("split "):
            assert int(re.search(r"shape=(-?\d+)", line).group(1)) >= 0
    for other in (L.options(precision=1), L.options(tile_bits=12)):
        assert "split" not in L.tpd_plan_describe(n, 0, other)[1]
    assert "split" not in L.tpd_plan_describe(n, 1, L.options())[1]
