"""Qudit levels fused into passes, at sizes that reach every kernel of the
pass rule (levels per pass, columns per tile, first and later passes,
remainders), and the out-of-place calls.

Reference: the level maps applied one after another in complex128 by plain
torch.  Tolerance: each level is an isometry up to a factor (in the weighted
norm for the Gell-Mann basis) and rounds each output at most 16 times at the
unit roundoff u of the arithmetic, so the error stays below 16 n u of the
result's norm, as in the other tests of these bases."""
import math

import pytest
import torch

SIZES = [(2, n) for n in range(1, 12)] + [(3, n) for n in range(1, 8)] + [(4, n) for n in range(1, 6)] + \
        [(5, n) for n in range(1, 6)]


def _levels(A, d, level):
    N, s = A.shape[0], 1
    A = A.to(torch.complex128)
    while s < N:
        v = A.view(N // (s * d), d, s, N // (s * d), d, s)
        out = torch.empty_like(v)
        level(lambda r, c: v[:, r, :, :, c, :], lambda r, c, x: out[:, r, :, :, c, :].copy_(x))
        A, s = out.view(N, N), s * d
    return A


def _weyl(A, d, dec):
    w = [complex(math.cos(2 * math.pi * k / d), math.sin(2 * math.pi * k / d)) for k in range(d)]

    def level(get, put):
        for a in range(d):
            for b in range(d):
                if dec:
                    put(b, (a + b) % d, sum(get((c + a) % d, c) * (w[-b * c % d] / d) for c in range(d)))
                else:
                    put((b + a) % d, b, sum(get(c, (a + c) % d) * w[b * c % d] for c in range(d)))

    return _levels(A, d, level)


def _gellmann(A, d, dec):
    f = [0.0] + [math.sqrt(2.0 / (k * (k + 1))) for k in range(1, d)]

    def level(get, put):
        for j in range(d):
            for k in range(j + 1, d):
                if dec:
                    put(j, k, (get(j, k) + get(k, j)) * 0.5)
                    put(k, j, (get(j, k) - get(k, j)) * 0.5j)
                else:
                    put(j, k, get(j, k) - 1j * get(k, j))
                    put(k, j, get(j, k) + 1j * get(k, j))
        for m in range(d):
            if dec:
                put(m, m, (sum(get(i, i) for i in range(m)) - m * get(m, m)) * (0.5 * f[m]) if m else
                    sum(get(i, i) for i in range(d)) / d)
            else:
                x = get(0, 0) + sum(f[k] * get(k, k) for k in range(m + 1, d))
                put(m, m, x - (m * f[m]) * get(m, m) if m else x)

    return _levels(A, d, level)


def _matrix(N, dtype, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(N, N, dtype=torch.complex128, device="cuda", generator=g).to(dtype)


def _calls(basis):
    import paper_2310_13421_gb300 as tpd
    return {"weyl": (tpd.weyl_decompose, tpd.weyl_compose, _weyl),
            "gellmann": (tpd.gellmann_decompose, tpd.gellmann_compose, _gellmann)}[basis]


@pytest.mark.gpu
@pytest.mark.parametrize("d,n", SIZES)
@pytest.mark.parametrize("basis", ["weyl", "gellmann"])
@pytest.mark.parametrize("dtype", [torch.complex64, torch.complex128])
def test_passes_against_levels(basis, d, n, dtype):
    dec, com, ref = _calls(basis)
    A = _matrix(d ** n, dtype, 10 * d + n)
    tol = 16 * n * (2.0 ** -24 if dtype == torch.complex64 else 2.0 ** -53)
    for call, want in ((dec(A, d), ref(A, d, True)), (com(A, d), ref(A, d, False)),
                       (com(A, d, scale=0.375), ref(A, d, False) * 0.375)):
        err = (call.to(torch.complex128) - want).norm() / want.norm()
        assert float(err) <= tol


@pytest.mark.gpu
@pytest.mark.parametrize("d,n", [(2, 1), (2, 7), (3, 1), (3, 4), (3, 6), (4, 3), (5, 3)])
@pytest.mark.parametrize("basis", ["weyl", "gellmann"])
@pytest.mark.parametrize("dtype", [torch.complex64, torch.complex128])
def test_out_of_place_equals_in_place(basis, d, n, dtype):
    dec, com, _ = _calls(basis)
    A = _matrix(d ** n, dtype, n)
    A[-1, 0] = float("inf")                               # classes with Inf / NaN take the IEEE path
    kept = torch.view_as_real(A).clone()
    as_bits = torch.int32 if dtype == torch.complex64 else torch.int64
    for call in (lambda X, p: dec(X, d, inplace=p), lambda X, p: com(X, d, scale=0.5, inplace=p)):
        out = torch.view_as_real(call(A, False)).view(as_bits)
        assert torch.equal(torch.view_as_real(A).view(as_bits), kept.view(as_bits))
        assert torch.equal(out, torch.view_as_real(call(A.clone(), True)).view(as_bits))


def test_argument_errors():
    from paper_2310_13421_gb300 import _lib as L, buildlib
    buildlib.build()
    size = 16 * 3 ** 6
    for call in (lambda a, w: L.tpd_weyl_decompose_to(a, w, 3, 3, L.TPD_C128),
                 lambda a, w: L.tpd_weyl_compose_to(a, w, 3, 3, L.TPD_C128, 1.0),
                 lambda a, w: L.tpd_gellmann_decompose_to(a, w, 3, 3, L.TPD_C128),
                 lambda a, w: L.tpd_gellmann_compose_to(a, w, 3, 3, L.TPD_C128, 1.0)):
        assert call(0, 4096) == L.TPD_ERR_INVALID_ARG
        assert call(4096, 0) == L.TPD_ERR_INVALID_ARG
        assert call(4096, 4096 + size - 16) == L.TPD_ERR_INVALID_ARG          # overlap
        assert call(4096 + 8, 1 << 20) == L.TPD_ERR_MISALIGNED
        assert call(4096, (1 << 20) + 8) == L.TPD_ERR_MISALIGNED
