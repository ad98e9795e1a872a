"""The work a user of this package has it do, as cases to be timed.

A case is a dict of plain values: "kind" names the call, the rest its sizes and
options.  The kinds and what they stand for:

  dec       decompose(A): the Pauli weights of a dense matrix, kept beside it
  string    decompose(A) and to_string_layout: the weights in base-4 string
            order, as a program that indexes them by Pauli string wants them
  com       compose(C): the matrix of a full set of weights
  train     the differentiable decomposition inside a model: forward, and
            backward from the gradient that arrives at the weights
  batch     a kept Batch of matrices of uneven sizes, refilled and decomposed
  list      a structured Hamiltonian held densely: decompose with zero skipping,
            then the paper's list of nonzero weights
  coo       the same Hamiltonian given by its nonzero entries
  weyl      qudits, Weyl basis (either direction)
  gellmann  qudits, generalized Gell-Mann basis (either direction)
"""
import math

import torch

import paper_2310_13421_gb300 as tpd
from paper_2310_13421_gb300 import synth

DEV = "cuda"
_TYPE = {"c128": torch.complex128, "c64": torch.complex64}


def listed():
    return [
        # one small molecule's or gate's matrix: the smallest call, all latency
        {"name": "dec-c128-n6", "kind": "dec", "n": 6, "dtype": "c128", "precision": "default", "hermitian": True},
        # an ordinary matrix (67 MB, it fits in L2), odd qubit count
        {"name": "dec-c128-n11", "kind": "dec", "n": 11, "dtype": "c128", "precision": "default", "hermitian": True},
        # the headline size: a dense 4.3 GB Hermitian matrix
        {"name": "dec-c128-n14", "kind": "dec", "n": 14, "dtype": "c128", "precision": "default", "hermitian": True},
        # complex64 with its default arithmetic, weights wanted in string order
        {"name": "string-c64-n13", "kind": "string", "n": 13, "dtype": "c64", "precision": "default",
         "hermitian": True},
        # complex64 with error-compensated sums at the largest size (8.6 GB)
        {"name": "dec-c64-comp-n15", "kind": "dec", "n": 15, "dtype": "c64", "precision": "compensated",
         "hermitian": True},
        # a matrix rebuilt from (non-real) weights
        {"name": "com-c128-n13", "kind": "com", "n": 13, "dtype": "c128", "precision": "default"},
        # one training step's worth of the decomposition layer, both directions
        {"name": "train-c128-n12", "kind": "train", "n": 12, "dtype": "c128"},
        # thousands of matrices, n uniform in 3..10
        {"name": "batch-c128-n3-10", "kind": "batch", "count": 4096, "n_lo": 3, "n_hi": 10, "dtype": "c128"},
        # a Heisenberg chain, dense and as its entries
        {"name": "list-c128-n14", "kind": "list", "n": 14, "dtype": "c128"},
        {"name": "coo-n14", "kind": "coo", "n": 14},
        # nine qutrits (a side that is no power of two), both bases and types
        {"name": "weyl-c128-d3-n9", "kind": "weyl", "d": 3, "n": 9, "dtype": "c128", "dec": True},
        {"name": "gellmann-c64-d3-n9", "kind": "gellmann", "d": 3, "n": 9, "dtype": "c64", "dec": True},
    ]


# largest qubit count of a drawn case: no drawn case costs more than the largest listed one
_DEC_MAX = {("c128", "default"): 14, ("c128", "plain"): 13, ("c64", "default"): 15, ("c64", "compensated"): 15,
            ("c64", "fixed"): 14}
# qudit counts: d^n up to 19,683 (complex128 with d = 5 up to 3,125)
_QUDIT_MAX = {2: 14, 3: 9, 4: 7, 5: 6}


def draw(rng):
    kind = rng.choice(["dec", "dec", "dec", "string", "com", "train", "batch", "list", "coo", "weyl", "gellmann"])
    if kind == "dec":
        dtype, precision = rng.choice(sorted(_DEC_MAX) + [("c128", "default"), ("c64", "default")])
        return {"kind": kind, "n": rng.randint(2, _DEC_MAX[dtype, precision]), "dtype": dtype, "precision": precision,
                "hermitian": rng.random() < 0.7}
    if kind == "string":
        dtype = rng.choice(["c128", "c64"])
        return {"kind": kind, "n": rng.randint(3, 13 if dtype == "c128" else 14), "dtype": dtype,
                "precision": "default", "hermitian": rng.random() < 0.7}
    if kind == "com":
        dtype = rng.choice(["c128", "c64"])
        return {"kind": kind, "n": rng.randint(2, 13 if dtype == "c128" else 14), "dtype": dtype,
                "precision": "default"}
    if kind == "train":
        dtype = rng.choice(["c128", "c64"])
        return {"kind": kind, "n": rng.randint(3, 12 if dtype == "c128" else 13), "dtype": dtype}
    if kind == "batch":
        lo = rng.randint(1, 6)
        hi = rng.randint(lo, 10)
        # at most as many elements as the listed batch holds
        mean = sum(4 ** n for n in range(lo, hi + 1)) / (hi - lo + 1)
        most = min(4096.0, 7e8 / mean)
        return {"kind": kind, "count": round(math.exp(rng.uniform(math.log(8), math.log(most)))), "n_lo": lo,
                "n_hi": hi, "dtype": rng.choice(["c128", "c128", "c64"])}
    if kind == "list":
        return {"kind": kind, "n": rng.randint(6, 14), "dtype": "c128"}
    if kind == "coo":
        return {"kind": kind, "n": rng.randint(6, 14)}
    d = rng.choice([2, 3, 3, 4, 5])
    dtype = rng.choice(["c128", "c64"])
    return {"kind": kind, "d": d, "n": rng.randint(2, 5 if (d, dtype) == (5, "c128") else _QUDIT_MAX[d]),
            "dtype": dtype, "dec": rng.random() < 0.7}


# ------------------------------------------------------------------ inputs


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _general(shape, dtype, g):
    """Complex entries with N(0, 1) real and imaginary parts."""
    real = torch.float64 if dtype == torch.complex128 else torch.float32
    return torch.view_as_complex(torch.randn(*shape, 2, generator=g, device=DEV, dtype=real))


def _hermitian(N, dtype, g):
    B = _general((N, N), dtype, g)
    return (B + B.mH).mul_(0.5)


def _matrix(case, N, seed):
    make = _hermitian if case.get("hermitian", True) else (lambda N, t, g: _general((N, N), t, g))
    return make(N, _TYPE[case["dtype"]], _gen(seed))


def _batch_sizes(case):
    """The sizes belong to the case, the entries to the seed: a refilled batch keeps its sizes."""
    return [int(n) for n in synth.batch_sizes(case["count"], 2024, case["n_lo"], case["n_hi"])]


def _batch_views(flat, ns):
    out, at = [], 0
    for n in ns:
        out.append(flat[at:at + 4 ** n].view(2 ** n, 2 ** n))
        at += 4 ** n
    return out


def _batch_source(case, seed):
    ns = _batch_sizes(case)
    return ns, _general((sum(4 ** n for n in ns),), _TYPE[case["dtype"]], _gen(seed))


def _chain(case, seed):
    """A Heisenberg chain with seeded couplings and fields, dense."""
    n = case["n"]
    J, h = synth.heisenberg_params(n, seed)
    H = torch.zeros(2 ** n, 2 ** n, dtype=_TYPE[case.get("dtype", "c128")], device=DEV)
    return synth.heisenberg_into(H, n, J, h)


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("dec", "string"):
        return {"kind": kind, "A": _matrix(case, 2 ** case["n"], seed), "precision": case["precision"]}
    if kind == "com":
        return {"kind": kind, "C": _general((2 ** case["n"],) * 2, _TYPE[case["dtype"]], _gen(seed)),
                "precision": case["precision"]}
    if kind == "train":
        N, t, g = 2 ** case["n"], _TYPE[case["dtype"]], _gen(seed)
        return {"kind": kind, "A": _hermitian(N, t, g).requires_grad_(), "grad": _general((N, N), t, g)}
    if kind == "batch":
        ns, source = _batch_source(case, seed)
        flat = torch.empty_like(source)
        return {"kind": kind, "source": source, "flat": flat, "batch": tpd.Batch(_batch_views(flat, ns))}
    if kind == "list":
        return {"kind": kind, "A": _chain(case, seed)}
    if kind == "coo":
        H = _chain(case, seed)
        rows, cols = torch.nonzero(H, as_tuple=True)
        return {"kind": kind, "n": case["n"], "rows": rows.to(torch.int32), "cols": cols.to(torch.int32),
                "values": H[rows, cols].contiguous()}
    N = case["d"] ** case["n"]
    if case["dec"]:
        A = _hermitian(N, _TYPE[case["dtype"]], _gen(seed))
    else:
        A = _general((N, N), _TYPE[case["dtype"]], _gen(seed))
    return {"kind": kind, "A": A, "d": case["d"], "dec": case["dec"]}


def run(s):
    kind = s["kind"]
    if kind == "dec":
        return tpd.decompose(s["A"], precision=s["precision"])
    if kind == "string":
        return tpd.to_string_layout(tpd.decompose(s["A"], precision=s["precision"]))
    if kind == "com":
        return tpd.compose(s["C"], precision=s["precision"])
    if kind == "train":
        W = tpd.tpd(s["A"])
        (gA,) = torch.autograd.grad(W, s["A"], s["grad"])
        return W.detach(), gA
    if kind == "batch":
        s["flat"].copy_(s["source"])
        s["batch"].decompose()
        return s["flat"]
    if kind == "list":
        W = tpd.decompose(s["A"], skip_zero=True)
        strings, weights = tpd.nonzero_list(W)
        return W, strings, weights
    if kind == "coo":
        return tpd.decompose_coo(s["rows"], s["cols"], s["values"], s["n"])
    if kind == "weyl":
        return (tpd.weyl_decompose if s["dec"] else tpd.weyl_compose)(s["A"], s["d"])
    return (tpd.gellmann_decompose if s["dec"] else tpd.gellmann_compose)(s["A"], s["d"])


def work(case):
    kind = case["kind"]
    esize = 8 if case.get("dtype", "c128") == "c64" else 16
    if kind == "batch":
        # expected sizes: every n equally often
        ns = range(case["n_lo"], case["n_hi"] + 1)
        elems = case["count"] / len(ns) * sum(4 ** n for n in ns)
        flops = case["count"] / len(ns) * sum(2 * n * 4 ** n for n in ns)
        return {"bytes": 2 * esize * elems, "flops": flops}
    n = case["n"]
    if kind == "coo":
        # the chain's entries: the diagonal and, per bond, half the rows; 12 + 16 bytes an entry with its indices,
        # each entry meeting its n levels twice
        nnz = 2 ** n * (1 + (n - 1) / 2)
        return {"bytes": 24 * nnz + 24 * (4 * n - 3), "flops": 4 * n * nnz}
    if kind in ("weyl", "gellmann"):
        d = case["d"]
        elems = float(d ** (2 * n))
        per = {2: 2, 3: 4, 4: 4, 5: 16}[d] if kind == "weyl" else 3
        return {"bytes": 2 * esize * elems, "flops": per * n * elems}
    elems = float(4 ** n)
    passes = 2 if kind == "train" else 1
    return {"bytes": passes * 2 * esize * elems, "flops": passes * 2 * n * elems}


# ------------------------------------------------------------------ the same results in 64 bits


def _pauli(A, dec, scale=1.0):
    """Every qubit level of Eq. 4 (or its inverse) on a batch (m, N, N) in complex128."""
    m, N = A.shape[0], A.shape[1]
    n = N.bit_length() - 1
    A = A.to(torch.complex128)
    for b in range(n):
        v = A.view(m, N >> (b + 1), 2, 1 << b, N >> (b + 1), 2, 1 << b)
        out = torch.empty_like(v)
        p, q, r, t = (v[:, :, i, :, :, j, :] for i in (0, 1) for j in (0, 1))
        if dec:
            out[:, :, 0, :, :, 0, :] = (p + t) * 0.5
            out[:, :, 0, :, :, 1, :] = (q + r) * 0.5
            out[:, :, 1, :, :, 0, :] = (q - r) * 0.5j
            out[:, :, 1, :, :, 1, :] = (p - t) * 0.5
        else:
            out[:, :, 0, :, :, 0, :] = p + t
            out[:, :, 0, :, :, 1, :] = q - 1j * r
            out[:, :, 1, :, :, 0, :] = q + 1j * r
            out[:, :, 1, :, :, 1, :] = p - t
        A = out.view(m, N, N)
    return A if scale == 1.0 else A * scale


def _string_order(W):
    """(N, N) weights -> base-4 string order: the bits of row and column interleaved, row bit first."""
    n = W.shape[0].bit_length() - 1
    s = torch.arange(4 ** n, device=DEV)
    at = torch.zeros_like(s)
    for b in range(n):
        at += ((s >> (2 * b)) & 1) << b
        at += ((s >> (2 * b + 1)) & 1) << (n + b)
    return W.reshape(-1)[at]


def _levels(A, d, level):
    """`level` on the d x d blocks of every qudit: (d, d, ...) -> (d, d, ...)."""
    N = A.shape[0]
    A, s = A.to(torch.complex128), 1
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
    c = [0.0] + [math.sqrt(2.0 / (l * (l + 1))) for l in range(1, d)]

    def level(get, put):
        for j in range(d):
            for k in range(j + 1, d):
                if dec:
                    put(j, k, (get(j, k) + get(k, j)) * 0.5)
                    put(k, j, (get(j, k) - get(k, j)) * 0.5j)
                else:
                    put(j, k, get(j, k) - 1j * get(k, j))
                    put(k, j, get(j, k) + 1j * get(k, j))
        if dec:
            put(0, 0, sum(get(m, m) for m in range(d)) / d)
            for l in range(1, d):
                put(l, l, (sum(get(m, m) for m in range(l)) - l * get(l, l)) * (0.5 * c[l]))
        else:
            for m in range(d):
                x = get(0, 0) + sum(c[l] * get(l, l) for l in range(m + 1, d))
                put(m, m, x - (m * c[m]) * get(m, m) if m else x)

    return _levels(A, d, level)


def _chain_weights(case, seed):
    """The chain's nonzero weights in string order (positions, weights)."""
    n = case["n"]
    terms = synth.heisenberg_terms(n, *synth.heisenberg_params(n, seed))
    found = sorted((synth.string_index(t), float(w)) for t, w in terms.items() if w != 0.0)
    return ([i for i, _ in found],
            torch.tensor([w for _, w in found], dtype=torch.float64, device=DEV).to(torch.complex128))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("dec", "string"):
        W = _pauli(_matrix(case, 2 ** case["n"], seed)[None], True)[0]
        return W if kind == "dec" else _string_order(W)
    if kind == "com":
        return _pauli(_general((2 ** case["n"],) * 2, _TYPE[case["dtype"]], _gen(seed))[None], False)[0]
    if kind == "train":
        N, t, g = 2 ** case["n"], _TYPE[case["dtype"]], _gen(seed)
        A = _hermitian(N, t, g)
        grad = _general((N, N), t, g)
        return _pauli(A[None], True)[0], _pauli(grad[None], False, 1.0 / N)[0]
    if kind == "batch":
        ns, source = _batch_source(case, seed)
        out = torch.empty(source.shape, dtype=torch.complex128, device=DEV)
        views, outs = _batch_views(source, ns), _batch_views(out, ns)
        for n in sorted(set(ns)):
            of = [i for i, x in enumerate(ns) if x == n]
            for i, W in zip(of, _pauli(torch.stack([views[i] for i in of]), True)):
                outs[i].copy_(W)
        return out
    if kind == "list":
        n = case["n"]
        at, weights = _chain_weights(case, seed)
        W = torch.zeros(4 ** n, dtype=torch.complex128, device=DEV)
        rows = [sum(((s >> (2 * b + 1)) & 1) << b for b in range(n)) for s in at]
        cols = [sum(((s >> (2 * b)) & 1) << b for b in range(n)) for s in at]
        W[torch.tensor(rows, device=DEV) * 2 ** n + torch.tensor(cols, device=DEV)] = weights
        return W.view(2 ** n, 2 ** n), None, weights
    if kind == "coo":
        return None, _chain_weights(case, seed)[1]
    if case["dec"]:
        A = _hermitian(case["d"] ** case["n"], _TYPE[case["dtype"]], _gen(seed))
    else:
        A = _general((case["d"] ** case["n"],) * 2, _TYPE[case["dtype"]], _gen(seed))
    return (_weyl if kind == "weyl" else _gellmann)(A, case["d"], case["dec"])
