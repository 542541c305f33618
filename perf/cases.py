"""What a user of this library has it do, as measurable cases.

Every case is one pass through the public entry points (trsm, trmm, Factor,
trsm_refined_async, Batch) on column-major CUDA tensors. TRSM and TRMM work in
place, so a pass first restores the right-hand side from its kept copy, as a
program does that solves into a buffer of its own and keeps the original.

Factors are triangles as an LU or Cholesky factorisation of a well-conditioned
matrix leaves them: diagonal 1 + |N(0,1)|, off-diagonal entries
uniform(-1, 1)/sqrt(k) (a row's off-diagonal part is of the diagonal's size),
and other finite numbers in the triangle that the call does not reference.
Right-hand sides are N(0,1).

Cost is counted in the m^2 n convention: k^2 nrhs operations, k the order of
the triangle.
"""
import math

import numpy as np
import torch

import paper_2504_13821_gb300 as trx

# Largest k^2 nrhs of a drawn case, by what it runs: the largest listed ones.
F32_WORK = 16384.0 ** 3
F64_WORK = 4096.0 ** 3
REFINED_WORK = 4096.0 ** 2 * 256


def _case(name, op, dtype, variant, m, n, alpha=1.0, api="call", pad=0):
    side, uplo, trans, diag = variant
    return {"name": name, "api": api, "op": op, "dtype": dtype, "side": side, "uplo": uplo,
            "trans": trans, "diag": diag, "m": m, "n": n, "alpha": alpha, "pad": pad}


def listed():
    return [
        # the smallest calls: a filter or a block of a larger algorithm, where
        # launches and latency are the time
        _case("trsm_f32_small", "trsm", "f32", "LLNN", 256, 256),
        _case("trmm_f32_odd", "trmm", "f32", "RUTU", 500, 300, 0.5, pad=3),
        # few right-hand sides: a solve with a kept factor, back substitution
        _case("trsm_f32_thin", "trsm", "f32", "LLTN", 8191, 16),
        _case("trsm_f32_factor", "trsm", "f32", "LLNN", 4096, 256, api="factor"),
        # block steps of a factorisation: middle sizes, both sides of B
        _case("trsm_f32_mid", "trsm", "f32", "RLNN", 2000, 2000, -1.0),
        _case("trmm_f32_mid", "trmm", "f32", "LUNN", 4096, 4096),
        # the square problem that the library is usually quoted on
        _case("trsm_f32_large", "trsm", "f32", "LLNN", 16384, 16384, 1.5),
        # the same in FP64
        _case("trsm_f64_small", "trsm", "f64", "LUNN", 1000, 200),
        _case("trsm_f64_large", "trsm", "f64", "LLNN", 4096, 4096, 1.5),
        _case("trmm_f64_mid", "trmm", "f64", "RUNU", 2500, 1500, 2.0, pad=5),
        # an FP64-accurate solution from FP32 data, as a server refines it
        _case("trsm_refined", "trsm", "f32", "LLNN", 4096, 256, api="refined"),
        # many small uneven problems in one launch (orders 16 .. 512)
        {"name": "batch_f32", "api": "batch", "dtype": "f32", "count": 4096, "sizes": 4096},
    ]


def _log_int(rng, lo, hi):
    """A whole number of [lo, hi], uniform over the logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["f32", "f32", "f32", "f32", "f64", "f64", "f64", "refined", "batch"])
    if kind == "batch":
        return {"api": "batch", "dtype": rng.choice(["f32", "f32", "f64"]),
                "count": _log_int(rng, 256, 4096), "sizes": rng.randrange(1 << 30)}
    work = {"f32": F32_WORK, "f64": F64_WORK, "refined": REFINED_WORK}[kind]
    k = _log_int(rng, 256, {"f32": 16384, "f64": 8192, "refined": 4096}[kind])
    n = _log_int(rng, 16, int(min(16384, work / k ** 2)))
    if rng.random() < 0.4:                   # the sizes that programs like to use
        k = max(256, k // 256 * 256)
    if rng.random() < 0.3:
        n = max(16, n // 16 * 16)
    side = rng.choice("LR")
    api, op = "call", rng.choice(["trsm", "trsm", "trmm"])
    if kind == "refined":
        api, op = "refined", "trsm"
    elif kind == "f32" and rng.random() < 0.25:
        api = "factor"
    m, n = (k, n) if side == "L" else (n, k)
    return {"api": api, "op": op, "dtype": "f64" if kind == "f64" else "f32", "side": side,
            "uplo": rng.choice("LU"), "trans": rng.choice("NNT"), "diag": rng.choice("NNNU"),
            "m": m, "n": n, "alpha": rng.choice([1.0, -1.0, 1.5, 0.5]),
            "pad": rng.choice([0, 0, 0, 1, 8])}


def _dtype(case):
    return torch.float64 if case["dtype"] == "f64" else torch.float32


def _order(case):
    return case["m"] if case["side"] == "L" else case["n"]


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _triangle(out, g):
    """Fill the k x k view `out` with a factor and, beside it, other numbers."""
    k = out.shape[0]
    out.uniform_(-1.0, 1.0, generator=g).div_(math.sqrt(k))
    d = torch.empty(k, dtype=out.dtype, device="cuda").normal_(generator=g)
    out.diagonal().copy_(d.abs_().add_(1.0))


def _colmajor(rows, cols, dtype, pad=0):
    """An uninitialised column-major rows x cols view with leading dimension rows + pad."""
    return torch.zeros((cols, rows + pad), dtype=dtype, device="cuda").t()[:rows]


def _inputs(case, seed):
    g, dtype, k = _generator(seed), _dtype(case), _order(case)
    A = _colmajor(k, k, dtype, case["pad"])
    _triangle(A, g)
    B = _colmajor(case["m"], case["n"], dtype, case["pad"])
    B.copy_(torch.empty((case["n"], case["m"]), dtype=dtype, device="cuda").normal_(generator=g).t())
    return A, B


def _batch_shapes(case):
    """[(op, side, uplo, k, nrhs, offset of A, offset of B)] and the two totals."""
    r = np.random.default_rng(case["sizes"])
    out, na, nb = [], 0, 0
    for i in range(case["count"]):
        k = int(round(math.exp(r.uniform(math.log(16), math.log(512)))))
        nrhs = int(r.integers(1, 65))
        side, uplo = "LR"[int(r.integers(2))], "LU"[int(r.integers(2))]
        out.append(("SM"[i % 2], side, uplo, k, nrhs, na, nb))
        na += k * k
        nb += (k * nrhs + 3) // 4 * 4
    return out, na, nb


def _batch_inputs(case, seed):
    shapes, na, nb = _batch_shapes(case)
    g, dtype = _generator(seed), _dtype(case)
    a = torch.empty(na, dtype=dtype, device="cuda").uniform_(-1.0, 1.0, generator=g)
    b = torch.empty(nb, dtype=dtype, device="cuda").normal_(generator=g)
    # scale by 1/sqrt(k) and set the diagonals in two passes over all problems
    ks = torch.tensor([s[3] for s in shapes], device="cuda")
    a.div_(torch.repeat_interleave(ks.to(dtype).sqrt(), ks * ks))
    first = torch.repeat_interleave(torch.cumsum(ks * ks, 0) - ks * ks, ks)
    step = torch.repeat_interleave(ks + 1, ks)
    index = torch.arange(first.numel(), device="cuda") - torch.repeat_interleave(
        torch.cumsum(ks, 0) - ks, ks)
    d = torch.empty(first.numel(), dtype=dtype, device="cuda").normal_(generator=g)
    a[first + index * step] = d.abs_().add_(1.0)
    return shapes, a, b


def _batch_views(shape, a, b):
    op, side, uplo, k, nrhs, oa, ob = shape
    m, n = (k, nrhs) if side == "L" else (nrhs, k)
    return a[oa:oa + k * k].view(k, k).t(), b[ob:ob + m * n].view(n, m).t()


def prepare(case, seed):
    if case["api"] == "batch":
        shapes, a, b = _batch_inputs(case, seed)
        x = b.clone()
        problems = [(s[0], s[1], s[2], "N", "N", 1.0) + _batch_views(s, a, x) for s in shapes]
        return {"case": case, "A": a, "B": b, "X": x, "batch": trx.Batch(problems)}
    A, B = _inputs(case, seed)
    state = {"case": case, "A": A, "B": B}
    if case["api"] == "refined":
        state["X"] = _colmajor(case["m"], case["n"], torch.float64)
    else:
        state["X"] = _colmajor(case["m"], case["n"], B.dtype, case["pad"])
    if case["api"] == "factor":
        state["factor"] = trx.Factor(case["side"], case["uplo"], case["trans"], case["diag"], A)
    return state


def run(state):
    case, A, B, X = state["case"], state["A"], state["B"], state["X"]
    if case["api"] == "batch":
        X.copy_(B)
        state["batch"].run()
        return X
    variant = case["side"], case["uplo"], case["trans"], case["diag"]
    if case["api"] == "refined":
        return trx.trsm_refined_async(*variant, case["alpha"], A, B, corrections=2, out=X)
    X.copy_(B)
    if case["api"] == "factor":
        call = state["factor"].trsm if case["op"] == "trsm" else state["factor"].trmm
        return call(case["alpha"], X)
    call = trx.trsm if case["op"] == "trsm" else trx.trmm
    return call(*variant, case["alpha"], A, X)


def work(case):
    if case["api"] == "batch":
        w = 8 if case["dtype"] == "f64" else 4
        shapes, _, _ = _batch_shapes(case)
        return {"bytes": sum(w * (k * (k + 1) // 2 + 2 * k * r) for _, _, _, k, r, _, _ in shapes),
                "flops": sum(k * k * r for _, _, _, k, r, _, _ in shapes)}
    w = 8 if case["dtype"] == "f64" else 4
    k, elements = _order(case), case["m"] * case["n"]
    out = 8 if case["api"] == "refined" else w
    return {"bytes": w * k * (k + 1) // 2 + (w + out) * elements, "flops": k * elements}


def _apply(op, side, uplo, trans, diag, alpha, A, B):
    """alpha op(A)^-1 B, alpha B op(A)^-1, or the products, in 64 bits."""
    A, B = A.to(torch.float64), B.to(torch.float64) * alpha
    upper = uplo == "U"
    if trans == "T":
        A, upper = A.mT, not upper
    if op in ("S", "trsm"):
        return torch.linalg.solve_triangular(A, B, upper=upper, left=side == "L",
                                             unitriangular=diag == "U")
    A = A.triu() if upper else A.tril()
    if diag == "U":
        A.diagonal().fill_(1.0)
    return A @ B if side == "L" else B @ A


def exact(case, seed):
    if case["api"] == "batch":
        shapes, a, b = _batch_inputs(case, seed)
        x = b.to(torch.float64)
        for s in shapes:
            A, B = _batch_views(s, a, b)
            _batch_views(s, a, x)[1].copy_(_apply(s[0], s[1], s[2], "N", "N", 1.0, A, B))
        return x
    A, B = _inputs(case, seed)
    return _apply(case["op"], case["side"], case["uplo"], case["trans"], case["diag"],
                  case["alpha"], A, B)
