"""Performance cases of the library: what its callers have it do, through the binding's entry points.

A case is one pass of a caller's loop over one problem, as a dict of plain values.  Its "kind":

  vectors     the level-1 routines on vectors of one length: copy, scal, axpy, swap, rot and the
              reductions dot, asum, nrm2, iamax -- what an iterative solver does between its
              matrix products
  matvec      gemv with A, then with A transposed: the two products of a least-squares,
              bidiagonalisation or primal-dual iteration
  update      ger, syr or syr2 on a matrix that stays on the device: quasi-Newton and
              eliminations
  symmetric   symv on the upper, then on the lower triangle
  multiply    trmv with a triangular factor, then with its transpose
  solve       trsv with a triangular factor, then with its transpose: the two substitutions
              behind a factorisation, or one application of such a preconditioner

Sizes run from those where a call is all latency to those that fill the memory bus for a
millisecond.  Half of the drawn dimensions are multiples of 16, as padded problems have them, the
others are whatever they are: the leading dimension is then often odd, and rows do not start on
16-byte boundaries.
"""
import math

import torch

from paper_2411_07211_b200 import binding as b2

_DTYPES = {"f32": torch.float32, "f64": torch.float64}
_SIZE = {"f32": 4, "f64": 8}
_ORDERS = {"row": b2.ROW_MAJOR, "col": b2.COL_MAJOR}
_UPLO = {"upper": b2.UPPER, "lower": b2.LOWER}
_DIAG = {"unit": b2.UNIT, "non-unit": b2.NON_UNIT}
_LARGEST_MATRIX = 1 << 30  # bytes


def listed():
    return [
        # short vectors that stay in L2: nine calls of a few microseconds each
        {"name": "vectors_65536_f32", "kind": "vectors", "dtype": "f32", "n": 65536, "inc": 1, "offset": 0},
        # an ordinary length that is no multiple of anything; two of the vectors are slices that
        # start off a 16-byte boundary
        {"name": "vectors_1000003_f64", "kind": "vectors", "dtype": "f64", "n": 1000003, "inc": 1, "offset": 1},
        # 256 MiB per vector: memory bandwidth
        {"name": "vectors_64Mi_f32", "kind": "vectors", "dtype": "f32", "n": 1 << 26, "inc": 1, "offset": 0},
        # a small dense operator inside a host-driven loop
        {"name": "matvec_512x512_f32", "kind": "matvec", "dtype": "f32", "m": 512, "n": 512, "order": "row", "pad": 0, "beta": 0.0},
        # ragged in both dimensions, rows on odd boundaries
        {"name": "matvec_5003x3001_f64", "kind": "matvec", "dtype": "f64", "m": 5003, "n": 3001, "order": "row", "pad": 0, "beta": 0.5},
        # 1 GiB of matrix
        {"name": "matvec_16384x16384_f32", "kind": "matvec", "dtype": "f32", "m": 16384, "n": 16384, "order": "row", "pad": 0, "beta": 0.0},
        # tall and narrow: a block of 64 basis vectors or features, stored column after column
        {"name": "matvec_1Mix64_f32", "kind": "matvec", "dtype": "f32", "m": 1 << 20, "n": 64, "order": "col", "pad": 0, "beta": 0.5},
        # rank-1 update of a square matrix
        {"name": "update_ger_4096x4096_f64", "kind": "update", "routine": "ger", "dtype": "f64", "m": 4096, "n": 4096, "order": "row", "pad": 0, "uplo": "upper"},
        # a symmetric operator that is a little larger than L2
        {"name": "symmetric_8192_f32", "kind": "symmetric", "dtype": "f32", "n": 8192, "order": "row", "pad": 0, "beta": 0.5},
        # a triangular factor of odd order in column-major storage
        {"name": "multiply_3001_f32", "kind": "multiply", "dtype": "f32", "n": 3001, "order": "col", "pad": 0, "uplo": "lower", "diag": "non-unit"},
        # substitutions with a factor that fits in L2: the chain of dependences
        {"name": "solve_1024_f64", "kind": "solve", "dtype": "f64", "n": 1024, "order": "row", "pad": 0, "uplo": "lower", "diag": "non-unit"},
        # substitutions with a large factor
        {"name": "solve_11520_f32", "kind": "solve", "dtype": "f32", "n": 11520, "order": "row", "pad": 0, "uplo": "lower", "diag": "non-unit"},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _dimension(rng, lo, hi):
    n = _log_uniform(rng, lo, hi)
    if rng.random() < 0.5:
        n = (n + 15) // 16 * 16
    return max(lo, min(hi, n))


def draw(rng):
    dtype = rng.choice(["f32", "f64"])
    size = _SIZE[dtype]
    kind = rng.choice(["vectors", "matvec", "update", "symmetric", "multiply", "solve"])
    if kind == "vectors":
        inc = rng.choice([1, 1, 1, 2, 3])
        return {"kind": kind, "dtype": dtype, "n": _dimension(rng, 1 << 10, (1 << 26) * 4 // (size * inc)), "inc": inc,
                "offset": rng.choice([0, 0, 1])}
    order = rng.choice(["row", "col"])
    pad = rng.choice([0, 0, 0, rng.randint(1, 64)])
    if kind == "matvec" or (kind == "update" and rng.random() < 0.5):
        most = _LARGEST_MATRIX // size // (2 if kind == "update" else 1)
        while True:
            m, n = _dimension(rng, 16, 1 << 20), _dimension(rng, 16, 1 << 20)
            minor = (n if order == "row" else m) + pad
            if m * n >= 1 << 12 and minor * (m if order == "row" else n) <= most:
                break
        if kind == "matvec":
            return {"kind": kind, "dtype": dtype, "m": m, "n": n, "order": order, "pad": pad, "beta": rng.choice([0.0, 0.5])}
        return {"kind": kind, "routine": "ger", "dtype": dtype, "m": m, "n": n, "order": order, "pad": pad, "uplo": "upper"}
    n = _dimension(rng, 64, 16384 if dtype == "f32" else 11520)
    uplo = rng.choice(["upper", "lower"])
    if kind == "update":
        return {"kind": kind, "routine": rng.choice(["syr", "syr2"]), "dtype": dtype, "m": n, "n": n, "order": order, "pad": pad, "uplo": uplo}
    if kind == "symmetric":
        return {"kind": kind, "dtype": dtype, "n": n, "order": order, "pad": pad, "beta": rng.choice([0.0, 0.5])}
    return {"kind": kind, "dtype": dtype, "n": n, "order": order, "pad": pad, "uplo": uplo, "diag": rng.choice(["unit", "non-unit"])}


# ---- inputs ---------------------------------------------------------------------------------
def _matrix(gen, rows, lda, dtype):
    return torch.rand(rows, lda, generator=gen, dtype=dtype, device="cuda").mul_(2).sub_(1)


def _vector(gen, n, dtype, inc=1, offset=0):
    buf = torch.rand(offset + 1 + (n - 1) * inc, generator=gen, dtype=dtype, device="cuda").mul_(2).sub_(1)
    return buf[offset:]


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    dtype = _DTYPES[case["dtype"]]
    s = {"case": case, "ctx": b2.Context("cuda")}
    if case["kind"] == "vectors":
        n, inc, off = case["n"], case["inc"], case["offset"]
        s["x"] = _vector(gen, n, dtype, inc)
        s["y"] = _vector(gen, n, dtype, inc, off).mul_(0.25).add_(s["x"], alpha=0.75)  # residuals and directions are correlated
        s["u"] = _vector(gen, n, dtype, inc)
        s["v"] = _vector(gen, n, dtype, inc, off)
        s["w"] = torch.zeros_like(s["x"])
        for name in ("dot", "asum", "nrm2"):
            s[name] = torch.zeros(1, dtype=dtype, device="cuda")
        s["iamax"] = torch.zeros(1, dtype=torch.int64, device="cuda")
        return s
    m, n = case.get("m", case["n"]), case["n"]
    rows, cols = (m, n) if case["order"] == "row" else (n, m)
    s["order"], s["lda"] = _ORDERS[case["order"]], cols + case["pad"]
    s["a"] = _matrix(gen, rows, s["lda"], dtype)
    if case["kind"] in ("multiply", "solve"):  # a well-conditioned factor: diagonal in [1, 2), off-diagonal ~ 1/sqrt(n)
        d = s["a"].diagonal()
        diag = d * 0.5 + 1.5
        s["a"].mul_(n ** -0.5)
        d.copy_(diag)
        s["uplo"], s["diag"] = _UPLO[case["uplo"]], _DIAG[case["diag"]]
        s["b"] = _vector(gen, n, dtype)
        s["x"] = torch.zeros_like(s["b"])
    else:
        s["xn"], s["ym"] = _vector(gen, n, dtype), _vector(gen, m, dtype)
        s["xm"], s["yn"] = _vector(gen, m, dtype), _vector(gen, n, dtype)
    return s


# ---- one pass -------------------------------------------------------------------------------
def run(s):
    c, ctx = s["case"], s["ctx"]
    kind, n = c["kind"], c["n"]
    if kind == "vectors":
        inc, x, y, u, v, w = c["inc"], s["x"], s["y"], s["u"], s["v"], s["w"]
        b2.copy(ctx, n, x, inc, w, inc)
        b2.scal(ctx, n, 0.75, w, inc)
        b2.axpy(ctx, n, 0.01, x, inc, y, inc)
        b2.swap(ctx, n, u, inc, v, inc)
        b2.rot(ctx, n, u, inc, v, inc, 0.8, 0.6)
        b2.dot(ctx, n, x, inc, y, inc, s["dot"])
        b2.asum(ctx, n, y, inc, s["asum"])
        b2.nrm2(ctx, n, y, inc, s["nrm2"])
        b2.iamax(ctx, n, x, inc, s["iamax"])
        return {"w": w, "y": y, "u": u, "v": v, "dot": s["dot"], "asum": s["asum"], "nrm2": s["nrm2"], "iamax": s["iamax"]}
    a, lda, order = s["a"], s["lda"], s["order"]
    if kind == "matvec":
        m, beta = c["m"], c["beta"]
        b2.gemv(ctx, order, b2.NO_TRANS, m, n, 1.25, a, lda, s["xn"], 1, beta, s["ym"], 1)
        b2.gemv(ctx, order, b2.TRANS, m, n, 1.25, a, lda, s["xm"], 1, beta, s["yn"], 1)
        return {"ym": s["ym"], "yn": s["yn"]}
    if kind == "update":
        if c["routine"] == "ger":
            b2.ger(ctx, order, c["m"], n, 1e-3, s["xm"], 1, s["xn"], 1, a, lda)
        elif c["routine"] == "syr":
            b2.syr(ctx, order, _UPLO[c["uplo"]], n, 1e-3, s["xn"], 1, a, lda)
        else:
            b2.syr2(ctx, order, _UPLO[c["uplo"]], n, 1e-3, s["xn"], 1, s["xm"], 1, a, lda)
        return {"a": a}
    if kind == "symmetric":
        b2.symv(ctx, order, b2.UPPER, n, 1.25, a, lda, s["xn"], 1, c["beta"], s["ym"], 1)
        b2.symv(ctx, order, b2.LOWER, n, 1.25, a, lda, s["xm"], 1, c["beta"], s["yn"], 1)
        return {"ym": s["ym"], "yn": s["yn"]}
    call = b2.trmv if kind == "multiply" else b2.trsv
    b2.copy(ctx, n, s["b"], 1, s["x"], 1)
    call(ctx, order, s["uplo"], b2.NO_TRANS, s["diag"], n, a, lda, s["x"], 1)
    call(ctx, order, s["uplo"], b2.TRANS, s["diag"], n, a, lda, s["x"], 1)
    return {"x": s["x"]}


# ---- what a pass cannot do without ----------------------------------------------------------
def work(case):
    size, n = _SIZE[case["dtype"]], case["n"]
    kind = case["kind"]
    if kind == "vectors":
        # copy 2, scal 2, axpy 3, swap 4, rot 4, dot 2, asum 1, nrm2 1, iamax 1 vectors; memory moves
        # whole 32-byte sectors, so a strided vector costs its span up to one sector per element
        return {"bytes": 20 * n * min(size * case["inc"], 32), "flops": n * (1 + 2 + 6 + 2 + 1 + 2)}
    if kind == "matvec":
        m = case["m"]
        vectors = m + n + (m + n) * (2 if case["beta"] else 1)
        return {"bytes": size * (2 * m * n + vectors), "flops": 4 * m * n}
    triangle = n * (n + 1) // 2
    if kind == "update":
        if case["routine"] == "ger":
            return {"bytes": size * (2 * case["m"] * n + case["m"] + n), "flops": 2 * case["m"] * n}
        k = 1 if case["routine"] == "syr" else 2
        return {"bytes": size * (2 * triangle + k * n), "flops": 2 * k * triangle}
    if kind == "symmetric":
        return {"bytes": size * (2 * triangle + 2 * n * (3 if case["beta"] else 2)), "flops": 4 * n * n}
    return {"bytes": size * (2 * triangle + 6 * n), "flops": 2 * n * n}


def tolerance(case):
    # rounding of sums in the case's own precision; "max" allows for single sums that cancel
    return {"rel": 1e-5, "max": 1e-3} if case["dtype"] == "f32" else {"rel": 1e-13, "max": 1e-11}
