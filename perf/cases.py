"""The solves that programs run through this library, as cases to time and compare.

A case is one call of the C ABI (through its ctypes binding) on device-resident
data: a triangular solve of one system, a solve with LU or Cholesky factors, or
a varlen batch of small solves.  Every entry point overwrites B with X, so a
pass copies the right-hand sides into the buffer that is solved in place, as a
program that keeps B does, and returns that buffer.

Sizes are those of the library's configurations, tests and serving stream
(m up to 4096 and n up to 512 there), with odd and padded ones among them.
Values follow the seeded recipe of inputs.py: off-diagonal entries U(-1, 1) / m,
diagonal 1 + U(0, 1), right-hand sides U(-1, 1), complex parts drawn alike.
"""
import math

import numpy as np
import torch

from paper_2608_25469_gb300 import hsma as H

# dtype code of the C ABI, torch element type, the 64-bit type of exact()
_DTYPES = {
    "f64": (H.R64, torch.float64),
    "c128": (H.C128, torch.complex128),
    "f32": (H.R32, torch.float32),
    "c64": (H.C64, torch.complex64),
    "f32_bf16": (H.R32_BF16, torch.float32),  # FP32 result, BF16 tensor-core products
    "f64_ir": (H.R64_IR, torch.float64),  # FP64 result by refinement of FP32 solves
}
_COMPLEX = ("c128", "c64")
_TRANS = {"n": H.NO_TRANS, "t": H.TRANS, "c": H.CONJ_TRANS}


def _one(name, dtype, m, n, **more):
    """One system: side / uplo / trans / unit / pad (rows of ld beyond the matrix) / factor
    (none, lu = getrs with interchanges, chol = potrs) / emulated FP64 products."""
    c = {"op": "one", "dtype": dtype, "m": m, "n": n, "side": "left", "uplo": "lower", "trans": "n", "unit": False,
         "pad": 0, "factor": "none", "emulated": False, "alpha": 1.0}
    c.update(more)
    return dict(c, name=name) if name else c


def _batch(name, dtype, batch, lo, hi, **more):
    """A varlen batch, m and n uniform in lo .. hi (<= 64) each, drawn from `sizes`."""
    c = {"op": "batch", "dtype": dtype, "batch": batch, "lo": lo, "hi": hi, "sizes": 1, "uplo": "lower", "trans": "n",
         "unit": False, "factor": "none", "alpha": 1.5}
    c.update(more)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one small system, the latency of a single call (the library's first configuration)
        _one("one_f64_64x64", "f64", 64, 64, alpha=1.5),
        # a small ragged variant call: U^H X = B with padded leading dimensions
        _one("one_c128_upper_37x19", "c128", 37, 19, uplo="upper", trans="c", pad=3, alpha=1.5),
        # many small complex systems at once (the headline configuration)
        _batch("batch_c128_8192", "c128", 8192, 8, 64),
        # LU-factor solves of many small real systems with row interchanges
        _batch("batch_f64_lu_4097", "f64", 4097, 8, 64, factor="lu"),
        # the same kind of batch in single precision complex
        _batch("batch_c64_8192", "c64", 8192, 8, 64),
        # the middle of the serving stream: one moderate system, few right-hand sides
        _one("one_f64_512x64", "f64", 512, 64),
        # one LU-factor solve of an odd size with interchanges, complex
        _one("one_c128_lu_777x129", "c128", 777, 129, factor="lu"),
        # the largest request of the serving stream, default FP64 products
        _one("one_f64_4096x512", "f64", 4096, 512),
        # large systems with FP64 products emulated on the tensor cores (real; complex, odd sizes)
        _one("emulated_f64_8192x4096", "f64", 8192, 4096, emulated=True),
        _one("emulated_c128_3001x1000", "c128", 3001, 1000, emulated=True, pad=1),
        # the reduced-precision configuration: FP32 result, and FP64 result by refinement
        _one("f32_bf16_8192x4096", "f32_bf16", 8192, 4096),
        _one("f64_ir_8192x4096", "f64_ir", 8192, 4096),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("small", "batch", "batch", "serve", "serve", "emulated", "reduced"))
    if kind == "small":  # m <= 64, any variant
        uplo, trans = rng.choice((("lower", "n"), ("lower", "n"), ("upper", "n"), ("lower", "t"), ("upper", "c")))
        return _one(None, rng.choice(("f64", "c128", "f32", "c64")), rng.randint(1, 64), _log(rng, 1, 512), uplo=uplo,
                    trans=trans, unit=rng.random() < 0.2, pad=rng.choice((0, 0, 1, 3)), alpha=1.5)
    if kind == "batch":
        factor = rng.choice(("none", "none", "lu", "chol"))
        uplo = "upper" if factor == "none" and rng.random() < 0.25 else "lower"
        lo = rng.randint(1, 32)
        return _batch(None, rng.choice(("f64", "c128", "f32", "c64")), _log(rng, 64, 8192), lo, rng.randint(lo, 64),
                      sizes=rng.randint(1, 1 << 20), factor=factor, uplo=uplo)
    if kind == "serve":  # one system of the serving stream's range
        dtype = rng.choice(("f64", "f64", "c128", "f32", "c64"))
        right = rng.random() < 0.15
        m, n = _log(rng, 65, 4096 if dtype != "c128" else 2500), _log(rng, 1, 512)
        if right:
            return _one(None, dtype, n, m, side="right", uplo=rng.choice(("lower", "upper")))
        return _one(None, dtype, m, n, factor=rng.choice(("none", "none", "none", "lu", "chol")),
                    pad=rng.choice((0, 0, 0, 1, 2)))
    if kind == "emulated":
        if rng.random() < 0.5:
            return _one(None, "f64", _log(rng, 400, 8192), _log(rng, 64, 4096), emulated=True,
                        factor=rng.choice(("none", "none", "chol")), pad=rng.choice((0, 0, 1)))
        return _one(None, "c128", _log(rng, 400, 4096), _log(rng, 64, 2048), emulated=True)
    return _one(None, rng.choice(("f32_bf16", "f32_bf16", "f64_ir")), _log(rng, 400, 8192), _log(rng, 16, 4096),
                unit=rng.random() < 0.2)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _uniform(gen, shape, cplx):
    """U(0, 1) entries; complex: real and imaginary parts alike."""
    if not cplx:
        return torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64)
    return torch.view_as_complex(torch.rand(tuple(shape) + (2,), generator=gen, device="cuda", dtype=torch.float64))


def _one_plus_i(cplx):
    return (1 + 1j) if cplx else 1.0


def _pivots(rs, m):
    """getrf-style interchanges: row k with row ipiv[k] >= k (1-based)."""
    return (np.arange(m) + np.floor(rs.random_sample(m) * (m - np.arange(m))) + 1).astype(np.int32)


def _permutation(ipiv):
    p = np.arange(len(ipiv))
    for k, q in enumerate(ipiv):
        p[k], p[q - 1] = p[q - 1], p[k]
    return p


def _one_data(case, seed):
    """The operands as torch matrices of the mathematical shape, in the case's element type."""
    _, tt = _DTYPES[case["dtype"]]
    cplx = case["dtype"] in _COMPLEX
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    na = case["m"] if case["side"] == "left" else case["n"]
    u = _uniform(gen, (na, na), cplx)
    d = torch.diagonal(u).clone() + 1.0 * _one_plus_i(cplx)
    A = u.mul_(2.0).sub_(_one_plus_i(cplx)).div_(na)
    torch.diagonal(A).copy_(d)
    if case["factor"] != "lu":
        A = torch.tril(A) if case["uplo"] == "lower" else torch.triu(A)
    B = _uniform(gen, (case["m"], case["n"]), cplx).mul_(2.0).sub_(_one_plus_i(cplx))
    piv = _pivots(np.random.RandomState(seed % (1 << 32)), case["m"]) if case["factor"] == "lu" else None
    return A.to(tt), B.to(tt), piv


def _column_major(M, pad):
    """(cols, ld) buffer holding M column by column, ld = rows + pad."""
    buf = torch.zeros((M.shape[1], M.shape[0] + pad), dtype=M.dtype, device=M.device)
    buf[:, : M.shape[0]] = M.T
    return buf


def _batch_sizes(case):
    rs = np.random.RandomState(case["sizes"])
    return (rs.randint(case["lo"], case["hi"] + 1, case["batch"]).astype(np.int64),
            rs.randint(case["lo"], case["hi"] + 1, case["batch"]).astype(np.int64))


def _batch_index(m, cols):
    """Instance, row and column of every element of consecutive m_i x cols_i column-major arrays."""
    dm = torch.from_numpy(m).cuda()
    inst = torch.repeat_interleave(torch.arange(len(m), device="cuda"), torch.from_numpy(m * cols).cuda())
    start = torch.from_numpy(np.concatenate([[0], np.cumsum(m * cols)[:-1]])).cuda()
    loc = torch.arange(inst.numel(), device="cuda") - start[inst]
    mi = dm[inst]
    return inst, loc % mi, loc // mi, mi, start


def _batch_data(case, seed):
    _, tt = _DTYPES[case["dtype"]]
    cplx = case["dtype"] in _COMPLEX
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    m, n = _batch_sizes(case)
    inst, row, col, mi, startA = _batch_index(m, m)
    u = _uniform(gen, (inst.numel(),), cplx)
    A = torch.where(row == col, u + 1.0 * _one_plus_i(cplx), (2.0 * u - _one_plus_i(cplx)) / mi)
    if case["factor"] != "lu":
        A = torch.where((row >= col) if case["uplo"] == "lower" else (row <= col), A, torch.zeros_like(A))
    startB = torch.from_numpy(np.concatenate([[0], np.cumsum(m * n)[:-1]])).cuda()
    B = _uniform(gen, (int((m * n).sum()),), cplx).mul_(2.0).sub_(_one_plus_i(cplx))
    rs = np.random.RandomState(seed % (1 << 32))
    piv = [_pivots(rs, int(k)) for k in m] if case["factor"] == "lu" else None
    return m, n, A.to(tt), startA, B.to(tt), startB, piv


def prepare(case, seed):
    code = _DTYPES[case["dtype"]][0]
    s = {"case": case, "code": code, "alpha": case["alpha"]}
    if case["op"] == "one":
        A, B, piv = _one_data(case, seed)
        s["A"] = _column_major(A, case["pad"])
        s["B"] = _column_major(B, case["pad"])
        s["X"] = torch.empty_like(s["B"])
        s["out"] = s["X"][:, : case["m"]]
        s["piv"] = torch.from_numpy(piv).cuda() if piv is not None else None
        s["opts"] = None
        if case["emulated"]:
            s["opts"] = H.Opts()
            s["opts"].fp64_products = 1
        return s
    m, n, A, startA, B, startB, piv = _batch_data(case, seed)
    s["A"], s["B"], s["X"] = A, B, torch.empty_like(B)
    s["out"] = s["X"]
    es = A.element_size()
    s["pA"] = startA * es + A.data_ptr()
    s["pX"] = startB * es + s["X"].data_ptr()
    s["m"] = torch.from_numpy(m.astype(np.int32)).cuda()
    s["n"] = torch.from_numpy(n.astype(np.int32)).cuda()
    s["max"] = case["hi"]
    if piv is not None:
        s["piv"] = torch.from_numpy(np.concatenate(piv)).cuda()
        start = np.concatenate([[0], np.cumsum(m)[:-1]])
        s["pP"] = torch.from_numpy(start * 4).cuda() + s["piv"].data_ptr()
    return s


def run(s):
    c, code, alpha = s["case"], s["code"], s["alpha"]
    st = H.stream_ptr()
    s["X"].copy_(s["B"])
    if c["op"] == "batch":
        m, n, a, x = s["m"].data_ptr(), s["n"].data_ptr(), s["pA"].data_ptr(), s["pX"].data_ptr()
        if c["factor"] == "lu":
            H.hsma_getrs_vbatched(code, c["batch"], m, n, alpha, a, m, s["pP"].data_ptr(), x, m, s["max"], s["max"],
                                  stream=st)
        elif c["factor"] == "chol":
            H.hsma_potrs_vbatched(code, c["batch"], m, n, alpha, a, m, x, m, s["max"], s["max"], stream=st)
        elif c["uplo"] == "lower":
            H.hsma_trsm_llnn_vbatched(code, int(c["unit"]), c["batch"], m, n, alpha, a, m, x, m, s["max"], s["max"],
                                      stream=st)
        else:
            H.hsma_trsm_vbatched(code, H.LEFT, H.UPPER, _TRANS[c["trans"]], int(c["unit"]), c["batch"], m, n, alpha, a,
                                 m, x, m, s["max"], s["max"], stream=st)
        return s["out"]
    a, lda, x, ldb = s["A"].data_ptr(), s["A"].shape[1], s["X"].data_ptr(), s["X"].shape[1]
    if c["factor"] == "lu":
        H.hsma_getrs(code, c["m"], c["n"], alpha, a, lda, s["piv"].data_ptr(), x, ldb, st, opts=s["opts"])
    elif c["factor"] == "chol":
        H.hsma_potrs(code, c["m"], c["n"], alpha, a, lda, x, ldb, st, opts=s["opts"])
    elif c["side"] == "left" and c["uplo"] == "lower" and c["trans"] == "n":
        H.hsma_trsm_llnn_ex(code, int(c["unit"]), c["m"], c["n"], alpha, a, lda, x, ldb, st, opts=s["opts"])
    else:
        H.hsma_trsm(code, H.LEFT if c["side"] == "left" else H.RIGHT, H.LOWER if c["uplo"] == "lower" else H.UPPER,
                    _TRANS[c["trans"]], int(c["unit"]), c["m"], c["n"], alpha, a, lda, x, ldb, st, opts=s["opts"])
    return s["out"]


# ---------------------------------------------------------------------------
# work, tolerance and the 64-bit results
# ---------------------------------------------------------------------------
def work(case):
    tt = _DTYPES[case["dtype"]][1]
    es = torch.empty((), dtype=tt).element_size()
    mul = (4 if case["dtype"] in _COMPLEX else 1) * (2 if case["factor"] != "none" else 1)
    if case["op"] == "one":
        m, n = np.array([case["m"]], float), np.array([case["n"]], float)
    else:
        m, n = (v.astype(float) for v in _batch_sizes(case))
    na, nb = (m, n) if case.get("side", "left") == "left" else (n, m)
    tri = na * na if case["factor"] == "lu" else na * (na + 1) / 2
    return {"bytes": float(((tri + 2 * m * n) * es).sum()), "flops": float((mul * na * na * nb).sum())}


def tolerance(case):
    """About four times the measured error against exact()."""
    one_blocked = case["op"] == "one" and (case["m"] if case["side"] == "left" else case["n"]) > 64
    if case["dtype"] == "f32_bf16" or (case["dtype"] == "f32" and one_blocked):
        return {"rel": 6e-6}  # BF16 pairs of a two-way split, FP32 sums: 1.4e-6 measured
    if case["dtype"] in ("f32", "c64"):
        return {"rel": 1e-6}  # 2.3e-7 measured
    if case["dtype"] == "f64_ir":
        return {"rel": 2e-14}  # stops at a residual ratio of 1e-15: 5.5e-15 measured
    return {"rel": 4e-15}  # 1e-15 at most measured


def _tri_solve(M, B, upper=False, unit=False):
    return torch.linalg.solve_triangular(M, B, upper=upper, unitriangular=unit)


def exact(case, seed):
    w = torch.complex128 if case["dtype"] in _COMPLEX else torch.float64
    if case["op"] == "one":
        A, B, piv = _one_data(case, seed)
        A, B = A.to(w), B.to(w) * case["alpha"]
        if case["factor"] == "lu":
            Y = _tri_solve(A, B[torch.from_numpy(_permutation(piv)).cuda()], unit=True)
            X = _tri_solve(A, Y, upper=True)
        elif case["factor"] == "chol":
            X = _tri_solve(A.mH, _tri_solve(A, B), upper=True)
        else:
            up = case["uplo"] == "upper"
            if case["trans"] != "n":
                A, up = (A.mH if case["trans"] == "c" else A.mT), not up
            if case["side"] == "left":
                X = _tri_solve(A, B, upper=up, unit=case["unit"])
            else:
                X = _tri_solve(A.mT, B.mT, upper=not up, unit=case["unit"]).mT
        return X.T.contiguous()
    m, n, A, _, B, _, piv = _batch_data(case, seed)
    ia, ra, ca, _, _ = _batch_index(m, m)
    ib, rb, cb, _, _ = _batch_index(m, n)
    P = torch.eye(64, dtype=w, device="cuda").repeat(case["batch"], 1, 1)
    P[ia, ra, ca] = A.to(w)
    Q = torch.zeros((case["batch"], 64, 64), dtype=w, device="cuda")
    if piv is not None:
        where = np.tile(np.arange(64), (case["batch"], 1))
        for i, p in enumerate(piv):
            q = np.empty(len(p), np.int64)
            q[_permutation(p)] = np.arange(len(p))
            where[i, : len(p)] = q  # row r of B goes to row where[r] of P^T B
        Q[ib, torch.from_numpy(where).cuda()[ib, rb], cb] = B.to(w) * case["alpha"]
    else:
        Q[ib, rb, cb] = B.to(w) * case["alpha"]
    if case["factor"] == "lu":
        X = _tri_solve(torch.triu(P), _tri_solve(torch.tril(P, -1) + torch.eye(64, dtype=w, device="cuda"), Q,
                                                 unit=True), upper=True)
    elif case["factor"] == "chol":
        X = _tri_solve(P.mH, _tri_solve(P, Q), upper=True)
    else:
        up = case["uplo"] == "upper"
        if case["trans"] != "n":
            P, up = (P.mH if case["trans"] == "c" else P.mT), not up
        X = _tri_solve(P, Q, upper=up, unit=case["unit"])
    return X[ib, rb, cb]
