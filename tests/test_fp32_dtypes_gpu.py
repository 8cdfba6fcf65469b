"""Native FP32 and complex64 dtypes (HSMA_R32, HSMA_C64): the small direct solve
and the varlen batch compute in FP32; larger m runs the FP32-result blocked
solve (R32) or a complex128 emulated-FP64 solve rounded back (C64).

Reference: the FP64 oracle applied to the same FP32 inputs (widened exactly).
Tolerance 2e-5 relative Frobenius forward error: FP32 substitution errs by at
most about m u_32 cond(L) (m <= 64, u_32 = 6e-8, cond <= 2 for these
generators: < 8e-6), and the blocked FP32-result path is held to the same
bound as HSMA_R32_BF16."""
import numpy as np
import pytest

import oracle
from paper_2608_25469_gb300 import inputs as I
from tests import gpu_util as U

pytestmark = pytest.mark.gpu

TOL32 = 2e-5


@pytest.fixture(scope="module")
def H():
    import torch
    assert torch.cuda.is_available()
    return U.lib()


def _f32(code64, X):
    return np.asfortranarray(X.astype(np.float32 if code64 == I.R64 else np.complex64))


def _solve(H, code, A, B, alpha, unit=False, opts=None):
    import torch
    dA, dB = H.to_device(A), H.to_device(B)
    m, n = B.shape
    H.hsma_trsm_llnn_ex(code, int(unit), A.shape[1], n, alpha, dA.data_ptr(), A.shape[0], dB.data_ptr(), m,
                        H.stream_ptr(), opts=opts)
    torch.cuda.synchronize()
    assert H.hsma_device_status() == 0
    return H.from_device(dB)


def _ref(A32, B32, alpha, unit=False):
    wide = np.complex128 if np.iscomplexobj(A32) else np.float64
    return oracle.solve(np.asfortranarray(A32.astype(wide)), np.asfortranarray(B32.astype(wide)), alpha, unit=unit)


@pytest.mark.parametrize("code64,code", [(I.R64, 4), (I.C128, 5)])
@pytest.mark.parametrize("n", [1, 5, 33, 64])
def test_small_fp32_every_m(H, code64, code, n):
    alpha = 1.5 if code64 == I.R64 else 1.5 - 0.5j
    for m in list(range(1, 65, 3)) + [64]:
        A32, B32 = _f32(code64, I.gen_A(m, m, code64)), _f32(code64, I.gen_B(m, m, n, code64))
        X = _solve(H, code, A32, B32, alpha)
        assert X.dtype == A32.dtype
        err = oracle.forward_error(X.astype(np.complex128 if code == 5 else np.float64), _ref(A32, B32, alpha))
        assert err <= TOL32, (m, err)


@pytest.mark.parametrize("code64,code", [(I.R64, 4), (I.C128, 5)])
def test_small_fp32_unit_diagonal_not_read(H, code64, code):
    m, n = 40, 17
    A32, B32 = _f32(code64, I.gen_A(3, m, code64)), _f32(code64, I.gen_B(3, m, n, code64))
    A = A32.copy(order="F")
    A[np.diag_indices(m)] = np.nan
    X = _solve(H, code, A, B32, 1.0, unit=True)
    assert np.all(np.isfinite(X))
    assert oracle.forward_error(X.astype(np.complex128 if code == 5 else np.float64),
                                _ref(A32, B32, 1.0, unit=True)) <= TOL32


@pytest.mark.parametrize("code64,code", [(I.R64, 4), (I.C128, 5)])
def test_batched_fp32_parity_and_alone(H, code64, code):
    import torch
    alpha = 1.5 if code64 == I.R64 else 1.5 - 0.5j
    ms, ns = I.batched_sizes(21, 600)
    As = [_f32(code64, I.gen_A(21, int(m), code64, inst=b)) for b, m in enumerate(ms)]
    Bs = [_f32(code64, I.gen_B(21, int(m), int(n), code64, inst=b)) for b, (m, n) in enumerate(zip(ms, ns))]

    def run(As_, Bs_):
        bt = U.Batch(As_, Bs_)
        H.hsma_trsm_llnn_vbatched(code, 0, bt.batch, bt.args()[0], bt.args()[1], alpha, bt.args()[2],
                                  bt.args()[3], bt.args()[4], bt.args()[5], max_m=64, max_n=0,
                                  d_status=bt.d_status.data_ptr(), stream=H.stream_ptr())
        torch.cuda.synchronize()
        assert bt.status() == 0
        return bt.results()
    mix = run(As, Bs)
    wide = np.complex128 if code == 5 else np.float64
    for b in range(len(As)):
        assert oracle.forward_error(mix[b].astype(wide), _ref(As[b], Bs[b], alpha)) <= TOL32, b
    for b in range(0, len(As), 37):
        assert np.array_equal(run([As[b]], [Bs[b]])[0], mix[b]), b


@pytest.mark.parametrize("code64,code", [(I.R64, 4), (I.C128, 5)])
@pytest.mark.parametrize("m,n", [(65, 7), (300, 100), (1000, 64)])
def test_blocked_fp32_dtypes(H, code64, code, m, n):
    alpha = 1.0 if code64 == I.R64 else 1.5 - 0.5j
    A32, B32 = _f32(code64, I.gen_A(m + 1, m, code64)), _f32(code64, I.gen_B(m + 1, m, n, code64))
    A = A32.copy(order="F")
    A[np.triu_indices(m, 1)] = np.nan  # only the lower triangle is read
    X = _solve(H, code, A, B32, alpha)
    wide = np.complex128 if code == 5 else np.float64
    assert oracle.forward_error(X.astype(wide), _ref(A32, B32, alpha)) <= TOL32


def test_host_batch_complex64_equals_device_batch(H):
    import torch
    alpha = 0.5 + 2.0j
    ms, ns = I.batched_sizes(4, 300)
    As = [_f32(I.C128, I.gen_A(4, int(m), I.C128, inst=b)) for b, m in enumerate(ms)]
    Bs = [_f32(I.C128, I.gen_B(4, int(m), int(n), I.C128, inst=b)) for b, (m, n) in enumerate(zip(ms, ns))]
    bt = U.Batch(As, Bs)
    H.hsma_trsm_llnn_vbatched(5, 0, bt.batch, bt.args()[0], bt.args()[1], alpha, bt.args()[2], bt.args()[3],
                              bt.args()[4], bt.args()[5], max_m=64, stream=H.stream_ptr())
    torch.cuda.synchronize()
    dev = bt.results()
    m32, n32 = ms.astype(np.int32), ns.astype(np.int32)
    offA = np.concatenate([[0], np.cumsum(ms.astype(np.int64) ** 2)[:-1]]).astype(np.int64)
    offB = np.concatenate([[0], np.cumsum(ms.astype(np.int64) * ns)[:-1]]).astype(np.int64)
    hA = np.concatenate([a.ravel(order="F") for a in As])
    hB = np.concatenate([b.ravel(order="F") for b in Bs])
    hX = np.empty_like(hB)
    H.hsma_trsm_llnn_vbatched_host(5, 0, len(As), m32, n32, alpha, hA.ctypes.data, offA, hB.ctypes.data, offB,
                                   hX.ctypes.data, stream=H.stream_ptr())
    torch.cuda.synchronize()
    for b in range(len(As)):
        got = hX[offB[b]:offB[b] + ms[b] * ns[b]].reshape((ms[b], ns[b]), order="F")
        assert np.array_equal(got, dev[b]), b


EDGES = [(1, 1), (7, 15), (8, 16), (9, 17), (15, 64), (16, 65), (17, 3), (31, 33), (32, 130), (33, 16), (63, 5), (64, 64)]


@pytest.mark.parametrize("code64,code", [(I.R64, 4), (I.C128, 5), (I.R64, 0)], ids=["f32", "c64", "f64"])
@pytest.mark.parametrize("kind", ["nn", "nn_unit", "un", "lt", "uc", "lc_unit", "lu", "chol"])
def test_batched_block_edges(H, code64, code, kind):
    """The batch kernel at the edges of its 4- and 8-row blocks, 16-column tiles and 64-column rounds,
    in every index map and both factor solves, with padded leading dimensions and NaN in whatever is
    not referenced.  Tolerance: the substitution bound of the type, twice for the factor solves."""
    import torch
    tol = TOL32 if code else 1e-13
    as_type = (lambda X: _f32(code64, X)) if code else np.asfortranarray
    uplo = 1 if kind[0] == "u" else 0
    trans = {"t": 1, "c": 2}.get(kind[1], 0) if kind not in ("lu", "chol") else 0
    unit = kind.endswith("unit")
    alpha = 1.5 if code64 == I.R64 else 1.5 - 0.5j
    As, Bs, raw, pivs = [], [], [], []
    rng = np.random.default_rng(5)
    for b, (m, n) in enumerate(EDGES):
        A = I.gen_LU(3, m, code64, inst=b) if kind == "lu" else I.gen_A(3, m, code64, inst=b)
        A = np.asfortranarray(A.T) if uplo else A
        A32, B32 = as_type(A), as_type(I.gen_B(3, m, n, code64, inst=b))
        raw.append((A32, B32))
        E = np.array(A32, order="F")
        if kind != "lu":
            E[np.tril_indices(m, -1) if uplo else np.triu_indices(m, 1)] = np.nan
        if unit:
            np.fill_diagonal(E, np.nan)
        As.append(I.embed(E, m + b % 3))
        Bs.append(I.embed(B32, m + b % 3))
        pivs.append((np.arange(m) + np.floor(rng.random(m) * (m - np.arange(m))) + 1).astype(np.int32))
    bt = U.Batch(As, Bs)
    bt.d_ldb = bt.d_lda
    a = bt.args()
    st, ds = H.stream_ptr(), bt.d_status.data_ptr()
    if kind == "lu":
        flat = torch.from_numpy(np.concatenate(pivs)).cuda()
        off = np.concatenate([[0], np.cumsum([len(p) for p in pivs])[:-1]]).astype(np.int64)
        ptr = torch.from_numpy(flat.data_ptr() + 4 * off).cuda()
        H.hsma_getrs_vbatched(code, bt.batch, a[0], a[1], alpha, a[2], a[3], ptr.data_ptr(), a[4], a[5], 64, 0, ds, st)
    elif kind == "chol":
        H.hsma_potrs_vbatched(code, bt.batch, a[0], a[1], alpha, a[2], a[3], a[4], a[5], 64, 0, ds, st)
    else:
        H.hsma_trsm_vbatched(code, 0, uplo, trans, int(unit), bt.batch, a[0], a[1], alpha, a[2], a[3], a[4], a[5], 64,
                             0, ds, st)
    torch.cuda.synchronize()
    assert bt.status() == 0
    wide = np.complex128 if code64 == I.C128 else np.float64
    for b, X in enumerate(bt.results()):
        A32, B32 = (np.asfortranarray(v.astype(wide)) for v in raw[b])
        m = A32.shape[0]
        if kind == "lu":
            ref = oracle.getrs(A32, pivs[b], B32, alpha)
        elif kind == "chol":
            ref = oracle.potrs(A32, B32, alpha)
        else:
            ref = oracle.solve_general(A32, B32, alpha, 0, uplo, trans, unit)
        assert np.all(np.isnan(X[m:])), EDGES[b]
        assert oracle.forward_error(X[:m].astype(wide), ref) <= tol * (2 if kind in ("lu", "chol") else 1), EDGES[b]


@pytest.mark.parametrize("code64,code", [(I.R64, 4), (I.C128, 5), (I.R64, 0)], ids=["f32", "c64", "f64"])
@pytest.mark.parametrize("uplo", [0, 1], ids=["lower", "upper"])
@pytest.mark.parametrize("what", ["nan_b", "inf_b", "zero_diagonal"])
def test_batched_non_finite_propagates(H, code64, code, uplo, what):
    """An infinity or NaN of B reaches its column from its row on (in the order of the substitution), a
    zero on the diagonal every column; nothing else changes by a bit, the other instances neither."""
    import torch
    sizes = [(64, 40), (13, 5), (37, 17)]
    as_type = (lambda X: _f32(code64, X)) if code else np.asfortranarray
    out = []
    for planted in (False, True):
        As, Bs = [], []
        for b, (m, n) in enumerate(sizes):
            A = I.gen_A(3, m, code64, inst=b)
            As.append(as_type(np.asfortranarray(A.T) if uplo else A).copy(order="F"))
            Bs.append(as_type(I.gen_B(3, m, n, code64, inst=b)).copy(order="F"))
        if planted and what == "zero_diagonal":
            As[0][21, 21] = 0
        elif planted:
            Bs[0][21, 33] = np.nan if what == "nan_b" else np.inf
        bt = U.Batch(As, Bs)
        a = bt.args()
        H.hsma_trsm_vbatched(code, 0, uplo, 0, 0, bt.batch, a[0], a[1], 1.5, a[2], a[3], a[4], a[5], 64, 0,
                             bt.d_status.data_ptr(), H.stream_ptr())
        torch.cuda.synchronize()
        assert bt.status() == 0
        out.append(bt.results())
    bad = np.zeros(sizes[0], bool)
    bad[slice(None, 22) if uplo else slice(21, None), slice(None) if what == "zero_diagonal" else 33] = True
    clean, got = out
    assert not np.any(np.isfinite(got[0][bad]))
    assert np.array_equal(got[0][~bad], clean[0][~bad])
    assert all(np.array_equal(p, q) for p, q in zip(got[1:], clean[1:]))
