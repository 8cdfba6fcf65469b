"""Blocked large-case path (Section 4.3) against the oracle, through the C ABI."""
import numpy as np
import pytest

import oracle
from paper_2608_25469_gb300 import inputs as I
from tests import gpu_util as U

pytestmark = pytest.mark.gpu

TOL = 1e-12


@pytest.fixture(scope="module")
def H():
    import torch
    assert torch.cuda.is_available()
    return U.lib()


def _dt(code):
    return np.float64 if code == I.R64 else np.complex128


def _run(H, code, A, B, alpha, nb, unit=False, **cfg):
    import torch
    dA, dB = H.to_device(A), H.to_device(B)
    opts = H.Opts()
    opts.path = H.PATH_BLOCKED
    opts.nb = nb
    for k, v in cfg.items():
        setattr(opts, k, v)
    info = H.Info()
    H.hsma_trsm_llnn_ex(code, int(unit), A.shape[1], B.shape[1], alpha, dA.data_ptr(), A.shape[0], dB.data_ptr(),
                        B.shape[0], H.stream_ptr(), opts=opts, info=info)
    torch.cuda.synchronize()
    assert info.plan.path == H.PATH_BLOCKED and info.plan.nb == nb
    return H.from_device(dB)


CASES = [(65, 7, 32), (127, 64, 64), (128, 1, 64), (129, 33, 128), (300, 200, 128), (1000, 100, 256),
         (700, 50, 512), (2048, 300, 256), (96, 97, 32), (513, 5, 512)]


@pytest.mark.parametrize("code", [I.R64, I.C128])
@pytest.mark.parametrize("pad", [0, 3])
@pytest.mark.parametrize("m,n,nb", CASES)
def test_blocked_parity(H, code, m, n, nb, pad):
    """Ragged sizes, every N_B, leading dimensions with (pad 0, even m) and without TMA (odd fp64 ld)."""
    alpha = 1.0 if code == I.R64 else 1.5 - 0.5j
    seed = m * 7 + n
    A0, B0 = I.gen_A(seed, m, code), I.gen_B(seed, m, n, code)
    A = I.embed(A0, m + pad, fill=np.nan)
    A[:m][np.triu_indices(m, 1)] = np.nan  # the strict upper triangle is never read
    B = I.embed(B0, m + pad, fill=np.nan)
    X = _run(H, code, A, B, alpha, nb)
    assert np.all(np.isnan(X[m:])), "padding rows written"
    ref = oracle.solve(A0, B0, alpha)
    err = oracle.forward_error(X[:m], ref)
    assert err <= TOL, err
    assert H.hsma_device_status() == 0


@pytest.mark.parametrize("code", [I.R64, I.C128])
def test_blocked_unit_diagonal_and_alpha(H, code):
    m, n, nb = 333, 41, 128
    A0, B0 = I.gen_A(2, m, code), I.gen_B(2, m, n, code)
    A = np.array(A0, order="F")
    np.fill_diagonal(A, np.nan)
    alpha = -0.75 if code == I.R64 else 0.25 + 1j
    X = _run(H, code, A, B0, alpha, nb, unit=True)
    A1 = np.array(A0, order="F")
    np.fill_diagonal(A1, 1.0)
    assert oracle.forward_error(X, oracle.solve(A1, B0, alpha)) <= TOL
    # alpha = 0 on the blocked path: B := 0, A not read
    Anan = np.full((m, m), np.nan, dtype=_dt(code), order="F")
    X0 = _run(H, code, Anan, B0, 0.0, nb)
    assert np.all(X0 == 0)


@pytest.mark.parametrize("code", [I.R64, I.C128])
def test_planner_default_matches_oracle(H, code):
    """hsma_trsm_llnn with the planner's own N_B (the table lookup of Section 4.3.2)."""
    import torch
    m, n = 777, 129
    A, B = I.gen_A(4, m, code), I.gen_B(4, m, n, code)
    alpha = 1.5 if code == I.R64 else 1.5 - 0.5j
    dA, dB = H.to_device(A), H.to_device(B)
    H.hsma_trsm_llnn(code, 0, m, n, alpha, dA.data_ptr(), m, dB.data_ptr(), m, H.stream_ptr())
    torch.cuda.synchronize()
    X = H.from_device(dB)
    assert oracle.forward_error(X, oracle.solve(A, B, alpha)) <= TOL
    assert oracle.backward_error(A, B, X, alpha) <= 1e-14


@pytest.mark.parametrize("code", [I.R64, I.C128])
@pytest.mark.parametrize("m,nb", [(33, 64), (4100, 512), (2050, 256), (2050, 64), (1055, 128)])
def test_inverse_levels_parity(H, code, m, nb):
    """Diagonal inverses whose last block has a part of one base block of 32 rows, one row more, or
    one row alone, and blocks of two to sixteen base blocks."""
    n = 3
    A, B = I.gen_A(m, m, code), I.gen_B(m, m, n, code)
    A[np.triu_indices(m, 1)] = np.nan
    X = _run(H, code, A, B, 1.0, nb)
    ref = oracle.solve(I.gen_A(m, m, code), B, 1.0)
    assert oracle.forward_error(X, ref) <= TOL


def _substituted(T, B, nb):
    """Blocked solve in numpy whose diagonal blocks are inverted by row-by-row substitution."""
    X = np.array(B)
    for r in range(0, len(T), nb):
        D = T[r:r + nb, r:r + nb]
        d = 1.0 / np.diag(D)
        S, inv = D * d[:, None], np.diag(d)
        for k in range(len(D) - 1):
            inv[k + 1:, :k + 1] -= np.outer(S[k + 1:, k], inv[k, :k + 1])
        X[r:r + nb] = inv @ X[r:r + nb]
        X[r + nb:] -= T[r + nb:, r:r + nb] @ X[r:r + nb]
    return X


@pytest.mark.parametrize("code", [I.R64, I.C128])
@pytest.mark.parametrize("factor", ["L", "UT"])
@pytest.mark.parametrize("m,nb", [(512, 512), (700, 256)])
def test_inverse_accuracy_on_lu_factors(H, code, factor, m, nb):
    """LU factors of random matrices, whose blocks are ill conditioned as the seeded recipe's are not:
    the residual stays at that of row-by-row substitution.  Six matrices, the mean of the ratios: two
    orders of the same sums differ by up to 10% in it, inverses joined by doubling give 1.5 to 2.7."""
    la = pytest.importorskip("scipy.linalg")
    ratios = []
    for seed in range(6):
        rng = np.random.default_rng(seed)
        G = rng.standard_normal((m, m)) + (1j * rng.standard_normal((m, m)) if code == I.C128 else 0.0)
        lu = la.lu_factor(G)[0]
        T = np.asfortranarray(np.tril(lu, -1) + np.eye(m) if factor == "L" else np.triu(lu).T)
        B = I.gen_B(seed, m, 8, code)
        got = oracle.backward_error(T, B, _run(H, code, T, B, 1.0, nb), 1.0)
        ratios.append(got / oracle.backward_error(T, B, _substituted(T, B, nb), 1.0))
    assert np.exp(np.mean(np.log(ratios))) <= 1.25, ratios


def test_solve_products_round_once_at_the_size_of_the_result(H):
    """m = 512 with two blocks, left-looking, on the seeded recipe, where the diagonal dominates: an
    entry sees the rounding of 1/a_ii and of the solve product, in the second block that of the update
    too, each at most u = 2^-53 relative and of root mean square at most u / sqrt(3).  The mean over
    both blocks, sqrt(2.5 / 3) u, bounds the error from the exact solution; partial sums added to a
    partial sum that holds the diagonal's term give 1.4 times that bound."""
    m, n, nb = 512, 24, 256
    A, B = I.gen_A(21, m, I.R64), I.gen_B(21, m, n, I.R64)
    X = _run(H, I.R64, A, B, 1.0, nb, looking=2).astype(np.longdouble)
    exact = B.astype(np.longdouble)
    for k in range(m):
        exact[k] /= A[k, k]
        exact[k + 1:] -= np.outer(A[k + 1:, k].astype(np.longdouble), exact[k])
    err = float(np.sqrt(((X - exact) ** 2).sum() / (exact ** 2).sum()))
    assert err <= np.sqrt(2.5 / 3.0) * 2.0 ** -53, err


@pytest.mark.parametrize("code", [I.R64, I.C128])
@pytest.mark.parametrize("n", [3, 600])
@pytest.mark.parametrize("what,row", [("nan_b", 300), ("inf_b", 511), ("zero_diagonal", 389)])
def test_blocked_non_finite_propagates(H, code, n, what, row):
    """An infinity or NaN of B reaches its column from its row on, and at most 7 rows above (the 8 x 8
    part of the inverse that holds its row); a zero on the diagonal every column from its row on."""
    m, nb, col = 640, 256, 2
    A0, B0 = I.gen_A(5, m, code), I.gen_B(5, m, n, code)
    A, B = A0.copy(order="F"), B0.copy(order="F")
    if what == "zero_diagonal":
        A[row, row] = 0
    else:
        B[row, col] = np.nan if what == "nan_b" else np.inf
    X = _run(H, code, A, B, 1.0, nb)
    reach = slice(None) if what == "zero_diagonal" else col
    assert not np.any(np.isfinite(X[row:, reach]))
    bad = np.zeros((m, n), bool)
    bad[row if what == "zero_diagonal" else row // 8 * 8:, reach] = True
    ref = oracle.solve(A0, B0, 1.0)
    assert np.linalg.norm((X - ref)[~bad]) <= TOL * np.linalg.norm(ref)


SMALL_TILE_CASES = [(66, 1, 64, 1), (129, 8, 64, 1), (300, 9, 128, 2), (520, 31, 256, 1), (1000, 33, 128, 2),
                    (1031, 200, 512, 1), (1500, 257, 128, 2), (1031, 517, 128, 1), (2051, 515, 128, 1)]


def _small_tiles(code, m, n, nb, look, sms):
    """The tile (in units of 8 x 8) and warps per CTA of every product of one blocked solve."""
    cdiv = lambda a, b: -(-a // b)
    products = []
    for r0 in range(0, m, nb):
        sr = min(nb, m - r0)
        products.append((sr, sr))
        if look == 2 and r0 > 0:
            products.append((sr, r0))
        elif look == 1 and r0 + sr < m:
            products.append((m - r0 - sr, sr))
    shapes = set()
    for M, K in products:
        tiles = lambda w: cdiv(cdiv(M, 8), w) * cdiv(cdiv(n, 8), w)
        if code == I.R64 and cdiv(n, 8) >= 4 and tiles(4) >= 4 * sms:
            shapes.add((4, 4))
        elif cdiv(n, 8) >= 2 and tiles(2) >= 4 * sms:
            shapes.add((2, 4))
        else:
            shapes.add((1, 4 if tiles(1) >= 2 * sms or K <= 64 else 16))
    return shapes


@pytest.mark.parametrize("code", [I.R64, I.C128])
@pytest.mark.parametrize("m,n,nb,look", SMALL_TILE_CASES)
def test_small_tile_products_parity(H, code, m, n, nb, look):
    """Every small-tile shape (by the number of tiles) at ragged sizes, odd leading dimensions,
    alpha, both update directions, NaN in what is never read."""
    alpha = -0.5 if code == I.R64 else 0.5 + 2j
    A0, B0 = I.gen_A(m, m, code), I.gen_B(m, m, n, code)
    A = I.embed(A0, m + 1, fill=np.nan)
    A[:m][np.triu_indices(m, 1)] = np.nan
    B = I.embed(B0, m + 3, fill=np.nan)
    assert H.hsma_plan(code, m, n).tile == 0
    X = _run(H, code, A, B, alpha, nb, looking=look)
    assert np.all(np.isnan(X[m:]))
    assert oracle.forward_error(X[:m], oracle.solve(A0, B0, alpha)) <= TOL


@pytest.mark.parametrize("code", [I.R64, I.C128])
def test_small_tile_cases_cover_every_shape(H, code):
    """The cases above select every compiled shape on this device."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    got = set().union(*(_small_tiles(code, *c, sms) for c in SMALL_TILE_CASES))
    assert got == {(2, 4), (1, 4), (1, 16)} | ({(4, 4)} if code == I.R64 else set())


CFG_CASES = [(65, 7, 32), (300, 200, 128), (700, 50, 512), (1000, 9, 64), (513, 130, 256)]


@pytest.mark.parametrize("code", [I.R64, I.C128])
@pytest.mark.parametrize("looking", [1, 2], ids=["right", "left"])
@pytest.mark.parametrize("tile", [1, 2, 3], ids=["64x64", "128x16", "128x8"])
@pytest.mark.parametrize("split_k", [1, 2], ids=["split", "nosplit"])
@pytest.mark.parametrize("m,n,nb", CFG_CASES)
def test_blocked_configurations_parity(H, code, looking, tile, split_k, m, n, nb):
    """Every configuration the autotuner may choose (update direction, product tile, split
    K) at ragged sizes, with NaN in the never-read upper triangle and padding rows."""
    import torch
    alpha = 1.25 if code == I.R64 else 0.5 - 1.5j
    seed = m + 3 * n + nb
    A0, B0 = I.gen_A(seed, m, code), I.gen_B(seed, m, n, code)
    A = I.embed(A0, m + 2, fill=np.nan)
    A[:m][np.triu_indices(m, 1)] = np.nan
    B = I.embed(B0, m + 2, fill=np.nan)
    X = _run(H, code, A, B, alpha, nb, looking=looking, tile=tile, split_k=split_k)
    assert np.all(np.isnan(X[m:]))
    assert oracle.forward_error(X[:m], oracle.solve(A0, B0, alpha)) <= TOL
    assert H.hsma_device_status() == 0


@pytest.mark.parametrize("code", [I.R64, I.C128])
def test_left_looking_unit_diagonal(H, code):
    m, n, nb = 450, 33, 64
    A0, B0 = I.gen_A(6, m, code), I.gen_B(6, m, n, code)
    A = np.array(A0, order="F")
    np.fill_diagonal(A, np.nan)
    X = _run(H, code, A, B0, -2.0, nb, unit=True, looking=2)
    A1 = np.array(A0, order="F")
    np.fill_diagonal(A1, 1.0)
    assert oracle.forward_error(X, oracle.solve(A1, B0, -2.0)) <= TOL
