"""k_band: the product step where rows span consecutive columns, bitwise
against the oracle (and with its Algorithm 1 records): sizes around the tile's
four rows and 64 columns, both tile heights, shared and single-warp tiles,
ranges of A longer than one staged chunk, rows that lie apart or fall back to
the accumulator, entries that come out as exact zeros, and filtered rows that
keep holes."""
import numpy as np
import pytest

import synthetic as syn
from gpu_helpers import assert_csr_bitwise, check_same, dev, ocsr
from oracle import CSR, alg1, axpy, matmul_add, psscf

pytestmark = pytest.mark.gpu

psf = pytest.importorskip("paper_2208_05683_gb300")


def band(n, lo, hi, seed, spread=0):
    """Entries (i, i + d), lo <= d <= hi, U[-1, 1], magnitudes over 10^+-spread."""
    rng = np.random.default_rng(seed)
    rows = [[i + d for d in range(lo, hi + 1) if 0 <= i + d < n] for i in range(n)]
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
    col = np.array([c for r in rows for c in r], np.int32)
    val = rng.uniform(-1.0, 1.0, len(col)) * 10.0 ** rng.uniform(-spread, spread, len(col))
    return CSR(n, rp, col, val)


def scattered(n, width, seed):
    """Row i: `width` consecutive columns anywhere (rows apart from each other)."""
    rng = np.random.default_rng(seed)
    start = rng.integers(0, max(1, n - width + 1), n)
    col = (start[:, None] + np.arange(min(width, n))).reshape(-1).astype(np.int32)
    return CSR(n, (np.arange(n + 1) * min(width, n)).astype(np.int32), col, rng.uniform(-1.0, 1.0, len(col)))


def check(A, B, addends=(), threshold=0.0):
    X = None
    for alpha, M in addends:
        X = axpy(alpha, M, X, A.n)
    C = matmul_add(A, B, X)
    got = psf.product_filter(dev(A), dev(B), [(a, None if M is None else dev(M)) for a, M in addends], threshold)
    st = got.steps[0]
    fma = int(np.diff(B.rowptr)[A.col].sum()) + sum(A.n if M is None else M.nnz for _, M in addends)
    assert (st["nnz_pre"], st["fma"]) == (C.nnz, fma)
    if threshold > 0.0:
        ref = alg1(C, threshold / 1.1, 0.1)
        assert (st["nnz_post"], st["eps_f"], st["iters"], st["dropped"]) == (ref.kept.nnz, ref.eps_f, ref.iters, ref.c)
        C = ref.kept
    assert_csr_bitwise(got.csr, C)


PLAIN = [(1, 0, 0), (2, 1, 1), (3, 0, 2), (31, 2, 3), (64, 1, 31), (65, 5, 32), (333, 3, 14), (1001, 15, 40),
         (700, 90, 90), (2600, 200, 170)]


@pytest.mark.parametrize("n,wa,wb", PLAIN)
@pytest.mark.parametrize("threshold", [0.0, 1e-2, 3.0])
def test_products_bitwise(n, wa, wb, threshold):
    A, B, M = band(n, -wa, wa, 1), band(n, -wb, wb + 1, 2, 3), band(n, -2, wa, 3)
    check(A, B, [(0.5, M), (-2.0, None), (0.25, B)], threshold)


@pytest.mark.parametrize("n", [34050, 40003])  # tiles of four rows
def test_tall_tiles_bitwise(n):
    check(band(n, -3, 2, 4), band(n, -20, 11, 5, 2), [(1.0, None), (0.5, band(n, 0, 1, 6))], 1e-3)


def test_rows_apart_and_one_sided_bitwise():
    for n, w in [(500, 1), (500, 7), (900, 40)]:
        check(scattered(n, w, n), scattered(n, 3, w), [(0.5, None)], 1e-3)
        check(band(n, 4, 9, 1), scattered(n, w, 2))
        check(scattered(n, 1, 3), band(n, -w, w, 4), (), 1e-2)


def test_empty_rows_and_exact_zeros_bitwise():
    n = 300
    Z = band(n, -4, 4, 7)
    rp, col, val = Z.rowptr, Z.col, Z.val
    keep = np.ones(len(col), bool)
    for r in range(0, n, 7):  # empty rows
        keep[rp[r]:rp[r + 1]] = False
    lens = [int(keep[rp[r]:rp[r + 1]].sum()) for r in range(n)]
    A = CSR(n, np.concatenate([[0], np.cumsum(lens)]).astype(np.int32), col[keep], val[keep])
    check(A, A, [(1.0, A)], 1e-3)
    ones = CSR(n, rp, col, np.where(col % 2 == 0, 1.0, -1.0))  # sums that cancel exactly
    check(ones, ones, [(-1.0, None)], 0.0)
    check(ones, ones, [], 2.0)


@pytest.mark.parametrize("n,w,tol,kind", [(257, 1, 1e-12, "exp"), (1500, 6, 1e-8, "cosh"), (1100, 3, 1e-6, "exp"),
                                          (5000, 8, 1e-10, "cos")])
@pytest.mark.parametrize("opts", [{}, {"square": True}, {"filtered": False}])
def test_series_keep_holes_bitwise(n, w, tol, kind, opts):
    if kind == "exp" and "square" in opts:
        pytest.skip("exp has both parities")
    Z, a = ocsr(syn.banded_random(n, w, n, 2.5)), syn.coeffs(kind)
    ref = psscf(Z, a, tol, **opts)
    s = psf.Series(a, tol, **opts)
    for _ in range(2):  # the first evaluation, and one with its records
        check_same(s.eval(dev(Z)), ref, kind)
    got = psf.eval_batch([psf.Series(a, tol, **opts)] * 3, [dev(Z), dev(ocsr(syn.laplacian_2d(9))), dev(Z)])
    for i in (0, 2):
        check_same(got[i], ref, "batch")
