"""Matrices whose rows are runs of consecutive columns and whose products' rows
are not: runs at unrelated places, permuted blocks, bands that the filter cuts
to pieces.  They take the general product kernels (by the check of the input,
or by what the previous evaluation recorded); bitwise against the oracle over
several evaluations of one series, as products and in batches."""
import numpy as np
import pytest

import synthetic as syn
from gpu_helpers import assert_csr_bitwise, check_same, dev, ocsr
from oracle import CSR, alg1, axpy, matmul_add, psscf

pytestmark = pytest.mark.gpu

psf = pytest.importorskip("paper_2208_05683_gb300")


def runs(n, start, width, seed, norm):
    """Row i: columns start[i] .. start[i] + width - 1, scaled to a 1-norm."""
    rng = np.random.default_rng(seed)
    col = (np.asarray(start)[:, None] + np.arange(width)).reshape(-1).astype(np.int32)
    val = rng.uniform(-1.0, 1.0, len(col))
    val *= norm / np.bincount(col, weights=np.abs(val), minlength=n).max()
    return CSR(n, (np.arange(n + 1) * width).astype(np.int32), col, val)


def scattered(n, width, seed, norm=0.5):
    return runs(n, np.random.default_rng(seed).integers(0, n - width + 1, n), width, seed, norm)


def blocks(n, m, seed, norm=1.5):
    """Block g's rows hold the columns of block p[g]."""
    p = np.random.default_rng(seed).permutation(n // m)
    return runs(n, p[np.arange(n) // m] * m, m, seed, norm)


def weak(n, amps, seed, norm=2.0):
    """A band whose diagonals d have magnitude amps[|d|]: the filter drops the weak ones."""
    rng = np.random.default_rng(seed)
    w = len(amps) - 1
    rows = [[j for j in range(i - w, i + w + 1) if 0 <= j < n] for i in range(n)]
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
    col = np.concatenate(rows).astype(np.int32)
    val = rng.uniform(0.5, 1.0, len(col)) * np.asarray(amps)[np.abs(col - np.repeat(np.arange(n), np.diff(rp)))]
    val *= norm / np.bincount(col, weights=np.abs(val), minlength=n).max()
    return CSR(n, rp, col, val)


SERIES = {
    "scattered 1000 w20": (scattered(1000, 20, 1), "exp", 1e-8, {}),
    "scattered 900 w3": (scattered(900, 3, 2), "cosh", 1e-8, {"square": True}),
    "scattered 6001 w3": (scattered(6001, 3, 3, 0.01), "exp", 1e-4, {"submult": True}),
    "scattered 20000 w2": (scattered(20000, 2, 4, 0.01), "exp", 1e-4, {"submult": True}),
    "blocks 1000 m8": (blocks(1000, 8, 5), "exp", 1e-10, {}),
    "blocks 5005 m7": (blocks(5005, 7, 6), "exp", 1e-8, {"filtered": False}),
    "weak odd 700": (weak(700, [1, 1e-9, 1, 1e-9, 1], 7), "exp", 1e-8, {}),
    "weak odd 6000 submult": (weak(6000, [1, 1e-9, 1, 1e-9, 1], 8), "exp", 1e-8, {"submult": True}),
    "far pair 3000": (weak(3000, [1] + [1e-10] * 11 + [1], 9), "cos", 1e-8, {}),
}


@pytest.mark.parametrize("name", list(SERIES))
def test_series_bitwise(name):
    Z, kind, tol, opts = SERIES[name]
    a = syn.coeffs(kind)
    ref = psscf(Z, a, tol, **opts)
    s = psf.Series(a, tol, **opts)
    for _ in range(3):
        check_same(s.eval(dev(Z)), ref, name)


def test_a_series_on_pieces_and_bands_of_one_size_bitwise():
    a, tol = syn.coeffs("exp"), 1e-8
    Zs = [weak(1500, [1, 1e-9, 1, 1e-9, 1], 1), ocsr(syn.banded_random(1500, 4, 2, 2.0)), scattered(1500, 5, 3),
          ocsr(syn.banded_random(1100, 4, 2, 2.0))]
    refs = [psscf(Z, a, tol) for Z in Zs]
    s = psf.Series(a, tol)
    for k in (0, 0, 1, 2, 1, 3, 0, 2, 1):
        check_same(s.eval(dev(Zs[k])), refs[k], str(k))


@pytest.mark.parametrize("n,w", [(1000, 20), (6001, 3), (1064, 1), (5000, 9)])
@pytest.mark.parametrize("threshold", [0.0, 1e-2])
def test_products_bitwise(n, w, threshold):
    A, B, D = scattered(n, w, 1), scattered(n, w + 1, 2), ocsr(syn.banded_random(n, 2, 3))
    for X, Y, M in ((A, B, None), (D, B, A), (A, D, B), (blocks(n // w * w, w, 4),) * 3):
        C = matmul_add(X, Y, axpy(0.5, M, None, X.n))
        got = psf.product_filter(dev(X), dev(Y), [(0.5, None if M is None else dev(M))], threshold)
        assert_csr_bitwise(got.csr, alg1(C, threshold / 1.1, 0.1).kept if threshold else C)


def test_few_rows_apart_stay_a_band_bitwise():
    Z = ocsr(syn.banded_random(3000, 3, 5, 2.0))
    keep = ~np.isin(np.repeat(np.arange(3000), np.diff(Z.rowptr)), (700, 701, 702, 703, 704, 705, 706, 707))
    rp = np.concatenate([[0], np.cumsum(np.bincount(np.repeat(np.arange(3000), np.diff(Z.rowptr))[keep],
                                                    minlength=3000))]).astype(np.int32)
    H = CSR(3000, rp, Z.col[keep], Z.val[keep])  # eight empty rows
    two = CSR(3000, Z.rowptr, Z.col.copy(), Z.val)
    s, e = two.rowptr[1500], two.rowptr[1501]
    two.col[s:e] = np.arange(e - s)  # one row's run far from the others
    a = syn.coeffs("exp")
    for M in (H, two):
        ref = psscf(M, a, 1e-8)
        s_ = psf.Series(a, 1e-8)
        for _ in range(2):
            check_same(s_.eval(dev(M)), ref)


def test_batches_bitwise():
    a, tol = syn.coeffs("exp"), 1e-6
    Zs = [ocsr(syn.banded_random(5000, 3, 1, 2.0)), scattered(700, 6, 2), ocsr(syn.scale(syn.laplacian_2d(30), 0.25)),
          blocks(1200, 12, 3), ocsr(syn.laplacian_1d(3000)), weak(900, [1, 1e-9, 1], 4)]
    refs = [psscf(Z, a, tol) for Z in Zs]
    s = psf.Series(a, tol)
    for pick in ((0, 1, 2, 3, 4, 5), (0, 4, 5, 3), (1, 3)):
        for _ in range(2):
            got = psf.eval_batch([s] * len(pick), [dev(Zs[k]) for k in pick])
            for g, k in zip(got, pick):
                check_same(g, refs[k], str(k))
