"""A row of a band that comes out with an exact zero between its entries keeps
the zero's place.  That place is no entry: where a power of Z has overflowed,
its infinity must not meet it (0 * inf), for an entry that is not there gives
nothing."""
import numpy as np
import pytest

from gpu_helpers import dev, ocsr
import synthetic as syn
from oracle import CSR, axpy, matmul_add

pytestmark = pytest.mark.gpu

psf = pytest.importorskip("paper_2208_05683_gb300")


def overflowing(n):
    """Half-bandwidth 2, diagonal 1; (Z^2)[r, r + 2] overflows for every tenth r."""
    rng = np.random.default_rng(n)
    rows = [[j for j in range(i - 2, i + 3) if 0 <= j < n] for i in range(n)]
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
    r = np.repeat(np.arange(n), np.diff(rp))
    c = np.concatenate(rows).astype(np.int32)
    v = rng.uniform(0.5, 1.5, len(c))
    v[r == c] = 1.0
    v[(c == r + 1) & ((r % 10 == 4) | (r % 10 == 5))] = 1e200
    return CSR(n, rp, c, v)


def ps(Z, a):
    """The unfiltered scheme for six coefficients (q = 2, b = 3), step by step."""
    def block(i):
        return axpy(a[2 * i + 1], Z, axpy(a[2 * i], None, None, Z.n), Z.n)
    Z2 = matmul_add(Z, Z)
    S = block(2)
    for i in (1, 0):
        S = matmul_add(Z2, S, block(i))
    return S


def same(got, ref):
    assert (got.info["q"], got.info["b"], got.info["g"]) == (2, 3, 0)
    rp, col, val = got.csr.to_host()
    assert np.array_equal(rp, ref.rowptr) and np.array_equal(col, ref.col)
    nan = np.isnan(ref.val)
    assert np.array_equal(np.isnan(val), nan)
    assert np.array_equal(val[~nan].view(np.int64), ref.val[~nan].view(np.int64))


@pytest.mark.parametrize("n", [40, 333, 5000])
def test_overflow_does_not_meet_holes(n):
    Z = overflowing(n)
    a = [0.5, 0.25, 0.125, 0.5, -0.25, 0.25]  # S_0 = a_4 I + a_5 Z: the diagonal cancels
    opts = dict(poly=True, submult=True, filtered=False)
    ref = ps(Z, a)
    inf, nan = np.isinf(ref.val), np.isnan(ref.val)
    assert inf.any() and (~inf & ~nan).any()
    s = psf.Series(a, 1e-8, **opts)
    for _ in range(2):
        same(s.eval(dev(Z)), ref)
    # in a batch of enough rows that bands have a kernel of their own
    L = ocsr(syn.laplacian_1d(9000))
    got = psf.eval_batch([psf.Series(a, 1e-8, **opts) for _ in range(2)], [dev(L), dev(Z)])
    same(got[0], ps(L, a))
    same(got[1], ref)


def test_powers_of_the_norm_phase_bring_no_holes():
    # exact norms: the second evaluation, and a batch, take the baby steps from
    # the norm phase's rows, whose zeros keep their places
    Z = overflowing(400)
    off = Z.col - np.repeat(np.arange(400), np.diff(Z.rowptr))
    Z.val[np.abs(off) < 2] = 1.0  # (Z^2)[r, r] = sums of +-1: exact zeros on the diagonal
    Z.val[off == -1] = -1.0
    Z.val[np.abs(off) == 2] = np.where(off[np.abs(off) == 2] > 0, 0.5, 1.0)
    Z.val[(off == 1) & np.isin(np.repeat(np.arange(400), np.diff(Z.rowptr)) % 10, (4, 5))] = 1e160
    a = [0.5, 0.25, 0.125, 0.5, 1e160, -1e160]
    ref = ps(Z, a)
    assert np.isinf(ref.val).any()
    s = psf.Series(a, 1e-8, poly=True, filtered=False)
    for _ in range(3):
        same(s.eval(dev(Z)), ref)
    same(psf.eval_batch([s], [dev(Z)])[0], ref)
