"""The list map (wide windows of few words) bitwise against the oracle: long
thin grids, runs that start and end anywhere in a word, rows with more words
than the map holds (its window is halved), rows of more entries than slots,
and windows wider than the map's 32768 columns; the first evaluation, which
predicts its windows, and the later ones, which have records."""
import numpy as np
import pytest

import synthetic as syn
from gpu_helpers import check_same, dev, ocsr
from oracle import CSR, psscf

pytestmark = pytest.mark.gpu

psf = pytest.importorskip("paper_2208_05683_gb300")


def diagonals(n, offsets, seed, norm):
    """Random entries U[-1, 1] on the given diagonals, scaled to a 1-norm."""
    rng = np.random.default_rng(seed)
    i = np.arange(n)
    rows = np.concatenate([i[(i + d >= 0) & (i + d < n)] for d in offsets])
    cols = np.concatenate([i[(i + d >= 0) & (i + d < n)] + d for d in offsets])
    vals = rng.uniform(-1.0, 1.0, len(rows))
    vals *= norm / np.bincount(cols, weights=np.abs(vals), minlength=n).max()
    order = np.lexsort((cols, rows))
    rp = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=n))]).astype(np.int32)
    return CSR(n, rp, cols[order].astype(np.int32), vals[order])


CASES = {
    "grid 9 x 700": (9 * 700, [-700, -1, 0, 1, 700], 2.0, "exp", 1e-10, {}),
    "grid 13 x 611 cos": (13 * 611, [-611, -1, 0, 1, 611], 2.0, "cos", 1e-8, {}),
    "grid 9 x 640 square": (9 * 640, [-640, -1, 0, 1, 640], 1.5, "cosh", 1e-10, {"square": True}),
    "unfiltered": (10 * 523, [-523, -1, 0, 1, 523], 1.0, "exp", 1e-6, {"filtered": False}),
    "many words": (9001, [-977, -311, -53, 0, 71, 401, 1201], 1.0, "exp", 1e-6, {}),
    "past the window": (45000, [-7001, 0, 1, 7000], 0.5, "exp", 1e-7, {}),
}


@pytest.mark.parametrize("name", list(CASES))
def test_wide_rows_bitwise(name):
    n, offsets, norm, kind, tol, opts = CASES[name]
    Z, a = diagonals(n, offsets, n, norm), syn.coeffs(kind)
    ref = psscf(Z, a, tol, **opts)
    s = psf.Series(a, tol, **opts)
    for _ in range(3):
        check_same(s.eval(dev(Z)), ref, name)
