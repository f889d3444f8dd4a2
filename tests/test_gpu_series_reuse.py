"""One series evaluated on matrices of different sizes: what it recorded on the
larger one (column windows, words, row lengths) must not choose a form that
the smaller one's kernel cannot take.  Bitwise against the oracle."""
import numpy as np
import pytest

import synthetic as syn
from gpu_helpers import check_same, dev, ocsr
from oracle import CSR, psscf

pytestmark = pytest.mark.gpu

psf = pytest.importorskip("paper_2208_05683_gb300")


def grid(rows, cols, norm, seed):
    """Five-point operator with random entries, scaled to a 1-norm."""
    n = rows * cols
    i = np.arange(n)
    parts = [(i, i)] + [(i[k], i[k] + d) for d, k in
                        ((1, i % cols < cols - 1), (-1, i % cols > 0), (cols, i < n - cols), (-cols, i >= cols))]
    r, c = (np.concatenate(x) for x in zip(*parts))
    v = np.random.default_rng(seed).uniform(-1.0, 1.0, len(r))
    v *= norm / np.bincount(c, weights=np.abs(v), minlength=n).max()
    o = np.lexsort((c, r))
    rp = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=n))]).astype(np.int32)
    return CSR(n, rp, c[o].astype(np.int32), v[o])


@pytest.mark.parametrize("small", [(30, 30), (7, 150), (1, 1064), (40, 40)])
def test_list_steps_then_a_small_matrix_bitwise(small):
    # 9 x 700: the late steps' rows span more than 4608 columns in few words
    # (the list map); the small matrices have few enough rows for one block a
    # row, and their B rows are expected as long as the large one's
    a, tol = syn.coeffs("exp"), 1e-10
    large, little = grid(9, 700, 2.0, 1), grid(*small, 2.0, 2)
    refs = [psscf(large, a, tol), psscf(little, a, tol)]
    s = psf.Series(a, tol)
    for k in (0, 0, 1, 1, 0):
        check_same(s.eval(dev((large, little)[k])), refs[k], f"{small} {k}")


def test_a_batch_between_evaluations_bitwise():
    # a batch records its windows and no words: the next evaluation must not
    # pair them with an older matrix's
    a, tol = syn.coeffs("exp"), 1e-8
    rng = np.random.default_rng(4)
    n = 9001
    c = np.sort(rng.integers(0, n, (n, 3)), axis=1)
    c += np.arange(3)  # distinct
    c = np.minimum(c, n - 3 + np.arange(3)).astype(np.int32)
    many = CSR(n, (3 * np.arange(n + 1)).astype(np.int32), c.reshape(-1), rng.uniform(-0.05, 0.05, 3 * n))
    Zs = [grid(9, 700, 2.0, 1), many, grid(60, 160, 2.0, 3)]
    s = psf.Series(a, tol, submult=True)
    refs = [psscf(Z, a, tol, submult=True) for Z in Zs]
    for k, batch in ((0, False), (1, True), (0, False), (1, False), (0, True), (1, False), (2, True), (0, False)):
        got = psf.eval_batch([s], [dev(Zs[k])])[0] if batch else s.eval(dev(Zs[k]))
        check_same(got, refs[k], f"{k} {batch}")
