"""Algorithm 1 as one cluster of blocks (small steps) and as the whole grid:
both sides of the line between them, bitwise against the oracle with every
step's records (passes, eps_f, dropped), through an evaluation and through a
single product; candidates that overflow the narrow threshold's exponents
(values over many magnitudes) included."""
import numpy as np
import pytest

import synthetic as syn
from gpu_helpers import assert_csr_bitwise, check_same, dev, ocsr
from oracle import CSR, alg1, matmul_add, psscf

pytestmark = pytest.mark.gpu

psf = pytest.importorskip("paper_2208_05683_gb300")


@pytest.mark.parametrize("n", [1, 2, 31, 33, 700, 1300, 2100, 4096, 4097])
def test_evaluations(n):
    Z = syn.banded_random(n, 5, n) if n > 5 else (np.arange(n + 1, dtype=np.int32), np.arange(n, dtype=np.int32),
                                                 np.linspace(0.5, 1.0, n))
    a = syn.coeffs("exp")
    ref = psscf(ocsr(Z), a, 1e-12)
    s = psf.Series(a, 1e-12)
    for _ in range(2):
        check_same(s.eval(dev(ocsr(Z))), ref, f"n = {n}")


def scattered(n, per_row, spread, seed):
    rng = np.random.default_rng(seed)
    rp, cols, vals = [0], [], []
    for _ in range(n):
        c = np.sort(rng.choice(n, size=min(n, per_row), replace=False))
        cols.append(c)
        vals.append(rng.uniform(-1, 1, len(c)) * 10.0 ** rng.uniform(-spread, 0, len(c)))
        rp.append(rp[-1] + len(c))
    return CSR(n, np.array(rp, np.int32), np.concatenate(cols).astype(np.int32), np.concatenate(vals))


@pytest.mark.parametrize("n,per_row", [(40, 20), (600, 9), (1500, 40), (5000, 6)])
@pytest.mark.parametrize("spread", [0, 12])
def test_products(n, per_row, spread):
    A, B = scattered(n, per_row, spread, 1), scattered(n, per_row, spread, 2)
    for eps in (1e-6, 0.3):
        ref = alg1(matmul_add(A, B), eps / 1.1, 0.1)
        got = psf.product_filter(dev(A), dev(B), [], eps, 0.1)
        assert_csr_bitwise(got.csr, ref.kept)
        assert got.steps[0]["iters"] == ref.iters and got.steps[0]["dropped"] == ref.c
