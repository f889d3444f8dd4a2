"""Batches whose instances all have rows of consecutive columns: k_band alone
runs and ends every stage, in tiles of one row and (from three rounds of the
chip's warps on) of four; bitwise against the oracle, instance by instance."""
import pytest

import synthetic as syn
from gpu_helpers import check_same, dev, ocsr
from oracle import psscf

pytestmark = pytest.mark.gpu

psf = pytest.importorskip("paper_2208_05683_gb300")


def instance(k, n):
    return syn.laplacian_1d(n) if k % 2 else syn.banded_random(n, 4, 11 + n)


# 8512 rows: the least that k_band gets; 51072: three rounds of tiles of four
@pytest.mark.parametrize("sizes", [(64, 5001, 3447), (333, 1, 9000, 700), (17024, 16001, 18047), (30000, 2, 21071)])
@pytest.mark.parametrize("filtered", [True, False])
def test_banded_batch_bitwise(sizes, filtered):
    a, tol = syn.coeffs("exp"), 1e-8
    Zs = [ocsr(instance(k, n)) for k, n in enumerate(sizes)]
    s = psf.Series(a, tol, filtered=filtered)
    refs = [psscf(Z, a, tol, filtered=filtered) for Z in Zs]
    for _ in range(2):
        got = psf.eval_batch([s] * len(Zs), [dev(Z) for Z in Zs])
        for i, ref in enumerate(refs):
            check_same(got[i], ref, f"instance {i}")
