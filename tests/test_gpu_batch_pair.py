"""Batches with instances whose rows span consecutive columns and others (the
step is then two overlapping launches), below and above the row count at
which the banded ones are computed four rows at a time; bitwise against
the oracle, instance by instance and step by step."""
import pytest

import synthetic as syn
from gpu_helpers import check_same, dev, ocsr
from oracle import psscf

pytestmark = pytest.mark.gpu

psf = pytest.importorskip("paper_2208_05683_gb300")


def instance(kind, n, seed):
    if kind == "band":
        return syn.banded_random(n, 3, seed)
    if kind == "grid":
        m = int(round(n ** 0.5))
        return syn.scale(syn.laplacian_2d(m), 1.0 / 4.0)
    return syn.laplacian_1d(n)


@pytest.mark.parametrize("sizes", [(2, 5, 9), (33, 64, 100, 257), (1700, 2500, 8100), (9000, 10000, 6001, 64)])
@pytest.mark.parametrize("filtered", [True, False])
def test_mixed_batch_bitwise(sizes, filtered):
    kinds = ["grid", "band", "lap"]
    Zs = [instance(kinds[i % 3], n, 7 + n) for i, n in enumerate(sizes)]
    a = syn.coeffs("exp")
    tol = 1e-8
    s = psf.Series(a, tol, filtered=filtered)
    refs = [psscf(ocsr(Z), a, tol, filtered=filtered) for Z in Zs]
    for _ in range(2):
        got = psf.eval_batch([s] * len(Zs), [dev(ocsr(Z)) for Z in Zs])
        for i, ref in enumerate(refs):
            check_same(got[i], ref, f"instance {i}")
