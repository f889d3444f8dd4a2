"""The workspace an evaluation reads back as one piece: a plan with more steps
than the front's records, and repeated evaluations of it."""
import pytest

import synthetic as syn
from gpu_helpers import check_same, dev, ocsr
from oracle import psscf

pytestmark = pytest.mark.gpu

psf = pytest.importorskip("paper_2208_05683_gb300")


@pytest.mark.parametrize("terms", [79, 80, 81, 150])
def test_long_plan_bitwise(terms):
    Z = ocsr(syn.banded_random(90, 2, 5, 0.9))
    a = [0.5 ** i for i in range(terms)]
    ref = psscf(Z, a, 1e-9, poly=True, s=1)
    s = psf.Series(a, 1e-9, poly=True, s=1)
    for _ in range(2):
        check_same(s.eval(dev(Z)), ref, f"{terms} terms")
