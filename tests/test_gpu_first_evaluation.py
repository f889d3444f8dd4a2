"""The first evaluation of a series sizes its pool for what the warps' arenas
leave unused too: the norm phase of a band runs once (by its launches)."""
import ctypes

import pytest

import synthetic as syn
from gpu_helpers import check_same, dev, ocsr
from oracle import psscf

pytestmark = pytest.mark.gpu

psf = pytest.importorskip("paper_2208_05683_gb300")


def launches(f):
    a, b = ctypes.c_int64(), ctypes.c_int64()
    psf.lib().psf_launch_count(ctypes.byref(a))
    r = f()
    psf.lib().psf_launch_count(ctypes.byref(b))
    return r, b.value - a.value


@pytest.mark.parametrize("n,w", [(256, 1), (1000, 2), (4000, 2), (4000, 6), (9000, 1)])
def test_a_bands_norm_phase_runs_once(n, w):
    Z, a = ocsr(syn.banded_random(n, w, n, 1.0)), syn.coeffs("exp")
    s, Zd = psf.Series(a, 1e-10), dev(Z)
    ref = psscf(Z, a, 1e-10)
    got, first = launches(lambda: s.eval(Zd))
    check_same(got, ref)
    s.eval(Zd)
    got, later = launches(lambda: s.eval(Zd))
    check_same(got, ref)
    # a second pass of the norm phase alone is 13 launches; a first evaluation
    # differs by its pool's reset and copy and the rows it can't reuse
    assert first <= later + 4


@pytest.mark.parametrize("opts", [{"submult": True}, {"filtered": False}, {"square": True}, {"estimate": True}])
def test_an_evaluations_phases_run_once(opts):
    # other schemes, whose second phase has the pool to itself or ends with a product
    Z = ocsr(syn.banded_random(5000, 7, 3, 2.5))
    a = syn.coeffs("sinh" if "square" in opts else "exp")
    s, Zd = psf.Series(a, 1e-12, **opts), dev(Z)
    _, first = launches(lambda: s.eval(Zd))
    s.eval(Zd)
    _, later = launches(lambda: s.eval(Zd))
    assert first <= later + 4
