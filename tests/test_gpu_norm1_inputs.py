"""psf_norm1 and psf_norm1_noalloc reject malformed inputs, whose entries they
read in place: their check bounds the entry count before any entry is read."""
import ctypes

import numpy as np
import pytest

from gpu_helpers import dev, ocsr
import synthetic as syn
from oracle import norm1

pytestmark = pytest.mark.gpu

psf = pytest.importorskip("paper_2208_05683_gb300")
from paper_2208_05683_gb300 import _abi  # noqa: E402


def i32(*x):
    return np.array(x, np.int32)


BAD = {
    "order": (i32(0, 2, 2, 2, 2, 2), i32(3, 1), np.array([1.0, 2.0])),
    "range": (i32(0, 1, 1, 1, 1, 1), i32(7), np.array([1.0])),
    "nan": (i32(0, 1, 1, 1, 1, 1), i32(0), np.array([np.nan])),
    "repeated": (i32(0, 2, 2, 2, 2, 2), i32(1, 1), np.array([1.0, 2.0])),
    "negative": (i32(0, 1, 1, 1, 1, 1), i32(-1), np.array([1.0])),
    "inf": (i32(0, 1, 1, 1, 1, 1), i32(0), np.array([np.inf])),
    "decreasing": (i32(0, 2, 1, 2, 2, 2), i32(0, 1), np.array([1.0, 2.0])),
    "first": (i32(1, 1, 1, 1, 1, 1), i32(0), np.array([1.0])),
    "last": (i32(0, 1, 1, 1, 1, 0), i32(0), np.array([1.0])),
}


@pytest.mark.parametrize("name", list(BAD))
def test_malformed_input_is_rejected(name):
    for f in (psf.norm1, psf.norm1_noalloc):
        with pytest.raises(psf.PsfError) as e:
            f(dev(BAD[name]))
        assert e.value.code == _abi.PSF_EINVAL
    Z = ocsr(syn.laplacian_2d(20))  # the next call is not disturbed
    assert psf.norm1(dev(Z)) == psf.norm1_noalloc(dev(Z)) == norm1(Z)


@pytest.mark.parametrize("claimed", [2**20, 2**31 - 1])
def test_an_entry_count_past_the_arrays_is_rejected(claimed):
    # well-formed rows, and an entry count that is not theirs
    Z = dev(ocsr(syn.laplacian_2d(20)))
    for f in (psf.lib().psf_norm1, psf.lib().psf_norm1_noalloc):
        m, out = Z._struct(), ctypes.c_double()
        m.nnz = claimed
        assert f(ctypes.byref(m), psf._stream_ptr(None), ctypes.byref(out)) == _abi.PSF_EINVAL
