"""psf_result_copy into device arrays: every alignment of source and
destination (a batch's results start anywhere in shared storage), null and
unaligned destinations, results without entries; the bytes are the result's."""
import ctypes

import numpy as np
import pytest

import synthetic as syn
from gpu_helpers import dev, ocsr

pytestmark = pytest.mark.gpu

psf = pytest.importorskip("paper_2208_05683_gb300")
torch = pytest.importorskip("torch")


def results(sizes):
    s = psf.Series(syn.coeffs("exp"), 1e-10)
    Zs = [dev(ocsr(syn.banded_random(n, 2, n))) for n in sizes]
    L = psf.lib()
    sh = (ctypes.c_void_p * len(Zs))(*[s._h.value] * len(Zs))
    zs = (psf.CSRStruct * len(Zs))(*[z._struct() for z in Zs])
    outs = (ctypes.c_void_p * len(Zs))()
    psf.check(L.psf_eval_batch(sh, zs, len(Zs), None, outs))
    return L, [ctypes.c_void_p(o) for o in outs], [s.eval(z).csr.to_host() for z in Zs]


@pytest.mark.parametrize("shift", [0, 4, 8, 12, 2])
def test_copies_are_the_result(shift):
    sizes = [3, 4, 8, 57, 130, 4099]
    L, outs, refs = results(sizes)
    for out, (rp, col, val) in zip(outs, refs):
        n, nnz = len(rp) - 1, len(col)
        sizes_b = [4 * (n + 1), 4 * nnz, 8 * nnz]
        bufs = [torch.full((b + 64,), 7, dtype=torch.uint8, device="cuda") for b in sizes_b]
        for skip in (None, 0, 2):
            ptrs = [ctypes.c_void_p(None if i == skip else b.data_ptr() + shift) for i, b in enumerate(bufs)]
            psf.check(L.psf_result_copy(out, *ptrs, None))
        torch.cuda.synchronize()
        for b, nb, ref in zip(bufs, sizes_b, (rp, col, val)):
            got = b.cpu().numpy()
            assert got[shift:shift + nb].tobytes() == np.ascontiguousarray(ref).tobytes()
            assert (got[:shift] == 7).all() and (got[shift + nb:] == 7).all()
        psf.check(L.psf_result_destroy(out))


def test_into_host_arrays_and_empty():
    Z = psf.DeviceCSR.from_host(np.zeros(6, np.int32), np.zeros(0, np.int32), np.zeros(0))
    r = psf.Series([0.0, 1.0], 1e-8, poly=True).eval(Z)
    assert r.csr.to_host()[0].tolist() == [0] * 6
    rp, col, val = syn.banded_random(300, 2, 1)
    s = psf.Series(syn.coeffs("exp"), 1e-10)
    (hr, hc, hv), _, _ = s.eval_host(rp, col, val)
    dr, dc, dv = s.eval(dev(ocsr((rp, col, val)))).csr.to_host()
    assert np.array_equal(hr, dr) and np.array_equal(hc, dc) and hv.tobytes() == dv.tobytes()
