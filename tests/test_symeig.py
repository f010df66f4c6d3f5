"""The host eigensolver of the M2L compression at sizes around its blocks of 8 rows and its
split over threads (128 and more).  A backward stable reduction leaves residuals and departures
from orthogonality of a small multiple of n eps; the bar is 50 n eps."""
import ctypes

import numpy as np
import pytest


@pytest.mark.parametrize("n", [1, 2, 3, 8, 9, 10, 27, 64, 125, 128, 216, 343])
@pytest.mark.parametrize("kind", ["dense", "multiplets", "diagonal"])
def test_symmetric_eigenvectors(n, kind):
    import paper_1710_06316_gb300 as pb
    f = pb.load()._ZN5afmpb12sym_eig_descEiPdS0_S0_
    f.restype = ctypes.c_int
    rng = np.random.default_rng(n)
    if kind == "dense":
        a = rng.standard_normal((n, n))
        a = a @ a.T
    elif kind == "diagonal":
        a = np.diag(rng.uniform(-1, 1, n))
    else:                                # eigenvalues in groups, over ten decades
        q, _ = np.linalg.qr(rng.standard_normal((n, n)))
        a = (q * 10.0 ** -(10 * (np.arange(n) // 3) / n)) @ q.T
        a = 0.5 * (a + a.T)
    w, zt = np.zeros(n), np.full((n, n), np.nan)
    keep = a.copy()
    p = lambda v: v.ctypes.data_as(ctypes.c_void_p)
    assert f(ctypes.c_int(n), p(keep), p(w), p(zt)) == 0
    bar = 50 * n * np.finfo(float).eps
    assert (np.diff(w) <= 0).all()
    assert np.abs(zt @ zt.T - np.eye(n)).max() < bar
    assert np.linalg.norm(a @ zt.T - zt.T * w) < bar * np.linalg.norm(a)
    assert np.allclose(w, np.linalg.eigvalsh(a)[::-1], rtol=0, atol=bar * np.linalg.norm(a))
