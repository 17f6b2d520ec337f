"""The FP64 factorization's diagonal-tile and row kernels on a panel of their own (tests/fp64_panel.cu): matrices that a
covariance reaches only by accident, at the ends of the fixed-point ranges.
"""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

HERE = os.path.dirname(os.path.abspath(__file__))
EPS = 2.0 ** -53


@pytest.fixture(scope="module")
def panel(tmp_path_factory):
    from paper_2411_05869_gb300 import build
    so = str(tmp_path_factory.mktemp("panel") / "panel.so")
    cmd = [build.nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-shared", "--cudart", "static", "-o", so,
           os.path.join(HERE, "fp64_panel.cu")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    fn = ctypes.CDLL(so).fp64_panel

    def run(A, diag):
        """A: m x bw lower part of a covariance, diag: its m variances. (L, inverse of its diagonal block, first failing
        column or None)"""
        m, bw = A.shape
        P = np.asfortranarray(A, dtype=np.float64).copy(order="F")
        d = np.ascontiguousarray(diag, dtype=np.float64)
        D = np.zeros((64, 64))
        st = (ctypes.c_int32 * 2)()
        torch.cuda.synchronize()
        e = fn(P.ctypes.data_as(ctypes.c_void_p), m, bw, d.ctypes.data_as(ctypes.c_void_p),
               D.ctypes.data_as(ctypes.c_void_p), st)
        assert e == 0 and st[1] == 0
        P[:bw] = np.tril(P[:bw])
        return P, D, None if st[0] == 0x7fffffff else st[0]

    return run


@pytest.mark.parametrize("v", [0.75 * 2.0 ** -33, 0.99 * 2.0 ** -33, 0.75 * 2.0 ** -32, 0.99 * 2.0 ** -32, 0.99 * 2.0 ** -31])
@pytest.mark.parametrize("a", [0.9375, 1.0])
def test_inverse_whose_low_halves_have_one_sign(panel, a, v):
    """L = I but for the column -a and the row v, entries whose low 30 bits are all near the largest: the inverse's cross
    sums add up 62 terms of one sign. The inverse is good to 2^-57 of each row's largest entry (its rows are cut at 2^-60 and
    come from at most 63 products), whose rows are at most 63 long against L's of at most 2: 2^-50 in the product."""
    L = np.eye(64)
    L[1:63, 0] = -a
    L[63, 1:63] = v
    A = np.tril(L @ L.T)
    P, D, bad = panel(A, np.diag(A))
    assert bad is None
    assert np.abs(D @ P - np.eye(64)).max() <= 2.0 ** -50
