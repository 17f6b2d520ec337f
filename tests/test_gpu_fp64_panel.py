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


@pytest.mark.parametrize("terms", [8, 15, 17, 33, 62])
@pytest.mark.parametrize("low", [0.99, -0.99, 0.6])
def test_inverse_whose_low_halves_have_one_sign(panel, low, terms):
    """Rows 1..62 of the inverse start with nearly the largest entry a row can have, and row 63 of L holds low 2^29 units of
    2^-60 (once at the scale of its row) in the first `terms` of them: all its cross products have one sign and add up to
    terms low 2^59. The inverse is good to 2^-57 of each row's largest entry (cut at 2^-60, from at most 63 products):
    2^-50 of it in a product with rows of L that are at most 2 long."""
    a, d, v = 255 / 128, 1027 / 8192, low * 2.0 ** -35   # exact squares: L L^T is exact but for its last diagonal entry
    L = np.diag(np.r_[1.0, np.full(62, d), 1.0])
    L[1:63, 0] = -a
    L[63, 1:terms + 1] = v
    A = np.tril(L @ L.T)
    P, D, bad = panel(A, np.diag(A))
    assert bad is None
    E = np.abs(D.astype(np.longdouble) @ P.astype(np.longdouble) - np.eye(64))
    assert (E <= 2.0 ** -49 * np.abs(D).max(1, keepdims=True)).all(), float(E.max())
