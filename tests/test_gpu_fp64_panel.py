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


def _first_failing(A):
    """First column whose pivot is not positive (None: positive definite); pivots are away from zero by construction."""
    A = A.astype(np.longdouble)
    for k in range(len(A)):
        if not A[k, k] > 0:
            return k
        c = A[k + 1:, k] / np.sqrt(A[k, k])
        A[k + 1:, k + 1:] -= np.outer(c, c)
    return None


@pytest.mark.parametrize("p", [1, 15, 16, 31, 32, 47, 63])
@pytest.mark.parametrize("scale", [1.0, 3.9])   # the ends of the rows' fixed-point range
def test_row_of_a_tile_that_breaks_definiteness_is_its_first_failing_column(panel, p, scale):
    """Uncorrelated columns and one row with the same entry in each: its pivot falls by r^2 per column, to below zero by a
    little, to any number of turns of a 64-bit integer, or to values beyond the fixed point."""
    for r in np.concatenate([np.linspace(0.05, 2.0, 80), [5.0, 30.0, 1e3, 1e6, 1e9, 1e30, 1e100]]):
        if abs(p * r * r - 1) < 1e-6:
            continue
        A = np.eye(64)
        A[p, :p] = r
        A *= scale
        want = p if p * r * r > 1 else None
        P, D, bad = panel(A, np.diag(A))
        assert bad == want, (p, r, bad)
        if bad is None:
            assert np.abs(P @ P.T - (A + np.tril(A, -1).T)).max() <= 64 * 2.0 ** -50 * scale


@pytest.mark.parametrize("bw", [1, 17, 33, 64])
def test_random_tiles_report_the_first_failing_pivot(panel, bw):
    rng = np.random.default_rng(bw)
    for k in range(40):
        Q = np.linalg.qr(rng.standard_normal((bw, bw)))[0]
        ev = np.exp(rng.uniform(-6, 0, bw))
        ev[rng.integers(bw)] *= rng.choice([-1.0, 1.0])
        d = 2.0 ** rng.integers(-20, 20, bw)
        A = (Q * ev) @ Q.T
        A = (A + A.T) / 2
        want = _first_failing(A)
        A = A * d[:, None] * d[None, :]
        P, D, bad = panel(np.tril(A), np.abs(np.diag(A)) + (np.diag(A) == 0))
        assert bad == want


@pytest.mark.parametrize("rows", [1, 64, 65, 128, 300])
def test_rows_below_are_flagged_only_beyond_their_variance(panel, rows):
    """A row of L longer than sqrt(C_ii) shows at its own pivot; one with an entry of many times that is recorded here."""
    rng = np.random.default_rng(rows)
    base = np.concatenate([np.eye(64), np.zeros((rows, 64))])
    diag = np.concatenate([np.ones(64), 10.0 ** rng.uniform(-3, 3, rows)])
    base[64:] = rng.uniform(-0.99, 0.99, (rows, 64)) * np.sqrt(diag[64:, None])
    P, D, bad = panel(base, diag)
    assert bad is None
    assert np.array_equal(P[64:], base[64:]) or np.abs(P[64:] - base[64:]).max() <= 2.0 ** -53 * np.sqrt(diag.max())
    for factor in (8.0, 1e3, 1e9, 1e40, 1e200):
        for col in (0, 31, 32, 63):
            i, j = rng.integers(rows), rng.integers(rows)
            A = base.copy()
            A[64 + i, col] = factor * math.sqrt(diag[64 + i])
            A[64 + j, col] = -factor * math.sqrt(diag[64 + j])
            P, D, bad = panel(A, diag)
            assert bad == 64 + min(i, j), (factor, col)


@pytest.mark.parametrize("kappa", [1e2, 1e6, 1e10, 1e13])
def test_ill_conditioned_positive_definite_panels_are_not_flagged(panel, kappa):
    rng = np.random.default_rng(int(math.log10(kappa)))
    for k in range(10):
        n = 64 + 150
        x = np.sort(rng.uniform(0, 1, n))
        K = np.exp(-0.5 * ((x[:, None] - x[None]) / 0.3) ** 2) + (10.0 / kappa) * np.eye(n)
        K *= 10.0 ** rng.uniform(-8, 8)
        P, D, bad = panel(np.concatenate([np.tril(K[:64, :64]), K[64:, :64]]), np.diag(K))
        assert bad is None


@pytest.mark.parametrize("bw,rows", [(64, 200), (64, 1), (17, 130)])
@pytest.mark.parametrize("noise", [1.0, 1e-2, 1e-4, 1e-8, 1e-12])
def test_rows_below_are_solved_backward_stably(panel, noise, bw, rows):
    """|B - X L^T| and |A - L L^T| within 4 units of 2^-53 of the products' scales whatever the tile's condition: X and L are
    rounded to 2^-53 each (2 units together, by Cauchy-Schwarz), the digits and the residual's integers to 2^-55 and less.
    Rows that are weakly correlated with the tile's columns keep to their own scale where its inverse is below 2^12."""
    rng = np.random.default_rng(bw + rows)
    n = bw + rows
    x = np.sort(rng.uniform(0, 1, n))
    K = np.exp(-0.5 * ((x[:, None] - x[None]) / 0.3) ** 2) + noise * np.eye(n)
    B = K[bw:, :bw].copy()
    weak = rng.uniform(size=rows) < 0.3
    B[weak] *= 2.0 ** -30
    P, D, bad = panel(np.concatenate([np.tril(K[:bw, :bw]), B]), np.diag(K))
    assert bad is None
    L, X = P[:bw].astype(np.longdouble), P[bw:].astype(np.longdouble)
    d = np.sqrt(np.diag(K))
    T = np.abs(np.tril(K[:bw, :bw] - L @ L.T)) / np.outer(d[:bw], d[:bw])
    assert T.max() <= 4 * EPS, float(T.max() / EPS)
    R = np.abs(B - X @ L.T) / d[None, :bw]
    assert (R <= 4 * EPS * d[bw:, None]).all(), float(R.max() / EPS)
    if noise >= 1e-4:
        size = np.sqrt((X * X).sum(1, keepdims=True))
        assert (R <= 4 * EPS * size).all(), float((R / size).max() / EPS)
