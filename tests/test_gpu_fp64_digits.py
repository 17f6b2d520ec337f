"""The FP64 factorization's tensor-core products (FP64 entries as 9-bit digits) at the sizes where its tiles, groups and
scales end: one dense front per case (every pair of points inside the core support), against the oracle.

Bounds: the log-likelihood within the FP64 parity bound 1e-10, and the residual |r - C alpha| / |r| within
n kappa 2^-53 of a backward stable solve, kappa <= 1e4 here (unit variances times n over the noise), which is below 1e-9
for every n below.
"""
import numpy as np
import pytest

import oracle
from paper_2411_05869_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


# one block and a remainder; 128-row tiles and one row more; whole groups of 256 columns and one column more or less
@pytest.mark.parametrize("n", [97, 127, 128, 129, 192, 193, 255, 256, 257, 320, 383, 513, 641])
def test_dense_fronts_of_every_remainder_match_the_oracle(n):
    from paper_2411_05869_gb300 import gp
    w = synth.spatial_2d(n=n, m=1, seed=1000 + n, rho=2.0, noise_var=0.1)
    settings = [w.hyper]
    for scale in (1e9, 1e-9):   # the digits' scales follow the covariance
        h = w.hyper.copy()
        h.core_var *= scale
        h.noise_var *= scale
        settings.append(h)
    rp, col = oracle.pattern(w.X, w.hyper.core_radius)
    assert len(col) == n * n
    perm = oracle.fill_order(w.X, w.hyper.core_radius, rp, col)
    ctx = gp.Context(0)
    ps = ctx.assemble(_dev(w.X), w.hyper.core_radius)
    f = ctx.factor(ps, settings, gp.GP_FP64)
    resid = np.stack([w.normals, w.normals * 1e4, w.normals * 1e-4])
    err = torch.empty(3, dtype=torch.float64, device="cuda")
    ll = f.loglik(_dev(resid), err=err).cpu().numpy()
    assert f.info()["not_pd_count"] == 0
    for h, r, got in zip(settings, resid, ll):
        want = oracle.sparse_loglik(h, w.X, rp, col, perm, r)["loglik"]
        assert abs(got - want) <= 1e-10 * abs(want), (n, got, want)
    assert float(err.max()) <= 1e-9
    f.free()
    ps.free()
