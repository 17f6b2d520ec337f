"""The FP64 path at the edges of its fixed-point arithmetic, through the C-ABI."""
import math

import numpy as np
import pytest

import oracle
from paper_2411_05869_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def _first_failing(C):
    """The first column whose pivot is not positive (None: positive definite), with pivots well away from zero."""
    A = C.copy()
    for k in range(len(A)):
        assert abs(A[k, k]) > 1e-9 * C[k, k]
        if A[k, k] <= 0:
            return k
        c = A[k + 1:, k] / math.sqrt(A[k, k])
        A[k + 1:, k + 1:] -= np.outer(c, c)
    return None


def _hyper(amplitude, core_var, r0, noise, r=0.1):
    return synth.Hyper(d=2, n1=1, n2=1, bump_dims=2, core_var=core_var, core_radius=np.full(2, 50.0), s0=0.0 if core_var < 0 else 1.0,
                       r0=np.full(2, r0), h=np.array([0.5, 0.5]), a=np.array([amplitude]), b=np.ones(1), r=np.full(1, r),
                       noise_var=noise)


def _grid(n, seed, jitter=0.2):
    rng = np.random.default_rng(seed)
    k = math.ceil(math.sqrt(n))
    g = np.stack(np.meshgrid(np.arange(k), np.arange(k)), -1).reshape(-1, 2)[:n]
    return (g + 0.5 + rng.uniform(-jitter, jitter, g.shape)) / k


def _check_flags(X, settings):
    """Batch of a good setting and `settings`: the flagged columns are the dense Cholesky's first failing pivots."""
    from paper_2411_05869_gb300 import gp
    n = len(X)
    good = _hyper(0.5, 1.0, 0.03, 0.3)
    hs = [good] + settings
    ctx = gp.Context(0)
    ps = ctx.assemble(_dev(X), good.core_radius)
    perm = ps.export("perm")
    want = [_first_failing(oracle.dense_cov(h, X)[np.ix_(perm, perm)]) for h in hs]
    f = ctx.factor(ps, hs, gp.GP_FP64)
    ll = f.loglik(_dev(np.ones((len(hs), n)))).cpu().numpy()
    info = f.info()
    got = [None if c < 0 else int(c) for c in info["not_pd_column"]]
    f.free()
    ps.free()
    assert got == want
    for v, w in zip(ll, want):
        assert v == -np.inf if w is not None else np.isfinite(v)
    return want


@pytest.mark.parametrize("noise", [-0.05, -0.9])
@pytest.mark.parametrize("n", [200, 600])
def test_pair_that_breaks_definiteness_is_flagged_at_its_own_column(n, noise):
    """Nearly uncorrelated points but one close pair, and a negative noise: the pair's later column fails, by a little or by
    far (its rows of L are then many times what their variances allow)."""
    seen = set()
    for seed in range(6):
        X = _grid(n, seed)
        rng = np.random.default_rng(100 + seed)
        i, j = rng.choice(n, 2, replace=False)
        X[i] = X[j] + 1e-4
        want = _check_flags(X, [_hyper(0.0, 1.0, 0.02, noise)])
        assert want[0] is None and want[1] is not None
        seen.add(want[1] // 64)
    assert len(seen) > 1   # several block columns


@pytest.mark.parametrize("ring", [40, 70, 120, 180, 240])
def test_variance_far_below_its_columns_share_is_flagged(ring):
    """C = tau^2 I - c f f^T with f large at one point: its row of L is as long as its variance allows in every column, and
    their squares add up to many times that."""
    n, radius = 320, 0.1
    rng = np.random.default_rng(ring)
    X = rng.uniform(3.0, 3.3, (n, 2))   # outside the bump
    phi = np.linspace(0, 2 * math.pi, ring, endpoint=False) + 0.01
    where = rng.permutation(n)
    X[where[:ring]] = 0.5 + radius * np.stack([np.cos(phi), np.sin(phi)], -1)
    X[where[ring]] = 0.5
    settings = []
    for share in (0.3, 0.45, 0.6, 0.75, 0.9):    # c |f_ring|^2: the ring alone is positive definite
        for var in (0.5, 0.1, 0.02, 0.004):      # 1 - c f_middle^2, the middle's variance (tau^2 = 1)
            c = 1 - var
            fk = math.sqrt(share / (c * ring))   # f on the ring: exp(1 - 1 / (1 - t))
            t = 1 - 1 / (1 - math.log(fk))
            settings.append(_hyper(1.0, -c, 0.02, 1.0, r=radius / math.sqrt(t)))
    want = _check_flags(X, settings)
    assert sum(w is not None for w in want) >= 10


def test_sparse_fronts_report_the_first_failing_column():
    from paper_2411_05869_gb300 import gp
    w = synth.spatial_2d(n=2500, m=1, seed=5, rho=0.15, noise_var=0.05)
    bad = w.hyper.copy()
    bad.noise_var = -2e-4
    ctx = gp.Context(0)
    ps = ctx.assemble(_dev(w.X), w.hyper.core_radius)
    perm = ps.export("perm")
    C = oracle.dense_cov(bad, w.X)[np.ix_(perm, perm)]
    A = C.copy()
    want = None
    for k in range(len(A)):
        if A[k, k] <= 0:
            want = k
            break
        c = A[k + 1:, k] / math.sqrt(A[k, k])
        nz = np.flatnonzero(c)
        A[np.ix_(k + 1 + nz, k + 1 + nz)] -= np.outer(c[nz], c[nz])
    f = ctx.factor(ps, [w.hyper, bad], gp.GP_FP64)
    cols = f.info()["not_pd_column"]
    assert cols[0] == -1 and want is not None and cols[1] == want


@pytest.mark.parametrize("where", ["alone", "pair", "pair_apart"])
def test_infinite_covariances(where):
    """A bump whose square overflows. One point inside: its variance is infinite, so is the log-determinant, and nothing
    else is affected; no pivot fails. Two points inside: their covariance is infinite too, and the later one fails."""
    from paper_2411_05869_gb300 import gp
    n = 300
    X = _grid(n, 3)
    d = np.linalg.norm(X - 0.5, axis=1)
    i, j = np.argsort(d)[:2]
    X[i] = 0.5
    if where != "alone":
        X[j] = 0.503
    huge = _hyper(1e160, 1.0, 0.03, 0.3, r=0.006)
    if where == "pair_apart":   # one point changes places with the pair's: other columns of the elimination order
        huge.h = huge.h * 0 + X[0]
        X[1] = X[0] + 0.003
    inside = np.flatnonzero(np.linalg.norm(X - huge.h, axis=1) < 0.006)
    assert len(inside) == (1 if where == "alone" else 2)
    good = _hyper(0.5, 1.0, 0.03, 0.3, r=0.006)
    good.h = huge.h.copy()
    ctx = gp.Context(0)
    ps = ctx.assemble(_dev(X), good.core_radius)
    f = ctx.factor(ps, [good, huge], gp.GP_FP64)
    ll = f.loglik(_dev(np.ones((2, n)))).cpu().numpy()
    pos = np.argsort(ps.export("perm"))[inside]
    assert np.isfinite(ll[0]) and ll[1] == -np.inf
    assert list(f.info()["not_pd_column"]) == [-1, -1 if where == "alone" else pos.max()]


@pytest.mark.parametrize("k", [-960, -1000, -40, 900])
@pytest.mark.parametrize("n", [200, 513])
def test_covariances_of_any_scale(n, k):
    """C times 2^k and r times 2^(k / 2) move the log-likelihood by -n k / 2 log 2 and nothing else: the entries of C keep
    their digits, down to 2^-74 of the variances where 2^-1000 leaves the normal range."""
    from paper_2411_05869_gb300 import gp
    w = synth.spatial_2d(n=n, m=1, seed=70 + n, rho=2.0, noise_var=0.1)
    h = w.hyper.copy()
    h.core_var, h.noise_var = math.ldexp(h.core_var, k), math.ldexp(h.noise_var, k)
    ctx = gp.Context(0)
    ps = ctx.assemble(_dev(w.X), w.hyper.core_radius)
    f = ctx.factor(ps, [w.hyper, h], gp.GP_FP64)
    ll = f.loglik(_dev(np.stack([w.normals, w.normals * 2.0 ** (k // 2)]))).cpu().numpy()
    want = ll[0] - 0.5 * n * k * math.log(2.0)
    # kappa <= 1e5 here: the quadratic form and the log-determinant are good to n kappa 2^-53 < 1e-8 at worst; a backward
    # error of 2^-53 in general position gives about sqrt(n) kappa 2^-53 of the quadratic form
    assert abs(ll[1] - want) <= 1e-11 * max(abs(want), abs(ll[0])), (ll, want)


def _reference(C, R):
    """Log-likelihoods of the residuals R (rows) by a Cholesky factorization in the matrix's own type."""
    A = C.copy()
    n = len(A)
    Y = R.T.astype(A.dtype).copy()
    logdet = A.dtype.type(0)
    for k in range(n):
        p = np.sqrt(A[k, k])
        logdet += 2 * np.log(p)
        c = A[k + 1:, k] / p
        Y[k] /= p
        Y[k + 1:] -= np.outer(c, Y[k])
        A[k + 1:, k + 1:] -= np.outer(c, c)
    return -(logdet + (Y * Y).sum(0) + n * np.log(2 * A.dtype.type(np.pi))) / 2


@pytest.mark.parametrize("noise", [1e-2, 1e-5, 1e-8])
@pytest.mark.parametrize("n", [130, 321])
def test_log_likelihoods_are_as_accurate_as_an_fp64_cholesky(n, noise):
    """Against extended precision, over several point sets and residuals: the root mean square error is at most 16 times
    that of a column-by-column FP64 elimination in the same order, whose backward error is a few units of 2^-53 of the
    variances; the device's covariances carry up to ten or so of their own. Digits cut one level short would give 2^-43."""
    from paper_2411_05869_gb300 import gp
    assert np.finfo(np.longdouble).nmant > 60
    ctx = gp.Context(0)
    got, host = [], []
    for seed in range(4):
        w = synth.spatial_2d(n=n, m=1, seed=900 + seed, rho=2.0, noise_var=noise)
        ps = ctx.assemble(_dev(w.X), w.hyper.core_radius)
        perm = ps.export("perm")
        C = oracle.csr_values(w.hyper, w.X, *oracle.pattern(w.X, w.hyper.core_radius)).reshape(n, n)
        C = C[np.ix_(perm, perm)]
        L = np.linalg.cholesky(C)
        for b in range(4):   # likely residuals and rough ones
            rng = np.random.default_rng(10 * seed + b)
            r = np.empty(n)
            r[perm] = L @ rng.standard_normal(n) if b % 2 else rng.standard_normal(n)
            f = ctx.factor(ps, [w.hyper], gp.GP_FP64)
            ll = float(f.loglik(_dev(r[None])).cpu()[0])
            f.free()
            ref = _reference(C.astype(np.longdouble), r[None, perm])[0]
            got.append(float((ll - ref) / ref))
            host.append(float((_reference(C, r[None, perm])[0] - ref) / ref))
        ps.free()
    rms = lambda v: math.sqrt(np.mean(np.square(v)))
    assert rms(got) <= 16 * rms(host), (rms(got), rms(host))


def test_digit_planes_take_no_memory_of_their_own_beside_update_matrices():
    """The operands of a level lie where its children's update matrices were: the factor of this plan takes 114,011,904
    bytes without them (panels, update matrices, inverses, values and the solves' vectors), and at most 1 % more with."""
    from paper_2411_05869_gb300 import gp
    w = synth.uniform_spacetime(9000, 0, 60.0, 16, 1, ndays=66)
    ctx = gp.Context(0)
    ps = ctx.assemble(_dev(w.X), w.hyper.core_radius)
    need = ps.factor_bytes(w.hyper, 1, gp.GP_FP64)
    assert need <= 1.01 * 114011904
    f = ctx.factor(ps, [w.hyper], gp.GP_FP64)
    assert f.info()["bytes"] == need
    f.free()
    ps.free()
