"""The FP64 factorization's bounded waits, made to run out on purpose (one poll, zero nanoseconds): the tensor-core kernels
wind down and the factor reports GP_ERR_TIMEOUT, a log-likelihood of NaN, and the context stays usable.

The limits of the context apply to the tensor-core kernels of both precisions; the waits inside a diagonal tile's cluster
keep the default limits. Nothing here faults: a wait that runs out is a return value.
"""
import numpy as np
import pytest

import oracle
from paper_2411_05869_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("batch", [1, 3])
def test_fp64_waits_that_run_out_report_timeout_and_the_context_recovers(batch):
    from paper_2411_05869_gb300 import gp
    w = synth.uniform_spacetime(12000, 0, 60.0, 8, seed=79, ndays=80)
    hp = w.hyper
    rp, col = oracle.pattern(w.X, hp.core_radius)
    perm = oracle.fill_order(w.X, hp.core_radius, rp, col)
    ref = oracle.sparse_loglik(hp, w.X, rp, col, perm, w.resid)["loglik"]
    ctx = gp.Context(0)
    ps = ctx.assemble(_dev(w.X), hp.core_radius)
    r = _dev(np.tile(w.resid, (batch, 1)))
    ctx.set_option("wait_polls", 1)
    ctx.set_option("wait_ns", 0)
    f = ctx.factor(ps, [hp] * batch, gp.GP_FP64)
    ctx.set_option("wait_polls", 1 << 26)
    ctx.set_option("wait_ns", 1_000_000_000)
    assert f.info(allow_timeout=True)["timed_out"] == 1
    f.update([hp] * batch)   # a factor keeps the limits it was made with
    assert f.info(allow_timeout=True)["timed_out"] == 1
    with pytest.raises(gp.GpError) as e:
        f.info()
    assert e.value.status == 5
    out = torch.empty(batch, dtype=torch.float64, device="cuda")
    f.loglik(r, out=out)   # asynchronous: the outputs tell
    torch.cuda.synchronize()
    assert np.isnan(out.cpu().numpy()).all()
    f.free()
    f2 = ctx.factor(ps, [hp] * batch, gp.GP_FP64)
    assert f2.info()["timed_out"] == 0
    for ll in f2.loglik(r).cpu().numpy():
        assert abs(ll - ref) <= 1e-10 * abs(ref), (ll, ref)
    f2.free()
    ps.free()
