"""The batched transform passes with few work items, and with more than one row of
their grid holds: every instance as by itself."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_util import dev, empty, host, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [(8,), (64,), (16, 1024, 32), (1024, 512, 1024, 1024), (128,) * 40 + (256,) * 40])
def test_batch_equals_single_evaluations(sizes):
    """Bound: the 1e-9 between batched and single evaluations of the batch tests.  The
    single problems' data before the batched solve leave no trace in it."""
    from paper_2309_05965_gb300 import kfbi
    rng = np.random.default_rng(len(sizes))
    ps = [kfbi.Problem(2, n, -1.0, 1.0, W.LS_ELLIPSE, [0.0, 0.0, 0.7, 0.6, 0.0], kfbi.DIRICHLET_INTERIOR, kappa=1.0,
                       precision=kfbi.MIXED, order=2 if n < 32 else 4) for n in sizes]
    B = kfbi.Batch(ps)
    keep = [dict(g1=dev(rng.standard_normal(P.nb)), f_in=dev(rng.standard_normal(P.grid_shape))) for P in ps]
    ds = [kfbi.make_data(**k) for k in keep]
    opts = kfbi.GmresOpts(rtol=1e-8, restart=100, max_iter=100, x0=None)
    x = [empty(P.nb) for P in ps]
    B.gmres_solve(ds, opts, x)
    first = [host(v).copy() for v in x]
    us = [empty(P.grid_shape) for P in ps]
    B.evaluate(ds, x, us)
    for P, d, v, u in zip(ps, ds, x, us):
        one = empty(P.grid_shape)
        kfbi.kfbi_evaluate(P.handle, d, v, one)
        assert rel_err(host(u), host(one)) < 1e-9
    B.gmres_solve(ds, opts, x)
    for v, a in zip(x, first):
        assert np.array_equal(host(v), a)
    B.close()
