"""Batched evaluation into the buffers that hold the outer boundary values."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_util import dev, empty, host

pytestmark = pytest.mark.gpu


def test_batch_evaluates_into_its_boundary_data():
    """Instances 0 and 1 share one grid of boundary values, which is also the
    output of instance 0; instance 2 writes into its own."""
    from paper_2309_05965_gb300 import kfbi
    shapes = [(128, 0.5), (128, 0.45), (64, 0.55)]
    ps = [kfbi.Problem(2, n, -1.0, 1.0, W.LS_STAR, [0.0, 0.0, r, 0.05, 3.0], kfbi.INTERFACE_MU, sigma_in=10.0,
                       precision=kfbi.MIXED) for n, r in shapes]
    B = kfbi.Batch(ps)
    rng = np.random.default_rng(11)
    gb = [rng.standard_normal(P.grid_shape) for P in ps]
    gb[1] = gb[0]
    jumps = [(dev(rng.standard_normal(P.nb)), dev(rng.standard_normal(P.nb))) for P in ps]
    x = [dev(rng.standard_normal(P.nb)) for P in ps]

    def evaluate(grids, us):
        B.evaluate([kfbi.make_data(g1=a, g2=b, g_b=g) for (a, b), g in zip(jumps, grids)], x, us)
        return [host(u).copy() for u in us]

    apart = [dev(g) for g in gb]
    ref = evaluate(apart, [empty(P.grid_shape) for P in ps])
    y = [empty(P.nb) for P in ps]
    for P, xi, yi in zip(ps, x, y):
        kfbi.kfbi_apply_operator(P.handle, xi, yi)
    before = [host(v).copy() for v in y]
    shared, own = dev(gb[0]), dev(gb[2])
    got = evaluate([shared, shared, own], [shared, empty(ps[1].grid_shape), own])
    for a, b, g in zip(got, ref, gb):
        assert np.array_equal(a, b)
        assert np.array_equal(a[0], g[0]) and np.array_equal(a[:, -1], g[:, -1])
    # the outer data stay out of the operator
    for P, xi, yi, b in zip(ps, x, y, before):
        kfbi.kfbi_apply_operator(P.handle, xi, yi)
        assert np.array_equal(host(yi), b)
    B.close()
