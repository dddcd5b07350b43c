"""The boundary layer of a mixed box solve's output is zero whatever the buffer
held and however many refinement steps ran, also of non-finite data."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_util import dev, host

pytestmark = pytest.mark.gpu


def _layer(u, d, n):
    return np.concatenate([np.take(u, [0, n], axis=a).ravel() for a in range(d)])


def _solve(G, R, fill):
    import torch
    from paper_2309_05965_gb300 import kfbi
    u = torch.full(G.grid_shape, fill, dtype=torch.float64, device="cuda")
    kfbi.kfbi_box_solve(G.handle, dev(R), u)
    return host(u)


@pytest.mark.parametrize("d,n,order", [(2, 8, 2), (2, 64, 4), (2, 256, 4), (3, 16, 2), (3, 32, 4), (3, 64, 4)])
@pytest.mark.parametrize("steps,rtol", [(1, 0.0), (2, 1e-30), (3, 1e-30), (4, 1e-11)])
def test_layer_is_zero(d, n, order, steps, rtol):
    """steps, rtol: no refinement, every step run (no correction is ever below
    1e-30 of the solution), a refinement that stops before its last step."""
    from paper_2309_05965_gb300 import kfbi
    shape = (W.LS_ELLIPSE, [0.0, 0.0, 0.7, 0.6, 0.0]) if d == 2 else (W.LS_ELLIPSOID, [0.0, 0.0, 0.0, 0.75, 0.7, 0.65])
    G = kfbi.Problem(d, n, -1.0, 1.0, *shape, kfbi.DIRICHLET_INTERIOR, kappa=1.0, precision=kfbi.MIXED, order=order,
                     box_max_iters=steps, box_rtol=rtol)
    R = np.random.default_rng(n + steps).standard_normal(G.grid_shape)
    a, b = _solve(G, R, 3.0), _solve(G, R, np.nan)
    assert not _layer(a, d, n).any() and not _layer(b, d, n).any()
    assert np.array_equal(a, b) and a.any()
    R[(n // 2,) * d] = np.nan
    c = _solve(G, R, 3.0)
    assert not _layer(c, d, n).any()
    assert not np.isfinite(c[(slice(1, n),) * d]).any()
    G.close()


@pytest.mark.parametrize("kind", ["mu", "spheres"])
def test_operator_after_nonfinite_solve(kind):
    """The operator is the same after an application to NaN data."""
    from paper_2309_05965_gb300 import kfbi
    from tests.gpu_util import empty
    if kind == "spheres":
        G = kfbi.Problem.from_workload(W.hetero_spheres_3d(64), precision=kfbi.MIXED, box_max_iters=2, box_rtol=1e-30)
    else:
        # an interface whose trace stencils come near the edge of the box
        G = kfbi.Problem(2, 64, -1.0, 1.0, W.LS_STAR, [0.0, 0.0, 0.75, 0.1, 5.0], kfbi.INTERFACE_MU, sigma_in=10.0,
                         precision=kfbi.MIXED, box_max_iters=2, box_rtol=1e-30)
    size = G.nb * (2 if kind == "spheres" else 1)
    x, y = dev(np.random.default_rng(3).standard_normal(size)), empty(size)
    kfbi.kfbi_apply_operator(G.handle, x, y)
    first = host(y).copy()
    assert np.isfinite(first).all()
    kfbi.kfbi_apply_operator(G.handle, dev(np.full(size, np.nan)), y)
    assert not np.isfinite(host(y)).all()
    kfbi.kfbi_apply_operator(G.handle, x, y)
    assert np.array_equal(host(y), first)
    G.close()


@pytest.mark.parametrize("steps", [1, 2])
def test_layer_of_batched_evaluation(steps):
    """A batch without and with refinement, one instance of NaN data."""
    from paper_2309_05965_gb300 import kfbi
    from tests.gpu_util import empty
    ps = [kfbi.Problem(2, n, -1.0, 1.0, W.LS_ELLIPSE, [0.0, 0.0, 0.7, 0.6, 0.0], kfbi.DIRICHLET_INTERIOR,
                       precision=kfbi.MIXED, box_max_iters=steps, box_rtol=1e-30) for n in (64, 128)]
    B = kfbi.Batch(ps)
    x = [dev(np.random.default_rng(P.n).standard_normal(P.nb)) for P in ps]
    x[0][5] = float("nan")
    us = [dev(np.full(P.grid_shape, 3.0)) for P in ps]
    B.evaluate([kfbi.make_data(g1=empty(P.nb)) for P in ps], x, us)
    for P, u in zip(ps, us):
        assert not _layer(host(u), 2, P.n).any()
    assert np.isfinite(host(us[1])).all() and host(us[1]).any() and np.isnan(host(us[0])).any()
    B.close()
