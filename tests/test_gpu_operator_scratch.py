"""The operator keeps a right-hand side of its own, and expects zeros on the
boundary layer of its solution: neither may show what data with sources and
outer boundary values left behind."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_util import dev, empty, host

pytestmark = pytest.mark.gpu


def _problem(name):
    from paper_2309_05965_gb300 import kfbi
    if name == "spheres":      # general kind: two box operators, several interfaces
        return kfbi.Problem.from_workload(W.hetero_spheres_3d(64))
    kw = {"fp64": dict(precision=kfbi.FP64), "mixed": dict(precision=kfbi.MIXED),
          "mg": dict(precision=kfbi.FP64, box_solver=kfbi.BOX_MG)}[name]
    # an interface whose trace stencils come near the edge of the box
    return kfbi.Problem(2, 64, -1.0, 1.0, 2, [0.0, 0.0, 0.75, 0.1, 5.0], kfbi.INTERFACE_MU, sigma_in=10.0, **kw)


@pytest.mark.parametrize("name", ["fp64", "mixed", "mg", "spheres"])
def test_operator_is_the_same_after_solves_with_data(name):
    import torch
    from paper_2309_05965_gb300 import kfbi
    P = _problem(name)
    size = P.nb * (2 if name == "spheres" else 1)
    rng = np.random.default_rng(5)
    x, y = dev(rng.standard_normal(size)), empty(size)
    kfbi.kfbi_apply_operator(P.handle, x, y)
    first = host(y).copy()
    keep = {k: dev(rng.standard_normal(P.grid_shape)) for k in ("f_in", "f_out", "lapf_in", "lapf_out", "g_b")}
    keep.update(g1=dev(rng.standard_normal(P.nb)), g2=dev(rng.standard_normal(P.nb)))
    data, u, b = kfbi.make_data(**keep), empty(P.grid_shape), empty(size)

    kfbi.kfbi_bie_rhs(P.handle, data, b)
    kfbi.kfbi_apply_operator(P.handle, x, y)
    assert np.array_equal(host(y), first)
    kfbi.kfbi_evaluate(P.handle, data, x, u)
    kfbi.kfbi_apply_operator(P.handle, x, y)
    assert np.array_equal(host(y), first)
    b_first = host(b).copy()
    kfbi.kfbi_bie_rhs(P.handle, data, b)
    assert np.array_equal(host(b), b_first)
    torch.cuda.synchronize()
    P.close()
