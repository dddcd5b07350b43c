"""FP64 sine-transform box solves of data among the subnormal numbers."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_util import dev, empty, host

pytestmark = pytest.mark.gpu

# the FFT kernel (32) and the fixed-point kernel
SIZES = [(2, 32), (3, 32), (2, 64), (2, 256), (2, 1024), (3, 64)]


@pytest.mark.parametrize("d,n", SIZES)
@pytest.mark.parametrize("e", [-1035, -1024, -1012])
def test_subnormal_data(d, n, e):
    """The solve of R 2^e is that of R times 2^e but for the roundings of what is
    stored and scaled to multiples of 2^-1074: half of one each, grown by at most N in
    every further transform and by the largest spectral scale (2/N)^d / |lambda|, |lambda| > 2 d."""
    from paper_2309_05965_gb300 import kfbi
    shape = (W.LS_ELLIPSE, [0.0, 0.0, 0.7, 0.6, 0.0]) if d == 2 else (W.LS_ELLIPSOID, [0.0, 0.0, 0.0, 0.75, 0.7, 0.65])
    G = kfbi.Problem(d, n, -1.0, 1.0, *shape, kfbi.DIRICHLET_INTERIOR, kappa=2.5, precision=kfbi.FP64)
    R = np.round(np.random.default_rng(n + d).standard_normal((n + 1,) * d) * 2.0 ** 20) / 2.0 ** 20
    assert np.array_equal(np.ldexp(np.ldexp(R, e), -e), R)
    out = []
    for x in (R, np.ldexp(R, e)):
        u = empty(G.grid_shape)
        kfbi.kfbi_box_solve(G.handle, dev(x), u)
        out.append(host(u))
    G.close()
    half, err = 2.0 ** -75, 0.0                       # in units of 2^-1000
    for _ in range(d):
        err = n * err + half
    err = (2.0 / n) ** d / (2 * d) * err + half
    for _ in range(d):
        err = n * err + half
    ref = np.ldexp(out[0], e + 1000)
    assert np.abs(ref).max() > 100 * err
    assert np.abs(np.ldexp(out[1], 1000) - ref).max() <= err + 1e-13 * np.abs(ref).max()
