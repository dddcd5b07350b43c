"""The FP64 sine-transform box solve on the tensor cores (fixed-point lines):
wide ranges within a line, scaling by powers of two, non-finite data."""
import numpy as np
import pytest

import workloads as W
from oracle import boxsolve as BS
from tests.gpu_util import dev, empty, host

pytestmark = pytest.mark.gpu

# every transform length of the kernel; few and many line groups
SIZES = [(2, 64), (2, 128), (2, 256), (2, 512), (2, 1024), (3, 64), (3, 128)]


def _problem(d, n):
    from paper_2309_05965_gb300 import kfbi
    w = W.ellipse_dirichlet_2d(n) if d == 2 else W.torus_helmholtz_3d(n)
    w.kappa = 2.5
    return w, kfbi.Problem.from_workload(w, precision=kfbi.FP64)


def _solve(G, R):
    from paper_2309_05965_gb300 import kfbi
    u = empty(G.grid_shape)
    kfbi.kfbi_box_solve(G.handle, dev(R), u)
    return host(u)


@pytest.mark.parametrize("d,n", SIZES)
def test_lines_of_wide_range(d, n):
    """Peaks 10^6 times the rest: FP64 rounding of a transform of log2(2N)
    stages, per axis and direction, on both sides of the comparison."""
    w, G = _problem(d, n)
    rng = np.random.default_rng(n + d)
    R = rng.standard_normal((n + 1,) * d)
    peaks = rng.integers(1, n, size=(40, d))
    R[tuple(peaks.T)] *= 1e6
    ref = BS.dst_solve(R, d, 4, w.h, w.kappa)
    tol = 2 * 2 * d * np.log2(2 * n) * 2.0 ** -53
    assert np.linalg.norm(_solve(G, R) - ref) <= tol * np.linalg.norm(ref)


@pytest.mark.parametrize("d,n", [(2, 64), (2, 256), (2, 1024), (3, 64)])
def test_power_of_two_scaling_is_exact(d, n):
    """Lines are scaled by their own exponent, so a power of two passes through
    bit for bit, also far from 1."""
    _, G = _problem(d, n)
    R = np.random.default_rng(7).standard_normal((n + 1,) * d)
    u = _solve(G, R)
    for e in (-900, -40, 600):
        assert np.array_equal(_solve(G, np.ldexp(R, e)), np.ldexp(u, e))
    assert not _solve(G, np.zeros_like(R)).any()


@pytest.mark.parametrize("d,n", [(2, 64), (2, 512), (3, 64)])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_nonfinite_data_reach_every_node(d, n, bad):
    _, G = _problem(d, n)
    R = np.ones((n + 1,) * d)
    R[(n // 3,) * d] = bad
    u = _solve(G, R)
    assert not np.isfinite(u[(slice(1, n),) * d]).any()
