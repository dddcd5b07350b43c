"""Device memory of a problem, in FP64 grids of its size."""
import pytest

pytestmark = pytest.mark.gpu


# R, u and a work grid; FP64: the spectral scales; mixed: half a grid of FP32 work and
# two of fixed point.  The set-up takes 3.5 grids.
@pytest.mark.parametrize("precision,grids", [(0, 4.0), (1, 5.5)])
def test_grids_of_a_problem(precision, grids):
    import torch
    from paper_2309_05965_gb300 import kfbi
    n = 512

    def create():
        return kfbi.Problem(3, n, -1.0, 1.0, 3, [0.0, 0.0, 0.0, 0.1, 0.1, 0.1], kfbi.DIRICHLET_INTERIOR, kappa=1.0,
                            precision=precision)

    kfbi.Problem(2, 64, -1.0, 1.0, 1, [0.0, 0.0, 0.6, 0.5, 0.0], 0, precision=precision).close()
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    G = create()
    used = (free - torch.cuda.mem_get_info()[0]) / (8.0 * (n + 1) ** 3)
    G.close()
    print("grids", precision, used)
    assert used < grids + 3.5 + 0.5
