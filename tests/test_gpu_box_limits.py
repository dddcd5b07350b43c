"""Box solves at the largest 3D grid the library takes."""
import math

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("box,precision,tol", [("dst", 1, 5e-12), ("mg", 1, 5e-12), ("dst", 0, 1e-12)])
def test_box_solve_1024_cubed(box, precision, tol):
    """The right-hand side of one discrete sine mode, whose solution is that mode.
    Bounds: those of the oracle tests."""
    import torch
    from paper_2309_05965_gb300 import kfbi
    n, kappa, mode = 1024, 1.0, (3, 5, 2)
    if torch.cuda.mem_get_info()[0] < 110e9:
        pytest.skip("needs 110 GB of free device memory")
    G = kfbi.Problem(3, n, -1.0, 1.0, 3, [0.0, 0.0, 0.0, 0.05, 0.05, 0.05], kfbi.DIRICHLET_INTERIOR, kappa=kappa,
                     precision=precision, box_solver=kfbi.BOX_MG if box == "mg" else kfbi.BOX_DST)
    x = torch.arange(n + 1, dtype=torch.float64, device="cuda")
    ax = [torch.sin(x * (math.pi * k / n)).reshape([-1 if i == j else 1 for j in range(3)])
          for i, k in enumerate(mode)]
    for s in ax:
        s.view(-1)[-1] = 0.0
    S = [math.sin(k * math.pi / (2 * n)) ** 2 for k in mode]
    s1, s2, h = sum(S), S[0] * S[1] + S[1] * S[2] + S[2] * S[0], 2.0 / n
    lam = (-4.0 * s1 + 8.0 / 3.0 * s2 - 4.0 / 3.0 * S[0] * S[1] * S[2]) / h ** 2 - kappa * (1.0 - s1 / 3.0)
    u = torch.zeros(G.grid_shape, dtype=torch.float64, device="cuda")
    kfbi.kfbi_box_solve(G.handle, ax[0] * ax[1] * ax[2] * lam, u)
    err = 0.0
    for i in range(0, n + 1, 64):
        err = max(err, float((u[i:i + 64] - ax[0][i:i + 64] * ax[1] * ax[2]).abs().max()))
    G.close()
    del u, ax
    torch.cuda.empty_cache()
    assert err < tol
