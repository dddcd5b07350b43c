"""Network gradients at the edges of the GEMM tiles: widths and input counts
that are and are not multiples of four, under and over a 64-wide tile, with
row counts around a CTA's share."""
import numpy as np
import pytest

from oracle import mlp as OM
from tests.gpu_util import empty, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_in,width,n", [(1, 1, 1), (5, 20, 33), (16, 64, 32), (3, 65, 129), (16, 100, 700), (7, 300, 31)])
def test_gradient_matches_oracle(n_in, width, n):
    """FP32 sums against FP64 at the same rounded weights: the bounds of the
    network tests at width 256 (2e-5 outputs, 1e-4 gradients)."""
    import torch
    from paper_2309_05965_gb300 import kfbi
    rng = np.random.default_rng(width + n)
    flat = rng.standard_normal(width * (n_in + width + 3) + 1 + n_in).astype(np.float32) / np.float32(np.sqrt(width))
    P = OM.Params.from_flat(flat.astype(np.float64), n_in, width)
    m = kfbi.kfbi_mlp_create(n_in, width)
    kfbi.kfbi_mlp_set_params(m, torch.from_numpy(flat).cuda())
    kfbi.kfbi_mlp_set_affine(m, np.zeros(n_in), np.ones(n_in), 0.0, 1.0)
    X, t = rng.standard_normal((n, n_in)).astype(np.float32), rng.standard_normal(n).astype(np.float32)
    Xd, y, loss, g = torch.from_numpy(X).cuda(), empty(n, "f32"), empty(1, "f32"), empty(flat.size, "f32")
    kfbi.kfbi_mlp_forward(m, Xd, y)
    kfbi.kfbi_mlp_loss_grad(m, Xd, torch.from_numpy(t).cuda(), loss=loss)
    kfbi.kfbi_mlp_get_params(m, grads=g)
    y_ref, _ = OM.forward(P, X.astype(np.float64))
    L_ref, G_ref = OM.loss_and_grad(P, X.astype(np.float64), t.astype(np.float64))
    assert np.abs(host(y) - y_ref).max() < 2e-5 * max(1.0, np.abs(y_ref).max())
    assert abs(float(host(loss)[0]) - L_ref) <= 2e-5 * L_ref
    gg = OM.Params.from_flat(host(g).astype(np.float64), n_in, width)
    top = max(np.abs(v).max() for v in (G_ref.W1, G_ref.W2, G_ref.W3))
    for name in ("W1", "b1", "W2", "b2", "W3", "b3", "WL"):
        a, b = getattr(gg, name), getattr(G_ref, name)
        assert np.abs(a - b).max() < 1e-4 * max(np.abs(b).max(), 1e-2 * top), name
    kfbi.kfbi_mlp_destroy(m)
