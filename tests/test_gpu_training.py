"""The tiled gradient kernel of the learned correction at the edges of its
64-sample tiles, against the oracle's binary64 gradient: one sample, one less
and one more than a tile, several tiles with a ragged end."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O  # noqa: E402
from paper_1509_07370_gb300 import bhgrav as B  # noqa: E402
from paper_1509_07370_gb300 import learned as L  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 63, 64, 65, 1000])
def test_gradient_at_tile_edges(n):
    rng = np.random.default_rng(n)
    x = rng.normal(0, 1, (n, 10)).astype(np.float32)
    z = rng.normal(0, 1, n).astype(np.float32)
    w = (L.init_weights(3) + rng.normal(0, 0.1, B.MLP_NW)).astype(np.float32)
    dx, dz, dw = (torch.as_tensor(a).cuda() for a in (x, z, w))
    grad, loss = torch.empty(B.MLP_NW, device="cuda"), torch.empty(1, device="cuda")
    B.bh_mlp_grad(dx, dz, dw, grad, loss)
    want_loss, want = O.mlp_loss_grad(w.astype(np.float64), x.astype(np.float64),
                                      z.astype(np.float64))
    got = grad.cpu().numpy()
    # the bar of the parity test: binary32 sums against binary64
    assert np.abs(got - want).max() <= 1e-4 * np.abs(want).max()
    assert abs(float(loss.item()) - want_loss) <= 1e-4 * want_loss
