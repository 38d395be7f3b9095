"""The tensor-core network evaluation where a CTA takes several tiles of 128
rows (6 CTAs on each of the SMs take one each first) and where the features
allow no pair loads.

Bar: a row's value does not depend on where it lies: the bits of the same rows
in calls of at most one tile a CTA, which the other tests compare with the
oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1509_07370_gb300 import bhgrav as B  # noqa: E402
from paper_1509_07370_gb300 import learned as L  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset", [0, 1])  # words before the first feature
@pytest.mark.parametrize("tiles,more", [(1, -1), (1, 0), (1, 1), (2, 129), (3, -128)])
def test_several_tiles_a_cta(tiles, more, offset):
    once = 6 * torch.cuda.get_device_properties(0).multi_processor_count * 128
    n = tiles * once + more
    w = L.init_weights(5) + np.random.default_rng(1).normal(0, 0.05, B.MLP_NW).astype(np.float32)
    s = B.Solver(learned=True)
    s.set_mlp(w)
    g = torch.Generator(device="cuda").manual_seed(n)
    buf = torch.randn(10 * n + offset, generator=g, device="cuda")
    x = buf[offset:].view(n, 10)
    assert x.data_ptr() % 8 == 4 * offset
    got = s.mlp_eval(x)
    want = torch.cat([s.mlp_eval(p.clone()) for p in x.split(once // 2)])
    assert torch.isfinite(got).all() and torch.equal(got, want)
