"""Tree construction where its branches meet: masses and products that are
exact in binary64 beside ones that round.

Bar: the oracle's masses, centres of mass and extents, bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O  # noqa: E402
from paper_1509_07370_gb300 import bhgrav as B  # noqa: E402
from paper_1509_07370_gb300 import meshgen as mg  # noqa: E402

pytestmark = pytest.mark.gpu


def corner(level, extra):
    return mg.refined_mesh(level, level + extra, lambda lev, ijk: np.all(ijk == 0, axis=1))


@pytest.mark.parametrize("box_len", [1.0, 3.0, 2.0 ** -90, 2.0 ** 60])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("level,extra", [(0, 0), (1, 9)])
def test_moments_of_exact_and_rounded_products(box_len, dtype, level, extra):
    """Per bottom node a mix of ordinary, zero, subnormal, smallest normal and
    (binary64) full-length or short densities; sides of a power of two and not."""
    m = corner(level, extra)
    rng = np.random.Generator(np.random.PCG64(5))
    n = m.nblocks * 512
    rho = rng.lognormal(0.0, 2.0, n).astype(dtype)
    pick = rng.integers(0, 40, n)
    rho[pick == 0] = 0.0
    rho[pick == 1] = 1e-40
    rho[pick == 2] = np.finfo(np.float32).tiny
    if dtype == np.float64:
        short = rng.integers(0, 2, n // 8).repeat(8) == 1  # whole bottom nodes of 24-bit values
        rho[short] = rho[short].astype(np.float32)
    rho = rho.reshape(m.nblocks, 8, 8, 8)
    t = O.Tree(m.level, m.ijk, rho.astype(np.float64), box_len=box_len).export()
    s = B.Solver(precision=B.BH_PREC_F64 if dtype == np.float64 else B.BH_PREC_F32)
    s.build(m.level, m.ijk, torch.as_tensor(rho.reshape(-1)).cuda(), box_len=box_len)
    e = {k: v.cpu().numpy() for k, v in s.export_nodes().items()}
    t["delta"] = t["delta"].astype(np.float32)
    for k in ("M", "R", "delta"):
        assert np.array_equal(e[k], t[k]), k
