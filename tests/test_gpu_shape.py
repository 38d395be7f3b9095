"""The launch shape on trees whose octants several warps share (up to 76
blocks): it has no part in their walks, so bh_autotune must not choose one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1509_07370_gb300 import bhgrav as B  # noqa: E402
from paper_1509_07370_gb300 import meshgen as mg  # noqa: E402

pytestmark = pytest.mark.gpu


def field(level, extra, seed=0):
    m = mg.refined_mesh(level, level + extra, lambda lev, ijk: np.all(ijk == 0, axis=1))
    rho = np.random.Generator(np.random.PCG64(seed)).lognormal(size=m.nblocks * 512)
    return m, torch.as_tensor(rho.astype(np.float32)).cuda()


def built(level, extra, **opt):
    m, rho = field(level, extra)
    s = B.Solver(**opt)
    s.build(m.level, m.ijk, rho)
    return s, rho


@pytest.mark.parametrize("level,extra", [(0, 0), (0, 1), (1, 1), (2, 0), (2, 1)])  # 1 to 71 blocks
def test_autotune_of_a_small_tree_keeps_the_shape(level, extra):
    s, _ = built(level, extra)
    for theta in (0.3, 0.6, 0.9):
        assert s.autotune(theta) == (4, 1, 1, 0)  # the default: one group a take
    s.set_walk_shape(8, 2, 2)
    assert s.autotune(0.6) == (8, 2, 2, 0)
    want = s.potential(0.6).cpu().numpy()
    s.set_walk_shape(4, 1, 1, 1)  # the order is there, as for any tree
    assert np.array_equal(s.potential(0.6).cpu().numpy(), want)


def test_autotune_of_a_larger_tree_after_a_small_one():
    s, _ = built(2, 1)
    assert s.autotune(0.6) == (4, 1, 1, 0)
    m, rho = field(2, 2)  # 127 blocks
    s.build(m.level, m.ijk, rho)
    w, pairs, take, longest = s.autotune(0.6)
    assert w in (2, 4, 8, 16) and pairs in (1, 2) and take in (0, 1, 2, 4) and longest in (0, 1)


@pytest.mark.parametrize("level,extra", [(1, 1), (2, 2)])
def test_graph_as_the_first_walk_of_a_context(level, extra):
    s, rho = built(level, extra, stream=torch.cuda.Stream())
    out = torch.empty(s.ncells, device="cuda")
    s.solve_graph(rho, 0.5, 1.0, out)
    s.stream.synchronize()
    want = built(level, extra)[0].potential(0.5)
    assert torch.equal(out, want)
