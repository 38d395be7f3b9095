"""Tree construction where its branches meet: masses and products that are
exact in binary64 beside ones that round, and the two block sorts.

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


def test_shuffled_fields_of_a_batch_are_sorted_by_themselves():
    """1, 519 and 8 blocks, listed in random order, in one batch: the sort
    counts each field's blocks alone."""
    rng = np.random.Generator(np.random.PCG64(9))
    fs = []
    for i, (level, extra) in enumerate([(0, 0), (3, 1), (1, 0)]):
        m = corner(level, extra)
        fs.append(mg.shuffled(m, rng.lognormal(size=(m.nblocks, 8, 8, 8)).astype(np.float32), i))
    s = B.Solver()
    s.build_batch([m.nblocks for m, _ in fs], np.concatenate([m.level for m, _ in fs]),
                  np.concatenate([m.ijk for m, _ in fs]),
                  torch.as_tensor(np.concatenate([r.reshape(-1) for _, r in fs])).cuda())
    e = {k: v.cpu().numpy() for k, v in s.export_nodes().items()}
    at = 0
    for m, rho in fs:
        t = O.Tree(m.level, m.ijk, rho.astype(np.float64)).export()
        n = t["M"].size
        assert np.array_equal(e["M"][at:at + n], t["M"]) and np.array_equal(e["R"][at:at + n], t["R"])
        at += n
    assert at == e["M"].size


def split_first(level, split):
    """All cubes of `level` with the first `split` of them refined once, in
    Morton order."""
    n = 1 << level
    ijk = np.stack(np.meshgrid(*[np.arange(n)] * 3, indexing="ij"), -1).reshape(-1, 3)
    fine = (2 * ijk[:split, None, :] + np.indices((2, 2, 2)).reshape(3, 8).T).reshape(-1, 3)
    lev = np.r_[np.full(len(ijk) - split, level), np.full(len(fine), level + 1)].astype(np.int32)
    ijk = np.concatenate([ijk[split:], fine]).astype(np.int32)
    key = np.zeros(len(lev), np.int64)  # Morton key of the lower corner at the finer level
    c = ijk.astype(np.int64) << (level + 1 - lev)[:, None]
    for b in range(level + 1):
        for d in range(3):
            key |= ((c[:, d] >> b) & 1) << (3 * b + d)
    order = np.argsort(key)
    return lev[order], ijk[order]


@pytest.mark.parametrize("split", [585, 586])
def test_trees_around_one_tile_of_the_scan(split):
    """8,191 and 8,198 blocks: the scan's tile holds 8,192."""
    lev, ijk = split_first(4, split)
    rho = np.random.default_rng(3).random((len(lev), 512), dtype=np.float32)
    t = O.Tree(lev, ijk, rho.reshape(-1, 8, 8, 8).astype(np.float64)).export()
    s = B.Solver()
    s.build(lev, ijk, torch.as_tensor(rho.reshape(-1)).cuda())
    e = {k: v.cpu().numpy() for k, v in s.export_nodes().items()}
    assert np.array_equal(e["level"], t["level"]) and np.array_equal(e["M"], t["M"])


@pytest.mark.parametrize("split", [4681, 4682])
def test_both_sorts_restore_the_morton_order(split):
    """65,535 blocks (sorted by counting) and 65,542 (by radix), listed in
    random order: the tree of the list in Morton order, whose potentials and
    masses the other tests compare with the oracle."""
    lev, ijk = split_first(5, split)
    rho = torch.rand((len(lev), 512), generator=torch.Generator().manual_seed(1))
    trees = []
    for p in (np.arange(len(lev)), np.random.default_rng(2).permutation(len(lev))):
        s = B.Solver()
        s.build(np.ascontiguousarray(lev[p]), np.ascontiguousarray(ijk[p]),
                rho[torch.as_tensor(p)].reshape(-1).cuda())
        trees.append(s.export_nodes())
    for k in ("level", "M", "R"):
        assert torch.equal(trees[0][k], trees[1][k]), k


@pytest.mark.parametrize("extra", [1, 10, 11, 18])
@pytest.mark.parametrize("shuffled", [False, True])
def test_children_of_top_nodes_in_deep_trees(extra, shuffled):
    """Top nodes of every level at one corner (8, 463 blocks: the geometry in
    one launch; 519 and 911: in several), alone and as the last of a batch
    behind single blocks and a shallow tree, whose slots come first: the
    oracle's tree and masses, which the child lists carry upwards."""
    m = corner(0, extra)
    rng = np.random.Generator(np.random.PCG64(extra))
    fs = [(corner(l, e), None) for l, e in ((0, 0), (1, 1), (0, 0))] + [(m, None)]
    fs = [(x, rng.lognormal(size=(x.nblocks, 8, 8, 8)).astype(np.float32)) for x, _ in fs]
    if shuffled:
        fs = [mg.shuffled(x, r, i) for i, (x, r) in enumerate(fs)]
    s = B.Solver()
    for batch in ([fs[-1]], fs):
        s.build_batch([x.nblocks for x, _ in batch], np.concatenate([x.level for x, _ in batch]),
                      np.concatenate([x.ijk for x, _ in batch]),
                      torch.as_tensor(np.concatenate([r.reshape(-1) for _, r in batch])).cuda())
        e = {k: v.cpu().numpy() for k, v in s.export_nodes().items()}
        at = 0
        for x, rho in batch:
            t = O.Tree(x.level, x.ijk, rho.astype(np.float64)).export()
            n = t["M"].size
            for k in ("level", "M", "R"):
                assert np.array_equal(e[k][at:at + n], t[k]), k
            at += n
        assert at == e["M"].size


def test_device_bytes_of_the_binary64_arrays():
    """What a binary64 context holds more than a binary32 one of the same tree:
    a 32-byte moment for every place in sibling order (72 a block, 8 for each of
    nb // 7 + 1 top nodes) and 8 bytes a cell."""
    for m in (corner(0, 0), corner(2, 2), corner(4, 0)):
        nb, held = m.nblocks, []
        rho = torch.ones(512 * nb, device="cuda")
        for prec in (B.BH_PREC_F32, B.BH_PREC_F64):
            s = B.Solver(precision=prec)
            s.build(m.level, m.ijk, rho)
            held.append(s.stats()["device_bytes"])
        assert held[1] - held[0] == 32 * (72 * nb + 8 * (nb // 7 + 1)) + 8 * 512 * nb
