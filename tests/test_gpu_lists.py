"""The list walk (siblings tested eight at a time, accepted nodes and opened
bottom nodes collected per sub-brick and row) where its stack, rings and lists
run full or nearly empty: meshes refined about one corner (deep, ragged trees),
small opening angles (many opened nodes per octant), one block.

Bars: opening decisions equal the oracle's exactly; potentials within 1e-5 of
the oracle's walk (the binary32 bar of the parity tests) or 1e-12 (binary64);
a field in a batch keeps the bits of its own solve, whatever the depth of the
others."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O  # noqa: E402
from paper_1509_07370_gb300 import bhgrav as B  # noqa: E402
from paper_1509_07370_gb300 import meshgen as mg  # noqa: E402

pytestmark = pytest.mark.gpu


def corner(level, extra):
    return mg.refined_mesh(level, level + extra, lambda lev, ijk: np.all(ijk == 0, axis=1))


def field(level, extra, seed):
    m = corner(level, extra)
    rng = np.random.Generator(np.random.PCG64(seed))
    return m, rng.lognormal(0.0, 1.5, size=(m.nblocks, 8, 8, 8)).astype(np.float32)


CASES = [(0, 0, 0.3), (0, 4, 0.12), (1, 2, 0.25), (2, 1, 1.0), (1, 9, 0.6)]


@pytest.mark.parametrize("level,extra,theta", CASES)
@pytest.mark.parametrize("vote", [False, True])
def test_decisions_and_potentials_match_oracle(level, extra, theta, vote):
    m, rho = field(level, extra, 10 * level + extra)
    t = O.Tree(m.level, m.ijk, rho.astype(np.float64))
    for quad in (False, True):
        s = B.Solver(criterion=B.BH_CRIT_WARP_VOTE if vote else B.BH_CRIT_PER_CELL,
                     quadrupole=quad)
        s.build(m.level, m.ijk, torch.as_tensor(rho.reshape(-1)).cuda())
        got = s.potential(theta).cpu().numpy().astype(np.float64)
        ni, nt = (x.cpu().numpy() for x in s.walk_counts(theta))
        if vote:  # (32 cells per brick in local Morton order)
            got, ni, nt = (x.reshape(-1, 512)[:, O.local_morton_order()].reshape(-1)
                           for x in (got, ni, nt))
            want, wi, wt = t.walk_vote(theta, quad=quad)
        else:
            want, wi, wt = t.walk(theta, quad=quad)
        assert np.array_equal(ni, wi) and np.array_equal(nt, wt)
        assert np.max(np.abs(got / want - 1.0)) <= 1e-5


@pytest.mark.parametrize("quad", [False, True])
def test_deep_and_shallow_fields_keep_their_bits_in_a_batch(quad):
    fs = [field(1, 14, 1), field(0, 0, 2), field(1, 1, 3), field(0, 5, 4)]
    nb = [m.nblocks for m, _ in fs]
    s = B.Solver(quadrupole=quad)
    rho = torch.as_tensor(np.concatenate([r.reshape(-1) for _, r in fs])).cuda()
    s.build_batch(nb, np.concatenate([m.level for m, _ in fs]),
                  np.concatenate([m.ijk for m, _ in fs]), rho)
    got = s.potential(0.4).cpu().numpy()
    at = 0
    for m, r in fs:
        a = B.Solver(quadrupole=quad)
        a.build(m.level, m.ijk, torch.as_tensor(r.reshape(-1)).cuda())
        want = a.potential(0.4).cpu().numpy()
        assert np.array_equal(got[at:at + want.size], want)
        at += want.size


@pytest.mark.parametrize("level,extra", [(0, 0), (0, 1), (3, 0), (3, 1)])
@pytest.mark.parametrize("shuffled", [False, True])
def test_block_lists_around_the_small_geometry_limit(level, extra, shuffled):
    """1, 8, 512 (the most that one launch takes) and 519 blocks, in Morton
    order and shuffled: the oracle's tree and masses, bit for bit."""
    m, rho = field(level, extra, 77)
    if shuffled:
        m, rho = mg.shuffled(m, rho, seed=3)
    t = O.Tree(m.level, m.ijk, rho.astype(np.float64)).export()
    s = B.Solver()
    s.build(m.level, m.ijk, torch.as_tensor(rho.reshape(-1)).cuda())
    e = {k: v.cpu().numpy() for k, v in s.export_nodes().items()}
    assert np.array_equal(e["level"], t["level"]) and np.array_equal(e["M"], t["M"])
    assert np.array_equal(e["R"], t["R"])


@pytest.mark.parametrize("kahan", [True, False])
@pytest.mark.parametrize("quad,vote", [(False, False), (True, False), (True, True)])
def test_octants_shared_by_warps_keep_their_bits(kahan, quad, vote):
    """1, 15, 36 (4 warps to an octant), 64 and 71 blocks (2 warps) alone: the
    bits that the fields have in a batch of 187 blocks, a warp to an octant."""
    fs = [field(0, 0, 1), field(1, 1, 2), field(0, 5, 3), field(2, 0, 4), field(2, 1, 5)]
    crit = B.BH_CRIT_WARP_VOTE if vote else B.BH_CRIT_PER_CELL
    s = B.Solver(criterion=crit, quadrupole=quad, kahan=kahan)
    s.build_batch([m.nblocks for m, _ in fs], np.concatenate([m.level for m, _ in fs]),
                  np.concatenate([m.ijk for m, _ in fs]),
                  torch.as_tensor(np.concatenate([r.reshape(-1) for _, r in fs])).cuda())
    got = s.potential(0.5).cpu().numpy()
    at = 0
    for m, r in fs:
        a = B.Solver(criterion=crit, quadrupole=quad, kahan=kahan)
        a.build(m.level, m.ijk, torch.as_tensor(r.reshape(-1)).cuda())
        want = a.potential(0.5).cpu().numpy()
        assert np.array_equal(got[at:at + want.size], want)
        at += want.size


@pytest.mark.parametrize("level,extra", [(1, 0), (2, 0), (2, 3)])
@pytest.mark.parametrize("quad", [False, True])
def test_sums_of_a_cell_that_holds_the_mass_stay_compensated(level, extra, quad):
    """8, 64 and 239 blocks (4, 2 and 1 warps to an octant).  A cell is no term
    of its own sum and of no node that it accepts, so its potential is the same
    sum of the same terms whether it is empty or holds 10^7 times the mass of
    the others (the mass unit is a power of two).  Compensated sums of some
    1,000 terms are within 2^-35 of it, so both round to the same value but
    for one case in some 2^10 (in 2^5 for sums that start from zero: the
    rounding of their first terms), and the factor -G/L that follows keeps
    neighbours within two units in the last place; uncompensated ones are
    about 2^-23 apart."""
    m, rho = field(level, extra, 31)
    vol = np.repeat(8.0 ** -m.level.astype(np.float64), 512)
    rho = rho.reshape(-1)
    total = float((rho * vol).sum())
    s = B.Solver(quadrupole=quad)
    cells = np.random.default_rng(level + extra).choice(rho.size, 40, replace=False)
    same = 0
    for c in cells:
        phi = []
        for heavy in (0.0, 1e7 * total / vol[c]):
            r = rho.copy()
            r[c] = heavy
            s.build(m.level, m.ijk, torch.as_tensor(r).cuda())
            phi.append(s.potential(0.4)[int(c)].item())
        assert abs(phi[1] / phi[0] - 1.0) <= 2.0 ** -22
        same += phi[0] == phi[1]
    assert same >= 30


@pytest.mark.parametrize("depth", [16, 17, 18])
@pytest.mark.parametrize("theta", [0.35, 0.8])
def test_deepest_meshes_match_the_oracle(depth, theta):
    """Blocks down to levels 16 to 18 about opposite corners of the box, where the
    stack has little or no room for four nodes of any kind: sampled cells of
    every level."""
    m = mg.refined_mesh(1, depth, lambda lev, ijk: np.all(ijk == 0, axis=1) |
                        np.all(ijk == (1 << lev) - 1, axis=1))
    rng = np.random.Generator(np.random.PCG64(depth))
    rho = rng.lognormal(0.0, 1.5, size=(m.nblocks, 8, 8, 8)).astype(np.float32)
    tg = 512 * np.arange(m.nblocks) + rng.integers(0, 512, m.nblocks)
    t = O.Tree(m.level, m.ijk, rho.astype(np.float64))
    for quad in (False, True):
        want, wi, wt = t.walk(theta, targets=tg, quad=quad)
        for prec, bar in ((B.BH_PREC_F32, 1e-5), (B.BH_PREC_F64, 1e-12)):
            s = B.Solver(precision=prec, quadrupole=quad)
            s.build(m.level, m.ijk, torch.as_tensor(rho.reshape(-1)).cuda())
            got = s.potential(theta).cpu().numpy().astype(np.float64)[tg]
            ni, nt = (x.cpu().numpy()[tg] for x in s.walk_counts(theta))
            assert np.array_equal(ni, wi) and np.array_equal(nt, wt)
            assert np.max(np.abs(got / want - 1.0)) <= bar


@pytest.mark.parametrize("level,extra,theta", CASES)
@pytest.mark.parametrize("vote", [False, True])
def test_binary64_walk_matches_oracle(level, extra, theta, vote):
    """Terms within 2 2^-53 each and plain sums of runs of up to some 600 terms:
    an rms error of about 2^-53 (2 + sqrt(600) / 2), 1.6e-15, and 1e-14 is six
    times that (the oracle's own sums are compensated)."""
    m, rho = field(level, extra, 10 * level + extra)
    t = O.Tree(m.level, m.ijk, rho.astype(np.float64))
    for quad in (False, True):
        s = B.Solver(precision=B.BH_PREC_F64, quadrupole=quad,
                     criterion=B.BH_CRIT_WARP_VOTE if vote else B.BH_CRIT_PER_CELL)
        s.build(m.level, m.ijk, torch.as_tensor(rho.reshape(-1)).cuda())
        got = s.potential(theta).cpu().numpy()
        if vote:
            got = got.reshape(-1, 512)[:, O.local_morton_order()].reshape(-1)
        want = (t.walk_vote if vote else t.walk)(theta, quad=quad)[0]
        assert np.max(np.abs(got / want - 1.0)) <= 1e-14


@pytest.mark.parametrize("quad", [False, True])
def test_binary64_fields_keep_their_bits_in_a_batch(quad):
    fs = [field(1, 14, 1), field(0, 0, 2), field(1, 1, 3), field(0, 5, 4)]
    s = B.Solver(precision=B.BH_PREC_F64, quadrupole=quad)
    s.build_batch([m.nblocks for m, _ in fs], np.concatenate([m.level for m, _ in fs]),
                  np.concatenate([m.ijk for m, _ in fs]),
                  torch.as_tensor(np.concatenate([r.reshape(-1) for _, r in fs])).cuda())
    got = s.potential(0.6).cpu().numpy()
    at = 0
    for m, r in fs:
        a = B.Solver(precision=B.BH_PREC_F64, quadrupole=quad)
        a.build(m.level, m.ijk, torch.as_tensor(r.reshape(-1)).cuda())
        want = a.potential(0.6).cpu().numpy()
        assert np.array_equal(got[at:at + want.size], want)
        at += want.size


@pytest.mark.parametrize("heavy", [0, -1])
def test_binary64_reciprocal_distance(heavy):
    """All mass in one cell, a power of two at an exact centre: each potential is
    one 1/sqrt of an exact d2 (180,000 cells of 9 levels).  The approximation's
    relative error of 2^-20 makes e = 1 - d2 y y at most 2^-19, so the third-order
    step leaves 5/16 e^3, 2^-58.7; rounding d2 y costs half of 2^-53, the last
    operation 2^-53: 1.6 2^-53 in all."""
    m, rho = field(0, 8, 0)
    rho[:] = 0.0
    rho[heavy, 3, 5, 2] = 1.0
    s = B.Solver(precision=B.BH_PREC_F64)
    s.build(m.level, m.ijk, torch.as_tensor(rho.reshape(-1)).cuda())
    got = s.potential(0.5).cpu().numpy().reshape(m.nblocks, 8, 8, 8)
    h = 2.0 ** -(m.level.astype(np.float64) + 3)
    c = [((8 * m.ijk[:, d, None] + np.arange(8)) + 0.5) * h[:, None] for d in range(3)]  # [b][i]
    at = c[0][heavy, 2], c[1][heavy, 5], c[2][heavy, 3]
    d2 = (((c[2] - at[2]) ** 2)[:, :, None, None] + ((c[1] - at[1]) ** 2)[:, None, :, None] +
          ((c[0] - at[0]) ** 2)[:, None, None, :])  # exact: 23-bit differences
    mine = d2 == 0.0
    assert mine.sum() == 1 and got[mine][0] == 0.0
    want = -np.longdouble(h[heavy] ** 3) / np.sqrt(np.longdouble(d2[~mine]))
    assert np.abs(got[~mine] / want - 1).max() <= 1.6 * 2.0 ** -53


@pytest.mark.parametrize("level,extra,theta", [(0, 0, 0.3), (0, 4, 0.25), (1, 2, 0.4), (2, 1, 1.0),
                                               (1, 9, 0.6), (0, 18, 0.9)])
def test_periodic_walk_matches_oracle(level, extra, theta):
    """Counts exactly; potentials by the bar of the periodic tests (1e-5 of the
    field's largest: they change sign).  Sampled cells of every block."""
    m, rho = field(level, extra, 10 * level + extra)
    t = O.Tree(m.level, m.ijk, rho.astype(np.float64))
    tg = (512 * np.arange(m.nblocks)[:, None] +
          np.random.default_rng(extra).integers(0, 512, (m.nblocks, 4))).reshape(-1)
    want, wi, wt = t.walk_periodic(theta, targets=tg)
    for kahan in (True, False):
        s = B.Solver(periodic=True, kahan=kahan)
        s.build(m.level, m.ijk, torch.as_tensor(rho.reshape(-1)).cuda())
        got = s.potential(theta).cpu().numpy().astype(np.float64)
        ni, nt = (x.cpu().numpy()[tg] for x in s.walk_counts(theta))
        assert np.array_equal(ni, wi) and np.array_equal(nt, wt)
        assert np.max(np.abs(got[tg] - want)) <= 1e-5 * np.abs(got).max()
