"""Calls at changing opening angles on one context: the opening radii of the
records in sibling order (list walks, counts) and of those in pre-order
(learned walks, pair listing) are made apart, each only when its own reader
needs another angle.  Every call must give what a fresh context gives."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1509_07370_gb300 import bhgrav as B  # noqa: E402
from paper_1509_07370_gb300 import learned as L  # noqa: E402
from paper_1509_07370_gb300 import meshgen as mg  # noqa: E402

pytestmark = pytest.mark.gpu

MESH = mg.refined_mesh(2, 4, lambda lev, ijk: np.all(ijk == 0, axis=1))
RHO = [np.random.Generator(np.random.PCG64(i)).lognormal(size=MESH.nblocks * 512).astype(np.float32)
       for i in (1, 2)]
TARGETS = np.arange(5, MESH.nblocks * 512, 4099)


def solver(which, **opt):
    s = B.Solver(**opt)
    if opt.get("learned"):
        s.set_mlp(L.init_weights(3))
    s.build(MESH.level, MESH.ijk, torch.as_tensor(RHO[which]).cuda())
    return s


def call(s, what, theta, density):
    if what == "potential":
        with torch.cuda.stream(s.stream):
            out = [s.potential(theta)]
    elif what == "counts":
        with torch.cuda.stream(s.stream):
            out = list(s.walk_counts(theta))
    elif what == "graph":
        out = [s.solve_graph(density, theta)]
    else:  # the pairs come in no particular order
        with torch.cuda.stream(s.stream):
            feat, eps, n, node = s.learn_pairs(theta, torch.as_tensor(TARGETS).cuda(), 1 << 16, True)
            at = torch.argsort(node * 1024.0 + feat[:, 3].double() * 64 + feat[:, 0].double())
            out = [feat[at], eps[at], node[at]]
    s.stream.synchronize()
    return [x.cpu().numpy() for x in out]


@pytest.mark.parametrize("learned", [0, 1, 2])
def test_calls_at_changing_angles(learned):
    opt = dict(learned=learned) if learned else dict(quadrupole=True)
    steps = [("pairs", 0.5), ("potential", 0.8), ("pairs", 0.8), ("counts", 0.6), ("potential", 0.8),
             ("pairs", 0.6), ("counts", 0.8), ("potential", 0.6), ("graph", 0.7), ("pairs", 0.7),
             ("counts", 0.7), ("pairs", 0.9), ("graph", 0.7), ("potential", 0.9), ("graph", 0.9),
             ("counts", 0.5), ("update", 0), ("counts", 0.5), ("pairs", 0.9), ("potential", 0.7)]
    s = solver(0, stream=torch.cuda.Stream(), **opt)
    which, dens = 0, [torch.as_tensor(r).cuda() for r in RHO]
    torch.cuda.synchronize()
    for what, theta in steps:
        if what == "update":
            which = 1
            s.update_density(dens[1])
            continue
        got = call(s, what, theta, dens[which])
        fresh = solver(which, **opt)
        want = call(fresh, "potential" if what == "graph" else what, theta, None)
        for a, b in zip(got, want):
            assert np.array_equal(a, b), (what, theta)
