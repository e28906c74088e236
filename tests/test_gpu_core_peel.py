"""Core numbers where the one-kernel peeling can go wrong: hubs of several
removal entries (more than 256 neighbours, exactly 256 and 257), a removal
that exposes more vertices than a warp's queue holds, long chains, isolated
vertices, more and fewer vertices than the grid has threads."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1701_01772_gb300 as gs  # noqa: E402


def _pairs(n, ab):
    ab = np.array(ab, dtype=np.int32).reshape(-1, 2)
    return synth.from_pairs(n, ab[:, 0].copy(), ab[:, 1].copy())


def _star(k):
    return _pairs(k + 1, [(0, i) for i in range(1, k + 1)])


def _fans(k, r):
    """r hubs, each with k leaf pairs (a leaf's other neighbour is the next
    leaf): removing a hub exposes all its leaves."""
    e = []
    for h in range(r):
        b = r + h * k
        e += [(h, b + i) for i in range(k)] + [(b + i, b + i + 1) for i in range(k - 1)]
    return _pairs(r + r * k, e)


MAKERS = {
    "star_255": lambda: _star(255), "star_256": lambda: _star(256), "star_257": lambda: _star(257),
    "star_5000": lambda: _star(5000),
    "path_4000": lambda: _pairs(4000, [(i, i + 1) for i in range(3999)]),
    "cycle_301": lambda: _pairs(301, [(i, (i + 1) % 301) for i in range(301)]),
    "bipartite_3_700": lambda: _pairs(703, [(a, 3 + b) for a in range(3) for b in range(700)]),
    "fans_97": lambda: _fans(97, 5), "fans_300": lambda: _fans(300, 9),
    "isolated": lambda: _pairs(2000, [(5, 1999), (5, 77)]),
    "one_edge": lambda: _pairs(2, [(0, 1)]),
    "cl_30000": lambda: synth.chung_lu(30000, 300000, 2.1, 3000.0, seed=3),
    "rmat_15": lambda: synth.rmat(15, 14, seed=4),
}


@pytest.mark.parametrize("name", sorted(MAKERS))
def test_core_numbers(name):
    gs.build()
    rp, col = MAKERS[name]()
    want = oracle.core_numbers(rp, col)
    g = gs.Graph.from_numpy(rp, col)
    for _ in range(2):  # the workspace keeps the first run's contents
        core = torch.full((len(rp) - 1,), 7, dtype=torch.int32, device="cuda")
        mx = gs.gs_core_numbers(g.handle, g.ws.handle, core)
        assert np.array_equal(core.cpu().numpy(), want) and mx == want.max()
    g.close()
