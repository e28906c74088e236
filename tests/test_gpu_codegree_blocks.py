"""8-bit co-degree blocks of small graphs, where they can go wrong: rows that
are no multiple of 16 bytes, pairs with 254, 255 and more common neighbours
(255 is not held), the largest graph that has a block and the first that has
none. Exact integers against the oracle."""
import itertools

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1701_01772_gb300 as gs  # noqa: E402


def _two_hubs(common):
    """Two adjacent hubs with `common` shared neighbours, some of them joined."""
    a = [0] + [0] * common + [1] * common + list(range(2, common, 3))
    b = [1] + list(range(2, 2 + common)) * 2 + list(range(3, common + 1, 3))
    return synth.from_pairs(common + 2, np.array(a, dtype=np.int32), np.array(b, dtype=np.int32))


def _clique(n):
    p = np.array(list(itertools.combinations(range(n), 2)), dtype=np.int32)
    return synth.from_pairs(n, p[:, 0].copy(), p[:, 1].copy())


MAKERS = {
    "two_hubs_253": lambda: _two_hubs(253), "two_hubs_254": lambda: _two_hubs(254),
    "two_hubs_255": lambda: _two_hubs(255), "two_hubs_300": lambda: _two_hubs(300),
    "k17": lambda: _clique(17), "k257": lambda: _clique(257),
    "er_33": lambda: synth.er(33, 200, seed=4), "er_1000": lambda: synth.er(1000, 9000, seed=5),
    "cl_3000": lambda: synth.chung_lu(3000, 40000, 2.1, 900.0, seed=6),
    "er_16384": lambda: synth.er(16384, 50000, seed=7), "er_16385": lambda: synth.er(16385, 50000, seed=8),
}


@pytest.mark.parametrize("name", sorted(MAKERS))
def test_exact_counts_of_one_graph(name):
    gs.build()
    rp, col = MAKERS[name]()
    want = oracle.exact_counts(rp, col)
    for use_hubs in (True, False):
        g = gs.Graph.from_numpy(rp, col)
        g.ws.set_tuning(use_hubs=use_hubs)
        got = gs.gs_estimate(g.count(None)).as_dict()
        g.close()
        assert {k: got[k]["exact"] for k in want} == want, use_hubs


def test_exact_counts_in_a_batch():
    gs.build()
    graphs = [MAKERS[k]() for k in sorted(MAKERS)]
    for budget in (0, 64 << 20, 1):  # blocks of every graph, too large for the budget, no index
        b = gs.Batch.from_graphs(graphs, autotune=False, hub_budget_bytes=budget)
        got = b.exact()
        b.close()
        for i, (rp, col) in enumerate(graphs):
            assert got[i] == oracle.exact_counts(rp, col), (budget, i)
