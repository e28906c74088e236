"""Branches that only larger graphs reach: co-degree rows built by CTAs of 512
threads, a largest degree too large for the degree table of the registration,
a sampler-key bucket that is split again before it is read back, and samples
on either side of the sizes at which the T lists change hands. Integers equal
to the oracle's or to closed forms."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1701_01772_gb300 as gs  # noqa: E402


def test_tables_of_a_graph_with_rows_of_17000_columns():
    gs.build()
    rp, col = synth.rmat(18, 16, seed=3)
    g = gs.Graph.from_numpy(rp, col)
    assert 13000 < g.info["big_hubs"] < 25000  # the shape of 512-thread rows
    pairs = synth.explicit_sample(rp, col, 400 / (len(col) / 2), seed=6)
    per = torch.empty((len(pairs), 3), dtype=torch.int64, device="cuda")
    g.count(torch.as_tensor(pairs, device="cuda"), gs.GS_CONNECTED, per)
    lc = oracle.local_counts(rp, col, pairs)
    want = np.stack([np.asarray(lc[k], dtype=np.int64) for k in ("t", "k", "q")], axis=1)
    assert np.array_equal(per.cpu().numpy(), want)
    g.close()


def test_star_with_more_leaves_than_the_degree_table_has_bins():
    gs.build()
    leaves = (1 << 22) + 5
    row = torch.empty(leaves + 2, dtype=torch.int64)
    row[0], row[1:] = 0, torch.arange(leaves, 2 * leaves + 1)
    col = torch.zeros(2 * leaves, dtype=torch.int32)
    col[:leaves] = torch.arange(1, leaves + 1, dtype=torch.int32)
    g = gs.Graph(row.cuda(), col.cuda(), hub_budget_bytes=2 << 30)
    got = gs.gs_estimate(g.count(None, gs.GS_THREE_NODE)).as_dict()
    assert got[3]["exact"] == 0 and got[4]["exact"] == leaves * (leaves - 1) // 2
    pairs = g.sample(0.001, 1)
    s = g.count(pairs, gs.GS_CONNECTED).sums()
    d = leaves - 1  # N(v) without u; u has no other neighbour
    assert s[4][0] == pairs.shape[0] * d and s[10][0] == 0 and s[12][0] == 0
    assert s[11][0] == pairs.shape[0] * d * (d - 1)
    g.close()


def _keys(m, seed):
    """oracle.sample_keys for many edges (its definition, on arrays)."""
    def sm(x):
        z = x + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))

    with np.errstate(over="ignore"):
        return sm(np.uint64(seed) ^ sm(np.arange(m, dtype=np.uint64))) >> np.uint64(11)


def test_fixed_size_samples_of_36_million_edges():
    gs.build()
    small = synth.er(300, 900, seed=1)
    assert np.array_equal(_keys(900, 77), oracle.sample_keys(*small, 77))
    rp, col = synth.er(1_200_000, 36_000_000, seed=9)
    g = gs.Graph.from_numpy(rp, col, validate=False, hub_budget_bytes=1)
    order = np.argsort(_keys(g.m, 77), kind="stable")
    up = synth.upper_pairs(rp, col)
    buf = torch.empty((g.m, 2), dtype=torch.int32, device="cuda")
    for lo, hi in ((0, 1), (0, 20001), (20001, 20005), (17_999_999, 18_000_000), (g.m - 3, g.m)):
        got = gs.gs_sample_ranks(g.handle, g.ws.handle, lo, hi, 77, buf).cpu().numpy()
        assert np.array_equal(got, up[np.sort(order[lo:hi])]), (lo, hi)
    g.close()


@pytest.mark.parametrize("edges", [1, 31, 32, 33, 32767, 32768])
def test_samples_at_the_sizes_where_the_t_lists_change_hands(edges):
    gs.build()
    rp, col = synth.chung_lu(60000, 600000, 2.1, 9000.0, seed=13)  # lists of up to 5,000 entries
    g = gs.Graph.from_numpy(rp, col)
    d = np.diff(rp)
    up = synth.upper_pairs(rp, col)
    order = np.argsort(-np.minimum(d[up[:, 0]], d[up[:, 1]]), kind="stable")
    # the longest lists and a spread of the rest
    idx = np.unique(np.concatenate([order[:min(edges, 40)],
                                    order[np.linspace(0, len(up) - 1, edges).astype(np.int64)]]))[:edges]
    pairs = up[idx]
    per = torch.empty((len(pairs), 3), dtype=torch.int64, device="cuda")
    g.count(torch.as_tensor(pairs, device="cuda"), gs.GS_CONNECTED, per)
    few = np.arange(0, len(pairs), max(1, len(pairs) // 150))
    lc = oracle.local_counts(rp, col, pairs[few])
    want = np.stack([np.asarray(lc[k], dtype=np.int64) for k in ("t", "k", "q")], axis=1)
    assert np.array_equal(per.cpu().numpy()[few], want)
    g.close()


def test_three_node_samples_with_long_lists_equal_the_unpadded_pass():
    gs.build()
    rp, col = synth.rmat(18, 16, seed=3)
    g = gs.Graph.from_numpy(rp, col, hub_budget_bytes=2 << 30)
    for fraction in (0.2, 0.01):  # above and below the line for padded chunks
        pairs = g.sample(fraction, 5)
        per = torch.empty((pairs.shape[0], 3), dtype=torch.int64, device="cuda")
        got = g.count(pairs, gs.GS_THREE_NODE, per)
        assert got.sums() == gs.gs_count3_static(g.handle, pairs, pairs.shape[0]).sums()
        few = np.arange(0, pairs.shape[0], pairs.shape[0] // 300)
        lc = oracle.local_counts(rp, col, pairs.cpu().numpy()[few], four=False)
        assert np.array_equal(per[:, 0].cpu().numpy()[few], np.asarray(lc["t"]))
    g.close()
