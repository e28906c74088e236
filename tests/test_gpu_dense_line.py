"""Samples on either side of the number of dense edges from which k_dense_pairs
runs in small CTAs: the same per-edge counts, and those of the oracle."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1701_01772_gb300 as gs  # noqa: E402


def test_counts_on_both_sides_of_the_line():
    gs.build()
    rp, col = synth.chung_lu(60_000, 1_500_000, 2.1, 9000.0, seed=13)
    g = gs.Graph.from_numpy(rp, col)
    up = synth.upper_pairs(rp, col)
    d = np.diff(rp)
    order = np.argsort(-np.minimum(d[up[:, 0]], d[up[:, 1]]), kind="stable")
    line = 80 * torch.cuda.get_device_properties(0).multi_processor_count * 6
    sides = []
    for k in (90_000, 30_000):
        pairs = up[order[:k]]
        per = torch.empty((k, 3), dtype=torch.int64, device="cuda")
        g.count(torch.as_tensor(pairs, device="cuda"), gs.GS_CONNECTED, per)
        sides.append((g.ws.stats()["dense_edges"], per.cpu().numpy()))
    g.close()
    (many, a), (few, b) = sides
    assert few < line <= many, (few, line, many)
    assert np.array_equal(a[:30_000], b)
    some = np.arange(0, 90_000, 900)
    lc = oracle.local_counts(rp, col, up[order[some]])
    want = np.stack([np.asarray(lc[k], dtype=np.int64) for k in ("t", "k", "q")], axis=1)
    assert np.array_equal(a[some], want)
