"""Samples on either side of the sizes from which longer T lists stay with one
warp, on a graph with lists of 2,049 to 4,097 and more positions."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1701_01772_gb300 as gs  # noqa: E402


def _graph():
    """Hubs of 2,047 to 4,200 neighbours, all joined to one another, over a
    random part."""
    n, sizes = 60_000, (2047, 2048, 2049, 4095, 4096, 4097, 4200)
    rp, col = synth.er(n, 200_000, seed=5)
    ab = [synth.upper_pairs(rp, col)]
    rng = np.random.default_rng(6)
    for h, k in enumerate(sizes):
        to = rng.choice(n, k - len(sizes) + 1, replace=False)
        ab.append(np.stack([np.full(len(to), n + h), to], 1))
    hubs = [(n + a, n + b) for a in range(len(sizes)) for b in range(a)]
    ab = np.concatenate(ab + [np.array(hubs)]).astype(np.int32)
    return synth.from_pairs(n + len(sizes), ab[:, 0].copy(), ab[:, 1].copy())


def test_counts_on_both_sides_of_the_lines():
    gs.build()
    rp, col = _graph()
    g = gs.Graph.from_numpy(rp, col)
    up = synth.upper_pairs(rp, col)
    d = np.diff(rp)
    up = up[np.argsort(-np.minimum(d[up[:, 0]], d[up[:, 1]]), kind="stable")]
    assert sorted(d)[-7:] == [2047, 2048, 2049, 4095, 4096, 4097, 4200]
    pers = {}
    for k in (1 << 15, (1 << 17) - 1, 1 << 17):
        per = torch.empty((k, 3), dtype=torch.int64, device="cuda")
        g.count(torch.as_tensor(up[:k], device="cuda"), gs.GS_CONNECTED, per)
        pers[k] = per.cpu().numpy()
    g.close()
    for k, per in pers.items():
        assert np.array_equal(per[:1 << 15], pers[1 << 15]), k
    assert np.array_equal(pers[1 << 17][:-1], pers[(1 << 17) - 1])
    some = np.concatenate([np.arange(60), np.arange(60, 1 << 17, 4000)])
    lc = oracle.local_counts(rp, col, up[some])
    want = np.stack([np.asarray(lc[k], dtype=np.int64) for k in ("t", "k", "q")], axis=1)
    assert np.array_equal(pers[1 << 17][some], want)
