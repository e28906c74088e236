"""Algorithm 7's probe kernel at the edges of its two walks: items of 31, 32,
33 and more probes, chunks with one live position, windows that wrap round the
end of a list, endpoints answered by a dense row, a bitmap, the matrix, a
directory and a search, and probability low enough for one probe an item.
Bit-exact at p_e = 1, within 1e-12 of the terms' size below."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1701_01772_gb300 as gs  # noqa: E402


def _wheels():
    """Hubs of degree 31, 32, 33, 64, 65 and 500 joined to one another, with
    shared rims."""
    e, at, hubs = [], 6, range(6)
    e += [(a, b) for a in hubs for b in hubs if a < b]
    for h, d in zip(hubs, (31, 32, 33, 64, 65, 500)):
        rim = range(at, at + d - 5)
        e += [(h, r) for r in rim] + [(r, r + 1) for r in rim[:-1]] + [((h + 1) % 6, r) for r in rim[::2]]
        at += d - 5
    a = np.array(e, dtype=np.int32)
    return synth.from_pairs(at, a[:, 0].copy(), a[:, 1].copy())


MAKERS = {
    "wheels": (_wheels, 0), "wheels_no_index": (_wheels, 1),
    "cl_20k": (lambda: synth.chung_lu(20000, 150000, 2.1, 1500.0, seed=77), 0),
    "cl_20k_small_index": (lambda: synth.chung_lu(20000, 150000, 2.1, 1500.0, seed=77), 3 << 20),
    # bitmap rows longer than 32 KB: matrix rows answer first
    "cl_300k": (lambda: synth.chung_lu(300000, 900000, 2.1, 4000.0, seed=5), 0),
}


@pytest.mark.parametrize("p_e", [1.0, 0.37, 1e-9])
@pytest.mark.parametrize("name", sorted(MAKERS))
def test_rows(name, p_e):
    gs.build()
    make, budget = MAKERS[name]
    rp, col = make()
    up = synth.upper_pairs(rp, col)
    pairs = up if len(up) < 4000 else synth.explicit_sample(rp, col, 600 / len(up), seed=2)
    want, om = oracle.micro(rp, col, pairs, p_e, 11)
    g = gs.Graph.from_numpy(rp, col, hub_budget_bytes=budget)
    out = torch.empty((len(pairs), 15), dtype=torch.float64, device="cuda")
    gs.gs_micro(g.handle, g.ws.handle, torch.as_tensor(pairs, device="cuda"), len(pairs), p_e, 11, out)
    g.close()
    got = out.cpu().numpy()
    if p_e == 1.0:
        assert np.array_equal(got, want)
        return
    col_of = {i: j for j, i in enumerate(gs.MICRO)}
    scale = np.abs(want) + (np.abs(want[:, [col_of[7], col_of[9], col_of[10]]]).sum(1) + np.abs(om) + 1.0)[:, None]
    assert (np.abs(got - want) <= 1e-12 * scale).all()
