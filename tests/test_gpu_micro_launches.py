"""The launches that gs_micro reports: preparation, chunks, fill, items, probes,
rows and their maxima, and two scans of one kernel up to 16,384 elements and
three beyond."""
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1701_01772_gb300 as gs  # noqa: E402


@pytest.mark.parametrize("k", [1, 7000, 9000, 20000])
def test_launches(k):
    gs.build()
    rp, col = synth.er(2000, 20000, seed=1)
    up = synth.upper_pairs(rp, col)[:k]
    chunks = sum(int((rp[x + 1] - rp[x] + 31) // 32) for x in up.reshape(-1))
    want = 7 + sum(1 if elements <= 16384 else 3 for elements in (k, chunks))
    g = gs.Graph.from_numpy(rp, col)
    x = torch.empty((k, 15), dtype=torch.float64, device="cuda")
    gs.gs_micro(g.handle, g.ws.handle, torch.as_tensor(up, device="cuda"), k, 0.5, 3, x)
    assert g.ws.stats()["launches"] == want
    g.close()
