"""Graphs with millions of empty ids between two blocks of edges (reserved or
padded id ranges) cost what the same graphs cost with the empty ids at the end,
and give the same results up to the shift of the second block's ids."""
import time

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1701_01772_gb300 as gs  # noqa: E402

N, GAP = 50_000, 8_000_000
# A search over the gap is about 2 log2(GAP) = 46 dependent loads of at most a
# microsecond; 0.5 ms more than the noise of two equal calls.
RATIO, SLACK = 1.5, 0.5e-3


def _two_blocks(shift):
    """Two random blocks of N vertices, the second `shift` ids further on."""
    ab = []
    for k in range(2):
        rp, col = synth.er(N, 500_000, seed=20 + k)
        ab.append(synth.upper_pairs(rp, col) + k * (N + shift))
    ab = np.concatenate(ab).astype(np.int32)
    return synth.from_pairs(2 * N + GAP, ab[:, 0].copy(), ab[:, 1].copy())


def _best(f):
    best = 1e9
    for _ in range(6):
        torch.cuda.synchronize()
        t = time.perf_counter()
        r = f()
        torch.cuda.synchronize()
        best = min(best, time.perf_counter() - t)
    return best, r


def _shifted(pairs):
    p = pairs.cpu().numpy().astype(np.int64)
    return np.where(p >= N, p + GAP, p)


def test_weighted_sample():
    gs.build()
    times, kept = [], []
    for shift in (0, GAP):
        g = gs.Graph.from_numpy(*_two_blocks(shift), hub_budget_bytes=1 << 30)
        w = torch.ones(2 * N + GAP, dtype=torch.int32, device="cuda")
        buf = torch.empty((50_000, 2), dtype=torch.int32, device="cuda")
        t, (k, _) = _best(lambda: gs.gs_sample_weighted(g.handle, g.ws.handle, w, 0.02, 7, buf))
        times.append(t)
        kept.append(buf[:k].clone())
        g.close()
    assert np.array_equal(_shifted(kept[0]), kept[1].cpu().numpy())
    assert times[1] <= RATIO * times[0] + SLACK, times


def test_registration_and_exact_triangles():
    gs.build()
    times, sums = [], []
    for shift in (0, GAP):
        rp, col = _two_blocks(shift)
        rp, col = torch.as_tensor(rp, device="cuda"), torch.as_tensor(col, device="cuda")

        def register():
            g = gs.Graph(rp, col, hub_budget_bytes=1 << 30)
            s = g.count(None, gs.GS_THREE_NODE).sums()
            g.close()
            return s

        t, s = _best(register)
        times.append(t)
        sums.append(s)
    assert sums[0] == sums[1]
    assert times[1] <= RATIO * times[0] + SLACK, times
