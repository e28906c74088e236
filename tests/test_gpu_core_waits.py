"""The grid-wide waits of the core-number kernel: a long chain of removals is cut
into rounds and needs no long wait; a wait that runs out ends the call with
GS_ETIMEOUT, and the workspace serves the next call."""
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1701_01772_gb300 as gs  # noqa: E402

GS_ETIMEOUT = 11


def test_a_long_path_takes_longer_than_the_limit():
    # two chains of 200,000 removals, 0.25 s; 20,000 looks are 2 to 40 ms, a
    # round's 17 steps about 20 us
    gs.build()
    n = 400_000
    row = torch.arange(-1, 2 * n - 1, 2, device="cuda")
    row = torch.cat((row, torch.tensor([2 * n - 2], device="cuda"))).clamp_(min=0)
    i = torch.arange(n, device="cuda")
    col = torch.stack((i - 1, i + 1), 1).reshape(-1)[1:-1].to(torch.int32)
    g = gs.Graph(row, col, hub_budget_bytes=1)
    g.ws.set_wait_limit(20_000)
    core = torch.zeros(n, dtype=torch.int32, device="cuda")
    assert gs.gs_core_numbers(g.handle, g.ws.handle, core) == 1
    assert bool((core == 1).all())
    g.close()


def test_a_wait_that_runs_out():
    gs.build()
    rp, col = synth.chung_lu(40_000, 200_000, 2.1, 900.0, seed=8)
    g = gs.Graph.from_numpy(rp, col)
    core = torch.zeros(len(rp) - 1, dtype=torch.int32, device="cuda")
    g.ws.set_wait_limit(0)
    for _ in range(3):
        with pytest.raises(gs.GraphletError) as e:
            gs.gs_core_numbers(g.handle, g.ws.handle, core)
        assert e.value.status == GS_ETIMEOUT
    g.ws.set_wait_limit(1 << 28)
    want = oracle.core_numbers(rp, col)
    assert gs.gs_core_numbers(g.handle, g.ws.handle, core) == want.max()
    assert (core.cpu().numpy() == want).all()
    with pytest.raises(gs.GraphletError):
        g.ws.set_wait_limit(-1)
    g.close()
