"""Validation of graphs whose hubs have neighbouring ids: long rows are checked
(errors in them are found wherever they lie) and are not all one block's work."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1701_01772_gb300 as gs  # noqa: E402


def _bipartite(a, b):
    """K_{a,b}, the a hubs first."""
    row = torch.cat((torch.arange(a) * b, a * b + torch.arange(b + 1) * a))
    col = torch.cat((torch.arange(a, a + b).repeat(a), torch.arange(a).repeat(b))).to(torch.int32)
    return row, col


def _best(f):
    best = 1e9
    for _ in range(4):
        torch.cuda.synchronize()
        t = time.perf_counter()
        f()
        torch.cuda.synchronize()
        best = min(best, time.perf_counter() - t)
    return best


def test_time_of_the_checks():
    gs.build()
    row, col = (t.cuda() for t in _bipartite(300, 60_000))
    with_checks = _best(lambda: gs.Graph(row, col, hub_budget_bytes=1).close())
    without = _best(lambda: gs.Graph(row, col, validate=False, hub_budget_bytes=1).close())
    # 18M edges in 300 rows: 7.2 ms with a warp per row, 35 ms in seven blocks
    assert with_checks - without <= 8e-3, (with_checks, without)


@pytest.mark.parametrize("hub,pos", [(0, 0), (0, 1023), (7, 1024), (7, 1025), (39, 2999)])
def test_errors_in_long_rows(hub, pos):
    gs.build()
    row, col = _bipartite(40, 3000)
    bad = col.numpy().copy()
    at = hub * 3000 + pos
    for value, status in ((-1, "GS_EINVAL"), (40 + 3000, "GS_EINVAL"), (hub, "GS_ESELFLOOP")):
        bad[at] = value
        with pytest.raises(gs.GraphletError) as e:
            gs.Graph(row.cuda(), torch.as_tensor(bad).cuda(), hub_budget_bytes=1)
        # a value out of order is reported too; either is an error of the input
        assert gs.STATUS[e.value.status] in (status, "GS_ENOTSORTED", "GS_EDUP", "GS_EASYM")
    bad[at] = np.int32(col[at])
    gs.Graph(row.cuda(), torch.as_tensor(bad).cuda(), hub_budget_bytes=1).close()
