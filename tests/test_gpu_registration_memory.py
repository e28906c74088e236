"""Registration on a nearly full GPU: the blocks of small graphs are optional
and give way to the index, also when they were built first."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1701_01772_gb300 as gs  # noqa: E402

GIB = 1 << 30


def test_batch_whose_blocks_do_not_fit_beside_its_index():
    gs.build()
    # 64 members with bit matrices of 32 MiB each (2 GiB; their co-degree blocks,
    # 16 GiB, are beyond half of the budget) and one without a block, whose
    # vertices fill the co-degree tables
    ring = np.arange(16384, dtype=np.int32)
    small = synth.from_pairs(16384, ring, (ring + 1) % 16384)
    graphs = [small] * 64 + [synth.er(70_000, 3_000_000, seed=3)]

    def make():
        return gs.Batch.from_graphs(graphs, mask=gs.GS_THREE_NODE, autotune=False,
                                    hub_budget_bytes=4 * GIB)

    def counts(b):
        return [s.sums() for s in b.count()]

    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    b = make()
    used = before - torch.cuda.mem_get_info()[0]
    want = counts(b)
    b.close()
    assert used > 5 * GIB  # bit matrices, index, workspace
    torch.cuda.empty_cache()
    # room for the index and the workspace and what registration needs beside
    # them for a while, but not for the bit matrices
    fill = torch.empty(torch.cuda.mem_get_info()[0] - (used - GIB // 2), dtype=torch.uint8,
                       device="cuda")
    b = make()
    got = counts(b)
    b.close()
    del fill
    torch.cuda.empty_cache()
    assert got == want
