"""What a stage kernel's wait that ran out is called: orders 8 and 9, whose FP32 stage waits
for its operator's bulk copies, have no tensor-core stage to blame."""
from __future__ import annotations

import pytest

from workloads import kuhn_box_mesh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [4, 9])
def test_message_fits_every_stage(N):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_0901_1024_gb300 as dg
    verts, tets = kuhn_box_mesh(2, 0.1, 1)
    _, msg, _ = dg.Mesh(verts, tets, N).check_wait_timeout(100)
    assert "timed out" in msg and "copy" in msg
