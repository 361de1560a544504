"""dg_step_host against dg_step: the overlapped copies and the last stage run in ranges
give the same bits, for meshes below and above the size where ranges start, odd and
even numbers of stages, with and without a host RK register."""
from __future__ import annotations

import numpy as np
import pytest

from workloads import kuhn_box_mesh, random_fields

pytestmark = pytest.mark.gpu


# 6 K Np floats: 0.6 MB; 12 MB (order 3) and 18 MB (order 4), one or two waves of tiles;
# 36 MB (order 1), several ranges with a last one that is no whole wave
@pytest.mark.parametrize("n,N,cut", [(5, 4, 0), (16, 3, 0), (16, 4, 1), (40, 1, 5)])
@pytest.mark.parametrize("nsteps", [0, 1, 2])
def test_matches_device_step(n, N, cut, nsteps):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_0901_1024_gb300 as dg
    verts, tets = kuhn_box_mesh(n, 0.1, 2)
    tets = tets[:len(tets) - cut]
    mesh = dg.Mesh(verts, tets, N)
    u0 = random_fields(mesh.K, mesh.Np, 7).astype(np.float32)
    u = torch.from_numpy(u0).cuda()
    res = torch.zeros_like(u)
    mesh.step(u, res, mesh.dt_cfl, nsteps)
    e = mesh.energy(u)
    for pinned in (True, False):
        for with_res in (False, True):
            uh = torch.from_numpy(u0.copy())
            uh = uh.pin_memory() if pinned else uh
            rh = torch.zeros_like(uh) if with_res else None
            for _ in range(2):                        # the second call reuses streams and buffers
                uh.copy_(torch.from_numpy(u0))
                if with_res:
                    rh.zero_()
                eh = mesh.step_host(uh, rh, mesh.dt_cfl, nsteps)
                assert eh == e
                assert np.array_equal(uh.numpy(), u.cpu().numpy())
                if with_res:
                    assert np.array_equal(rh.numpy(), res.cpu().numpy())
