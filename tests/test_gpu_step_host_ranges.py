"""dg_step_host with its last stage split into ranges of tiles, on every kind of stage: the
same bits as dg_step, and the launch count proves that the stage was split."""
from __future__ import annotations

import numpy as np
import pytest

from workloads import kuhn_box_mesh, random_fields

pytestmark = pytest.mark.gpu


# fields of 24 to 40 MB and at least two waves of tiles twice over: 2 to 4 ranges
@pytest.mark.parametrize("N,n,cut,ext,check", [
    (2, 30, 0, False, False),        # tensor cores, two CTAs an SM
    (3, 24, 0, False, False), (3, 24, 4, True, True),
    (4, 20, 0, False, True), (6, 14, 0, False, False), (6, 14, 1, True, False),
    (7, 13, 0, False, False), (8, 11, 0, False, False), (9, 10, 0, True, True)])
def test_split_last_stage(N, n, cut, ext, check):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_0901_1024_gb300 as dg
    verts, tets = kuhn_box_mesh(n, 0.1, 2)
    tets = tets[:len(tets) - cut]
    mesh = dg.Mesh(verts, tets, N)
    K = mesh.K
    if ext:
        rng = np.random.default_rng(K)
        mesh.set_materials(rng.uniform(0.5, 4.0, K), rng.uniform(0.5, 3.0, K))
        mesh.set_boundary(rng.integers(0, 2, (K, 4)).astype(np.int8))
    u0 = random_fields(K, mesh.Np, 7).astype(np.float32)
    u = torch.from_numpy(u0).cuda()
    res = torch.zeros_like(u)
    mesh.step(u, res, mesh.dt_cfl, 1)
    e = mesh.energy(u)
    want_u, want_r = u.cpu().numpy(), res.cpu().numpy()
    if check:
        mesh.set_energy_check(1e-3)
    for pinned, with_res in ((True, False), (True, True), (False, False)):
        uh = torch.from_numpy(u0.copy())
        uh = uh.pin_memory() if pinned else uh
        rh = torch.zeros_like(uh) if with_res else None
        eh = mesh.step_host(uh, rh, mesh.dt_cfl, 1)
        ranges = mesh.last_launch_count() - (4 if check else 2) - 4   # energies, whole stages
        assert 2 <= ranges <= 4
        assert eh == e
        assert np.array_equal(uh.numpy(), want_u)
        if with_res:
            assert np.array_equal(rh.numpy(), want_r)
