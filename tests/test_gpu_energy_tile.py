"""The tiled energy kernel at every order against the FP64 oracle's mass matrix:
passes that end inside a row set, ranges, unaligned field buffers, materials."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from workloads import kuhn_box_mesh, random_fields

pytestmark = pytest.mark.gpu

TOL = 1e-6          # relative, the library's bar for the energy


# 6 K rows against passes (orders 1 and 2: blocks of 256 threads)
# of 128 (64 at order 8): one row set, a ragged one, several passes
@pytest.mark.parametrize("K", [1, 5, 21, 22, 160])
@pytest.mark.parametrize("N", range(1, 10))
def test_energy_tiles(N, K):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_0901_1024_gb300 as dg
    verts, tets = kuhn_box_mesh(3, 0.15, N)
    tets = tets[:K]
    mesh, om = dg.Mesh(verts, tets, N), oracle.build_mesh(verts, tets, N)
    u32 = random_fields(K, om.Np, N).astype(np.float32)
    u = torch.from_numpy(u32).cuda()
    want = oracle.energy(om, u32.astype(np.float64))
    e = mesh.energy(u)
    assert abs(e - want) < TOL * want
    # the same fields 4 bytes off a 16-byte boundary: the same sums
    shifted = torch.empty(u.numel() + 1, device="cuda")[1:].copy_(u.reshape(-1)).view(u.shape)
    assert mesh.energy(shifted) == e
    # ranges add up (FP64 sums, other order)
    if K > 2:
        parts = mesh.energy_range(u, 0, K // 3) + mesh.energy_range(u, K // 3, K)
        assert abs(parts - e) <= 1e-12 * e
    eps, mu = np.linspace(0.5, 3.0, K), np.linspace(2.0, 0.7, K)
    mesh.set_materials(eps, mu)
    want = oracle.energy(om, u32.astype(np.float64), eps, mu)
    assert abs(mesh.energy(u) - want) < TOL * want
