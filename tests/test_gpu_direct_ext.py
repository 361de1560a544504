"""Order 1's one-thread-per-element stage with absorbing faces alone, materials alone and both,
below and above the size (half the SMs with a CTA) where the form changes: the tiles'
bits, which unaligned buffers give."""
from __future__ import annotations

import numpy as np
import pytest

from workloads import kuhn_box_mesh, random_fields

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["absorbing", "materials", "both"])
@pytest.mark.parametrize("K", [6, 1296, 9728, 9729, 10368])      # 76 CTAs of 128: 9 728
def test_same_bits_as_the_tiles(K, kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_0901_1024_gb300 as dg
    verts, tets = kuhn_box_mesh(12, 0.15, 3)
    mesh = dg.Mesh(verts, tets[:K], 1)
    rng = np.random.default_rng(K)
    if kind != "materials":
        mesh.set_boundary(rng.integers(0, 2, (K, 4)).astype(np.int8))
    if kind != "absorbing":
        mesh.set_materials(rng.uniform(0.5, 4.0, K), rng.uniform(0.5, 3.0, K))
    u = torch.from_numpy(random_fields(K, 4, 1).astype(np.float32)).cuda()
    res0 = torch.from_numpy(random_fields(K, 4, 2).astype(np.float32)).cuda()
    dt = float(np.float32(mesh.dt_cfl))

    def shifted(x):
        return torch.empty(x.numel() + 1, device="cuda")[1:].copy_(x.reshape(-1)).view(x.shape)
    out = []
    for src, r in ((u, res0.clone()), (shifted(u), shifted(res0))):
        rhs, nxt = torch.full_like(u, float("nan")), torch.full_like(u, float("nan"))
        mesh.rhs(src, rhs)
        mesh.rk_stage(src, nxt, r, 3, dt)
        out.append((rhs, nxt, r))
    for a, b in zip(*out):
        assert torch.isfinite(a).all() and torch.equal(a, b)
