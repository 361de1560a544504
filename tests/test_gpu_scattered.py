"""Order 3 on a mesh in random element order, whose launch takes the one-CTA form, against the
same mesh in its native order (two CTAs an SM): the same bits, element by element."""
from __future__ import annotations

import numpy as np
import pytest

from workloads import kuhn_box_mesh, random_fields

pytestmark = pytest.mark.gpu


def test_random_order_gives_the_same_bits():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_0901_1024_gb300 as dg
    verts, tets = kuhn_box_mesh(26, 0.1, 1)                  # 105 456: 0.63 of the faces far
    p = np.random.default_rng(1).permutation(len(tets))
    native, shuffled = dg.Mesh(verts, tets, 3), dg.Mesh(verts, tets[p], 3)
    order = torch.from_numpy(p).cuda()
    u = torch.from_numpy(random_fields(native.K, native.Np, 3).astype(np.float32)).cuda()
    res = torch.from_numpy(random_fields(native.K, native.Np, 4).astype(np.float32)).cuda()
    dt = float(np.float32(native.dt_cfl))
    want, got = torch.full_like(u, float("nan")), torch.full_like(u, float("nan"))
    r2 = res[:, order].contiguous()
    native.rk_stage(u, want, res, 2, dt)
    shuffled.rk_stage(u[:, order].contiguous(), got, r2, 2, dt)
    assert torch.isfinite(got).all()
    assert torch.equal(got, want[:, order]) and torch.equal(r2, res[:, order])
