"""Order 4's RK update with absorbing faces alone and with materials, several tiles a CTA and
a ragged last one, against the FP64 oracle (its register batches differ from the vacuum
form's)."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from workloads import kuhn_box_mesh, random_fields

pytestmark = pytest.mark.gpu

STEP_TOL = 1e-4


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


@pytest.mark.parametrize("kind", ["absorbing", "materials"])
def test_a_step(kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_0901_1024_gb300 as dg
    verts, tets = kuhn_box_mesh(12, 0.15, 3)
    K = 8488                                  # 424 tiles and 8 elements: 2 or 3 a CTA
    tets = tets[:K]
    mesh, om = dg.Mesh(verts, tets, 4), oracle.build_mesh(verts, tets, 4)
    mesh.set_stage_impl(dg.Mesh.STAGE_TC)
    rng = np.random.default_rng(3)
    kw = dict(bc=np.ones((K, 4), np.int8))
    mesh.set_boundary(kw["bc"])
    if kind == "materials":
        kw.update(eps=rng.uniform(0.5, 4.0, K), mu=rng.uniform(0.5, 3.0, K))
        mesh.set_materials(kw["eps"], kw["mu"])
    u0 = random_fields(K, om.Np, 5).astype(np.float32)
    u = torch.from_numpy(u0).cuda()
    res, dt = torch.zeros_like(u), mesh.dt_cfl
    mesh.step(u, res, dt, 1)
    ue, re_ = oracle.lserk4_run(om, u0.astype(np.float64), dt, 1, **kw)
    assert rel(u.cpu().numpy(), ue) < STEP_TOL and rel(res.cpu().numpy(), re_) < 10 * STEP_TOL
