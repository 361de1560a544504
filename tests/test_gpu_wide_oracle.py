"""The register-tiled FP32 stage of orders 8 and 9 against the FP64 oracle with materials and
absorbing faces, at order 8 above the one wave of tiles (1 216 tetrahedra on 152 SMs) up to
which the earlier stage runs."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from workloads import kuhn_box_mesh, random_fields

pytestmark = pytest.mark.gpu

RHS_TOL, STEP_TOL = 1e-5, 1e-4


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


@pytest.mark.parametrize("ext", [False, True])
@pytest.mark.parametrize("N,K", [(8, 1250), (9, 650)])
def test_rhs_and_a_step(N, K, ext):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_0901_1024_gb300 as dg
    verts, tets = kuhn_box_mesh(6, 0.15, N)
    tets = tets[:K]
    mesh, om = dg.Mesh(verts, tets, N), oracle.build_mesh(verts, tets, N)
    kw = {}
    if ext:
        rng = np.random.default_rng(N)
        kw = dict(eps=rng.uniform(0.5, 4.0, K), mu=rng.uniform(0.5, 3.0, K),
                  bc=rng.integers(0, 2, (K, 4)).astype(np.int8))
        mesh.set_materials(kw["eps"], kw["mu"])
        mesh.set_boundary(kw["bc"])
    u0 = random_fields(K, om.Np, 5).astype(np.float32)
    u = torch.from_numpy(u0).cuda()
    out = torch.full_like(u, float("nan"))
    mesh.rhs(u, out)
    assert rel(out.cpu().numpy(), oracle.rhs(om, u0.astype(np.float64), 1.0, **kw)) < RHS_TOL
    res, dt = torch.zeros_like(u), mesh.dt_cfl
    mesh.step(u, res, dt, 1)
    ue, re_ = oracle.lserk4_run(om, u0.astype(np.float64), dt, 1, **kw)
    assert rel(u.cpu().numpy(), ue) < STEP_TOL and rel(res.cpu().numpy(), re_) < 10 * STEP_TOL
