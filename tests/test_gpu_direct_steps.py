"""Order 1's RK update over several CTAs: the one-thread-per-element stage against the FP64
oracle, and the tiles (which unaligned buffers fall back to) against it bit for bit."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from workloads import kuhn_box_mesh, random_fields

pytestmark = pytest.mark.gpu

STEP_TOL = 1e-4


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_0901_1024_gb300 as dg
    return torch, dg


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


def _shifted(torch, u):
    return torch.empty(u.numel() + 1, device="cuda")[1:].copy_(u.reshape(-1)).view(u.shape)


@pytest.mark.parametrize("ext", [False, True])
@pytest.mark.parametrize("K", [130, 1296])                   # blocks of 128
def test_steps_and_the_unaligned_stage(env, K, ext):
    torch, dg = env
    verts, tets = kuhn_box_mesh(6, 0.15, 3)
    tets = tets[:K]
    mesh, om = dg.Mesh(verts, tets, 1), oracle.build_mesh(verts, tets, 1)
    kw = {}
    if ext:
        rng = np.random.default_rng(K)
        kw = dict(eps=rng.uniform(0.5, 4.0, K), mu=rng.uniform(0.5, 3.0, K),
                  bc=rng.integers(0, 2, (K, 4)).astype(np.int8))
        mesh.set_materials(kw["eps"], kw["mu"])
        mesh.set_boundary(kw["bc"])
    u0 = random_fields(K, 4, K).astype(np.float32)
    dt = float(np.float32(mesh.dt_cfl))
    u = torch.from_numpy(u0).cuda()
    res = torch.zeros_like(u)
    mesh.step(u, res, dt, 5)
    ue, re_ = oracle.lserk4_run(om, u0.astype(np.float64), dt, 5, **kw)
    assert rel(u.cpu().numpy(), ue) < STEP_TOL and rel(res.cpu().numpy(), re_) < 10 * STEP_TOL
    # one stage, scalar and per-element steps, all buffers 4 bytes off: the tiles
    u = torch.from_numpy(u0).cuda()
    res0 = torch.from_numpy(random_fields(K, 4, 2).astype(np.float32)).cuda()
    for elem in (False, True):
        out = []
        for shift in (False, True):
            src, r = (_shifted(torch, u), _shifted(torch, res0)) if shift else (u, res0.clone())
            dst = _shifted(torch, torch.full_like(u, float("nan"))) if shift else torch.full_like(u, float("nan"))
            if elem:
                mesh.rk_stage_elem(src, dst, r, 3, torch.linspace(0.5, 1.0, K, device="cuda") * dt)
            else:
                mesh.rk_stage(src, dst, r, 3, dt)
            out.append((dst, r))
        assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
