"""Order 1's one-thread-per-element stage against the FP64 oracle and, bit for bit
where the arithmetic is the same, across its entry points: element counts around
the block size, materials and absorbing faces, ranges, element steps, and the tiled
stage that unaligned buffers fall back to."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from workloads import kuhn_box_mesh, random_fields

pytestmark = pytest.mark.gpu

RHS_TOL = 1e-5


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


@pytest.mark.parametrize("ext", [False, True])
@pytest.mark.parametrize("K", [1, 19, 127, 128, 129, 162])
def test_rhs(env, K, ext):
    torch, dg = env
    verts, tets = kuhn_box_mesh(3, 0.15, 3)
    tets = tets[:K]
    mesh, om = dg.Mesh(verts, tets, 1), oracle.build_mesh(verts, tets, 1)
    kw = {}
    if ext:
        rng = np.random.default_rng(K)
        kw = dict(eps=rng.uniform(0.5, 4.0, K), mu=rng.uniform(0.5, 3.0, K),
                  bc=rng.integers(0, 2, (K, 4)).astype(np.int8))
        mesh.set_materials(kw["eps"], kw["mu"])
        mesh.set_boundary(kw["bc"])
    u32 = random_fields(K, 4, K).astype(np.float32)
    u32[:, ::5] *= 1e-4
    want = oracle.rhs(om, u32.astype(np.float64), 1.0, **kw)
    u = torch.from_numpy(u32).cuda()
    out = torch.full_like(u, float("nan"))
    mesh.rhs(u, out)
    assert rel(out.cpu().numpy(), want) < RHS_TOL
    # 4 bytes off: the tiled stage, which rounds the same way
    us = torch.empty(u.numel() + 1, device="cuda")[1:].copy_(u.reshape(-1)).view(u.shape)
    tiled = torch.full_like(u, float("nan"))
    mesh.rhs(us, tiled)
    assert rel(tiled.cpu().numpy(), want) < RHS_TOL
    assert torch.equal(tiled, out)


def test_ranges_and_element_steps(env):
    torch, dg = env
    verts, tets = kuhn_box_mesh(4, 0.15, 4)
    mesh = dg.Mesh(verts, tets, 1)
    K, dt = mesh.K, float(np.float32(mesh.dt_cfl))
    u = torch.from_numpy(random_fields(K, 4, 1).astype(np.float32)).cuda()
    res0 = torch.from_numpy(random_fields(K, 4, 2).astype(np.float32)).cuda()
    want, rw = torch.empty_like(u), res0.clone()
    mesh.rk_stage(u, want, rw, 3, dt)
    got, rg = torch.empty_like(u), res0.clone()
    mesh.rk_stage_elem(u, got, rg, 3, torch.full((K,), dt, device="cuda"))
    assert torch.equal(got, want) and torch.equal(rg, rw)
    E = mesh.stage_tile(u, got, rg)
    got, rg = torch.full_like(u, 7.0), res0.clone()
    mesh.rk_stage_range(u, got, rg, 3, dt, E, 9 * E)
    assert torch.equal(got[:, E:9 * E], want[:, E:9 * E])
    assert torch.equal(rg[:, :E], res0[:, :E]) and (got[:, 9 * E:] == 7.0).all()
    mesh.rk_stage_range(u, got, rg, 3, dt, 0, E)
    mesh.rk_stage_range(u, got, rg, 3, dt, 9 * E, K)
    assert torch.equal(got, want) and torch.equal(rg, rw)
