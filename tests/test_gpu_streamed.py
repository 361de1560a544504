"""The streamed-operator tensor-core stage (orders 8 and 9 by default) and the order-4
stage for field chunks off the 16-byte grid against the FP64 oracle and the FP32 stage: ragged and full tiles, several tiles per CTA,
field chunks off the 16-byte grid, materials and absorbing faces, per-element
steps, element ranges, and its accuracy against the FP32 stage's."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from workloads import cavity_mode, kuhn_box_mesh, random_fields

pytestmark = pytest.mark.gpu

RHS_TOL, STEP_TOL = 1e-5, 1e-4         # the library's bars (one evaluation, 100 steps)
FP32, AUTO = 1, 0


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


def _rhs(torch, mesh, u32, impl):
    mesh.set_stage_impl(impl)
    mesh.trace_enable(2)
    u = torch.from_numpy(u32).cuda()
    out = torch.full_like(u, float("nan"))
    mesh.rhs(u, out)
    torch.cuda.synchronize()
    _, kinds = mesh.trace_read()
    mesh.trace_enable(0)
    mesh.set_stage_impl(0)
    return out.cpu().numpy(), set(int(k) for k in kinds)


# K = 48 and 162 end in ragged tiles (of 20 at order 8, of 16 at order 9; 48 is whole at
# order 9); 160 is whole at both; 161 and 159 put order 8's chunks off the 16-byte grid, K
# not a multiple of 4 order 4's (tiles of 20; all three offsets)
@pytest.mark.parametrize("ext", [False, True])
@pytest.mark.parametrize("N,K", [(8, 4), (8, 48), (8, 160), (8, 161), (8, 162), (8, 159), (9, 1),
                                 (9, 48), (9, 160), (9, 161), (4, 1), (4, 2), (4, 3), (4, 21),
                                 (4, 22), (4, 23), (4, 161), (4, 162)])
def test_rhs_against_the_oracle(env, N, K, ext):
    torch, dg = env
    verts, tets = kuhn_box_mesh(3, 0.15, 10 + N)
    tets = tets[:K]
    mesh, om = dg.Mesh(verts, tets, N), oracle.build_mesh(verts, tets, N)
    kw = {}
    if ext:
        rng = np.random.default_rng(K)
        kw = dict(eps=rng.uniform(0.5, 4.0, K), mu=rng.uniform(0.5, 3.0, K),
                  bc=rng.integers(0, 2, (K, 4)).astype(np.int8))
        mesh.set_materials(kw["eps"], kw["mu"])
        mesh.set_boundary(kw["bc"])
    u32 = random_fields(K, om.Np, 20 + N).astype(np.float32)
    u32[:, ::7] *= 1e-6                                  # rows of very different scales
    got, kinds = _rhs(torch, mesh, u32, AUTO)
    assert kinds == {5}
    want = oracle.rhs(om, u32.astype(np.float64), 1.0, **kw)
    assert np.isfinite(got).all()
    assert rel(got, want) < RHS_TOL


@pytest.mark.parametrize("N,K", [(8, 3072 + 7), (8, 3072 + 8), (9, 2600), (4, 3041), (4, 4374 - 1)])
def test_several_tiles_per_cta(env, N, K):
    """More tiles than SMs: the rings wrap from tile to tile."""
    torch, dg = env
    verts, tets = kuhn_box_mesh(9, 0.15, 5)
    tets = tets[:K]
    mesh = dg.Mesh(verts, tets, N)
    u = torch.from_numpy(random_fields(K, mesh.Np, 3).astype(np.float32)).cuda()
    out = []
    for impl in (AUTO, FP32):
        mesh.set_stage_impl(impl)
        x, r = u.clone(), torch.zeros_like(u)
        mesh.step(x, r, mesh.dt_cfl, 2)
        out.append((x.cpu().numpy(), r.cpu().numpy()))
    mesh.set_stage_impl(0)
    for a, b in zip(*out):
        assert np.isfinite(a).all()
        assert rel(a, b.astype(np.float64)) < RHS_TOL * 10


@pytest.mark.parametrize("N,K", [(8, 162), (8, 164), (9, 162), (4, 162), (4, 163)])
def test_element_steps_and_ranges(env, N, K):
    """Per-element steps equal the scalar step bit for bit where they agree, and two
    ranges of tiles equal the whole mesh."""
    torch, dg = env
    verts, tets = kuhn_box_mesh(4, 0.15, 6)
    tets = tets[:K]
    mesh = dg.Mesh(verts, tets, N)
    u = torch.from_numpy(random_fields(K, mesh.Np, 4).astype(np.float32)).cuda()
    res0 = torch.from_numpy(random_fields(K, mesh.Np, 5).astype(np.float32)).cuda()
    dt = float(np.float32(mesh.dt_cfl))
    want, rw = torch.empty_like(u), res0.clone()
    mesh.rk_stage(u, want, rw, 2, dt)
    got, rg = torch.empty_like(u), res0.clone()
    mesh.rk_stage_elem(u, got, rg, 2, torch.full((K,), dt, device="cuda"))
    assert torch.equal(got, want) and torch.equal(rg, rw)
    tile = mesh.stage_tile(u, got, rg)
    got, rg = torch.empty_like(u), res0.clone()
    mesh.rk_stage_range(u, got, rg, 2, dt, 0, 3 * tile)
    mesh.rk_stage_range(u, got, rg, 2, dt, 3 * tile, K)
    assert torch.equal(got, want) and torch.equal(rg, rw)


@pytest.mark.parametrize("N", [8, 9])
def test_accuracy_is_the_fp32_stages_or_better(env, N):
    """Relative L2 error of one right-hand side against the oracle, smooth and random
    fields: no larger than the FP32 CUDA-core stage's."""
    torch, dg = env
    verts, tets = kuhn_box_mesh(4, 0.1, 2)
    mesh, om = dg.Mesh(verts, tets, N), oracle.build_mesh(verts, tets, N)
    for u in (cavity_mode(om.x, om.y, om.z, 0.3), random_fields(om.K, om.Np, 8)):
        u32 = u.astype(np.float32)
        want = oracle.rhs(om, u32.astype(np.float64))
        err = [rel(_rhs(torch, mesh, u32, impl)[0], want) for impl in (AUTO, FP32)]
        assert err[0] <= err[1], err
