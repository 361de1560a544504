"""The two-CTAs-an-SM form of the tensor-core stages of orders 2 and 3 where its rings of 5
and 4 field slots wrap, its barriers come to further phases and order 3's single A buffer
is waited for again and again: 2 058 tiles, the last one ragged, are 6 or 7 a CTA on 304
CTAs.  Against the FP64 oracle, and bit for bit against the one-CTA form, which a shared
launch (dg_rk_stage_multi) runs; also at the counts where the launch changes form."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from workloads import kuhn_box_mesh, random_fields

pytestmark = pytest.mark.gpu

RHS_TOL, STEP_TOL = 1e-5, 1e-4            # the library's bars, as in the tests of smaller meshes


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


def _ext(mesh, K):
    rng = np.random.default_rng(K)
    kw = dict(eps=rng.uniform(0.5, 4.0, K), mu=rng.uniform(0.5, 3.0, K),
              bc=rng.integers(0, 2, (K, 4)).astype(np.int8))
    mesh.set_materials(kw["eps"], kw["mu"])
    mesh.set_boundary(kw["bc"])
    return kw


@pytest.mark.parametrize("ext", [False, True])
@pytest.mark.parametrize("N", [2, 3])
def test_many_tiles_a_cta_against_the_oracle(env, N, ext):
    torch, dg = env
    verts, tets = kuhn_box_mesh(19, 0.15, 5)                 # 41 154 tetrahedra
    mesh, om = dg.Mesh(verts, tets, N), oracle.build_mesh(verts, tets, N)
    mesh.set_stage_impl(dg.Mesh.STAGE_TC)
    kw = _ext(mesh, om.K) if ext else {}
    u0 = random_fields(om.K, om.Np, 40 + N).astype(np.float32)
    u = torch.from_numpy(u0).cuda()
    out = torch.full_like(u, float("nan"))
    mesh.rhs(u, out)
    assert rel(out.cpu().numpy(), oracle.rhs(om, u0.astype(np.float64), 1.0, **kw)) < RHS_TOL
    res, dt = torch.zeros_like(u), mesh.dt_cfl
    mesh.step(u, res, dt, 1)
    ue, re_ = oracle.lserk4_run(om, u0.astype(np.float64), dt, 1, **kw)
    assert rel(u.cpu().numpy(), ue) < STEP_TOL
    assert rel(res.cpu().numpy(), re_) < 10 * STEP_TOL


# tiles: one CTA an SM (65), the first pair (153), order 3 in either form within a round
# (360 paired, 400 single, 460 paired, 740 single), seven rounds; elements off a tile
@pytest.mark.parametrize("ext", [False, True])
@pytest.mark.parametrize("tiles,cut", [(65, 0), (153, 4), (360, 0), (400, 12), (460, 0), (740, 0),
                                       (2058, 8)])
@pytest.mark.parametrize("N", [2, 3])
def test_same_bits_as_one_cta_an_sm(env, N, tiles, cut, ext):
    torch, dg = env
    verts, tets = kuhn_box_mesh(20, 0.15, 6)
    K = 20 * tiles - cut
    mesh = dg.Mesh(verts, tets[:K], N)
    mesh.set_stage_impl(dg.Mesh.STAGE_TC)
    if ext:
        _ext(mesh, K)
    u = torch.from_numpy(random_fields(K, mesh.Np, 3).astype(np.float32)).cuda()
    res0 = torch.from_numpy(random_fields(K, mesh.Np, 4).astype(np.float32)).cuda()
    dt = torch.full((K,), float(np.float32(mesh.dt_cfl)), device="cuda")
    want, rw = torch.full_like(u, float("nan")), res0.clone()
    dg.Mesh.rk_stage_multi([mesh], [u], [want], [rw], 2, dt_elem=[dt])
    got, rg = torch.full_like(u, float("nan")), res0.clone()
    mesh.rk_stage_elem(u, got, rg, 2, dt)
    assert torch.isfinite(got).all() and torch.equal(got, want) and torch.equal(rg, rw)
