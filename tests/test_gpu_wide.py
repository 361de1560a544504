"""The register-tiled FP32 stage of orders 8 and 9 against the tiled one (shape 1 of
dg_set_stage_shape, which the oracle tests pin): the same bits, for whole and ragged
tiles, one and several tiles per CTA, materials and absorbing faces, element steps and
ranges that start off its own tile boundaries."""
from __future__ import annotations

import numpy as np
import pytest

from workloads import kuhn_box_mesh, random_fields

pytestmark = pytest.mark.gpu


def _mesh(dg, N, K, ext):
    verts, tets = kuhn_box_mesh(8, 0.15, N)
    mesh = dg.Mesh(verts, tets[:K], N)
    if ext:
        rng = np.random.default_rng(K)
        mesh.set_materials(rng.uniform(0.5, 4.0, K), rng.uniform(0.5, 3.0, K))
        mesh.set_boundary(rng.integers(0, 2, (K, 4)).astype(np.int8))
    return mesh


# order 8 is register tiled (tiles of 16) above one wave of 8-element tiles (1 216
# tetrahedra on 152 SMs), order 9 (tiles of 8) always; 3 072 gives CTAs several tiles
@pytest.mark.parametrize("ext", [False, True])
@pytest.mark.parametrize("N,K", [(8, 1217), (8, 1232), (8, 3072), (8, 3059), (9, 1), (9, 7), (9, 8),
                                 (9, 9), (9, 1225), (9, 2433)])
def test_same_bits_as_the_tiles(N, K, ext):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_0901_1024_gb300 as dg
    mesh = _mesh(dg, N, K, ext)
    u = torch.from_numpy(random_fields(K, mesh.Np, 3).astype(np.float32)).cuda()
    res0 = torch.from_numpy(random_fields(K, mesh.Np, 4).astype(np.float32)).cuda()
    dt = float(np.float32(mesh.dt_cfl))
    out = []
    for shape in (1, 0):
        mesh.set_stage_shape(shape)
        rhs, nxt, res = torch.full_like(u, float("nan")), torch.full_like(u, float("nan")), res0.clone()
        mesh.rhs(u, rhs)
        mesh.rk_stage(u, nxt, res, 2, dt)
        out.append((rhs, nxt, res))
    for a, b in zip(*out):
        assert torch.equal(a, b)
    nxt, res = torch.full_like(u, float("nan")), res0.clone()
    mesh.rk_stage_elem(u, nxt, res, 2, torch.full((K,), dt, device="cuda"))
    assert torch.equal(nxt, out[1][1]) and torch.equal(res, out[1][2])
    tile = mesh.stage_tile(u, nxt, res)
    if K > 5 * tile:                        # three tiles, then the rest (enough for register tiles)
        nxt, res = torch.full_like(u, float("nan")), res0.clone()
        mesh.rk_stage_range(u, nxt, res, 2, dt, 0, 3 * tile)
        mesh.rk_stage_range(u, nxt, res, 2, dt, 3 * tile, K)
        assert torch.equal(nxt, out[1][1]) and torch.equal(res, out[1][2])
