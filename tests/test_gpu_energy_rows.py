"""How the energy kernels of orders 1 and 2 round a row u^T M u: one element with one nonzero
field gives that row's FP32 value times its Jacobian, which a NumPy restatement of the
sums (one chain of multiply-adds at order 1, two at order 2) reproduces exactly."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from workloads import kuhn_box_mesh

pytestmark = pytest.mark.gpu


def fma(a, b, c):
    # the product of two FP32 numbers is exact in FP64
    return (a.astype(np.float64) * b.astype(np.float64) + c.astype(np.float64)).astype(np.float32)


def rows(u, M, chains):
    n = M.shape[0]
    e = np.zeros(len(u), np.float32)
    for i in range(n):
        s = [np.zeros(len(u), np.float32) for _ in range(chains)]
        for j in range(i, n):
            w = np.full(len(u), (1 if i == j else 2) * M[i, j], np.float32)
            s[(j - i) % chains] = fma(w, u[:, j], s[(j - i) % chains])
        e = fma(u[:, i], s[0] if chains == 1 else s[0] + s[1], e)
    return e


# rows that round otherwise than the restatement: none, but for a constant of M or J that two
# FP64 computations round to FP32 differently (1e-8 each); one chain in place of two changes
# half of the rows
@pytest.mark.parametrize("N,chains", [(1, 1), (2, 2)])
def test_row_sums(N, chains):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_0901_1024_gb300 as dg
    verts, tets = kuhn_box_mesh(6, 0.15, 2)
    mesh, om = dg.Mesh(verts, tets, N), oracle.build_mesh(verts, tets, N)
    u = np.random.default_rng(N).standard_normal((om.K, om.Np)).astype(np.float32)
    fields = np.zeros((6, om.K, om.Np), np.float32)
    fields[np.arange(om.K) % 6, np.arange(om.K)] = u
    d = torch.from_numpy(fields).cuda()
    got = np.array([mesh.energy_range(d, k, k + 1) for k in range(om.K)])
    want = 0.5 * om.J.astype(np.float32).astype(np.float64) * rows(
        u, om.ref.M.astype(np.float32), chains).astype(np.float64)
    assert np.mean(np.abs(got - want) <= 1e-12 * want) > 0.99
    other = 0.5 * om.J.astype(np.float32).astype(np.float64) * rows(
        u, om.ref.M.astype(np.float32), 3 - chains).astype(np.float64)
    assert np.mean(np.abs(other - want) <= 1e-12 * want) < 0.9       # the two can be told apart
