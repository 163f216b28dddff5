"""Degree transfers and vector passes of the p-multigrid solve where their tiles and
vector widths can go wrong: every coarse degree's instance, the widest operator (10 -> 9),
lengths that no vector width divides, ragged last tiles, several right-hand sides, and a
solution vector off 16-byte alignment; the graph and the host-driven loop must agree bit
for bit and the oracle's residual must meet the tolerance."""
import numpy as np
import pytest

from dg_inputs import jittered_grid, uniform_field
from dg_inputs.mesh import rotate_local_vertices
from tests.gpu_util import cuda, pair, pkg
from tests.test_gpu_graph import _assert_same, _both, _oracle_relres

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("degrees", ([10, 9, 5, 2, 1], [8, 7, 6, 3, 1], [9, 8, 4, 1], [3, 2, 1], [6, 1]))
@pytest.mark.parametrize("mixed,B", ((1, 1), (0, 3)))
def test_transfer_chain(degrees, mixed, B):
    P = pkg()
    m = rotate_local_vertices(jittered_grid(9, 5, seed=4), 3)     # 90 triangles
    lib, ora = pair(m, degrees[0])
    bb = ora.mass_apply(uniform_field((B, m.K, ora.Np), seed=11))
    g, r, e = _both(lib, cuda(bb), precond=P.PREC_PMG, degrees=degrees, mixed=mixed, coarse_amg=1, tol=1e-10)
    _assert_same(g, e)
    _assert_same(r, e)
    for k in range(B):
        assert _oracle_relres(ora, g[0][k], bb[k]) <= 1.5e-10


def _off16(a):
    """A copy 8 bytes off 16-byte alignment."""
    import torch
    t = torch.empty(a.numel() + 1, dtype=a.dtype, device=a.device)[1:].view(a.shape)
    t.copy_(a)
    return t


@pytest.mark.parametrize("N,precond", ((2, "PREC_JACOBI"), (4, "PREC_PMG"), (5, "PREC_PMG")))
def test_vectors_off_alignment(N, precond):
    import torch
    P = pkg()
    m = rotate_local_vertices(jittered_grid(9, 5, seed=4), 3)
    lib, ora = pair(m, N)
    b = cuda(ora.mass_apply(uniform_field((2, m.K, ora.Np), seed=11)))
    kw = dict(precond=getattr(P, precond), degrees=[N, 1] if precond == "PREC_PMG" else None, tol=1e-10, graph=0,
              max_iter=3000)
    if kw["degrees"] is None:
        del kw["degrees"]
    x0, i0 = lib.solve(b, **kw)
    x1, i1 = lib.solve(_off16(b), x=_off16(torch.zeros_like(b)), **kw)
    assert torch.equal(x0, x1) and i0["iters"] == i1["iters"] and i0["relres"] == i1["relres"]
