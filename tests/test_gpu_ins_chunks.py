"""The flow step on meshes larger than the elements whose fluxes it holds at a time:
copies of a small mesh, side by side and not connected, flow like the small one, and
the memory it keeps is what include/dg.h says."""
import gc
from types import SimpleNamespace

import numpy as np
import pytest

from dg_inputs import jittered_grid
from dg_inputs.fields import kovasznay
from dg_inputs.mesh import ins_pressure_tags, rotate_local_vertices
from tests.gpu_util import cuda, pkg

pytestmark = pytest.mark.gpu


def _copies(m, n):
    """n copies of mesh m as one mesh (the same coordinates: each copy has its own vertices)."""
    nv = len(m.VX)
    return SimpleNamespace(VX=np.tile(m.VX, n), VY=np.tile(m.VY, n), bc=np.tile(m.bc, (n, 1)),
                           EToV=(m.EToV[None] + (nv * np.arange(n, dtype=m.EToV.dtype))[:, None, None]).reshape(-1, 3))


def _stepper(P, m, mp, N):
    nu, fu, fv, fp = kovasznay(40.0)
    mu_l, mp_l = (P.Mesh(N, q.VX, q.VY, q.EToV, q.bc) for q in (m, mp))
    x, y = (t.cpu().numpy() for t in mu_l.nodes())
    U, p = cuda(np.stack([fu(x, y), fv(x, y)])), cuda(fp(x, y))
    vel = P.default_opts(precond=P.PREC_INVMASS, tol=1e-13, max_iter=2000)
    pr = P.default_opts(precond=P.PREC_JACOBI, tol=1e-13, max_iter=50000)
    return P.InsStepper(mu_l, mp_l, nu, 0.01, 4, U, p, U.clone(), p.clone(), vel_opts=vel, pr_opts=pr)


# 60 elements: 66,000 are three chunks of 22,000, which cut through a copy; 32,820 are
# two. Both solves stop at 1e-13 of the right-hand side, with sums taken in another
# order: differences as in the parity tests with the oracle.
@pytest.mark.parametrize("N,copies", ((3, 1100), (6, 547), (9, 547)))
def test_copies_of_a_mesh_flow_like_one(N, copies):
    P = pkg()
    m = rotate_local_vertices(jittered_grid(6, 5, box=(-0.5, 1.0, -0.5, 1.5), jitter=0.1, seed=2,
                                            bc_sides=(1, 2, 1, 1)), 1)
    mp = ins_pressure_tags(m)
    one, many = _stepper(P, m, mp, N), _stepper(P, _copies(m, copies), _copies(mp, copies), N)
    for s in (one, many):
        s.step(3)
    U, p = one.U.unsqueeze(1), one.P.unsqueeze(0)
    assert float((many.U.view(2, copies, *one.P.shape) - U).norm() / U.norm()) <= 1e-9 * copies ** 0.5
    assert float((many.P.view(copies, *one.P.shape) - p).norm() / p.norm()) <= 1e-8 * copies ** 0.5


def test_workspace_is_what_the_header_says():
    import torch
    P = pkg()
    N, c, Np = 8, 13, 45
    K = 2 * 256 * 256
    m = jittered_grid(256, 256, box=(-0.5, 1.0, -0.5, 1.5), jitter=0.0)
    s = _stepper(P, m, ins_pressure_tags(m), N)
    for mesh in (s.mesh_u, s.mesh_p):  # the solves' workspaces, before
        B = 2 if mesh is s.mesh_u else 1
        o = P.default_opts(precond=P.PREC_INVMASS if B == 2 else P.PREC_JACOBI, tol=0.5, max_iter=1)
        mesh.solve(torch.rand(B, K, Np, dtype=torch.float64, device="cuda"), lam=1.0 if B == 2 else 0.0, opts=o, check=False)
    gc.collect()
    torch.cuda.empty_cache()
    s.st.vel_opts.max_iter = s.st.pr_opts.max_iter = 1
    before = torch.cuda.mem_get_info()[0]
    with pytest.raises(P.DgError):  # one iteration does not converge
        s.step()
    used = (before - torch.cuda.mem_get_info()[0]) / 8
    said = (27 * Np + 8 * c * (c + 3) + 9) * K + 4 * (c * (2 * c + 3) + Np) * 32768
    assert used <= 1.02 * said
