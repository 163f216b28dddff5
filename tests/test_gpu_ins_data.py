"""Velocity boundary data are defined on the velocity-Dirichlet faces: what the arrays
hold at every other node (unset memory, say) changes no bit of a step."""
import numpy as np
import pytest

from dg_inputs import jittered_grid
from dg_inputs.fields import kovasznay
from dg_inputs.mesh import DIRICHLET, ins_pressure_tags, rotate_local_vertices
from tests.gpu_util import cuda, pkg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", (2, 3, 8))
@pytest.mark.parametrize("timed", (False, True))
def test_only_the_nodes_of_dirichlet_faces_are_read(N, timed):
    import torch
    from oracle import refops
    P = pkg()
    m = rotate_local_vertices(jittered_grid(5, 4, box=(-0.5, 1.0, -0.5, 1.5), jitter=0.1, seed=2,
                                            bc_sides=(1, 2, 1, 1)), 1)
    mp = ins_pressure_tags(m)
    on = np.zeros((m.K, (N + 1) * (N + 2) // 2), dtype=bool)
    for f, nodes in enumerate(refops.reference_operators(N)["faces"]):
        on[np.ix_(m.bc[:, f] == DIRICHLET, nodes)] = True
    nu, fu, fv, fp = kovasznay(40.0)
    results = []
    for junk in (0.0, 1e30, np.nan):
        mu_l, mp_l = P.Mesh.from_inputs(m, N), P.Mesh.from_inputs(mp, N)
        x, y = (t.cpu().numpy() for t in mu_l.nodes())
        U, p = np.stack([fu(x, y), fv(x, y)]), fp(x, y)
        data = lambda t: cuda(np.where(on, (1 + t) * U, junk))  # noqa: E731
        flow = P.InsStepper(mu_l, mp_l, nu, 0.01, 4, cuda(U), cuda(p), None if timed else data(0.0), cuda(p),
                            bc=(lambda t: (data(t), cuda(p))) if timed else None)
        flow.step(2)
        results.append(torch.cat([flow.U.flatten(), flow.P.flatten()]))
    assert torch.isfinite(results[0]).all()
    for r in results[1:]:
        assert torch.equal(r, results[0])
