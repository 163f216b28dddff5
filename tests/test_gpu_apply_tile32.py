"""FP32 apply of the tile kernel at degrees 9 and 10: sixteen elements per tile whose
faces are sorted by the neighbour's local face. Element counts around the tile size,
tiles that span right-hand sides, rotated vertices (every pairing of local faces), all
of one pairing, and both kinds of boundary, against the host oracle."""
import numpy as np
import pytest

from dg_inputs import jittered_grid, uniform_field
from dg_inputs.mesh import rotate_local_vertices
from tests.gpu_util import abs_bound, cuda, pair, pkg

pytestmark = pytest.mark.gpu

# The longest chain has Np + 2 Np + Np + 6 (N + 1) + (N + 1) < 350 roundings of 2^-24; they
# are independent of each other, so in the 2-norm sqrt(350) of them, on terms that (|A||u|)
# underestimates by the cancellation inside the products that A is made of: two digits at
# degree 10. 2^-24 sqrt(350) 100 < 2^-13; a wrong face or slot gives an error of order 1.
NORM = 2.0 ** -13


@pytest.mark.parametrize("N", (9, 10))
@pytest.mark.parametrize("nx,ny,B,rot", ((1, 1, 1, 1), (1, 1, 17, 1), (5, 3, 1, 0), (4, 4, 1, 1), (17, 1, 2, 1),
                                         (9, 7, 3, 1)))
def test_tile_edges(N, nx, ny, B, rot):
    import torch
    P = pkg()
    mesh = jittered_grid(nx, ny, jitter=0.1, seed=3, bc_sides=(1, 2, 1, 1))
    lib, ora = pair(rotate_local_vertices(mesh, nx) if rot else mesh, N)
    u = uniform_field((B, lib.K, ora.Np), seed=N).astype(np.float32)
    x = torch.empty(u.size + 1, dtype=torch.float32, device="cuda")[1:].view(u.shape)  # 4 bytes off alignment
    x.copy_(cuda(u, torch.float32))
    for lam in (0.0, 3.0):
        lib.set_kernel(N, P.DG_F32, int(lam != 0), P.KERNEL_TILE)
        y0, y1 = lib.apply(cuda(u, torch.float32), lam=lam), lib.apply(x, lam=lam)
        assert torch.equal(y0, y1)
        for b in range(B):
            ref, bnd = ora.apply(u[b].astype(np.float64), lam=lam), abs_bound(ora, u[b], lam)
            assert np.linalg.norm(y0[b].cpu().numpy() - ref) <= NORM * np.linalg.norm(bnd)
