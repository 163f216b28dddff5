"""Entry-by-entry bounds, the library's own (1e-12 of (|A||u|)_i in FP64, 1e-5 in FP32),
where other files grant more: the FP64 tensor-core apply next to elements 2^60 larger
at every degree, and the FP32 tile kernel of degrees 9 and 10 at the edges of its tiles."""
import numpy as np
import pytest

from dg_inputs import jittered_grid, uniform_field
from dg_inputs.mesh import rotate_local_vertices
from tests.gpu_util import abs_bound, cuda, max_entry_err, pair, pkg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", (1, 3, 5, 8, 9, 10))
def test_fp64_neighbours_2_to_the_60_apart(N):
    P = pkg()
    lib, ora = pair(rotate_local_vertices(jittered_grid(6, 6, jitter=0.1, seed=3), 2), N)
    exps = np.random.default_rng(N).choice([-60.0, 0.0, 60.0], size=lib.K)
    u = uniform_field((lib.K, ora.Np), seed=50 + N) * np.exp2(exps)[:, None]
    u[::10] = 0.0
    for lam in (0.0, 1.5):
        lib.set_kernel(N, P.DG_F64, int(lam != 0), P.KERNEL_TC64)
        got = lib.apply(cuda(u), lam=lam).cpu().numpy()
        assert max_entry_err(got, ora.apply(u, lam=lam), abs_bound(ora, u, lam)) <= 1e-12


@pytest.mark.parametrize("N", (9, 10))
@pytest.mark.parametrize("nx,ny,B,rot", ((1, 1, 1, 1), (1, 1, 17, 1), (5, 3, 1, 0), (4, 4, 1, 1), (17, 1, 2, 1),
                                         (9, 7, 3, 1)))
def test_fp32_tile_edges(N, nx, ny, B, rot):
    import torch
    P = pkg()
    mesh = jittered_grid(nx, ny, jitter=0.1, seed=3, bc_sides=(1, 2, 1, 1))
    lib, ora = pair(rotate_local_vertices(mesh, nx) if rot else mesh, N)
    u = uniform_field((B, lib.K, ora.Np), seed=N).astype(np.float32)
    for lam in (0.0, 3.0):
        lib.set_kernel(N, P.DG_F32, int(lam != 0), P.KERNEL_TILE)
        got = lib.apply(cuda(u, torch.float32), lam=lam).cpu().numpy()
        for b in range(B):
            v = u[b].astype(np.float64)
            assert max_entry_err(got[b], ora.apply(v, lam=lam), abs_bound(ora, v, lam)) <= 1e-5
