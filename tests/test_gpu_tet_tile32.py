"""FP32 tetrahedral apply at degrees 4 and 5 on both sides of the size (one wave of
blocks) where the register-blocked kernels take over: below it, just past it with a ragged
last tile, and with more tiles than resident blocks; tiles span right-hand sides, and the
vertices are renumbered so that every pairing of local faces occurs."""
import pytest

from dg_inputs import uniform_field
from dg_inputs.tetmesh import jittered_tet_grid, permute_local_vertices
from tests.gpu_util import cuda, rel
from tests.test_gpu_tet import MIXED, TOL32, _pair

pytestmark = pytest.mark.gpu


# 2,058 elements; one wave of the small kernel is 2,432 elements at N = 5, 8,512 at N = 4
@pytest.mark.parametrize("N,batches", ((5, (1, 2, 3)), (4, (4, 5, 7))))
@pytest.mark.parametrize("lam", (0.0, 1.25))
def test_tet_fp32_around_one_wave(N, batches, lam):
    import torch
    m = permute_local_vertices(jittered_tet_grid(7, jitter=0.1, seed=9, bc_sides=MIXED), seed=N)
    lib, ora = _pair(m, N)
    u = uniform_field((max(batches), m.K, ora.Np), seed=40 + N)
    ref = ora.apply(u, lam=lam)
    for B in batches:
        x = torch.empty(u[:B].size + 1, dtype=torch.float32, device="cuda")[1:].view(u[:B].shape)  # 4 bytes off
        x.copy_(cuda(u[:B], torch.float32))
        y = lib.apply(cuda(u[:B], torch.float32), lam=lam)
        assert torch.equal(y, lib.apply(x, lam=lam))
        assert rel(y.cpu().numpy(), ref[:B]) <= TOL32
