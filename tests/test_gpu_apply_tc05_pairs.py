"""FP32 tensor-core apply where two blocks share an SM (degrees 1 to 5): more tiles than
SMs, so that both tensor-memory halves of an SM are in use, with a ragged last tile,
against the host oracle."""
import pytest

from dg_inputs import jittered_grid, uniform_field
from dg_inputs.mesh import rotate_local_vertices
from tests.gpu_util import cuda, pair, pkg, rel
from tests.test_gpu_apply import TOL32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", (1, 4, 5, 6))   # 6: one block per SM
@pytest.mark.parametrize("B,lam", ((1, 0.0), (2, 2.5)))
def test_more_tiles_than_sms(N, B, lam):
    import torch
    P = pkg()
    m = rotate_local_vertices(jittered_grid(101, 99, jitter=0.1, seed=5, bc_sides=(1, 2, 2, 1)), 7)
    lib, ora = pair(m, N)     # 19,998 triangles: 157 tiles, 313 with two right-hand sides
    lib.set_kernel(N, P.DG_F32, int(lam != 0), P.KERNEL_TC05)
    u = uniform_field((B, m.K, ora.Np), seed=N)
    y = lib.apply(cuda(u, torch.float32), lam=lam)
    assert torch.equal(y, lib.apply(cuda(u, torch.float32), lam=lam))
    for b in range(B):
        assert rel(y[b].cpu().numpy(), ora.apply(u[b], lam=lam)) <= TOL32
    assert P.lib().dg_tensor_timeouts() == 0
