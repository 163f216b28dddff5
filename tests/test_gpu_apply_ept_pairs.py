"""FP32 element-per-thread apply with two values to an access (even rows on 8 bytes) and
without (fields 4 bytes off, input or output), several right-hand sides, against the host
oracle."""
import pytest

from dg_inputs import jittered_grid, uniform_field
from dg_inputs.mesh import rotate_local_vertices
from tests.gpu_util import cuda, pair, pkg, rel
from tests.test_gpu_apply import TOL32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", (1, 2, 3))
@pytest.mark.parametrize("lam", (0.0, 2.5))
def test_rows_on_and_off_8_bytes(N, lam):
    import torch
    P = pkg()
    m = rotate_local_vertices(jittered_grid(7, 5, jitter=0.1, seed=3, bc_sides=(1, 2, 2, 1)), N)
    lib, ora = pair(m, N)
    lib.set_kernel(N, P.DG_F32, int(lam != 0), P.KERNEL_EPT)
    u = uniform_field((3, m.K, ora.Np), seed=N)
    ref = ora.apply(u, lam=lam)
    x = torch.empty(u.size + 1, dtype=torch.float32, device="cuda")[1:].view(u.shape)
    x.copy_(cuda(u, torch.float32))
    for src in (cuda(u, torch.float32), x):
        for off in (0, 1):
            out = torch.empty(u.size + off, dtype=torch.float32, device="cuda")[off:].view(u.shape)
            lib.apply(src, lam=lam, out=out)
            assert rel(out.cpu().numpy(), ref) <= TOL32
