"""Discrete conservation of the FP64 apply. With Neumann conditions all around, the
constant is in the kernel of the transposed operator: the entries of A u sum to zero
for every u. Errors that differ from element to element average out of that sum; one
that all elements share (a table's) does not, and the inverse operator amplifies it."""
import numpy as np
import pytest

from dg_inputs import jittered_grid
from tests.gpu_util import pkg

pytestmark = pytest.mark.gpu

# An element's sum has Np roundings of 2^-53 of terms up to 2^4 times its flux (the
# operator's largest entries): 66 2^-53 2^4 < 2^-42.9 at most, independent from one
# jittered element to the next, so 2^-42.9 / sqrt(2 256^2) < 2^-51 in the mean.
MEAN = 2.0 ** -51


@pytest.mark.parametrize("N", (3, 6, 8, 10))
def test_entries_sum_to_zero_under_neumann_conditions(N):
    import torch
    P = pkg()
    n = 256
    m = jittered_grid(n, n, jitter=0.1, seed=1, bc_sides=(2, 2, 2, 2))
    lib = P.Mesh.from_inputs(m, N)
    lib.set_kernel(N, P.DG_F64, 0, P.KERNEL_TC64)
    x, y = lib.nodes()
    for u, grad in ((x, 1.0), (y, 1.0), (x + y, np.sqrt(2.0)), (torch.sin(2 * x) * torch.cos(y), 1.0)):
        total = float(lib.apply(u.contiguous()).sum())
        assert abs(total) / (lib.K * grad / n) <= MEAN, (N, total)
