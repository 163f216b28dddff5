"""The fixed-point FP64 apply (DG_KERNEL_TC64) where its tiles, item groups and
scales can go wrong: rows just below, at and above a 128-row tile, every group
layout of the degrees, inputs off 16-byte alignment, a field that is smooth
across faces (jumps near zero), large offsets, and non-finite data."""
import numpy as np
import pytest

from dg_inputs import jittered_grid, uniform_field
from dg_inputs.mesh import rotate_local_vertices
from tests.gpu_util import abs_bound, cuda, max_entry_err, pair, pkg

pytestmark = pytest.mark.gpu

# Columns carry 56 bits of a bound at most 2^9 above their row's largest entry and
# sum up to 363 terms; inputs carry 53 bits: 2^-56 2^9 sqrt(363) < 2^-42.7 of
# (|A||u|)_i in the worst row, 2^-45 of it in the 2-norm.
ENTRY, NORM = 2.0 ** -42, 2.0 ** -45


def _mesh(nx, ny, seed=3):
    return rotate_local_vertices(jittered_grid(nx, ny, jitter=0.1, seed=seed, bc_sides=(1, 2, 1, 1)), seed)


def _check(lib, ora, u, lam, got):
    ref, bnd = ora.apply(u, lam=lam), abs_bound(ora, u, lam)
    assert max_entry_err(got, ref, bnd) <= ENTRY
    assert np.linalg.norm(got - ref) <= NORM * np.linalg.norm(bnd)


@pytest.mark.parametrize("N", (1, 2, 5, 6, 8, 9, 10))
@pytest.mark.parametrize("nx,ny,B", ((9, 7, 1), (8, 8, 1), (13, 5, 1), (1, 1, 3), (11, 6, 2)))
def test_tile_edges(N, nx, ny, B):
    import torch
    P = pkg()
    lib, ora = pair(_mesh(nx, ny), N)
    lib.set_kernel(N, P.DG_F64, 0, P.KERNEL_TC64)
    lib.set_kernel(N, P.DG_F64, 1, P.KERNEL_TC64)
    u = uniform_field((B, lib.K, ora.Np), seed=N)
    x = torch.empty(u.size + 1, dtype=torch.float64, device="cuda")[1:].view(u.shape)  # 8 bytes off alignment
    x.copy_(cuda(u))
    for lam in (0.0, 3.0):
        y0, y1 = lib.apply(cuda(u), lam=lam), lib.apply(x, lam=lam)
        assert torch.equal(y0, y1)
        for b in range(B):
            _check(lib, ora, u[b], lam, y0[b].cpu().numpy())
    assert P.lib().dg_tensor_timeouts() == 0


@pytest.mark.parametrize("N", (3, 6, 10))
def test_smooth_and_offset_fields(N):
    P = pkg()
    lib, ora = pair(_mesh(10, 9), N)
    for name, u in (("wave", np.sin(2 * ora.x) * np.cos(3 * ora.y)), ("constant", np.full_like(ora.x, 0.7)),
                    ("offset", 1e8 + np.sin(2 * ora.x)), ("one element", np.eye(lib.K)[5][:, None] + 0 * ora.x)):
        for lam in (0.0, 3.0):
            lib.set_kernel(N, P.DG_F64, int(lam != 0), P.KERNEL_TC64)
            _check(lib, ora, u, lam, lib.apply(cuda(u), lam=lam).cpu().numpy())


def test_non_finite_elements_stay_local():
    P = pkg()
    m = _mesh(8, 9)
    lib, ora = pair(m, 4)
    lib.set_kernel(4, P.DG_F64, 0, P.KERNEL_TC64)
    u = uniform_field((lib.K, ora.Np), seed=1)
    clean = lib.apply(cuda(u)).cpu().numpy()
    for value in (np.nan, np.inf):
        v = u.copy()
        v[40, 7] = value
        got = lib.apply(cuda(v)).cpu().numpy()
        near = {40} | {int(n) for n in ora.geo.EToE[40] if n >= 0}
        for e in range(lib.K):
            if e in near:
                assert np.all(np.isnan(got[e]))
            else:
                assert np.array_equal(got[e], clean[e])
