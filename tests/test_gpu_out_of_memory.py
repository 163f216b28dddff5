"""A call that runs out of device memory while it builds its workspace says so and
leaves nothing half-built: the same call succeeds once memory is there. The memory is
taken by an ordinary tensor; nothing here faults the GPU."""
import numpy as np
import pytest

from dg_inputs import jittered_grid
from dg_inputs.fields import kovasznay
from dg_inputs.mesh import ins_pressure_tags
from tests.gpu_util import cuda, pkg

pytestmark = pytest.mark.gpu

LEFT = 192 << 20  # bytes left free, below what each workspace needs


def _short_of_memory():
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.empty(torch.cuda.mem_get_info()[0] - LEFT, dtype=torch.uint8, device="cuda")


def _fails_then_works(call):
    import torch
    P = pkg()
    hog = _short_of_memory()
    try:
        for _ in range(2):  # the second call finds no trace of the first
            with pytest.raises(P.DgError) as e:
                call()
            assert e.value.name == "DG_ERR_OOM"
    finally:
        del hog
        torch.cuda.empty_cache()
    return call()


def test_flow_step():
    P = pkg()
    N, m = 8, jittered_grid(96, 96, box=(-0.5, 1.0, -0.5, 1.5), jitter=0.0)  # 18,432 triangles: 675 MB
    nu, fu, fv, fp = kovasznay(40.0)
    results = []
    for short in (False, True):
        mu_l, mp_l = P.Mesh.from_inputs(m, N), P.Mesh.from_inputs(ins_pressure_tags(m), N)
        x, y = (t.cpu().numpy() for t in mu_l.nodes())
        U, p = cuda(np.stack([fu(x, y), fv(x, y)])), cuda(fp(x, y))
        o = lambda: P.default_opts(precond=P.PREC_PMG, degrees=[8, 4, 1], tol=1e-8, max_iter=200, mixed=1,  # noqa: E731
                                   cheb_degree=3, coarse_tol=1e-2, coarse_max_iter=1, coarse_amg=1)
        s = P.InsStepper(mu_l, mp_l, nu, 0.001, 4, U, p, U.clone(), p.clone(), vel_opts=o(), pr_opts=o())
        _fails_then_works(s.step) if short else s.step()
        results.append((s.U.clone(), s.P.clone()))
        del s
        mu_l.close()
        mp_l.close()
    for a, b in zip(*results):
        assert bool((a == b).all())


@pytest.mark.parametrize("precond", ("jacobi", "pmg"))
def test_solve(precond):
    import torch
    P = pkg()
    N, B, m = 8, 16, jittered_grid(96, 96, jitter=0.1, seed=1)  # vectors of 106 MB, at least four of them
    kw = dict(precond=P.PREC_JACOBI) if precond == "jacobi" else dict(precond=P.PREC_PMG, degrees=[8, 4, 2, 1], mixed=1)
    o = P.default_opts(tol=1e-2, max_iter=200, **kw)
    results = []
    for short in (False, True):
        lib = P.Mesh.from_inputs(m, N)
        b = torch.rand(B, lib.K, 45, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
        x = torch.zeros_like(b)

        def solve():
            try:
                lib.solve(b, x, opts=o)
            except P.DgError as e:  # 200 iterations may be too few: the iterate is what is compared
                if e.name != "DG_ERR_NOT_CONVERGED":
                    raise
        _fails_then_works(solve) if short else solve()
        results.append(x.clone())
        lib.close()
    assert bool(results[0].any()) and bool((results[0] == results[1]).all())
