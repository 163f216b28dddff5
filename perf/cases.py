"""The work that a user of this library has it do, as measurable cases.

listed() names the cases, draw() gives more of the same ranges, prepare() makes
what a program has in hand before the call, run() is one pass through the
public entry points, work() says what a pass cannot do without and exact() what
it returns in 64 bits, from the bilinear form in plain torch.

A case is a dict of plain values:
  kind   "apply" (A u), "grad" (A u and its vector-Jacobian product through
         autograd), "solve" (A x = b by preconditioned CG), "step" (one
         incompressible Navier-Stokes step)
  dim    2 (triangles) or 3 (tetrahedra)
  degree, nx, ny (grid squares, two triangles each; tetrahedra: nx^3 cubes of
         six), batch, dtype, lam (0: Poisson)
  sides  "dirichlet" (all around) or "mixed" (Neumann on the x = x1 side)
  solver for kind "solve", the p-multigrid levels: "mixed" (FP32 inside an FP64
         outer iteration) or "double" (all FP64)
"""
import functools
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_1801_00246_gb300 as P
from paper_1801_00246_gb300.autograd import sipdg_apply

DEVICE = "cuda"
FACES = {2: ((0, 1), (1, 2), (2, 0)), 3: ((0, 1, 2), (0, 1, 3), (1, 2, 3), (0, 2, 3))}
UNIT_BOX = (0.0, 1.0, 0.0, 1.0)
KOVASZNAY_BOX = (-0.5, 1.0, -0.5, 1.5)


# ---------------------------------------------------------------- the cases

def _case(name, kind, degree, nx, ny=None, dim=2, batch=1, dtype="float64", lam=0.0, sides="dirichlet", solver=""):
    return dict(name=name, kind=kind, dim=dim, degree=degree, nx=nx, ny=nx if ny is None else ny, batch=batch,
                dtype=dtype, lam=lam, sides=sides, solver=solver)


def listed():
    return [
        # the smallest mesh a user starts with (16x16 squares, degree 3): launches count
        _case("poisson_f64_n3_512tri", "apply", 3, 16),
        # the operator at the headline size, in the precision the outer iteration needs
        _case("poisson_f64_n8_524k", "apply", 8, 512),
        # a mesh that fills no tile, three fields at once, screened, with an outflow side
        _case("helmholtz_f64_n5_29k_b3", "apply", 5, 151, 97, batch=3, lam=200.0, sides="mixed"),
        # low order in single precision: the smoother's work on a coarse multigrid degree
        _case("poisson_f32_n2_524k", "apply", 2, 512, dtype="float32"),
        # the smoother's work on the finest degree
        _case("poisson_f32_n8_524k", "apply", 8, 512, dtype="float32"),
        # the top of the degree range in single precision
        _case("helmholtz_f32_n10_32k", "apply", 10, 128, dtype="float32", lam=100.0),
        # forward and backward of the operator over an ensemble of 16 fields
        _case("grad_f64_n6_32k_b16", "grad", 6, 128, batch=16),
        # the pressure solve of the headline: p-multigrid in FP32 inside an FP64 iteration
        _case("pressure_mixed_n8_524k", "solve", 8, 512, solver="mixed"),
        # an ensemble of 16 pressure right-hand sides in one solve
        _case("pressure_mixed_n6_32k_b16", "solve", 6, 128, batch=16, solver="mixed"),
        # a flow's time step: advection, the two velocity components' viscous solve, the pressure increment
        _case("flow_step_n8_8k", "step", 8, 64),
        # the operator on tetrahedra, 32^3 cubes
        _case("tet_poisson_f64_n3_196k", "apply", 3, 32, dim=3, sides="mixed"),
        # tetrahedra in single precision on a ragged mesh, two fields, screened
        _case("tet_helmholtz_f32_n4_29k_b2", "apply", 4, 17, dim=3, batch=2, dtype="float32", lam=2.5),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("apply",) * 5 + ("grad", "solve", "solve", "step", "tet", "tet"))
    dtype = rng.choice(("float64", "float64", "float32"))
    lam = rng.choice((0.0, round(math.exp(rng.uniform(0.0, math.log(6000.0))), 3)))
    sides = rng.choice(("dirichlet", "mixed"))
    if kind == "tet":
        degree = rng.randint(1, 5)
        nx = _log(rng, 4, (44, 40, 32, 24, 20)[degree - 1])
        batch = rng.choice((1, 1, 2, 3))
        c = _case("", "apply", degree, nx, dim=3, batch=batch, dtype=dtype, lam=lam, sides=sides)
    elif kind == "solve":
        solver = rng.choice(("mixed", "mixed", "double"))
        degree = rng.randint(3, 9)
        batch = rng.choice((1, 1, 2, 4))
        nx = _log(rng, 16, {"mixed": 256, "double": 128}[solver])
        ny = max(8, int(nx * rng.uniform(0.5, 1.0)))
        while batch > 1 and batch * nx * ny * _np(2, degree) > (2000000 if solver == "double" else 7000000):
            batch //= 2
        c = _case("", "solve", degree, nx, ny, batch=batch, sides=sides, solver=solver)
    elif kind == "step":
        c = _case("", "step", rng.randint(3, 8), _log(rng, 12, 60), _log(rng, 12, 60))
    else:
        degree = rng.randint(1, 10)
        squares = _log(rng, 64, 262144)
        aspect = rng.uniform(0.4, 1.0)
        nx = max(4, int(round(math.sqrt(squares / aspect))))
        ny = max(4, squares // nx)
        batch = rng.choice((1, 1, 2, 3, 4, 16))
        while batch > 1 and batch * nx * ny * _np(2, degree) > 262144 * 45:
            batch //= 2
        c = _case("", kind, degree, nx, ny, batch=batch, dtype=dtype, lam=lam, sides=sides)
    del c["name"]
    return c


# ------------------------------------------------- meshes (jittered grids)

def _np(dim, N):
    return math.comb(N + dim, dim)


def _grid(dim, nx, ny, sides, box, jitter):
    """Vertices, elements (positive orientation), face tags of a jittered grid of
    squares cut in two or cubes cut in six; the jitter's seed is 0."""
    n = (nx, ny) if dim == 2 else (nx, nx, nx)
    lo = np.array(box[0::2][:dim] if dim == 2 else (0.0,) * 3)
    hi = np.array(box[1::2][:dim] if dim == 2 else (1.0,) * 3)
    idx = np.stack(np.meshgrid(*[np.arange(k + 1) for k in n], indexing="ij"), axis=-1)
    idx = idx.transpose(*range(dim - 1, -1, -1), dim).reshape(-1, dim)  # first coordinate fastest
    X = lo + idx * ((hi - lo) / np.array(n))
    inner = np.all((idx > 0) & (idx < np.array(n)), axis=1)
    X[inner] += jitter * np.random.default_rng(0).uniform(-1, 1, (int(inner.sum()), dim)) * ((hi - lo) / np.array(n))
    X[idx == np.array(n)] = np.broadcast_to(hi, X.shape)[idx == np.array(n)]
    stride = np.cumprod([1] + [k + 1 for k in n[:-1]])
    cell = np.stack(np.meshgrid(*[np.arange(k) for k in n], indexing="ij"), axis=-1)
    cell = cell.transpose(*range(dim - 1, -1, -1), dim).reshape(-1, dim) @ stride
    orders = ((0, 1), (1, 0)) if dim == 2 else ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0))
    elems = []
    for order in orders:
        path = [0]
        for ax in order:
            path.append(path[-1] + int(stride[ax]))
        elems.append(cell[:, None] + np.array(path))
    E = np.stack(elems, axis=1).reshape(-1, dim + 1)
    vol = np.linalg.det(X[E[:, 1:]] - X[E[:, :1]])
    E[vol < 0] = E[vol < 0][:, [0, 2, 1] + ([3] if dim == 3 else [])]
    # faces: a vertex set that occurs once lies on the boundary
    faces = np.sort(np.stack([E[:, list(f)] for f in FACES[dim]], axis=1), axis=2)
    key = faces[..., 0].astype(np.int64)
    for k in range(1, dim):
        key = key * X.shape[0] + faces[..., k]
    _, inv, cnt = np.unique(key.ravel(), return_inverse=True, return_counts=True)
    first = np.argsort(inv.ravel(), kind="stable")
    start = np.concatenate([[0], np.cumsum(cnt)[:-1]])
    pair = np.full(key.size, -1, dtype=np.int64)
    two = cnt == 2
    a, b = first[start[two]], first[start[two] + 1]
    pair[a], pair[b] = b, a
    pair = pair.reshape(key.shape)
    mid = X[faces, 0].mean(axis=2)
    neumann = {"dirichlet": mid > np.inf, "mixed": mid > hi[0] - 1e-9, "pressure": mid < hi[0] - 1e-9}[sides]
    bc = np.where(pair >= 0, 0, np.where(neumann, 2, 1)).astype(np.int8)
    return X, E.astype(np.int32), bc, pair


def _box(case):
    return KOVASZNAY_BOX if case["kind"] == "step" else UNIT_BOX


def _jitter(case):
    return 0.0 if case["kind"] == "step" else 0.1


@functools.lru_cache(maxsize=2)
def _grid_of(dim, nx, ny, sides, box, jitter):
    return _grid(dim, nx, ny, sides, box, jitter)


def _of(case):
    return _grid_of(case["dim"], case["nx"], case["ny"], case["sides"], _box(case), _jitter(case))


@functools.lru_cache(maxsize=4)
def _mesh_of(dim, N, nx, ny, sides, box, jitter):
    """The handle that a program keeps for all its fields on a mesh."""
    X, E, bc, _ = _grid_of(dim, nx, ny, sides, box, jitter)
    return (P.Mesh if dim == 2 else P.TetMesh)(N, *X.T, E, bc)


def _mesh(case, sides=""):
    return _mesh_of(case["dim"], case["degree"], case["nx"], case["ny"], sides or case["sides"], _box(case), _jitter(case))


def _elements(case):
    return 2 * case["nx"] * case["ny"] if case["dim"] == 2 else 6 * case["nx"] ** 3


# ------------------------------- the bilinear form in plain torch, 64 bits

def _lattice(dim, N):
    """Exponents (a_0, ..., a_dim), |a| = N, last coordinate slowest, a_1 fastest."""
    if dim == 1:
        return [(N - i, i) for i in range(N + 1)]
    if dim == 2:
        return [(N - i - j, i, j) for j in range(N + 1) for i in range(N + 1 - j)]
    return [(N - i - j - k, i, j, k) for k in range(N + 1) for j in range(N + 1 - k) for i in range(N + 1 - j - k)]


def _lobatto(N):
    """Legendre-Gauss-Lobatto points: the ends and the roots of P_N', polished in extended precision."""
    x = np.sort(np.polynomial.Legendre.basis(N).deriv().roots().real).astype(np.longdouble) if N > 1 else np.zeros(0)
    for _ in range(4):
        p0, p1 = np.ones_like(x), x.copy()
        for n in range(1, N):
            p0, p1 = p1, ((2 * n + 1) * x * p1 - n * p0) / (n + 1)
        # (1 - x^2) P_N' = N (P_{N-1} - x P_N), and Legendre's equation for its derivative
        x = x - (p0 - x * p1) / (-(N + 1) * p1) if N > 1 else x
    return np.concatenate([[-1.0], x, [1.0]]).astype(np.longdouble)


# blend parameters of Warburton (2006), Table 1, degrees 1 to 10
_ALPHA = (0.0, 0.0, 1.4152, 0.1001, 0.2751, 0.9800, 1.0999, 1.2832, 1.3648, 1.4773)


def _nodes(dim, N, even):
    """Barycentric coordinates of the nodes: equispaced (tetrahedra and their
    faces), or warp & blend (triangles and their edges)."""
    L = np.array(_lattice(dim, N), dtype=np.longdouble) / N
    if even:
        return L
    gl, eq = _lobatto(N), np.linspace(np.longdouble(-1), np.longdouble(1), N + 1)

    def warp(x):  # displacement from equispaced to Lobatto points, interpolated at x
        w = np.zeros_like(x)
        for i in range(N + 1):
            w += (gl[i] - eq[i]) * np.prod([(x - eq[j]) / (eq[i] - eq[j]) for j in range(N + 1) if j != i], axis=0)
        return w
    if dim == 1:
        return np.stack([(1 - gl) / 2, (1 + gl) / 2], axis=1)
    out = L.copy()
    for c in range(3):  # along the edge a -> b opposite vertex c
        a, b = (c + 1) % 3, (c + 2) % 3
        x = L[:, b] - L[:, a]
        inner = np.abs(x) < 1 - 1e-12
        w = np.where(inner, warp(x) / np.where(inner, 1 - x * x, 1), 0)
        move = 4 * L[:, a] * L[:, b] * w * (1 + (_ALPHA[N - 1] * L[:, c]) ** 2) / 2
        out[:, b] += move
        out[:, a] -= move
    return out


def _bernstein(exps, lam, N):
    """Values of the Bernstein polynomials of degree N at barycentric points."""
    p = np.ones((lam.shape[0], len(exps)), dtype=np.longdouble)
    for j, a in enumerate(exps):
        f = math.factorial(N)
        for i, k in enumerate(a):
            p[:, j] *= lam[:, i] ** k
            f //= math.factorial(k)
        p[:, j] *= f
    return p


def _inverse(V):
    X = np.linalg.inv(V.astype(np.float64)).astype(np.longdouble)
    for _ in range(4):
        X = X @ (2 * np.eye(len(V), dtype=np.longdouble) - V @ X)
    return X


@functools.lru_cache(maxsize=None)
def _reference(dim, N, even):
    """Nodal mass (of a unit-measure simplex) and derivatives along lambda_b - lambda_0, b = 1..dim."""
    ex = _lattice(dim, N)
    lam = _nodes(dim, N, even)
    Vi = _inverse(_bernstein(ex, lam, N))
    Mb = np.array([[math.prod(math.comb(p + q, p) for p, q in zip(a, b)) for b in ex] for a in ex], dtype=np.longdouble)
    Mb /= math.comb(2 * N, N) * math.comb(2 * N + dim, dim)
    lower = {a: i for i, a in enumerate(_lattice(dim, N - 1))}
    Bl = _bernstein(list(lower), lam, N - 1) * N
    D = []
    for i in range(dim + 1):
        d = np.zeros((len(ex), len(ex)), dtype=np.longdouble)
        for j, a in enumerate(ex):
            if a[i]:
                d[:, j] = Bl[:, lower[tuple(v - (k == i) for k, v in enumerate(a))]]
        D.append(d @ Vi)
    return Vi.T @ Mb @ Vi, [D[b] - D[0] for b in range(1, dim + 1)], lam


class _Form:
    """The SIPDG form on a mesh: volume term, {n.grad u} and [u] on the faces with
    the penalty (N+1)(N+d)/d max(1/h-, 1/h+), h = |E| / |face|; Dirichlet faces
    u+ = -u-, grad u+ = grad u-, Neumann faces none."""

    def __init__(self, case):
        d, N = self.d, self.N = case["dim"], case["degree"]
        X, E, bc, pair = _of(case)
        dev = DEVICE
        M, D, lam = _reference(d, N, d == 3)
        to = lambda a: torch.tensor(np.asarray(a, dtype=np.float64), device=dev)  # noqa: E731
        self.M, self.D, self.Mf = to(M), [to(x) for x in D], to(_reference(d - 1, N, d == 3)[0])
        V = X[E]                                                              # K, d+1, d
        T = V[:, 1:] - V[:, :1]
        self.vol = to(np.abs(np.linalg.det(T)) / math.factorial(d))
        g = to(np.linalg.inv(T).transpose(0, 2, 1))                           # grad lambda_1..d
        self.g = torch.cat([-g.sum(1, keepdim=True), g], 1)
        V = to(V)
        self.x = torch.einsum("nv,kvd->knd", to(lam), V)
        ex = _lattice(d, N)
        of = {a: i for i, a in enumerate(_lattice(d - 1, N))}
        opp = [next(v for v in range(d + 1) if v not in f) for f in FACES[d]]
        gv = self.g[:, opp]                                                   # K, nf, d
        self.n = -gv / gv.norm(dim=2, keepdim=True)
        h = d * gv.norm(dim=2)
        self.area = h * self.vol[:, None]
        self.pair = torch.tensor(pair, device=dev)
        self.bc = torch.tensor(bc.astype(np.int64), device=dev)
        other = torch.where(self.pair >= 0, h.reshape(-1)[self.pair.clamp(min=0).reshape(-1)].reshape(h.shape), h)
        self.tau = (N + 1) * (N + d) / d * torch.maximum(h, other)
        # each face's nodes in the order of its vertices' global numbers, so that both sides agree
        nf = len(of)
        idx = np.zeros((len(E), len(FACES[d]), nf), dtype=np.int64)
        for f, vs in enumerate(FACES[d]):
            on = [i for i, a in enumerate(ex) if a[opp[f]] == 0]
            order = np.argsort(E[:, list(vs)], axis=1)
            for p in {tuple(o) for o in order}:
                row = np.zeros(nf, dtype=np.int64)
                for i in on:
                    row[of[tuple(ex[i][vs[k]] for k in p)]] = i
                idx[np.all(order == np.array(p), axis=1), f] = row
        self.idx = torch.tensor(idx, device=dev)

    def apply(self, u, lam):
        return torch.stack([self._one(v.double(), lam) for v in u.reshape(-1, *u.shape[-2:])]).reshape(u.shape)

    def _one(self, u, lam):
        K, Np = u.shape
        grad = [u @ D.T for D in self.D]
        gr = sum(self.g[:, b + 1, None, :] * grad[b][..., None] for b in range(self.d))    # K, Np, d
        z = [self.vol[:, None] * ((gr * self.g[:, b + 1, None, :]).sum(-1) @ self.M.T) for b in range(self.d)]
        out = lam * self.vol[:, None] * (u @ self.M.T) if lam else torch.zeros_like(u)
        nf = self.idx.shape[1]
        um = torch.stack([torch.gather(u, 1, self.idx[:, f]) for f in range(nf)], 1)       # K, nf, nodes
        qm = torch.stack([torch.gather((gr * self.n[:, f, None, :]).sum(-1), 1, self.idx[:, f]) for f in range(nf)], 1)
        del gr, grad
        at = self.pair.clamp(min=0).reshape(-1)
        up = um.reshape(K * nf, -1)[at].reshape(um.shape)
        qp = -qm.reshape(K * nf, -1)[at].reshape(um.shape)
        bc = self.bc[..., None]
        up = torch.where(bc == 1, -um, torch.where(bc == 2, um, up))
        qp = torch.where(bc == 1, qm, torch.where(bc == 2, -qm, qp))
        jump = um - up
        F1 = self.area[..., None] * ((self.tau[..., None] * jump - 0.5 * (qm + qp)) @ self.Mf.T)
        F2 = self.area[..., None] * ((-0.5 * jump) @ self.Mf.T)
        for f in range(nf):
            out.scatter_add_(1, self.idx[:, f], F1[:, f])
            for b in range(self.d):
                s = (self.g[:, b + 1] * self.n[:, f]).sum(-1)
                z[b].scatter_add_(1, self.idx[:, f], s[:, None] * F2[:, f])
        for b in range(self.d):
            out += z[b] @ self.D[b]
        return out


@functools.lru_cache(maxsize=1)
def _form_of(*key):
    return _Form(dict(key))


def _form(case):
    return _form_of(*sorted((k, v) for k, v in case.items() if k in ("kind", "dim", "degree", "nx", "ny", "sides", "solver")))


# ------------------------------------------------------------------ inputs

def _uniform(case, seed):
    """Fields of random values in (-1, 1): what an apply meets inside an iteration."""
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    shape = (case["batch"], _elements(case), _np(case["dim"], case["degree"]))
    u = torch.rand(shape, generator=gen, device=DEVICE, dtype=torch.float64) * 2 - 1
    u = u.to(getattr(torch, case["dtype"]))
    return u[0] if case["batch"] == 1 else u


def _waves(case, seed):
    """The pressures that a right-hand side is made for: solutions of the Laplace
    problem whose source is a sum of 16 random Fourier modes."""
    rng = np.random.default_rng(seed)
    x, y = _form(case).x.unbind(-1)
    out = []
    for _ in range(case["batch"]):
        a, k = rng.standard_normal(16), rng.integers(1, 9, (16, 2))
        u = torch.zeros_like(x)
        for m in range(16):
            kx, ky = (float(v) * math.pi for v in k[m])
            u += a[m] / (kx * kx + ky * ky) * torch.sin(kx * x) * torch.sin(ky * y)
        out.append(u)
    return out[0] if case["batch"] == 1 else torch.stack(out)


def _options(degrees, mixed=True):
    return P.default_opts(precond=P.PREC_PMG, degrees=degrees, tol=1e-10, max_iter=200, cheb_degree=3, coarse_tol=1e-2,
                          coarse_max_iter=1, coarse_amg=1, mixed=int(mixed))


def _flow(case, seed):
    """A Kovasznay flow (Re = 40) with three weak random eddies, past its start-up
    step; 32 advection substeps at degree 8 on 64 squares, in proportion below."""
    N, Re, dt = case["degree"], 40.0, 0.01
    mu, mp = _mesh(case), _mesh(case, "pressure")
    x, y = mu.nodes()
    k = Re / 2 - math.sqrt(Re * Re / 4 + 4 * math.pi ** 2)
    U = torch.stack([1 - torch.exp(k * x) * torch.cos(2 * math.pi * y),
                     k / (2 * math.pi) * torch.exp(k * x) * torch.sin(2 * math.pi * y)])
    p = 0.5 * (1 - torch.exp(2 * k * x))
    gU = U.clone()
    rng = np.random.default_rng(seed)
    for a, xc, yc in zip(rng.uniform(-0.1, 0.1, 3), rng.uniform(0.0, 0.5, 3), rng.uniform(0.0, 1.0, 3)):
        e = a * torch.exp(-40 * ((x - xc) ** 2 + (y - yc) ** 2))
        U += torch.stack([-(y - yc) * e, (x - xc) * e]) * 10
    substeps = max(4, math.ceil(32 * max(case["nx"], case["ny"]) / 64 * (N + 1) ** 2 / 81))
    degrees = [N, N // 2, 1] if N > 3 else [N, 1]
    flow = P.InsStepper(mu, mp, 1 / Re, dt, substeps, U, p, gU, p.clone(), vel_opts=_options(degrees),
                        pr_opts=_options(degrees))
    flow.step()
    return flow


def prepare(case, seed):
    if case["kind"] == "step":
        return SimpleNamespace(case=case, flow=_flow(case, seed))
    s = SimpleNamespace(case=case, mesh=_mesh(case))
    if case["kind"] == "solve":
        degrees = [case["degree"]]
        while degrees[-1] > 1:
            degrees.append(degrees[-1] // 2)
        s.options = _options(degrees, case["solver"] == "mixed")
        s.b = _form(case).apply(_waves(case, seed), case["lam"])
    else:
        s.u = _uniform(case, seed)
        if case["kind"] == "grad":
            s.w = _uniform(case, seed + (1 << 31))
    return s


def run(s):
    c = s.case
    if c["kind"] == "apply":
        return s.mesh.apply(s.u, lam=c["lam"])
    if c["kind"] == "grad":
        u = s.u.detach().requires_grad_(True)
        y = sipdg_apply(s.mesh, u, lam=c["lam"])
        return y.detach(), torch.autograd.grad(y, u, s.w)[0]
    if c["kind"] == "step":
        s.flow.step()
        return s.flow.U, s.flow.P
    return s.mesh.solve(s.b, lam=c["lam"], opts=s.options)[0]


def work(case):
    """Each field read and written once, with the elements' geometry and
    connectivity; multiply-adds of the factored operator, counted as two. A solve
    cannot do with fewer than some twenty applications of the operator; a step's
    work is its advection (interpolation to and projection from the cubature
    points in five stages a substep, three times over) and some forty applications."""
    d, N, B, K = case["dim"], case["degree"], case["batch"], _elements(case)
    size = {"float64": 8, "float32": 4}[case["dtype"]]
    n, nf = _np(d, N), _np(d - 1, N)
    one = (10 * n * n + 24 * n * nf if d == 2 else 18 * n * n + 16 * nf * nf) + (2 * n * n if case["lam"] else 0)
    fields = {"apply": 2, "grad": 4, "solve": 2, "step": 8}[case["kind"]]
    applies = {"apply": 1, "grad": 2, "solve": 20, "step": 40}[case["kind"]]
    flops = applies * B * K * one
    if case["kind"] == "step":
        substeps = max(4, math.ceil(32 * max(case["nx"], case["ny"]) / 64 * (N + 1) ** 2 / 81))
        flops += 15 * substeps * K * 16 * n * math.ceil((3 * N + 1) / 2) ** 2
    return {"bytes": float(fields * B * K * n * size + K * (d * d * size + 4 * (d + 1))), "flops": float(flops)}


def exact(case, seed):
    if case["kind"] == "step":
        return None
    if case["kind"] == "solve":
        return _waves(case, seed)
    form = _form(case)
    y = form.apply(_uniform(case, seed), case["lam"])
    if case["kind"] == "grad":  # the operator is symmetric
        return y, form.apply(_uniform(case, seed + (1 << 31)), case["lam"])
    return y
