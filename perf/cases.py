"""Performance cases: the calls that a user of the library makes, from the
smallest tangent to the 4.34M-unknown one, through its public entry points.

Kinds of work:
  solve     one nested solve of a tangent whose preconditioner is built
  tangent   a new tangent on a known pattern: new values, preconditioner, solve
  numeric   the same on the kept aggregates (numeric re-setup)
  adjoint   a differentiable solve, forward and backward (dL/db, dL/dr)
  batch     many independent uneven tangents in one batched solve
  newton    one predictor multi-corrector time step with on-device assembly
  assemble  the VMS residual and its tangent values at one state

Solves run to a relative residual of 1e-11 (1e-12 in the adjoint): the outer
iteration is FP64 in every precision mode, and a solution to that tolerance
is one that users can difference or compare between modes.  All inputs come
from the seed: the perturbation of the velocity the tangent is linearised
about and the right-hand side (time step: Reynolds number, resistances).
"""
import dataclasses
import math

import numpy as np
import torch

import synth
from paper_1911_10814_gb300 import BatchSolver, Solver, Vms
from paper_1911_10814_gb300.autograd import nested_solve

DEV = "cuda:0"
RTOL = 1e-11


def _box(kind, name, nx, ny, nz, Lz, Re, n_out, Rmin, Rmax, precision):
    return dict(kind=kind, name=name, nx=nx, ny=ny, nz=nz, Lz=float(Lz), Re=float(Re), n_out=n_out,
                Rmin=float(Rmin), Rmax=float(Rmax), precision=precision)


def listed():
    return [
        # smallest call: the 2,916-unknown cube in plain FP64; latency and launches are all it costs
        _box("solve", "solve_cube8_fp64", 8, 8, 8, 1, 100, 1, 1e3, 1e3, 0),
        # a coarse mesh in a Newton loop: every tangent is new, the preconditioner is rebuilt for it
        _box("tangent", "tangent_cube16", 16, 16, 16, 1, 300, 2, 1e2, 1e4, 4),
        # an odd-sized vessel, no dimension a multiple of a warp or a slice; FP32 inner values
        _box("solve", "solve_19x23x61_fp32", 19, 23, 61, 3, 700, 3, 1e2, 1e4, 1),
        # plain FP64 at an ordinary size: what results are checked against
        _box("solve", "solve_24x24x96_fp64", 24, 24, 96, 4, 500, 1, 1e3, 1e3, 0),
        # the ordinary Newton tangent (0.56M unknowns): new values, full preconditioner, solve
        _box("tangent", "tangent_32x32x128", 32, 32, 128, 4, 2000, 4, 1e2, 1e5, 4),
        # the same on the aggregates of an earlier tangent of the time step
        _box("numeric", "numeric_32x32x128", 32, 32, 128, 4, 2000, 4, 1e2, 1e5, 3),
        # parameter estimation: gradient of a loss over outlet flows, forward and transposed solve
        _box("adjoint", "adjoint_32x32x128", 32, 32, 128, 4, 300, 4, 1e2, 1e4, 1),
        # many small independent tangents (cubes of 12 to 40 hexes a side) at once
        dict(kind="batch", name="batch_16", count=16, smin=12, smax=40, shapes=3, precision=4),
        # one time step: predictor, residuals, FP32 tangents, one preconditioner, nested solves, outlets
        _box("newton", "newton_32x32x128", 32, 32, 128, 4, 2000, 4, 1e3, 1e3, 3),
        # the assembly alone with the exact FP64 tangent
        _box("assemble", "assemble_32x32x128", 32, 32, 128, 4, 2000, 4, 1e3, 1e3, 0),
        # a large new tangent (1.85M unknowns): setup and solve
        _box("tangent", "tangent_48x48x192", 48, 48, 192, 4, 2000, 4, 1e2, 1e5, 4),
        # the largest: the 4,343,300-unknown box at Re 2000, preconditioner built before
        _box("solve", "solve_64x64x256", 64, 64, 256, 4, 2000, 4, 1e2, 1e5, 4),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case: a kind, a box of its range (log-uniform sizes, each side on
    its own, so most are odd), Reynolds number, outlets, precision mode."""
    kind = rng.choice(["solve", "solve", "tangent", "tangent", "numeric", "adjoint", "batch", "newton", "assemble"])
    if kind == "batch":
        smin = rng.randint(8, 16)
        return dict(kind=kind, count=rng.randint(3, 16), smin=smin, smax=smin + rng.randint(4, 20),
                    shapes=rng.randint(0, 999), precision=rng.choice([1, 3, 4]))
    top = {"solve": 56, "tangent": 48, "numeric": 40, "adjoint": 32, "newton": 32, "assemble": 32}[kind]
    n = _log(rng, 8, top)
    elong = rng.choice([1, 2, 3, 4])
    nx, ny = (max(6, round(n * rng.uniform(0.85, 1.15))) for _ in range(2))
    nz = max(8, round(n * elong * rng.uniform(0.85, 1.15)))
    precision = {"adjoint": 1, "newton": 3, "assemble": 0}.get(kind) or rng.choice([0, 1, 3, 4, 4])
    if precision == 0:   # FP64 everywhere costs about four times the mixed modes
        nx, ny, nz = min(nx, 32), min(ny, 32), min(nz, 128)
    Re = rng.uniform(500, 2000) if kind in ("newton", "assemble") else rng.uniform(100, 2000)
    Rmin, Rmax = (1e3, 1e3) if kind in ("newton", "assemble") else (1e2, 1e4)
    c = _box(kind, "", nx, ny, nz, elong, round(Re, 1), rng.randint(1, 4), Rmin, Rmax,
             0 if kind == "assemble" else precision)
    del c["name"]
    return c


# ------------------------------------------------------------------- inputs
def _spec(case, seed):
    u = synth.uniforms(seed ^ 0x5EED, 8)
    lo, hi = math.log10(case["Rmin"]), math.log10(case["Rmax"])
    if case["kind"] == "newton":   # equal outlets, no perturbation: a consistent start (see _newton)
        R, Re, pert = (case["Rmin"] * (0.9 + 0.2 * u[0]),) * case["n_out"], case["Re"] * (0.95 + 0.05 * u[1]), 0.0
    else:
        R, Re, pert = tuple(float(10.0 ** (lo + (hi - lo) * u[k])) for k in range(case["n_out"])), case["Re"], 0.05
    return synth.MeshSpec(case["nx"], case["ny"], case["nz"], Lz=case["Lz"], Re=Re, pert=pert, seed=seed, R=R)


def _gpu(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64), device=DEV)


def _values(d):
    return [_gpu(np.asarray(d[k]).reshape(-1)) for k in "ABCD"]


def _newton(case, spec, d):
    """Consistent start of a time step: smooth Poiseuille velocity, the outlet
    model at rest, a uniform pressure equal to the mean outlet pressure."""
    s = Solver(d, precision=case["precision"], rtol=RTOL)
    vm = Vms(s, synth.mesh(spec), spec.rho, spec.mu, spec.dt, spec.rho_inf)
    R, N = np.asarray(spec.R), d["n_nodes"]
    v0 = _gpu(d["vel"])
    Q0 = s.outlet_flows(v0)
    rcr = dict(Rp=_gpu(0.1 * R), Rd=_gpu(0.9 * R), C=_gpu(0.1 / R), Pd=_gpu(np.zeros(len(R))))
    rcr["Pi"] = rcr["Rd"] * Q0
    P0 = (rcr["Rp"] * Q0 + rcr["Pi"]).mean()
    y = torch.cat([v0, torch.ones(N, dtype=torch.float64, device=DEV) * P0])
    return dict(s=s, vm=vm, rcr=rcr, y=y, yd=torch.zeros_like(y))


def _vms_state(spec, d, seed):
    """A state off equilibrium: perturbed velocity, random accelerations and
    pressures, outlet pressures."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    N = d["n_nodes"]
    nrm = lambda n: torch.randn(n, dtype=torch.float64, device=DEV, generator=g)  # noqa: E731
    v = _gpu(d["vel"]) * (1.0 + 0.3 * nrm(3 * N))
    P = 1e3 * (1.0 + 0.3 * nrm(spec.n_out))
    return 40.0 * nrm(3 * N), v, 80.0 * nrm(N), P


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        specs = synth.batch(case["count"], case["shapes"], case["smin"], case["smax"])   # sizes, Re, outlets: the case's
        ds = [synth.generate(dataclasses.replace(sp, seed=1000 * seed + i)) for i, sp in enumerate(specs)]
        B = BatchSolver(ds, precision=case["precision"], rtol=RTOL)
        B.setup()
        return dict(kind=kind, B=B, bs=[_gpu(d["b"]) for d in ds])
    spec = _spec(case, seed)
    d = synth.generate(spec)
    if kind == "newton":
        return dict(kind=kind, **_newton(case, spec, d))
    if kind == "assemble":
        s = Solver(d)
        vm = Vms(s, synth.mesh(spec), spec.rho, spec.mu, spec.dt, spec.rho_inf, tangent_fp32=False)
        vd, v, p, P = _vms_state(spec, d, seed)
        return dict(kind=kind, s=s, vm=vm, vd=vd, v=v, p=p, P=P)
    s = Solver(d, precision=case["precision"], rtol=1e-12 if kind == "adjoint" else RTOL)
    st = dict(kind=kind, s=s, b=_gpu(d["b"]))
    if kind != "tangent":   # a tangent's preconditioner is part of its pass
        s.setup()
    if kind in ("tangent", "numeric"):
        st["values"] = _values(d)
    if kind == "adjoint":
        a = torch.zeros((spec.n_out, 3 * d["n_nodes"]), dtype=torch.float64)
        for k in range(spec.n_out):
            sl = slice(d["out_ptr"][k], d["out_ptr"][k + 1])
            a[k, torch.as_tensor(d["out_idx"][sl], dtype=torch.long)] = torch.as_tensor(d["out_val"][sl])
        st["b"].requires_grad_(True)
        st.update(a=a.to(DEV), r=torch.tensor(d["r"], dtype=torch.float64, device=DEV, requires_grad=True),
                  q=_gpu(synth.uniforms(seed ^ 0xA11, spec.n_out)))
    return st


def run(st):
    kind = st["kind"]
    if kind == "batch":
        xs, _ = st["B"].solve(st["bs"])
        return xs
    s = st["s"]
    if kind == "newton":
        y, yd, Pi, _ = st["vm"].newton_step(st["y"], st["yd"], st["rcr"], tol_R=1e-6, tol_A=1e-10, l_max=20, nts=10,
                                            pc_rebuild=1)
        return dict(y=y, yd=yd, Pi=Pi)
    if kind == "assemble":
        out = st["vm"].tangent(st["vd"], st["v"], st["p"])
        return dict(out, R=st["vm"].residual(st["vd"], st["v"], st["p"], st["P"]))
    if kind == "adjoint":
        x = nested_solve(st["b"], st["r"], s)
        flow = st["a"] @ x[:st["a"].shape[1]]
        gb, gr = torch.autograd.grad(((flow - st["q"]) ** 2).sum(), (st["b"], st["r"]))
        return dict(x=x.detach(), gb=gb, gr=gr)
    if kind in ("tangent", "numeric"):
        s.set_values(*st["values"])
        s.setup(numeric=kind == "numeric")
    x, _ = s.solve(st["b"])
    return x


# --------------------------------------------------------------------- work
def _nnz(nx, ny, nz):
    """Entries of the node graph: every node, and both ends of the tets' edges
    (three axis, three face-diagonal, one body-diagonal direction)."""
    edges = (nx * (ny + 1) * (nz + 1) + (nx + 1) * ny * (nz + 1) + (nx + 1) * (ny + 1) * nz + nx * ny * (nz + 1)
             + nx * (ny + 1) * nz + (nx + 1) * ny * nz + nx * ny * nz)
    return (nx + 1) * (ny + 1) * (nz + 1) + 2 * edges


def _solve_work(nx, ny, nz):
    """A solve reads the tangent (16 FP64 values and a column per entry) and b
    and writes x; its least arithmetic is one product with the tangent."""
    z, n = _nnz(nx, ny, nz), 4 * (nx + 1) * (ny + 1) * (nz + 1)
    return 132.0 * z + 16.0 * n, 32.0 * z


def work(case):
    if case["kind"] == "batch":
        mean = (case["smin"] + case["smax"]) / 2.0
        b, f = _solve_work(mean, mean, mean)
        return {"bytes": case["count"] * b, "flops": case["count"] * f}
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    z, n, E = _nnz(nx, ny, nz), (nx + 1) * (ny + 1) * (nz + 1), 6.0 * nx * ny * nz
    if case["kind"] == "assemble":
        # 4 node ids per tet, 3 coordinates and 7 state values per node in; 16 values per entry and
        # 4 residual rows per node out; about 5 kflop per tet for its 16 x 16 tangent and its rows
        return {"bytes": 16 * E + 80.0 * n + 132.0 * z + 32.0 * n, "flops": 5e3 * E}
    b, f = _solve_work(nx, ny, nz)
    if case["kind"] == "newton":   # state in and out, the mesh, and at least one tangent and its solve
        return {"bytes": b + 16 * E + 128.0 * n + 132.0 * z, "flops": f + 5e3 * E}
    if case["kind"] == "adjoint":  # forward and transposed solve
        return {"bytes": 2 * b, "flops": 2 * f}
    return {"bytes": b + (132.0 * z if case["kind"] in ("tangent", "numeric") else 0.0), "flops": f}


# -------------------------------------------------------------------- exact
def _dense(d, r):
    """The tangent [[A + sum r a a^T, B], [C, D]] as one dense FP64 matrix."""
    N = d["n_nodes"]
    rows = torch.repeat_interleave(torch.arange(N), torch.as_tensor(np.diff(d["rowptr"]))).to(DEV)
    cols = torch.as_tensor(d["col"], dtype=torch.long, device=DEV)
    M = torch.zeros((4 * N, 4 * N), dtype=torch.float64, device=DEV)
    A, B, C, D = (_gpu(d[k]) for k in "ABCD")
    for i in range(3):
        for j in range(3):
            M[3 * rows + i, 3 * cols + j] = A[:, i, j]
        M[3 * rows + i, 3 * N + cols] = B[:, i]
        M[3 * N + rows, 3 * cols + i] = C[:, i]
    M[3 * N + rows, 3 * N + cols] = D
    for k in range(len(r)):
        sl = slice(d["out_ptr"][k], d["out_ptr"][k + 1])
        i, v = torch.as_tensor(d["out_idx"][sl], dtype=torch.long, device=DEV), _gpu(d["out_val"][sl])
        M[i[:, None], i[None, :]] += r[k] * v[:, None] * v[None, :]
    return M


def _lu_solve(d, spec, b):
    """Dense LU of the equilibrated tangent, with three steps of refinement."""
    M = _dense(d, d["r"])
    sr = 1.0 / M.abs().amax(1, keepdim=True)
    Ms = M * sr
    sc = 1.0 / Ms.abs().amax(0, keepdim=True)
    LU, piv = torch.linalg.lu_factor(Ms * sc)

    def back(v):
        return (sc.T * torch.linalg.lu_solve(LU, piv, sr * v[:, None]))[:, 0]

    x = back(b)
    for _ in range(3):
        x = x + back(b - M @ x)
    return x


def _tet_rows(spec, w, u_tau, X):
    """The 16 residual rows of one tet (per node: momentum x, y, z, continuity)
    in the values w (4 nodes x (vdot, v, p)); tau at the velocity u_tau."""
    rho, mu = spec.rho, spec.mu
    ud, u, p = w[:, 0:3], w[:, 3:6], w[:, 6]
    e = X[1:] - X[0]
    det = torch.dot(e[0], torch.linalg.cross(e[1], e[2]))
    g = torch.stack([torch.linalg.cross(e[1], e[2]), torch.linalg.cross(e[2], e[0]), torch.linalg.cross(e[0], e[1])]) / det
    dN = torch.cat([-g.sum(0, keepdim=True), g])
    G = 2.0 ** (1.0 / 3.0) / 2.0 * dN.T @ dN
    grad, gp = u.T @ dN, p @ dN
    div = grad.diagonal().sum()
    hi, lo = (5.0 + 3.0 * math.sqrt(5.0)) / 20.0, (5.0 - math.sqrt(5.0)) / 20.0
    wq = det.abs() / 24.0
    Rm, Rp = 0.0, 0.0
    for q in range(4):
        Nq = torch.tensor([hi if k == q else lo for k in range(4)], dtype=torch.float64, device=w.device)
        uq, udq, ut, pq = Nq @ u, Nq @ ud, Nq @ u_tau, Nq @ p
        tauM = 1.0 / (rho * torch.sqrt(4.0 / spec.dt ** 2 + ut @ G @ ut + 36.0 * (mu / rho) ** 2 * (G * G).sum()))
        tauC = 1.0 / (tauM * G.diagonal().sum())
        cv = grad @ uq
        vp = -tauM * (rho * udq + rho * cv + gp)
        m = rho * Nq[:, None] * (udq + cv + grad @ vp)[None, :]
        m = m - (pq - tauC * div) * dN + mu * dN @ (grad + grad.T)
        m = m - rho * (dN @ (uq + vp))[:, None] * vp[None, :]
        Rm = Rm + wq * m
        Rp = Rp + wq * (Nq * div - dN @ vp)
    return torch.cat([Rm, Rp[:, None]], 1).reshape(16)


def _tri_rows(spec, u, X):
    """The 9 backflow rows of one outlet triangle (beta = 0.2)."""
    n = torch.linalg.cross(X[1] - X[0], X[2] - X[0])
    length = torch.linalg.norm(n)
    n = n / length
    out = 0.0
    for q in range(3):
        Nq = torch.tensor([2.0 / 3.0 if k == q else 1.0 / 6.0 for k in range(3)], dtype=torch.float64, device=u.device)
        uq = Nq @ u
        out = out - length / 6.0 * spec.rho * 0.2 * torch.clamp(uq @ n, max=0.0) * Nq[:, None] * uq[None, :]
    return out.reshape(9)


def _assemble(spec, d, m, vd, v, p, P):
    N = d["n_nodes"]
    X, tets = _gpu(m["X"]), torch.as_tensor(m["tets"], dtype=torch.long, device=DEV)
    tris = torch.as_tensor(m["tris"], dtype=torch.long, device=DEV)
    wall = torch.as_tensor(m["dir"], device=DEV) != 0
    am, cc = (3.0 - spec.rho_inf) / (2.0 * (1.0 + spec.rho_inf)), spec.alpha_f_gamma_dt
    U, UD = v.view(N, 3), vd.view(N, 3)
    rows = torch.repeat_interleave(torch.arange(N), torch.as_tensor(np.diff(d["rowptr"]))).to(DEV)
    cols = torch.as_tensor(d["col"], dtype=torch.long, device=DEV)
    key = rows * N + cols
    K = torch.zeros((len(cols), 4, 4), dtype=torch.float64, device=DEV)
    R = torch.zeros((N, 4), dtype=torch.float64, device=DEV)
    tet = torch.func.vmap(lambda w, ut, x: _tet_rows(spec, w, ut, x))
    tet_j = torch.func.vmap(torch.func.jacfwd(lambda w, ut, x: _tet_rows(spec, w, ut, x)))
    for nd in torch.split(tets, 1 << 16):
        w = torch.cat([UD[nd], U[nd], p[nd][..., None]], 2)
        R.index_add_(0, nd.reshape(-1), tet(w, U[nd], X[nd]).reshape(-1, 4))
        J = tet_j(w, U[nd], X[nd]).reshape(-1, 4, 4, 4, 7)
        J = torch.cat([am * J[..., 0:3] + cc * J[..., 3:6], cc * J[..., 6:]], -1).permute(0, 1, 3, 2, 4)
        slot = torch.searchsorted(key, (nd[:, :, None] * N + nd[:, None, :]).reshape(-1))
        K.index_add_(0, slot, J.reshape(-1, 4, 4))
    if len(tris):
        f = lambda u, x: _tri_rows(spec, u, x)  # noqa: E731
        R[:, :3].index_add_(0, tris.reshape(-1), torch.func.vmap(f)(U[tris], X[tris]).reshape(-1, 3))
        J = cc * torch.func.vmap(torch.func.jacfwd(f))(U[tris], X[tris]).reshape(-1, 3, 3, 3, 3).permute(0, 1, 3, 2, 4)
        slot = torch.searchsorted(key, (tris[:, :, None] * N + tris[:, None, :]).reshape(-1))
        K[:, :3, :3].index_add_(0, slot, J.reshape(-1, 3, 3))
    flat = torch.zeros(3 * N, dtype=torch.float64, device=DEV)
    for k in range(spec.n_out):
        sl = slice(d["out_ptr"][k], d["out_ptr"][k + 1])
        flat.index_add_(0, torch.as_tensor(d["out_idx"][sl], dtype=torch.long, device=DEV), P[k] * _gpu(d["out_val"][sl]))
    R[:, :3] += flat.view(N, 3)
    R[wall, :3] = 0.0
    A = K[:, :3, :3].clone()
    fixed = wall[rows] | wall[cols]
    keep = torch.eye(3, dtype=torch.float64, device=DEV)[None] * (rows == cols)[:, None, None]
    A[fixed] = (A * keep)[fixed]
    B = K[:, :3, 3] * (~wall[rows])[:, None]
    C = K[:, 3, :3] * (~wall[cols])[:, None]
    return dict(A=A.reshape(-1), B=B.reshape(-1), C=C.reshape(-1), D=K[:, 3, 3].clone(),
                R=torch.cat([R[:, :3].reshape(-1), R[:, 3]]))


def exact(case, seed):
    """The assembly by automatic differentiation and small tangents by dense LU,
    in FP64; None for the solves that a dense factorisation cannot do quickly."""
    if case["kind"] in ("batch", "newton", "adjoint"):
        return None
    spec = _spec(case, seed)
    if case["kind"] == "assemble":
        d = synth.generate(spec)
        vd, v, p, P = _vms_state(spec, d, seed)
        return _assemble(spec, d, synth.mesh(spec), vd, v, p, P)
    if 4 * spec.n_nodes > 20000:
        return None
    d = synth.generate(spec)
    return _lu_solve(d, spec, _gpu(d["b"]))
