"""The work this library is timed on: full time steps of the ADER-DG scheme with its subcell
limiter over the grids, degrees, precisions and boundary kinds that its tests, its benchmark and
its serving loop use, the limiter's stand-alone patch update, and a resume from host memory.

A stepping case holds a checkpoint of its whole grid in device memory, as a parameter study or a
slab of a decomposed grid does.  One pass puts the checkpoint into the state
(`Solver.unpack_cells`), takes the case's steps and hands the new level back in device memory
(`Solver.pack_cells`), so that every pass does the same work however often it runs.
"""
import numpy as np
import torch

from paper_1406_7416_gb300 import adg, inputs

GAMMA = 1.4
FP64, MIXED = adg.PREC_FP64, adg.PREC_MIXED_FP32
# scratch of the stand-alone patch update (include/adg.h): 32 MiB, less what its tables take
SCRATCH = 31 * 1024 * 1024


def _case(name, kind, N, n, steps, prec, **more):
    c = dict(kind=kind, N=N, nx=n[0], ny=n[1], nz=n[2] if len(n) > 2 else 0, steps=steps,
             prec="fp64" if prec == FP64 else "mixed")
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest grid of the benchmark's workloads: a step is a chain of short kernels
        _case("explosion2d_32_N3_mixed", "explosion", 3, (32, 32), 8, MIXED),
        # the benchmark's default workload: quadrants + vortex, 512 x 512, N = 5, mixed precision
        _case("quadvortex_512_N5_mixed", "quadvortex", 5, (512, 512), 8, MIXED),
        # the same data in the binding's default precision, on a grid that fits a shorter run
        _case("quadvortex_256_N5_fp64", "quadvortex", 5, (256, 256), 4, FP64),
        # the benchmark's highest degree: 200 x 200, N = 9, mixed (one FP64 sweep)
        _case("quadrants_200_N9_mixed", "quadrants", 9, (200, 200), 3, MIXED),
        # the 3D explosion of the benchmark at half its resolution, mixed precision
        _case("explosion3d_64_N3_mixed", "explosion", 3, (64, 64, 64), 4, MIXED),
        # the 3D explosion in FP64, on a ragged grid
        _case("explosion3d_33_N3_fp64", "explosion", 3, (33, 29, 30), 2, FP64),
        # the double Mach reflection on the paper's mesh: inflow, wall and moving-front faces
        _case("double_mach_350x100_N5_mixed", "dmr", 5, (350, 100), 8, MIXED),
        # a closed 3D box, reflecting walls on every face, odd extents, N = 2
        _case("box3d_37_N2_mixed", "box", 2, (37, 30, 26), 4, MIXED),
        # the smooth vortex of the convergence table in FP64, limiter quiet, odd extents, fixed steps
        _case("vortex_67_N6_fp64", "vortex", 6, (67, 53), 4, FP64),
        # the serving loop's shared launches: sixteen runs of the Riemann problems of mixed sizes
        _case("serving_batch16_mixed", "batch", 0, (0, 0), 8, MIXED, members=16, structure=4),
        # the limiter's patch update on caller-owned buffers, the most patches of 2D N = 5
        _case("subcell_update_N5_146", "subcell", 5, (0, 0), 1, FP64, dim=2, count=146),
        # resume from host memory: load, steps with the flags read back each step, read
        _case("resume_128_N5_mixed", "resume", 5, (128, 128), 4, MIXED),
    ]


# ---------------------------------------------------------------------------
# work of one pass
# ---------------------------------------------------------------------------
def _dim(case):
    if case["kind"] == "subcell":
        return case["dim"]
    return 3 if case["nz"] else 2


def _members(case):
    """(n, N, configuration) of each run of a batch, by the case alone."""
    rng = np.random.default_rng(case["structure"])
    return [(int(rng.choice((32, 64, 128))), int(rng.choice((3, 5))),
             int(rng.integers(len(inputs.RP2D)))) for _ in range(case["members"])]


def _step_flops(D, N):
    """Arithmetic of one cell's unlimited step: N + 1 Picard sweeps (the first on time-constant
    data), the final stage, face fluxes, corrector and the projection on the subcells."""
    n, nv, ns = N + 1, D + 2, 2 * N + 1
    nst, nd, nf = n ** (D + 1), n ** D, n ** (D - 1)
    flux = D * D + 5 * D + 5
    sweep = nst * flux + nv * nst * (D + 1) * 2 * n
    first = nd * flux + nv * nd * (D * 2 * n + 2 * n)
    final = nst * flux + D * nv * nst * 2 + nv * nd * D * 2 * n + 2 * D * nv * nf * n * 2 * n
    faces = D * nf * n * (2 * flux + 10)
    proj = sum(nv * ns ** (k + 1) * n ** (D - 1 - k) * 2 * n for k in range(D))
    return (N * sweep + first + final + faces + proj
            + nv * nd * D * 4 + ns ** D * (4 * D + 6))


def _patch_flops(D, N):
    """Arithmetic of one patch of the limiter: WENO3 sweeps, degree-2 predictors of the subcells
    and their face ghosts, sub-face fluxes and the update."""
    nv, ns = D + 2, 2 * N + 1
    L, ne = ns + 6, ns + 2
    weno = sum(nv * ne ** (k + 1) * L ** (D - 1 - k) * 3 ** k * 75 for k in range(D))
    subs = ns ** D + 2 * D * ns ** (D - 1)
    flux = D * D + 5 * D + 5
    nst, nd = 3 ** (D + 1), 3 ** D
    pred = subs * (2 * (nst * flux + nv * nst * (D + 1) * 6) + nd * flux + nv * nd * (D + 1) * 6)
    faces = D * (ns + 1) * ns ** (D - 1) * 3 ** D * (2 * flux + 10 + 12 * nv)
    return weno + pred + faces + nv * ns ** D * D * 3


def work(case):
    D = _dim(case)
    if case["kind"] == "subcell":
        N, nv, ns = case["N"], D + 2, 2 * case["N"] + 1
        vals = nv * ((ns + 6) ** D + ns ** D + 2 * D * ns ** (D - 1))
        return dict(bytes=8 * case["count"] * vals, flops=case["count"] * _patch_flops(D, N))
    if case["kind"] == "batch":
        cells = [(n * n, N) for n, N, _ in _members(case)]
    else:
        cells = [(case["nx"] * case["ny"] * max(1, case["nz"]), case["N"])]
    # the level in and out (DOFs, extrema, flag of each cell); limited cells' subcell rows and
    # their arithmetic depend on the data and are not counted
    nbytes = sum(c * 2 * (8 * (D + 2) * ((N + 1) ** D + 2) + 1) for c, N in cells)
    return dict(bytes=nbytes, flops=case["steps"] * sum(c * _step_flops(D, N) for c, N in cells))


# ---------------------------------------------------------------------------
# drawn cases
# ---------------------------------------------------------------------------
def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    """One more case of the listed families.  Grids are drawn over the logarithm of their size and
    are cut so that a pass stays below the largest listed one's cost in its precision."""
    kind = rng.choice(("explosion", "explosion", "quadvortex", "quadvortex", "quadrants", "riemann",
                       "dmr", "tube", "box", "vortex", "batch", "subcell", "resume"))
    if kind == "batch":
        return _case(None, "batch", 0, (0, 0), rng.randint(2, 8), MIXED, members=rng.randint(2, 20),
                     structure=rng.randint(0, 10 ** 6))
    if kind == "subcell":
        dim = rng.choice((2, 2, 3))
        N = rng.randint(1, 9 if dim == 2 else 3)
        return _case(None, "subcell", N, (0, 0), 1, FP64, dim=dim,
                     count=_log(rng, 1, _patches(dim, N)))
    dim = 3 if kind in ("explosion", "box") and rng.random() < 0.5 else 2
    N = rng.randint(1, 3) if dim == 3 else rng.randint(1, 9)
    prec = FP64 if kind in ("vortex", "tube") or rng.random() < 0.4 else MIXED
    steps = rng.randint(2, 4)
    if kind == "vortex":
        N = max(N, 3)                   # below it these grids are too coarse for a quiet limiter
    if kind == "resume":
        n = (_log(rng, 24, 160), _log(rng, 24, 160))
    elif kind == "dmr":
        nx = _log(rng, 70, 420)
        n = (nx, max(10, nx * 2 // 7))
    elif kind == "tube":
        n = (_log(rng, 20, 200), _log(rng, 5, 50))
    elif dim == 3:
        n = tuple(_log(rng, 10, 64) for _ in range(3))
    else:
        lo = 24 if kind == "vortex" else 16
        n = (_log(rng, lo, 512), _log(rng, lo, 512))
        if max(n) > 4 * min(n):         # cells no flatter than 1 : 4
            n = (max(n[0], n[1] // 4), max(n[1], n[0] // 4))
    limit = 4e10 if prec == FP64 else 3e11
    need = steps * _step_flops(dim, N)
    while need * int(np.prod(n)) > limit:
        n = tuple(max(16, x * 4 // 5) for x in n)
    more = {}
    if kind == "riemann":
        more["config"] = rng.randint(0, len(inputs.RP2D) - 1)
    return _case(None, kind, N, n, steps, prec, **more)


def _patches(dim, N):
    """Patches that the stand-alone update's scratch holds."""
    nv, ns = dim + 2, 2 * N + 1
    L, ne = ns + 6, ns + 2
    per = nv * ((ne * L * 3 + ne * ne * 9) if dim == 2 else
                (ne * L * L * 3 + ne * ne * L * 9 + ne ** 3 * 27))
    per += ne ** dim * nv * 3 ** (dim + 1) + dim * nv * (ns + 1) * ns ** (dim - 1)
    return max(1, SCRATCH // (8 * per))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _stretch(w, n):
    """The workload on its own domain with n[k] cells along axis k."""
    size = [w["dx"][k] * w["ncell"][k] for k in range(w["dim"])]
    w["ncell"] = tuple(n)
    w["dx"] = tuple(size[k] / n[k] for k in range(w["dim"]))
    return w


def _jitter(states, rng, by=0.02):
    """Densities and pressures scaled by a seeded factor, as the serving runs' are."""
    out = []
    for s in states:
        s = list(s)
        s[0] *= 1.0 + rng.uniform(-by, by)
        s[-1] *= 1.0 + rng.uniform(-by, by)
        out.append(tuple(s))
    return out


def _workload(case, seed):
    kind, N, D = case["kind"], case["N"], _dim(case)
    n = (case["nx"], case["ny"], case["nz"])[:D]
    rng = np.random.default_rng(seed)
    if kind == "explosion" and D == 3:
        w = _stretch(inputs.explosion_3d(n=2, N=N), n)
        w["problem"]["cell_rho_factor"] = 1.0 + 0.01 * rng.uniform(-1.0, 1.0, size=n)
    elif kind in ("explosion", "box"):
        w = inputs.closed_box(n=2, N=N, dim=D) if kind == "box" else inputs.explosion_2d(n=2, N=N)
        w = _stretch(w, n)
        pr = w["problem"]
        pr["inner"], pr["outer"] = _jitter((pr["inner"], pr["outer"]), rng)
        pr["radius"] *= 1.0 + rng.uniform(-0.05, 0.05)
    elif kind in ("quadvortex", "resume", "quadrants"):
        w = inputs.quadrants_2d(n=2, N=N) if kind == "quadrants" else inputs.quadrants_vortex_2d(n=2, N=N)
        w = _stretch(w, n)
        w["problem"]["states"] = _jitter(w["problem"]["states"], rng)
    elif kind == "riemann":
        w = _stretch(inputs.riemann_2d(2, N, case["config"], jitter=0.02, rng=rng), n)
    elif kind == "tube":
        w = inputs.shock_tube("sod" if seed % 2 else "lax", nx=n[0], ny=n[1], N=N)
        # the inflow faces keep the tube's printed states; the data start off them by up to 2%
        w["problem"]["states"] = [tuple(s) for s in w["problem"]["states"]]
        left, right = w["problem"]["states"][1], w["problem"]["states"][0]
        left, right = _jitter((left, right), rng)
        w["problem"]["states"] = [right, left, left, right]
    elif kind == "dmr":
        w = inputs.double_mach(nx=n[0], ny=n[1], N=N)
        pr = w["problem"]
        pr["inner"], pr["outer"] = _jitter((pr["inner"], pr["outer"]), rng, 0.005)
    else:
        raise ValueError(kind)
    return w


class Grid:
    """A state with its whole level in a device buffer, and a buffer for the level it reaches."""

    def __init__(self, solver, stream=0):
        self.solver = solver
        if stream:
            solver.set_stream(stream)
        self.hi = solver.ncell
        self.lo = (0,) * solver.dim
        count = solver.cells
        nbytes = solver.halo_bytes(count)
        words = (nbytes + 7) // 8
        self.start = torch.zeros(words, dtype=torch.float64, device="cuda")
        self.end = torch.zeros(words, dtype=torch.float64, device="cuda")
        a = count * solver.nvar * solver.nodes
        b = a + count * solver.nvar * solver.subcells
        c = b + count * solver.nvar * 2
        self.out = dict(
            dofs=self.end[:a].view(count, solver.nvar, solver.nodes),
            subcells=self.end[a:b].view(count, solver.nvar, solver.subcells),
            extrema=self.end[b:c].view(count, solver.nvar, 2),
            flags=self.end.view(torch.uint8)[8 * c:8 * c + count])
        torch.cuda.current_stream().synchronize()
        self.solver.pack_cells(self.lo, self.hi, self.start.data_ptr())

    def restore(self):
        self.solver.unpack_cells(self.lo, self.hi, self.start.data_ptr())

    def result(self):
        self.solver.pack_cells(self.lo, self.hi, self.end.data_ptr())
        return self.out


def _prec(case):
    return FP64 if case["prec"] == "fp64" else MIXED


def _vortex_setup(case, seed):
    """Nodal values of the isentropic vortex at the Gauss-Legendre nodes, the cell sizes and the
    step: the data a program with its own initial condition loads."""
    N, nx, ny = case["N"], case["nx"], case["ny"]
    rng = np.random.default_rng(seed)
    cx, cy = rng.uniform(-0.5, 0.5, 2)
    beta = 5.0 * (1.0 + rng.uniform(-0.02, 0.02))
    xi = 0.5 * (np.polynomial.legendre.leggauss(N + 1)[0] + 1.0)
    dx, dy = 10.0 / nx, 10.0 / ny
    x = (-5.0 + (np.arange(nx)[:, None] + xi) * dx).reshape(1, nx, 1, N + 1) - cx
    y = (-5.0 + (np.arange(ny)[:, None] + xi) * dy).reshape(ny, 1, N + 1, 1) - cy
    r2 = x * x + y * y
    g = beta / (2.0 * np.pi) * np.exp(0.5 * (1.0 - r2))
    T = 1.0 - (GAMMA - 1.0) / (2.0 * GAMMA) * g * g
    rho = T ** (1.0 / (GAMMA - 1.0))
    u, v, p = 1.0 - g * y, 1.0 + g * x, rho * T
    E = p / (GAMMA - 1.0) + 0.5 * rho * (u * u + v * v)
    q = np.stack([rho, rho * u, rho * v, E], axis=2)        # [ny][nx][var][b][a]
    # |v| + c stays below 3.6 for this vortex; half of the configured CFL factor
    dt = 0.45 / (2 * (2 * N + 1)) * min(dx, dy) / 3.6
    return np.ascontiguousarray(q.reshape(nx * ny, 4, -1)), dx, dy, dt


def _subcell_setup(case, seed):
    """Patches around a shock front of seeded place and direction on smooth data."""
    D, N, count = case["dim"], case["N"], case["count"]
    L, nv = 2 * N + 7, D + 2
    rng = np.random.default_rng(seed)
    ax = [np.linspace(-1.0, 1.0, L)] * D
    grid = np.meshgrid(*ax, indexing="ij")[::-1]           # grid[0] is x, fastest
    nrm = rng.normal(size=(count, D))
    nrm /= np.linalg.norm(nrm, axis=1, keepdims=True)
    off = rng.uniform(-1.0, 1.0, count)
    shape = (count,) + (1,) * D
    side = sum(nrm[:, k].reshape(shape) * grid[k] for k in range(D)) < off.reshape(shape)
    phase = rng.uniform(0, 2 * np.pi, size=(count, nv))
    wave = [1.0 + 0.05 * np.sin(phase[:, v].reshape(shape) + 2.0 * grid[v % D] - grid[(v + 1) % D])
            for v in range(nv)]
    rho = np.where(side, 1.0, 0.125) * wave[0]
    p = np.where(side, 1.0, 0.1) * wave[nv - 1]
    vel = [np.where(side, 0.7 * nrm[:, k].reshape(shape), 0.0) + 0.2 * (wave[1 + k] - 1.0)
           for k in range(D)]
    E = p / (GAMMA - 1.0) + 0.5 * rho * sum(v * v for v in vel)
    q = np.stack([rho] + [rho * v for v in vel] + [E], axis=1)
    h = [0.01 * (1.0 + 0.1 * k) for k in range(D)]
    return np.ascontiguousarray(q.reshape(count, nv, -1)), h, 0.3 * h[0] / (D * 2.5)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "subcell":
        q, h, dt = _subcell_setup(case, seed)
        D, ns, count = case["dim"], 2 * case["N"] + 1, case["count"]
        return dict(case=case, h=h, dt=dt, patches=torch.from_numpy(q).cuda(),
                    out=dict(averages=torch.empty((count, D + 2, ns ** D), dtype=torch.float64,
                                                  device="cuda"),
                             faces=torch.empty((count, D, 2, D + 2, ns ** (D - 1)),
                                               dtype=torch.float64, device="cuda")))
    if kind == "vortex":
        q, dx, dy, dt = _vortex_setup(case, seed)
        s = adg.Solver(2, (case["nx"], case["ny"]), (-5.0, -5.0), (dx, dy), (0, 0, 0, 0), case["N"],
                       GAMMA, _prec(case))
        s.load(q)
        return dict(case=case, grid=Grid(s), dt=dt)
    if kind == "batch":
        rng = np.random.default_rng(seed)
        stream = torch.cuda.Stream()
        grids = []
        for n, N, config in _members(case):
            w = inputs.riemann_2d(n, N, config, jitter=0.02, rng=rng)
            s = adg.Solver.from_workload(w, MIXED)
            s.set_option(adg.OPT_CFL, w["cfl"])
            s.init_problem(w["problem"])
            grids.append(Grid(s, stream.cuda_stream))
        batch = adg.Batch([g.solver for g in grids], stream.cuda_stream)
        return dict(case=case, grids=grids, batch=batch, stream=stream)
    w = _workload(case, seed)
    s = adg.Solver.from_workload(w, _prec(case))
    s.init_problem(w["problem"])
    if kind != "resume":
        return dict(case=case, grid=Grid(s), cfl=w["cfl"])
    dofs, flags, sub = (torch.from_numpy(x).pin_memory() for x in s.read_full())
    out = torch.empty(dofs.shape, dtype=torch.float64, pin_memory=True)
    return dict(case=case, solver=s, cfl=w["cfl"], dofs=dofs.numpy(), flags=flags.numpy(),
                sub=sub.numpy(), out=out.numpy(), pinned=(dofs, flags, sub, out))


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    case = state["case"]
    kind, steps = case["kind"], case["steps"]
    if kind == "subcell":
        out = state["out"]
        rc, msg = adg.subcell_update_noalloc(
            case["dim"], case["N"], GAMMA, state["h"], state["dt"], state["patches"].data_ptr(),
            case["count"], out["averages"].data_ptr(), out["faces"].data_ptr())
        if rc != adg.OK:
            raise RuntimeError(msg)
        return out
    if kind == "resume":
        s = state["solver"]
        s.load_full(state["dofs"], state["flags"], state["sub"])
        for _ in range(steps):
            s.step_cfl(state["cfl"])
            flags = s.flags()
        return dict(dofs=s.read(out=state["out"]), flags=flags)
    if kind == "batch":
        for g in state["grids"]:
            g.restore()
        for _ in range(steps):
            state["batch"].step()
        return [g.result() for g in state["grids"]]
    g = state["grid"]
    g.restore()
    if kind == "dmr":
        g.solver.set_time(0.0)          # its boundary front moves with the simulated time
    for _ in range(steps):
        if kind == "vortex":
            g.solver.step(state["dt"])
        else:
            g.solver.step_cfl(state["cfl"])
    return g.result()


# ---------------------------------------------------------------------------
# the same in plain 64-bit torch: the smooth vortex (the DG path with a quiet limiter) and the
# stand-alone patch update (the limiter's reconstruction, predictor and fluxes)
# ---------------------------------------------------------------------------
def _basis(N):
    """Gauss-Legendre nodes and weights on [0, 1] and the operators of the nodal basis."""
    z, wz = np.polynomial.legendre.leggauss(N + 1)
    xi, w, n = 0.5 * (z + 1.0), 0.5 * wz, N + 1
    bary = np.array([1.0 / np.prod([xi[a] - xi[b] for b in range(n) if b != a]) for a in range(n)])
    D = np.zeros((n, n))                                    # D[a][b] = phi_b'(xi_a)
    for a in range(n):
        for b in range(n):
            if a != b:
                D[a, b] = bary[b] / bary[a] / (xi[a] - xi[b])
        D[a, a] = sum(1.0 / (xi[a] - xi[b]) for b in range(n) if b != a)

    def phi(x):
        return np.array([np.prod([(x - xi[b]) / (xi[a] - xi[b]) for b in range(n) if b != a])
                         for a in range(n)])
    p0, p1 = phi(0.0), phi(1.0)
    K1 = np.outer(p1, p1) - (w[:, None] * D).T             # K1[m][l] = p1[m] p1[l] - w_l D[l][m]
    Kt = np.linalg.solve(K1, np.diag(w))
    return xi, w, D, Kt, p0, p1


def _t(x):
    x = torch.as_tensor(np.asarray(x), dtype=torch.float64)
    return x.cuda() if torch.cuda.is_available() else x


def _fluxes(q, D):
    """Euler fluxes along every axis; the variable is q's second dimension."""
    rho, m, E = q[:, 0], [q[:, 1 + k] for k in range(D)], q[:, D + 1]
    v = [x / rho for x in m]
    p = (GAMMA - 1.0) * (E - 0.5 * sum(a * b for a, b in zip(m, v)))
    out = []
    for k in range(D):
        f = [m[k]] + [m[j] * v[k] + (p if j == k else 0.0) for j in range(D)] + [v[k] * (E + p)]
        out.append(torch.stack(f, dim=1))
    return out, [x.abs() + torch.sqrt(GAMMA * p / rho) for x in v]


def _rusanov(qL, qR, k, D):
    fL, sL = _fluxes(qL, D)
    fR, sR = _fluxes(qR, D)
    s = torch.maximum(sL[k], sR[k]).unsqueeze(1)
    return 0.5 * (fL[k] + fR[k]) - 0.5 * s * (qR - qL)


def _exact_vortex(case, seed):
    q, dx, dy, dt = _vortex_setup(case, seed)
    N, nx, ny = case["N"], case["nx"], case["ny"]
    n = N + 1
    if nx * ny * n ** 3 > 2e7:
        return None
    _, w, Dm, Kt, p0, p1 = _basis(N)
    Mv = w[None, :] * Dm.T / w[:, None]                    # Mv[a][j] = w_j D[j][a] / w_a
    wt, Dm, Kt, Mv, t0, t1 = (_t(x) for x in (w, Dm, Kt, Mv, p0, p1))
    l0, l1 = _t(p0 / w), _t(p1 / w)
    u = _t(q).view(nx * ny, 4, n, n)                       # [cell][var][b][a]
    cx, cy = dt / dx, dt / dy
    for _ in range(case["steps"]):
        q = u.unsqueeze(2).expand(-1, -1, n, -1, -1)       # [cell][var][tau][b][a]
        for _ in range(N + 1):
            (fx, fy), _s = _fluxes(q, 2)
            S = cx * torch.einsum("aj,cvtbj->cvtba", Dm, fx) + cy * torch.einsum("bj,cvtja->cvtba", Dm, fy)
            q = u.unsqueeze(2) - torch.einsum("tj,cvjba->cvtba", Kt, S)
        (fx, fy), _s = _fluxes(q, 2)
        fx, fy = (torch.einsum("t,cvtba->cvba", wt, f) for f in (fx, fy))
        new = u + cx * torch.einsum("aj,cvbj->cvba", Mv, fx) + cy * torch.einsum("bj,cvja->cvba", Mv, fy)
        lo, hi = (torch.einsum("a,cvtba->cvtb", t, q).view(ny, nx, 4, n, n) for t in (t0, t1))
        G = _rusanov(hi.flatten(0, 1), lo.roll(-1, 1).flatten(0, 1), 0, 2)     # each cell's high x face
        G = torch.einsum("t,cvtb->cvb", wt, G).view(ny, nx, 4, n)
        new = new - cx * (G.flatten(0, 1).unsqueeze(3) * l1 - G.roll(1, 1).flatten(0, 1).unsqueeze(3) * l0)
        lo, hi = (torch.einsum("b,cvtba->cvta", t, q).view(ny, nx, 4, n, n) for t in (t0, t1))
        G = _rusanov(hi.flatten(0, 1), lo.roll(-1, 0).flatten(0, 1), 1, 2)
        G = torch.einsum("t,cvta->cva", wt, G).view(ny, nx, 4, n)
        u = new - cy * (G.flatten(0, 1).unsqueeze(2) * l1.view(n, 1)
                        - G.roll(1, 0).flatten(0, 1).unsqueeze(2) * l0.view(n, 1))
    return dict(dofs=u.reshape(nx * ny, 4, n * n), subcells=None, extrema=None, flags=None)


def _weno(u, axis, nodes):
    """WENO3 along `axis` of the subcell averages: the values at the three nodes of every target
    (its own dimension, last), over the targets that have two neighbours on each side."""
    m = u.shape[axis] - 4
    U = [u.narrow(axis, r, m) for r in range(5)]
    num, den = 0.0, 0.0
    for k, lam in ((0, 1.0), (1, 1e5), (2, 1.0)):
        # parabola c0 + c1 x + c2 x^2 with the averages U[k], U[k+1], U[k+2] over cells k-2 .. k
        rows = [[1.0, ((j + 1) ** 2 - j ** 2) / 2.0, ((j + 1) ** 3 - j ** 3) / 3.0] for j in range(k - 2, k + 1)]
        C = np.linalg.inv(np.array(rows, dtype=np.float64))
        c = [sum(float(C[r, j]) * U[k + j] for j in range(3)) for r in range(3)]
        sigma = c[1] * (c[1] + 2.0 * c[2]) + 16.0 / 3.0 * c[2] * c[2]
        wgt = (lam / (sigma + 1e-14) ** 8).unsqueeze(-1)
        p = torch.stack([c[0] + c[1] * x + c[2] * x * x for x in nodes], dim=-1)
        num, den = num + wgt * p, den + wgt
    return num / den


def _exact_subcell(case, seed):
    q, h, dt = _subcell_setup(case, seed)
    D, N, count = case["dim"], case["N"], case["count"]
    nv, ns, L = D + 2, 2 * N + 1, 2 * N + 7
    xi, w, Dm, Kt, p0, p1 = _basis(2)
    nodes = [float(x) for x in xi]
    Dm, Kt, p0, p1, w = (_t(x) for x in (Dm, Kt, p0, p1, w))
    v = _t(q).view((count, nv) + (L,) * D)
    u = v
    for k in range(D):                                     # x, then y[, z]; x is the last subcell axis
        u = _weno(u, 1 + D - k, nodes)
    # u: [count][var][z][y][x][node x][node y][node z] -> time before the nodes, z slowest
    perm = [0, 1] + list(range(2, 2 + D)) + list(range(1 + 2 * D, 1 + D, -1))
    u = u.permute(perm).unsqueeze(2 + D).contiguous()      # [count][var][z][y][x][tau][nz][ny][nx]
    ax = [u.dim() - 1 - k for k in range(D)]               # node axis of x, y, z
    c = [dt / x for x in h]

    def along(M, f, axis):
        return torch.movedim(torch.tensordot(f, M, dims=([axis], [1])), -1, axis)
    s = u.expand(*([-1] * (2 + D)), 3, *([-1] * D))
    for _ in range(3):
        f, _s = _fluxes(s, D)
        S = sum(c[k] * along(Dm, f[k], ax[k]) for k in range(D))
        s = u - along(Kt, S, 2 + D)
    inner = v[(slice(None), slice(None)) + (slice(3, -3),) * D]
    new, faces = inner.clone(), []
    for k in range(D):
        sub = 1 + D - k                                    # subcell axis of x, y, z in the array
        hi = torch.tensordot(s, p1, dims=([ax[k]], [0]))
        lo = torch.tensordot(s, p0, dims=([ax[k]], [0]))
        cut = [slice(None)] * hi.dim()
        for j in range(D):
            if j != k:
                cut[1 + D - j] = slice(1, -1)
        cutL, cutR = list(cut), list(cut)
        cutL[sub], cutR[sub] = slice(0, ns + 1), slice(1, ns + 2)
        G = _rusanov(hi[tuple(cutL)], lo[tuple(cutR)], k, D)
        for _ in range(D):
            G = torch.tensordot(G, w, dims=([G.dim() - 1], [0]))
        new = new - c[k] * (G.narrow(sub, 1, ns) - G.narrow(sub, 0, ns))
        ends = [G.select(sub, 0), G.select(sub, ns)]
        faces.append(torch.stack([x.reshape(count, nv, -1) for x in ends], dim=1))
    return dict(averages=new.reshape(count, nv, -1), faces=torch.stack(faces, dim=1))


def exact(case, seed):
    if case["kind"] == "vortex":
        return _exact_vortex(case, seed)
    if case["kind"] == "subcell":
        return _exact_subcell(case, seed)
    return None          # limited steps: no plain 64-bit restatement of the whole scheme here
