"""Performance cases of the topology-optimisation library, through its public
calls (the design loop's driver and the C ABI binding).

A design iteration filters the design, sets the moduli, solves K(rho) u = f by
multigrid-preconditioned CG (MGCG) or, later in a run, by the reduced model
(CARM), and updates the design from the sensitivities.  The cases are these
parts, from the smallest grid the workloads name to the largest:

  step    one whole design iteration of the driver from a given design
  solve   the density of an iteration and the cold MGCG solve that follows it
          (hierarchy rebuild and CG iterations)
  vcycle  one application of the multigrid preconditioner
  carm    the reduced model of an iteration: basis, reduced solve, residual
  update  compliance and sensitivity, their filter and the OC update
  batch   one served round of several jobs: both shared phases of each job

Inputs are synthetic, drawn from the seed: densities with solid flanges and a
random smooth web between near-void and solid (a design in mid-optimisation),
smooth displacement-like fields where a stored solution is an input.

Displacements of an iterative solve are returned as float32: a relative
residual of 1e-6 to 1e-8 leaves no more digits than that, and a program that
stores or draws them keeps no more.  The V-cycle of the mixed solver returns
float32 values widened to float64 and is narrowed back without loss.
"""

import math
from dataclasses import dataclass

import numpy as np
import torch

from paper_2205_00385_gb300 import binding as B
from paper_2205_00385_gb300.driver import TopoSolver

E0, EMIN, NU, PENAL, MOVE, OMEGA = 1.0, 1e-9, 0.3, 3.0, 0.2, 0.6
SERVED = ((32, 16, 16, 4), (64, 32, 32, 5), (96, 48, 48, 5), (128, 64, 64, 6))


def _case(kind, support, nx, ny, nz, levels, mixed, s=2, rmin=1.5, rtol=1e-8, jobs=0, **name):
    return dict(kind=kind, support=support, nx=nx, ny=ny, nz=nz, levels=levels, mixed=mixed, s=s,
                rmin=rmin, rtol=rtol, jobs=jobs, **name)


def listed():
    return [
        # the smallest workload: latency and launches of a whole 2D iteration
        _case("step", "mbb", 60, 20, 0, 3, False, 6, name="step 2D 60x20 fp64"),
        # a 2D study at its usual size: large-radius filter, tolerance 1e-6
        _case("step", "halfwheel", 640, 320, 0, 7, True, 2, 2.5, 1e-6,
              name="step 2D 640x320 mixed"),
        # the small 3D workload in plain float64, a whole iteration
        _case("step", "cantilever", 48, 24, 24, 4, False, 8, name="step 48x24x24 fp64"),
        # a served job's solve at its own tolerance: small grid, launch bound
        _case("solve", "bridge", 64, 32, 32, 5, True, 8, 1.5, 1e-6, name="solve 64x32x32 mixed"),
        # the headline workload's solve, where a design run spends its time
        _case("solve", "cantilever", 192, 96, 96, 6, True, 10, 2.0, name="solve 192x96x96 mixed"),
        # the preconditioner in plain float64, middle size
        _case("vcycle", "cantilever", 96, 48, 48, 5, False, name="vcycle 96x48x48 fp64"),
        # the preconditioner at the headline size and at the largest grid
        _case("vcycle", "cantilever", 192, 96, 96, 6, True, rmin=2.0,
              name="vcycle 192x96x96 mixed"),
        _case("vcycle", "bridge", 320, 160, 160, 6, True, rmin=2.5,
              name="vcycle 320x160x160 mixed"),
        # reduced model after its activation: small float64 and headline mixed
        _case("carm", "cantilever", 48, 24, 24, 4, False, 8, name="carm 48x24x24 fp64"),
        _case("carm", "cantilever", 192, 96, 96, 6, True, 10, 2.0, name="carm 192x96x96 mixed"),
        # the design side of the headline workload's iteration
        _case("update", "cantilever", 192, 96, 96, 6, True, 10, 2.0,
              name="update 192x96x96 mixed"),
        # a served round: the four served grids, both shared phases
        _case("batch", "cantilever", 0, 0, 0, 0, True, 8, 1.5, 1e-6, 4, name="batch of 4 served"),
    ]


def draw(rng):
    kind = rng.choice(["step", "step", "solve", "solve", "vcycle", "vcycle", "carm", "update",
                       "batch"])
    if kind == "batch":
        return _case("batch", rng.choice(["cantilever", "bridge"]), 0, 0, 0, 0, True, 8,
                     rng.choice([1.5, 2.0, 2.5]), 1e-6, rng.randint(1, 12))
    if kind == "step" and rng.random() < 0.6:
        # 2D: 3 to 7 grids above a coarsest grid of a few hundred elements at most
        levels = rng.randint(3, 6)
        unit = 1 << (levels - 1)
        nx = max(5, min(40, round(math.exp(rng.uniform(math.log(48), math.log(960))) / unit)))
        ny = max(3, min(24, round(nx * rng.uniform(0.25, 0.6))))
        return _case("step", rng.choice(["mbb", "halfwheel"]), nx * unit, ny * unit, 0, levels,
                     rng.random() < 0.5, rng.randint(1, 8), rng.choice([1.5, 2.0, 2.5]),
                     rng.choice([1e-6, 1e-8]))
    mixed = kind == "update" or rng.random() < (0.3 if kind == "step" else 0.7)
    # element counts, spread over their logarithm, up to the listed case of the kind
    top = {"step": 3e5 if mixed else 3e4, "solve": 1.7e6 if mixed else 6e4,
           "vcycle": 8e6 if mixed else 4e5, "carm": 1.7e6 if mixed else 6e4, "update": 1.7e6}[kind]
    nel = math.exp(rng.uniform(math.log(1.5e3), math.log(top)))
    ry, rz = rng.uniform(0.35, 0.75), rng.uniform(0.35, 0.75)
    nx = (nel / (ry * rz)) ** (1 / 3)
    levels = max(2, min(6, 1 + int(math.log2(nx * min(ry, rz) / 2.5))))
    unit = 1 << (levels - 1)
    c = [max(2, min(11, int(v / unit))) for v in (nx, nx * ry, nx * rz)]
    return _case(kind, rng.choice(["cantilever", "bridge"]), *[v * unit for v in c], levels, mixed,
                 rng.choice([2, 3, 4, 6, 8, 10]), rng.choice([1.5, 2.0, 2.5]),
                 rng.choice([1e-6, 1e-8]))


# ---------------------------------------------------------------------------
# Problem data
# ---------------------------------------------------------------------------
def _jobs(case):
    """The cases of a batch's jobs: served grids in turn."""
    return [_case("batch", case["support"], *SERVED[q % 4], True, case["s"], case["rmin"],
                  case["rtol"]) for q in range(case["jobs"])]


def _nel(case):
    return case["nx"] * case["ny"] * max(case["nz"], 1)


def _ndof(case):
    d3 = case["nz"] > 0
    return (3 if d3 else 2) * (case["nx"] + 1) * (case["ny"] + 1) * (case["nz"] + 1 if d3 else 1)


def _mesh(case):
    """(fixed uint8, f float64) per DOF: node i + (nx+1)(j + (ny+1)k), DOF dim*node + c."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    dim = 3 if nz else 2
    fixed = torch.zeros((nz + 1, ny + 1, nx + 1, dim), dtype=torch.uint8, device="cuda")
    f = torch.zeros(fixed.shape, dtype=torch.float64, device="cuda")

    def trapezoid(n):
        w = torch.full((n + 1,), 1.0 / n, dtype=torch.float64, device="cuda")
        w[0] = w[-1] = 0.5 / n
        return w

    if case["support"] == "mbb":            # symmetry edge, roller, point load
        fixed[0, :, 0, 0] = 1
        fixed[0, 0, nx, 1] = 1
        f[0, ny, 0, 1] = -1.0
    elif case["support"] == "halfwheel":    # pin, roller, point load at the bottom
        fixed[0, 0, 0, :] = 1
        fixed[0, 0, nx, 1] = 1
        f[0, 0, nx // 2, 1] = -1.0
    elif case["support"] == "cantilever":   # clamped face, line load
        fixed[:, :, 0, :] = 1
        f[:, 0, nx, 1] = -trapezoid(nz)
    else:                                   # bridge: four corner nodes, load on the top face
        for k in (0, nz):
            for i in (0, nx):
                fixed[k, 0, i, :] = 1
        f[:, ny, :, 1] = -trapezoid(nz)[:, None] * trapezoid(nx)[None, :]
    return fixed.reshape(-1), f.reshape(-1)


def _waves(case, rng, nodes, count, top):
    """Sum of `count` random plane waves with up to `top` periods per axis."""
    n = [case["nz"], case["ny"], case["nx"]]
    ax = [torch.arange(max(v, 1) + (1 if nodes and v else 0), dtype=torch.float64, device="cuda") /
          max(v, 1) for v in n]
    out = torch.zeros([len(a) for a in ax], dtype=torch.float64, device="cuda")
    for _ in range(count):
        k, ph = rng.uniform(-top, top, 3), rng.uniform(0, 2 * math.pi)
        out += torch.cos(2 * math.pi * (k[0] * ax[0][:, None, None] + k[1] * ax[1][None, :, None] +
                                        k[2] * ax[2][None, None, :]) + ph)
    return out


def _density(case, rng):
    """Flanges at the bottom and top, a random web with near-void between them."""
    web = _waves(case, rng, False, 8, 3.0) / 2.0
    y = (torch.arange(case["ny"], dtype=torch.float64, device="cuda") + 0.5) / case["ny"]
    flange = 25.0 * ((2.0 * y - 1.0).abs() - 0.85)
    rho = torch.sigmoid(torch.maximum(2.5 * web - 1.0, flange[None, :, None].expand_as(web)))
    return rho.reshape(-1).clamp(1e-3, 1.0).contiguous()


def _noise(n, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    return torch.rand(n, generator=g, dtype=torch.float64, device="cuda")


def _field(case, rng, fixed):
    """A smooth displacement-like field, zero on the fixed DOFs."""
    dim = 3 if case["nz"] else 2
    nx = case["nx"]
    x = (torch.arange(nx + 1, dtype=torch.float64, device="cuda") / nx) ** int(rng.integers(1, 4))
    u = torch.stack([_waves(case, rng, True, 2, 1.0) * x for _ in range(dim)], dim=-1)
    return (u.reshape(-1) * (1 - fixed.to(torch.float64))).contiguous()


def _inputs(case, seed):
    """Everything a call takes, from the case and the seed alone."""
    rng = np.random.default_rng([seed, case["nx"], case["ny"], case["nz"]])
    fixed, f = _mesh(case)
    rho = _density(case, rng)
    d = dict(fixed=fixed, f=f, rho=rho)
    if case["kind"] == "vcycle":
        r = 1e-3 * (2.0 * _noise(f.numel(), seed) - 1.0) + 1e-3 * _field(case, rng, fixed)
        d["r"] = (r + f) * (1 - fixed.to(torch.float64))
    if case["kind"] == "carm":
        bump = _waves(case, rng, False, 4, 2.0).reshape(-1) / 4.0
        d["rho_prev"] = (rho + 0.05 * bump).clamp(1e-3, 1.0)
        d["parm"] = [_field(case, rng, fixed) for _ in range(case["s"])]
        d["u_last"] = 40.0 * d["parm"][-1]
    if case["kind"] in ("update", "batch"):
        d["u"] = 40.0 * _field(case, rng, fixed)
        d["design"] = (rho + 0.02 * (_noise(rho.numel(), seed) - 0.5)).clamp(0.0, 1.0)
    d["volfrac"] = float(d.get("design", rho).mean())   # the running design meets its volume
    return d


class _Context:
    """A library context with its workspace and inputs, as a program keeps it."""

    def __init__(self, case, seed):
        self.case = case
        self.__dict__.update(_inputs(case, seed))
        dim = 3 if case["nz"] else 2
        desc = B.make_desc(dim, (case["nx"], case["ny"], case["nz"])[:dim], E0, EMIN, NU, PENAL,
                           case["rmin"], case["levels"], B.TO_MIXED if case["mixed"] else B.TO_FP64,
                           case["s"], case["s"])
        size = B.to_workspace_bytes(desc)
        raw = torch.empty(size + 256, dtype=torch.uint8, device="cuda")
        self.ws = raw[(-raw.data_ptr()) % 256:][:size]
        self.ctx = B.to_mesh_init(desc, self.fixed, self.f, self.ws,
                                  torch.cuda.current_stream().cuda_stream)
        f64 = dict(dtype=torch.float64, device="cuda")
        nel, n = _nel(case), _ndof(case)
        self.out = torch.zeros(n, **f64)
        kind = case["kind"]
        if kind in ("update", "batch"):
            self.dc, self.dc_f, self.dv_f = (torch.empty(nel, **f64) for _ in range(3))
            self.rho_phys, self.x = torch.empty(nel, **f64), torch.empty(nel, **f64)
            self.scalars = torch.zeros(2, **f64)
            B.to_filter(self.ctx, B.TO_FILTER_SENS, torch.ones(nel, **f64), self.dv_f)
            B.to_set_density(self.ctx, self.rho)
        elif kind == "vcycle":
            B.to_set_density(self.ctx, self.rho)
            B.to_vcycle(self.ctx, self.r, self.out)     # builds the hierarchy
        elif kind == "carm":
            B.to_set_density(self.ctx, self.rho_prev)
            B.to_set_density(self.ctx, self.rho)
            for v in self.parm:
                B.to_parm_push(self.ctx, v)

    def __del__(self):
        if getattr(self, "ctx", None) is not None:
            B.to_destroy(self.ctx)
            self.ctx = None

    def job(self):
        return dict(ctx=self.ctx, rho=self.x, rho_phys=self.rho_phys, u=self.u, dc=self.dc,
                    dc_f=self.dc_f, dv_f=self.dv_f, compliance_dev=self.scalars[0:1],
                    change_dev=self.scalars[1:2], volfrac=self.volfrac, move=MOVE)


@dataclass
class _Problem:
    """The attributes the driver reads from a problem."""
    dim: int
    nelx: int
    nely: int
    nelz: int
    fixed: np.ndarray
    f: np.ndarray
    rho0: np.ndarray
    volfrac: float
    rmin: float
    mg_levels: int
    precision: str
    n_parm: int
    n_carm: int
    rtol: float
    E0: float = E0
    Emin: float = EMIN
    nu: float = NU
    penal: float = PENAL
    move: float = MOVE
    n_on: int = 20
    eps_tol: float = 1e-3
    maxit: int = 200

    nel = property(lambda self: self.rho0.size)
    ndof = property(lambda self: self.f.size)

    def volfrac_at(self, k):
        return self.volfrac


class _Design:
    """A job of the driver and the design it starts its iteration from."""

    def __init__(self, case, seed):
        d = _inputs(case, seed)
        self.rho = d["rho"]
        host = [d[k].cpu().numpy() for k in ("fixed", "f", "rho")]
        self.solver = TopoSolver(_Problem(
            3 if case["nz"] else 2, case["nx"], case["ny"], case["nz"], *host, d["volfrac"],
            case["rmin"], case["levels"], "mixed" if case["mixed"] else "fp64", case["s"],
            case["s"], case["rtol"]))


class _Batch:
    """Jobs of a server: a stream per job, and one for the shared launches."""

    def __init__(self, case, seed):
        self.stream, self.jobs = torch.cuda.Stream(), []
        for q, c in enumerate(_jobs(case)):
            own = torch.cuda.Stream()
            with torch.cuda.stream(own):
                job = _Context(c, seed + q)
            job.stream = own
            self.stream.wait_stream(own)
            self.jobs.append(job)


def prepare(case, seed):
    if case["kind"] == "step":
        return _Design(case, seed)
    if case["kind"] == "batch":
        return _Batch(case, seed)
    return _Context(case, seed)


def run(state):
    if isinstance(state, _Design):
        s = state.solver
        s.rho.copy_(state.rho)
        s.k = 0
        s.history.clear()
        s.step()
        return {"u": s.u.float(), "rho_phys": s.rho_phys, "dc_f": s.dc_f.float(),
                "rho": s.rho.float(), "compliance": s.scalars[0].float()}
    if isinstance(state, _Batch):
        with torch.cuda.stream(state.stream):
            for c in state.jobs:
                c.x.copy_(c.design)
            jobs = [c.job() for c in state.jobs]
            B.to_batch_step(jobs, B.TO_PHASE_DENSITY, state.stream.cuda_stream)
            B.to_batch_step(jobs, B.TO_PHASE_UPDATE, state.stream.cuda_stream)
        torch.cuda.current_stream().wait_stream(state.stream)
        return [[c.rho_phys, c.x, c.dc_f, c.scalars] for c in state.jobs]
    c, kind = state, state.case["kind"]
    if kind == "solve":
        B.to_set_density(c.ctx, c.rho)
        B.to_mgcg_solve(c.ctx, c.case["rtol"], 200, 0, c.out)
        return c.out.float()
    if kind == "vcycle":
        B.to_vcycle(c.ctx, c.r, c.out)
        return c.out.float() if c.case["mixed"] else c.out
    if kind == "carm":
        B.to_carm_build(c.ctx, c.u_last)
        eps = B.to_carm_solve(c.ctx, c.out)
        return {"u": c.out, "eps": eps}
    c.x.copy_(c.design)
    B.to_sensitivity(c.ctx, c.u, c.scalars[0:1], c.dc)
    B.to_filter(c.ctx, B.TO_FILTER_SENS, c.dc, c.dc_f)
    B.to_oc_update(c.ctx, c.volfrac, MOVE, c.dc_f, c.dv_f, c.x, c.scalars[1:2])
    return {"dc": c.dc, "dc_f": c.dc_f, "rho": c.x, "scalars": c.scalars}


def work(case):
    """Bytes and operations one pass cannot do without: inputs and outputs once
    (float64 as the calls take them), and the arithmetic of the element
    operator in its factorised form (about 234 operations per hex8 element
    and product, 56 per Q4), of the filter and of the small dense parts."""
    if case["kind"] == "batch":
        parts = [work(dict(c, kind="update")) for c in _jobs(case)]
        return {k: 1.3 * sum(p[k] for p in parts) for k in ("bytes", "flops")}
    nel, n, s = _nel(case), _ndof(case), case["s"]
    op = (234.0 if case["nz"] else 56.0) * nel
    dim = 3 if case["nz"] else 2
    filt = 2.0 * nel * (math.pi * case["rmin"] ** 2 if dim == 2
                        else 4.19 * case["rmin"] ** 3)
    # a V-cycle: two operator products and the transfers on a geometric series of grids
    cycle = (2.0 * op + 14.0 * n) / (1.0 - 0.5 ** dim)
    kind = case["kind"]
    if kind == "vcycle":
        return {"bytes": 8.0 * nel + 16.0 * n, "flops": cycle}
    if kind == "carm":
        # operator products on s PARM columns, s - 1 basis vectors and up to s
        # reduced columns; Gram products and combinations of the blocks
        return {"bytes": 16.0 * nel + 8.0 * n * (s + 3), "flops": 3.0 * s * op + 12.0 * s * s * n}
    if kind == "update":
        return {"bytes": 8.0 * n + 7 * 8.0 * nel, "flops": op + filt + 20.0 * nel * 10}
    # a cold solve takes some 30 iterations to 1e-8, 20 to 1e-6
    its = 30.0 if case["rtol"] < 1e-7 else 20.0
    solve = {"bytes": 8.0 * nel + 16.0 * n, "flops": its * (cycle + op + 12.0 * n)}
    if kind == "solve":
        return solve
    return {"bytes": solve["bytes"] + 8.0 * n + 8 * 8.0 * nel,
            "flops": solve["flops"] + op + 2 * filt + 200.0 * nel}


# ---------------------------------------------------------------------------
# The same results in 64 bits with plain torch
# ---------------------------------------------------------------------------
def _stiffness(dim):
    """Unit-modulus KE of a unit square / cube by 2-point Gauss quadrature."""
    npe, nd = 1 << dim, dim << dim
    if dim == 2:
        D = np.array([[1, NU, 0], [NU, 1, 0], [0, 0, (1 - NU) / 2]]) / (1 - NU * NU)
        pairs = ((0, 1),)
    else:
        lam, mu = NU / ((1 + NU) * (1 - 2 * NU)), 0.5 / (1 + NU)
        D = np.diag([2 * mu] * 3 + [mu] * 3)
        D[:3, :3] += lam
        pairs = ((0, 1), (1, 2), (0, 2))
    KE = np.zeros((nd, nd))
    for q in range(npe):
        xi = [0.5 + (1 if (q >> d) & 1 else -1) * 0.5 / math.sqrt(3.0) for d in range(dim)]
        G = np.zeros((dim + len(pairs), nd))
        for a in range(npe):
            for d in range(dim):
                g = math.prod((1.0 if (a >> e) & 1 else -1.0) if e == d else
                              (xi[e] if (a >> e) & 1 else 1.0 - xi[e]) for e in range(dim))
                G[d, dim * a + d] = g
                for p, pr in enumerate(pairs):
                    if d in pr:
                        G[dim + p, dim * a + (pr[1] if d == pr[0] else pr[0])] = g
        KE += G.T @ D @ G / npe
    return torch.from_numpy(KE).cuda()


def _child_weights(dim):
    """P_c: nodal values of child c's corners from its parent's, per component."""
    npe = 1 << dim
    out = np.zeros((npe, dim * npe, dim * npe))
    for c in range(npe):
        for a in range(npe):
            for A in range(npe):
                pos = [0.5 * (((c >> d) & 1) + ((a >> d) & 1)) for d in range(dim)]
                w = math.prod(p if (A >> d) & 1 else 1 - p for d, p in enumerate(pos))
                for i in range(dim):
                    out[c, dim * a + i, dim * A + i] = w
    return torch.from_numpy(out).cuda()


class _Level:
    """One grid: element matrices E_e KE (A is None) or A[e], masked on fixed DOFs."""

    def __init__(self, nel, dim, fixed, KE, E=None, A=None):
        self.nel, self.dim, self.E, self.KE, self.A = nel, dim, E, KE, A
        self.nn = [v + 1 for v in nel[:dim]]
        self.free = 1.0 - fixed.to(torch.float64)
        el = torch.arange(math.prod(nel), device="cuda")
        ex, ey, ez = el % nel[0], el // nel[0] % nel[1], el // (nel[0] * nel[1])
        self.conn = torch.stack([(ex + (a & 1)) + self.nn[0] * ((ey + (a >> 1 & 1)) + (
            self.nn[1] * (ez + (a >> 2 & 1)) if dim == 3 else 0)) for a in range(1 << dim)], dim=1)

    def _scatter(self, F):
        y = torch.zeros(math.prod(self.nn), self.dim, dtype=torch.float64, device="cuda")
        y.index_add_(0, self.conn.reshape(-1), F.reshape(-1, self.dim))
        return y.reshape(-1)

    def gather(self, x):
        return (self.free * x).reshape(-1, self.dim)[self.conn].reshape(len(self.conn), -1)

    def unmasked(self, x, E=None):
        U = self.gather(x)
        if self.A is None:
            return self._scatter((U @ self.KE) * (self.E if E is None else E)[:, None])
        return self._scatter(torch.bmm(self.A, U[:, :, None]))

    def apply(self, x, E=None):
        return self.free * self.unmasked(x, E) + (1.0 - self.free) * x

    def dinv(self):
        d = (self.E[:, None] * self.KE.diagonal()[None, :] if self.A is None
             else self.A.diagonal(dim1=1, dim2=2))
        d = self._scatter(d.contiguous())
        return torch.where(self.free > 0, 1.0 / d, torch.ones_like(d))

    def grid(self, x):
        return x.reshape(*reversed(self.nn), self.dim)

    def dense(self):
        n, nd = self.free.numel(), self.KE.shape[0]
        dof = (self.dim * self.conn[:, :, None] + torch.arange(self.dim, device="cuda")).reshape(-1, nd)
        M = torch.zeros(n * n, dtype=torch.float64, device="cuda")
        A = self.A if self.A is not None else self.E[:, None, None] * self.KE
        M.index_add_(0, (dof[:, :, None] * n + dof[:, None, :]).reshape(-1), A.reshape(-1))
        M = M.reshape(n, n) * self.free[:, None] * self.free[None, :]
        return M + torch.diag(1.0 - self.free)


def _children(E, nel, dim):
    """E of the child c = 0 .. 2^dim - 1 of every coarse element, coarse order."""
    g = E.reshape(*([nel[2]] if dim == 3 else []), nel[1], nel[0], *E.shape[1:])
    for c in range(1 << dim):
        s = tuple(slice(c >> d & 1, None, 2) for d in reversed(range(dim)))
        yield g[s].reshape(-1, *E.shape[1:])


def _hierarchy(case, fixed, E):
    dim = 3 if case["nz"] else 2
    KE, P = _stiffness(dim), _child_weights(dim)
    nel = [case["nx"], case["ny"], max(case["nz"], 1)]
    lv = [_Level(nel, dim, fixed, KE, E=E)]
    for _ in range(1, case["levels"]):
        up = lv[-1]
        f = up.grid(1 - up.free)
        cf = f[tuple([slice(None, None, 2)] * dim)].reshape(-1)
        if up.A is None:
            A = sum(e[:, None, None] * (P[c].T @ KE @ P[c])
                    for c, e in enumerate(_children(up.E, up.nel, dim)))
        else:
            A = sum(P[c].T @ a @ P[c] for c, a in enumerate(_children(up.A, up.nel, dim)))
        nel = [v // 2 if d < dim else v for d, v in enumerate(up.nel)]
        lv.append(_Level(nel, dim, cf, KE, A=A))
    for l in lv:
        l.di = l.dinv()
    lv[-1].inv = torch.linalg.inv(lv[-1].dense())
    return lv


def _restrict(x, dim):
    for d in range(dim):
        x = x.movedim(d, 0)
        c = x[::2].clone()
        c[:-1] += 0.5 * x[1::2]
        c[1:] += 0.5 * x[1::2]
        x = c.movedim(0, d)
    return x


def _prolong(x, dim):
    for d in range(dim):
        x = x.movedim(d, 0)
        f = torch.empty((2 * x.shape[0] - 1, *x.shape[1:]), dtype=x.dtype, device=x.device)
        f[::2] = x
        f[1::2] = 0.5 * (x[:-1] + x[1:])
        x = f.movedim(0, d)
    return x


def _cycle(lv, b, q=0):
    """One V(1,1) cycle with damped Jacobi from a zero guess."""
    l = lv[q]
    if q == len(lv) - 1:
        return l.inv @ b
    z = OMEGA * l.di * b
    r = l.free * (b - l.apply(z))
    bc = lv[q + 1].free * _restrict(l.grid(r), l.dim).reshape(-1)
    zc = lv[q + 1].free * _cycle(lv, bc, q + 1)
    z = z + l.free * _prolong(lv[q + 1].grid(zc), l.dim).reshape(-1)
    return z + OMEGA * l.di * (b - l.apply(z))


def _solve(lv, f):
    """K u = f to the limit of 64 bits by CG with the V-cycle."""
    u = torch.zeros_like(f)
    r, fn = f.clone(), float(f.norm())
    z = _cycle(lv, r)
    p, rz = z, r @ z
    for it in range(400):
        q = lv[0].apply(p)
        a = rz / (p @ q)
        u = u + a * p
        r = r - a * q if it % 20 else f - lv[0].apply(u)
        if float(r.norm()) < 1e-13 * fn:
            break
        z = _cycle(lv, r)
        new = r @ z
        p, rz = z + (new / rz) * p, new
    return u


def _modulus(rho):
    return EMIN + (E0 - EMIN) * rho ** PENAL


def _filter_sum(case, x):
    """sum_j w_ij x_j with the cone weights max(0, rmin - distance)."""
    g = x.reshape(max(case["nz"], 1), case["ny"], case["nx"])
    R = math.ceil(case["rmin"])
    out = torch.zeros_like(g)
    for dz in range(-R if case["nz"] else 0, (R if case["nz"] else 0) + 1):
        for dy in range(-R, R + 1):
            for dx in range(-R, R + 1):
                w = case["rmin"] - math.sqrt(dx * dx + dy * dy + dz * dz)
                if w <= 0 or any(abs(d) >= n for d, n in zip((dz, dy, dx), g.shape)):
                    continue
                to = tuple(slice(max(0, -d), n - max(0, d)) for d, n in zip((dz, dy, dx), g.shape))
                fr = tuple(slice(max(0, d), n - max(0, -d)) for d, n in zip((dz, dy, dx), g.shape))
                out[to] += w * g[fr]
    return out.reshape(-1)


def _design_side(case, lv0, u, rho_phys, design, volfrac):
    """(dc, dc_f, new design, [compliance, change])."""
    U = lv0.gather(u)
    ce = ((U @ lv0.KE) * U).sum(1)
    dc = -PENAL * (E0 - EMIN) * rho_phys ** (PENAL - 1.0) * ce
    ones = torch.ones_like(dc)
    hs = _filter_sum(case, ones)
    dc_f, dv_f = _filter_sum(case, dc / hs), _filter_sum(case, ones / hs)
    a = design * torch.sqrt((-dc_f / dv_f).clamp(min=0.0))
    lo, hi = (design - MOVE).clamp(min=0.0), (design + MOVE).clamp(max=1.0)
    l1, l2, target = 0.0, 1e9, volfrac * dc.numel()
    while l2 - l1 > 1e-14 * (l1 + l2):
        mid = 0.5 * (l1 + l2)
        if float((dv_f * torch.minimum(hi, torch.maximum(lo, a / math.sqrt(mid)))).sum()) > target:
            l1 = mid
        else:
            l2 = mid
        if mid in (l1, l2) and (l1 + l2) * 0.5 in (l1, l2):
            break
    new = torch.minimum(hi, torch.maximum(lo, a / math.sqrt(0.5 * (l1 + l2))))
    c = (_modulus(rho_phys) * ce).sum()
    return dc, dc_f, new, torch.stack([c, (new - design).abs().max()])


def _reduced(lv0, d, s):
    """CARM: K_Phi, basis, truncated SVD, reduced solve and force residual."""
    E, Ep = _modulus(d["rho"]), _modulus(d["rho_prev"])
    Phi = torch.stack([v / v.norm() for v in d["parm"]], dim=1)
    KPhi = Phi.T @ torch.stack([lv0.apply(Phi[:, i], Ep) for i in range(s)], dim=1)
    Ki = torch.cholesky_inverse(torch.linalg.cholesky(0.5 * (KPhi + KPhi.T)))
    R = [d["u_last"]]
    for _ in range(1, s):
        R.append(-(Phi @ (Ki @ (Phi.T @ (lv0.free * lv0.unmasked(R[-1], E - Ep))))))
    R = torch.stack([v / v.norm() for v in R], dim=1)
    q, t = torch.linalg.qr(R)
    v, sig, _ = torch.linalg.svd(t)
    Rt = q @ v[:, sig > 1e-6 * sig[0]]
    KR = torch.stack([lv0.apply(Rt[:, i], E) for i in range(Rt.shape[1])], dim=1)
    A = Rt.T @ KR
    y = torch.linalg.solve(0.5 * (A + A.T), Rt.T @ d["f"])
    return Rt @ y, float((KR @ y - d["f"]).norm() / d["f"].norm())


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for q, c in enumerate(_jobs(case)):
            d = _inputs(c, seed + q)
            rp = _filter_sum(c, d["design"]) / _filter_sum(c, torch.ones_like(d["design"]))
            lv0 = _Level([c["nx"], c["ny"], c["nz"]], 3, d["fixed"], _stiffness(3), E=_modulus(rp))
            _, dc_f, new, sc = _design_side(c, lv0, d["u"], rp, d["design"], d["volfrac"])
            out.append([rp, new, dc_f, sc])
        return out
    d = _inputs(case, seed)
    dim = 3 if case["nz"] else 2
    nel = [case["nx"], case["ny"], max(case["nz"], 1)]
    if kind == "vcycle":
        return _cycle(_hierarchy(case, d["fixed"], _modulus(d["rho"])), d["r"])
    if kind == "solve":
        return _solve(_hierarchy(case, d["fixed"], _modulus(d["rho"])), d["f"])
    if kind == "step":
        rp = _filter_sum(case, d["rho"]) / _filter_sum(case, torch.ones_like(d["rho"]))
        lv = _hierarchy(case, d["fixed"], _modulus(rp))
        u = _solve(lv, d["f"])
        _, dc_f, new, sc = _design_side(case, lv[0], u, rp, d["rho"], d["volfrac"])
        return {"u": u, "rho_phys": rp, "dc_f": dc_f, "rho": new, "compliance": sc[0]}
    lv0 = _Level(nel, dim, d["fixed"], _stiffness(dim), E=_modulus(d["rho"]))
    if kind == "carm":
        u, eps = _reduced(lv0, d, case["s"])
        return {"u": u, "eps": eps}
    dc, dc_f, new, sc = _design_side(case, lv0, d["u"], d["rho"], d["design"], d["volfrac"])
    return {"dc": dc, "dc_f": dc_f, "rho": new, "scalars": sc}
