"""The work that users of this library give it, as sized cases, and the means to run them.

A case is a dict of plain values:

  kind       "step": one fractional step of a running simulation (Grid.step or
             Grid.step_graph) from a restart state, as an ensemble member, a restarted run
             or the adjoint's recomputation takes it; "adjoint": a forward run and its
             reverse sweep (AdjointRun); "checkpoint": the four state fields compressed to
             wavelet streams and decoded again
  flow       "channel": inflow past a fixed sphere with convective outflow; "cavity": the
             lid-driven cavity; "two_level": the channel with a refined block and rotating
             ellipsoids; "batch": many independent cavities and channels in one grid
  nx ny nz   level-0 cubes (cavity: nx per edge; batch: nx sims, cube counts ny .. nz)
  B          cells per cube edge
  prec       0 FP64, 1 FP32 state with FP64 defect correction, 2 FP64 state with it
  mg         multigrid preconditioner, else Jacobi
  graph      the step as a captured CUDA graph
  cn         QUICK + Crank-Nicolson momentum, else Adams-Bashforth + central
  particles  Lagrangian particles on the sphere, else the solid fraction
  bf16       lagged convection stored as bfloat16 (prec 1)
"""
import functools
import math

import numpy as np
import torch

from paper_1808_04099_gb300 import adjoint, bcm
from paper_1808_04099_gb300 import workloads as W

H = 1.0 / 64.0    # cell size of the channel flows, that of the sphere workload
RE = 300.0
LEAD = 2          # steps a run has behind it when a "step" case begins: the warm start of
                  # the pressure, the lagged convection and the outflow values are a run's
NOISE = 1e-2      # velocity fluctuations of the initial state
STATE = (bcm.U, bcm.V, bcm.W, bcm.P, bcm.NX, bcm.NY, bcm.NZ, bcm.UB)
NAMES = ("u", "v", "w", "p", "nx", "ny", "nz", "ub")


def _case(name, kind, flow, nx, ny, nz, B, prec, mg=False, graph=False, cn=False,
          particles=False, bf16=False):
    c = dict(kind=kind, flow=flow, nx=nx, ny=ny, nz=nz, B=B, prec=prec, mg=mg, graph=graph,
             cn=cn, particles=particles, bf16=bf16)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest run that is made in earnest (a sphere in 16 cubes of 8^3, parameter
        # scans and regression runs): latency and launches
        _case("channel_8k_fp64", "step", "channel", 4, 2, 2, 8, 0),
        # the 64^3 cavity, the plain FP64 method
        _case("cavity_262k_fp64", "step", "cavity", 4, 4, 4, 16, 0),
        # the sphere flow (4.2M cells) in FP64 with the production solver
        _case("channel_4M_fp64_mg", "step", "channel", 16, 8, 8, 16, 0, mg=True),
        # the same in mixed precision with the default solver, issued by the host
        _case("channel_4M_mixed", "step", "channel", 16, 8, 8, 16, 1),
        # ... and with multigrid as a captured step, the fastest way to run it
        _case("channel_4M_mixed_mg_graph", "step", "channel", 16, 8, 8, 16, 1, mg=True,
              graph=True),
        # moving bodies on the two-level grid at full size (83.1M cells)
        _case("two_level_83M_mixed_mg", "step", "two_level", 32, 16, 16, 16, 1, mg=True),
        # the same flow at half the extent (10.4M cells) with the default solver: the
        # vectors of the solver no longer fit the L2 cache
        _case("two_level_10M_mixed", "step", "two_level", 16, 8, 8, 16, 1),
        # 64 independent simulations of 8 .. 512 cubes in captured steps
        _case("batch64_mixed_mg_graph", "step", "batch", 64, 8, 512, 16, 1, mg=True, graph=True),
        # an ensemble of small simulations (cubes of 8^3) with the default solver
        _case("batch24_small_mixed_graph", "step", "batch", 24, 8, 64, 8, 1, graph=True),
        # QUICK + Crank-Nicolson, Lagrangian particles and multigrid together, on an
        # uneven grid: the method's production set-up
        _case("channel_1M6_cn_particles", "step", "channel", 11, 5, 7, 16, 1, mg=True, cn=True,
              particles=True),
        # a checkpoint of the sphere flow's state, written and read back
        _case("checkpoint_4M", "checkpoint", "channel", 16, 8, 8, 16, 1),
        # drag gradient over two steps (0.5M cells): forward, recomputation, reverse sweep
        _case("adjoint_524k_fp64", "adjoint", "channel", 16, 8, 8, 8, 0),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    # half the draws are plain steps of channels and cavities, as in use
    what = rng.choice(["channel", "channel", "channel", "cavity", "two_level", "batch",
                       "checkpoint", "adjoint"])
    B = rng.choice([4, 8, 8, 16, 16, 16])
    prec = rng.choice([0, 0, 1, 1, 1, 2])
    mg = rng.random() < 0.5
    graph = rng.random() < 0.4
    bf16 = prec == 1 and rng.random() < 0.2

    def box(cells, B):  # cubes per axis of an elongated box of about this many cells
        n = max(8.0, cells / B ** 3)
        m = (n / 2.0) ** (1.0 / 3.0)
        ny = max(2, round(m * rng.uniform(0.75, 1.35)))
        nz = max(2, round(m * rng.uniform(0.75, 1.35)))
        return max(2, round(n / (ny * nz))), ny, nz

    # the plain solver's iterations grow with the grid, the FP64 ones cost most
    top = 4.0e6 if mg else (0.6e6 if prec == 0 else 2.0e6)
    if B == 4:
        top = min(top, 0.5e6)
    if what == "channel":
        particles = rng.random() < 0.25
        return _case(None, "step", "channel", *box(_log(rng, 6e3, top), B), B, prec, mg,
                     graph, rng.random() < 0.25, particles, bf16)
    if what == "cavity":
        m = max(2, round((_log(rng, 6e3, min(top, 1.5e6)) / B ** 3) ** (1.0 / 3.0)))
        return _case(None, "step", "cavity", m, m, m, B, prec, mg, graph, bf16=bf16)
    if what == "two_level":
        n = rng.randint(5, 7) if B == 16 else rng.randint(5, 10)
        return _case(None, "step", "two_level", n + rng.randint(0, 4), n, n, B, max(prec, 1),
                     mg, graph, bf16=bf16)
    if what == "batch":
        B = max(B, 8)
        return _case(None, "step", "batch", rng.randint(2, 32), 8, rng.randint(16, 96), B,
                     max(prec, 1), mg, True, bf16=bf16)
    if what == "checkpoint":
        return _case(None, "checkpoint", "channel", *box(_log(rng, 6e3, 4e6), B), B,
                     rng.choice([0, 1, 1, 2]))
    return _case(None, "adjoint", "channel", *box(_log(rng, 6e3, 2.5e5), max(B, 8)), max(B, 8), 0)


# ------------------------------------------------------------------ grids and states

@functools.lru_cache(maxsize=4)
def _spec(flow, nx, ny, nz, B):
    if flow == "cavity":
        return W.cavity(nx, B)
    if flow == "two_level":
        # the refined block keeps its distance to the domain faces, as in the workload
        def lo(n):
            return max(1, round(n * 5 / 16))

        def cut(n):
            return max(1, n // 8)
        return W.two_level_channel(nx, ny, nz, B, (lo(nx), cut(ny), cut(nz)),
                                   (nx - lo(nx), ny - cut(ny), nz - cut(nz)), 1.0 / (4.0 * B))
    if flow == "batch":
        return W.batched_mix(nx, 0, B, ny, nz)
    length = tuple(n * B * H for n in (nx, ny, nz))
    side = min(length[1], length[2])
    return W.sphere_channel(nx, ny, nz, B, length, side / 8.0,
                            (length[0] / 4.0, length[1] / 2.0, length[2] / 2.0), RE)


def _spec_of(case):
    return _spec(case["flow"], case["nx"], case["ny"], case["nz"], case["B"])


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _base(spec):
    """1 on the cells of sims with an inflow of speed 1 along x, else 0."""
    has = torch.tensor([float(W.INFLOW in list(b)) for b in spec.sim_bc], dtype=torch.float64)
    counts = torch.tensor(np.diff(spec.sim_cube_offset) * spec.B ** 3)
    return torch.repeat_interleave(has.cuda(), counts.cuda())


def _initial(spec, seed, dtype):
    """The inflow everywhere plus seeded fluctuations, in the state's type."""
    g = _generator(seed)
    base = _base(spec)
    out = []
    for k in range(3):
        x = (torch.rand(spec.n_cells, generator=g, device="cuda", dtype=torch.float64) - 0.5)
        out.append((x * (2.0 * NOISE) + (base if k == 0 else 0.0)).to(dtype))
    return out


def _rtol(case):
    # FP32 states run at Grid.step's tolerance, FP64 states at Grid.solve_pressure's
    return 1e-10 if case["prec"] == 1 else 1e-12


def _advance(g, case, n):
    f = g.step_graph if case["graph"] else g.step
    f(n, rtol=_rtol(case), stats=False)


def prepare(case, seed):
    spec = _spec_of(case)
    if case["kind"] == "adjoint":
        modes = np.random.default_rng(seed).uniform(-0.05, 0.05, 8)
        u, v, w = (x.cpu().numpy() for x in _initial(spec, seed, torch.float64))
        st = W.initial_state(spec)
        body = spec.bodies[0][0]
        run_ = adjoint.AdjointRun(spec, modes, body.center, float(body.axes[0]), 2,
                                  state=W.State(u, v, w, st.p, st.ub))
        return {"case": case, "run": run_}
    g = bcm.Grid(spec, case["prec"], lagged_bf16=case["bf16"])
    if case["kind"] == "checkpoint":
        # smooth flow features over the box, a body's boundary layer, small fluctuations
        steps = []
        for k, f in enumerate(STATE[:4]):
            t = g.field(f)
            t.copy_(_smooth(spec, seed, k))
            steps.append(1e-4 * float(t.abs().max()))
        # a checkpoint buffer with one slot per field, of a word per value and the tables
        slots = torch.zeros(4, spec.n_cells + 2 * spec.n_cubes + 8, dtype=torch.int32,
                            device="cuda")
        return {"case": case, "grid": g, "steps": steps, "slots": slots}
    if case["mg"]:
        g.set_preconditioner(bcm.PRECOND_MULTIGRID)
    if case["cn"]:
        g.set_momentum_scheme(bcm.SCHEME_QUICK_CN)
    if case["particles"]:
        g.set_particles(W.surface_particles(spec))
    for f, t in zip(STATE[:3], _initial(spec, seed, g.field(bcm.U).dtype)):
        g.field(f).copy_(t)
    g.field(bcm.UB).view(-1, 3, spec.B * spec.B)[:, 0] = 1.0
    _advance(g, case, LEAD)
    return {"case": case, "grid": g, "restart": [g.field(f).clone() for f in STATE],
            "fields": [g.field(f) for f in STATE]}


def _smooth(spec, seed, k):
    """A seeded smooth field with fluctuations, cube by cube."""
    B, g = spec.B, _generator(4 * seed + k)
    ijk = torch.tensor(spec.cube_ijk, device="cuda", dtype=torch.float64)
    ax = torch.arange(B, device="cuda", dtype=torch.float64)
    n = float(spec.sim_extent[0].max())
    x = (ijk[:, 0, None] + ax)[:, None, None, :] / n
    y = (ijk[:, 1, None] + ax)[:, None, :, None] / n
    z = (ijk[:, 2, None] + ax)[:, :, None, None] / n
    a = torch.rand(12, generator=g, device="cuda", dtype=torch.float64) * 2 * math.pi
    f = torch.zeros(ijk.shape[0], B, B, B, device="cuda", dtype=torch.float64)
    for m in range(4):
        f += torch.sin((m + 1) * 3 * x + a[3 * m]) * torch.sin((m + 1) * 2 * y + a[3 * m + 1]) \
            * torch.cos((m + 1) * 2 * z + a[3 * m + 2]) / (m + 1)
    r = torch.sqrt((x - 0.25) ** 2 + (y - 0.25) ** 2 + (z - 0.25) ** 2)
    f *= torch.tanh(30.0 * r)
    f += (torch.rand(f.shape, generator=g, device="cuda", dtype=torch.float64) - 0.5) * 2e-3
    return f.reshape(-1)


def run(state):
    case = state["case"]
    if case["kind"] == "adjoint":
        J = state["run"].forward()
        da, dc = state["run"].backward()
        out = {n: state["run"].g.field(f) for n, f in zip(NAMES, STATE)}
        return dict(out, J=np.array([J]), da=da, dc=dc)
    g = state["grid"]
    if case["kind"] == "checkpoint":
        slots = state["slots"]
        sizes = []
        for slot, f, h in zip(slots, STATE[:4], state["steps"]):
            s = g.compress_field(f, h)
            sizes.append(s.numel())
            slot[:s.numel()].copy_(s)
            slot[s.numel():].zero_()
        back = (bcm.USTAR, bcm.VSTAR, bcm.WSTAR, bcm.RHS)
        for f, slot, n in zip(back, slots, sizes):
            g.decompress_field(f, slot[:n])
        return {"streams": slots, "sizes": sizes, "fields": [g.field(f) for f in back]}
    for t, s in zip(state["fields"], state["restart"]):
        t.copy_(s)
    g.set_step(LEAD)
    _advance(g, case, 1)
    out = dict(zip(NAMES, state["fields"]))
    if case["prec"] == 1:
        # an FP32 run hands its pressure on as it does its velocities: the digits beyond
        # are those of the FP32 momentum's rounding
        out["p"] = out["p"].float()
    return out


def work(case):
    """One pass: each input read once, each output written once; for the flops the
    explicit stencils and one application of the pressure operator."""
    cells = _spec_of(case).n_cells
    S = 4 if case["prec"] == 1 else 8
    if case["kind"] == "checkpoint":
        return {"bytes": 2 * cells * (3 * S + 8), "flops": 4 * 2 * 20 * cells}
    per = {"bytes": cells * (2 * (6 * S + 8) + S), "flops": 150 * cells}
    return {k: v * (6 if case["kind"] == "adjoint" else 1) for k, v in per.items()}


# ------------------------------------------------------------------------- in 64 bits

def _ghosted(x, d, lo, hi):
    """x with one layer before and after along axis d (arrays are [z, y, x]; d = 0 is x)."""
    ax = 2 - d
    return torch.cat([lo.unsqueeze(ax), x, hi.unsqueeze(ax)], ax)


def _ends(x, d):
    ax = 2 - d
    return x.select(ax, 0), x.select(ax, x.shape[ax] - 1)


class _Box:
    """One single-level simulation on monolithic arrays, in FP64: central convection with
    Adams-Bashforth, the solid-fraction forcing of fixed spheres, a direct solve of the
    pressure equation in the eigenvectors of its one-dimensional operators."""

    def __init__(self, spec, s):
        self.n = [int(e) for e in spec.sim_extent[s]]
        self.h, self.nu = float(spec.sim_h0[s]), float(spec.sim_nu[s])
        self.dt, self.uc = float(spec.sim_dt[s]), float(spec.sim_uconv[s])
        self.bc, self.vel = [int(b) for b in spec.sim_bc[s]], spec.sim_bc_vel[s]
        shape = (self.n[2], self.n[1], self.n[0])
        self.phi = torch.zeros(shape, device="cuda", dtype=torch.float64)
        x = [(torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) * self.h + float(o)
             for n, o in zip(self.n, spec.sim_origin[s])]
        for b in spec.bodies[s]:
            c = [float(v) for v in b.center]
            d = torch.sqrt((x[0] - c[0])[None, None, :] ** 2 + (x[1] - c[1])[None, :, None] ** 2
                           + (x[2] - c[2])[:, None, None] ** 2) - float(b.axes[0])
            eps = 1.5 * self.h
            self.phi = torch.where(d < 20 * eps, 0.5 * (1 - torch.tanh(d / eps)), 0.0)
        self.vec, self.val = [], []
        for d in range(3):
            n = self.n[d]
            t = 2 * torch.eye(n, dtype=torch.float64)
            t -= torch.diag(torch.ones(n - 1, dtype=torch.float64), 1)
            t -= torch.diag(torch.ones(n - 1, dtype=torch.float64), -1)
            for e, f in ((0, 2 * d), (n - 1, 2 * d + 1)):
                t[e, e] += 1.0 if self.bc[f] == W.OUTFLOW else -1.0
            val, vec = torch.linalg.eigh(t)
            self.val.append(val.cuda())
            self.vec.append(vec.cuda())
        self.singular = W.OUTFLOW not in self.bc
        self.p = torch.zeros(shape, device="cuda", dtype=torch.float64)
        self.ub = {f: [torch.full(shape[:2 - f // 2] + shape[3 - f // 2:], float(c == 0),
                                  device="cuda", dtype=torch.float64) for c in range(3)]
                   for f in range(6) if self.bc[f] == W.OUTFLOW}
        self.old = None

    def velocity_ghosts(self, x, c, d):
        out = []
        for side, u0 in zip((0, 1), _ends(x, d)):
            f = 2 * d + side
            if self.bc[f] == W.SLIP:
                out.append(-u0 if c == d else u0)
            elif self.bc[f] == W.OUTFLOW:
                out.append(2 * self.ub[f][c] - u0)
            else:
                out.append(2 * float(self.vel[f][c]) - u0)
        return _ghosted(x, d, *out)

    def poisson(self, b):
        # sum of the 1-D operators / h^2, p = -A^-1 b
        x = b
        if self.singular:
            x = x - x.mean()
        x = torch.einsum("zyx,xa->zya", x, self.vec[0])
        x = torch.einsum("zyx,yb->zbx", x, self.vec[1])
        x = torch.einsum("zyx,zc->cyx", x, self.vec[2])
        lam = self.val[0][None, None, :] + self.val[1][None, :, None] + self.val[2][:, None, None]
        if self.singular:
            lam[0, 0, 0] = 1.0
            x[0, 0, 0] = 0.0
        x = -x * self.h ** 2 / lam
        x = torch.einsum("cyx,zc->zyx", x, self.vec[2])
        x = torch.einsum("zbx,yb->zyx", x, self.vec[1])
        return torch.einsum("zya,xa->zyx", x, self.vec[0])

    def step(self, u):
        N, star = [], []
        for c in range(3):
            n, lap = 0.0, 0.0
            for d in range(3):
                gc = self.velocity_ghosts(u[c], c, d)
                gd = self.velocity_ghosts(u[d], d, d)
                m = gc.shape[2 - d] - 1
                fc = 0.5 * (gc.narrow(2 - d, 0, m) + gc.narrow(2 - d, 1, m))
                fd = 0.5 * (gd.narrow(2 - d, 0, m) + gd.narrow(2 - d, 1, m))
                n = n + torch.diff(fc * fd, dim=2 - d) / self.h
                lap = lap + torch.diff(gc, n=2, dim=2 - d) / self.h ** 2
            prev = n if self.old is None else self.old[c]
            t = u[c] + self.dt * (-(1.5 * n - 0.5 * prev) + self.nu * lap)
            N.append(n)
            star.append(t - self.phi * t)
        self.old = N
        for f, ub in self.ub.items():
            for c in range(3):
                u0 = _ends(u[c], f // 2)[f % 2]
                ub[c] = ub[c] - self.uc * self.dt / (0.5 * self.h) * (ub[c] - u0)
        div = 0.0
        for d in range(3):
            ends = []
            for side, u0 in zip((0, 1), _ends(star[d], d)):
                f = 2 * d + side
                if self.bc[f] == W.SLIP:
                    ends.append(torch.zeros_like(u0))
                elif self.bc[f] == W.OUTFLOW:
                    ends.append(self.ub[f][d])
                else:
                    ends.append(torch.full_like(u0, float(self.vel[f][d])))
            m = star[d].shape[2 - d] - 1
            inner = 0.5 * (star[d].narrow(2 - d, 0, m) + star[d].narrow(2 - d, 1, m))
            div = div + torch.diff(_ghosted(inner, d, *ends), dim=2 - d)
        self.p = self.poisson(div / (self.h * self.dt))
        out = []
        for d in range(3):
            ends = [-e if self.bc[2 * d + side] == W.OUTFLOW else e
                    for side, e in zip((0, 1), _ends(self.p, d))]
            grad = torch.diff(_ghosted(self.p, d, *ends), dim=2 - d) / self.h
            m = grad.shape[2 - d] - 1
            out.append(star[d] - 0.5 * self.dt * (grad.narrow(2 - d, 0, m)
                                                  + grad.narrow(2 - d, 1, m)))
        return out


def exact(case, seed):
    if case["kind"] != "step" or case["flow"] == "two_level" or case["cn"] or case["particles"] \
            or case["bf16"]:
        return None
    spec = _spec_of(case)
    B, B3 = spec.B, spec.B ** 3
    u0 = [x.double() for x in _initial(spec, seed, torch.float32 if case["prec"] == 1
                                       else torch.float64)]
    slots = W.outflow_slots(spec)
    out = {k: torch.zeros(spec.n_cells, device="cuda", dtype=torch.float64) for k in NAMES[:7]}
    out["ub"] = torch.zeros(len(slots), 3, B, B, device="cuda", dtype=torch.float64)
    ax = torch.arange(B, device="cuda")
    sim = spec.sim_of_cube()
    for s in range(spec.n_sims):
        a, b = int(spec.sim_cube_offset[s]), int(spec.sim_cube_offset[s + 1])
        box = _Box(spec, s)
        q = torch.tensor(spec.cube_ijk[a:b], device="cuda", dtype=torch.int64)
        at = ((q[:, 2, None] + ax)[:, :, None, None] * box.n[1]
              + (q[:, 1, None] + ax)[:, None, :, None]) * box.n[0] \
            + (q[:, 0, None] + ax)[:, None, None, :]
        at = at.reshape(-1)

        def whole(x):
            y = torch.empty(box.phi.numel(), device="cuda", dtype=torch.float64)
            y[at] = x[a * B3:b * B3]
            return y.reshape(box.phi.shape)
        u = [whole(x) for x in u0]
        for _ in range(LEAD + 1):
            u = box.step(u)
        for name, x in zip(NAMES[:7], u + [box.p] + box.old):
            out[name][a * B3:b * B3] = x.reshape(-1)[at]
        for k, (c, f) in enumerate(slots):
            if sim[c] != s:
                continue
            d = f // 2
            t1, t2 = (1 if d == 0 else 0), (1 if d == 2 else 2)
            i1, i2 = int(spec.cube_ijk[c, t1]), int(spec.cube_ijk[c, t2])
            for e in range(3):
                out["ub"][k, e] = box.ub[f][e][i2:i2 + B, i1:i1 + B]
    out["ub"] = out["ub"].reshape(-1)
    if not all(W.OUTFLOW in list(b) for b in spec.sim_bc):
        out["p"] = None  # without an outflow the pressure is known up to a constant only
    return out
