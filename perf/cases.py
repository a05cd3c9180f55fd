"""The workloads by which the speed of this solver is judged.

Every case goes through the Python API of ``paper_2109_04455_gb300.lbm`` the
way a user's program does: a flow solve, an ADR solve, a long-lived ADR solver,
the adjoint behind the catalyst gradients, a batched sweep, or the random walk
particle tracker.  ``exact`` restates the lattice schemes in plain torch
float64 (collide and pull with array shifts and masks), without the library.
"""
import math

import numpy as np
import torch

from paper_2109_04455_gb300 import lbm

PREC = {"f64": lbm.LBM_F64, "f32": lbm.LBM_F32, "f16dev": lbm.LBM_F16DEV}
U0 = 0.05           # inflow centreline velocity of every workload
TAU_FLOW = 0.8


def listed():
    return [
        # one catalyst cylinder in a 200 x 100 channel, the smallest lattice a
        # user starts with: a solve is thousands of steps of a few
        # microseconds each
        dict(name="fiber_flow_f64", kind="flow", nx=200, ny=100, fibers=1,
             prec="f64", steps=400),
        dict(name="fiber_adr_f64", kind="solve", nx=200, ny=100, fibers=1,
             ns=2, prec="f64", steps=400, pe=10.0, da=1.0),
        # the pure-diffusion cascade: a box periodic in both directions,
        # no flow, run for hundreds of thousands of steps
        dict(name="noflow_adr_f32", kind="solve", nx=300, ny=300, fibers=2,
             ns=3, prec="f32", steps=400, pe=1.5, da=15.0, periodic=3),
        # the 1000 x 300 membrane series, reduced precision
        dict(name="membrane_adr_f32", kind="solve", nx=1000, ny=300,
             fibers=12, ns=3, prec="f32", steps=400, pe=10.0, da=50.0),
        # the two-membrane cascade in the default precision: its flow and its
        # ADR lattices take 10^5 steps each to the steady state
        dict(name="cascade_flow_f64", kind="flow", nx=2048, ny=512, fibers=80,
             prec="f64", steps=200),
        dict(name="cascade_adr_f64", kind="solve", nx=2048, ny=512, fibers=80,
             ns=3, prec="f64", steps=200, pe=10.0, da=1.0),
        # gradients with respect to the catalysts: the backward pass of the
        # cascade
        dict(name="cascade_adjoint_f32", kind="adjoint", nx=2048, ny=512,
             fibers=80, ns=3, prec="f32", steps=400, pe=10.0, da=1.0),
        # the throughput lattice of the benchmark, single and half storage
        dict(name="large_adr_f32", kind="run", nx=16384, ny=4096, fibers=2000,
             ns=3, prec="f32", steps=60, pe=50.0, da=0.5),
        dict(name="large_adr_f16dev", kind="run", nx=8192, ny=4096,
             fibers=1000, ns=3, prec="f16dev", steps=100, pe=50.0, da=0.5),
        # a Pe x Da sweep: lattices of uneven size solved together
        dict(name="sweep_batch_f32", kind="batch", count=16, scale=32, ns=3,
             prec="f32", steps=200),
        dict(name="sweep_batch_f16dev", kind="batch", count=16, scale=32,
             ns=3, prec="f16dev", steps=200),
        # the particle method's cross-check of the efficiency, on a membrane
        dict(name="particles", kind="particles", nx=1000, ny=300, fibers=24,
             ns=3, density=1.0, steps=200),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["flow", "solve", "solve", "run", "adjoint", "batch",
                       "particles"])
    prec = rng.choice(["f64", "f32"] if kind in ("flow", "adjoint")
                      else ["f64", "f32", "f16dev"])
    ns = rng.choice([1, 2, 3] if kind in ("solve", "run") else [2, 3])
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(4, 24), ns=ns, prec=prec,
                    scale=rng.choice([17, 27, 32]),
                    steps=2 * rng.randint(25, 100))
    if kind == "particles":
        nx, ny = rng.randint(160, 1200), rng.randint(80, 320)
        return dict(kind=kind, nx=nx, ny=ny, ns=ns,
                    fibers=rng.randint(1, max(1, nx * ny // 8000)),
                    density=_log(rng, 0.2, 2.0), steps=rng.randint(50, 250))
    # channels from the smallest lattices up to millions of nodes, two to
    # four times as long as they are high, of any width
    nodes = _log(rng, 4e3, 1.2e7 if kind == "run" else 2e6)
    aspect = rng.uniform(1.5, 4.5)
    ny = max(24, int(math.sqrt(nodes / aspect)))
    nx = max(40, int(aspect * ny) + rng.randint(0, 31))
    case = dict(kind=kind, nx=nx, ny=ny, prec=prec,
                fibers=rng.randint(1, max(1, nx * ny // 12000)),
                steps=2 * int(min(400, max(20, 2e8 / (nx * ny)))) // 2)
    if kind == "flow":
        return case
    case.update(ns=ns, pe=_log(rng, 1.0, 50.0), da=_log(rng, 0.1, 20.0))
    if kind == "solve":
        option = rng.choice(["", "", "periodic", "nodewise", "abb"])
        if option == "periodic":
            case["periodic"] = rng.choice([1, 2, 3])
        elif option:
            case[option] = True
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _fiber_table(case, seed):
    """Fibers placed by rejection in two bands (A->B upstream, B->C
    downstream), as in the random membranes; radius 5 or 8."""
    rng = np.random.RandomState(seed % (1 << 31))
    nx, ny, n = case["nx"], case["ny"], case["fibers"]
    r = 8.0 if min(nx, ny) >= 60 and nx * ny / n > 1500 else \
        (5.0 if min(nx, ny) >= 40 else 3.0)
    bands = [(0.2 * nx, 0.45 * nx), (0.5 * nx, 0.75 * nx)]
    xs, ys, rows = np.empty(n), np.empty(n), []
    for i in range(n):
        x0, x1 = bands[i % 2]
        for _ in range(20000):
            cx = x0 + r + (x1 - x0 - 2 * r) * rng.random_sample()
            cy = r + 2 + (ny - 1 - 2 * r - 4) * rng.random_sample()
            m = len(rows)
            if m == 0 or np.min((xs[:m] - cx) ** 2 +
                                (ys[:m] - cy) ** 2) >= (2 * r + 4) ** 2:
                xs[m], ys[m] = cx, cy
                cat = 1 + i % 2
                angle = 0.0
                if case["kind"] == "batch" and rng.random_sample() < 0.5:
                    cat, angle = 3, 2 * math.pi * rng.random_sample()
                # the gradients are taken at relaxed catalyst weights
                weight = 0.2 + 0.6 * rng.random_sample() \
                    if case["kind"] == "adjoint" else -1.0
                rows.append([cx, cy, r, cat, angle, weight])
                break
    return np.array(rows, dtype=np.float64).reshape(-1, 6), r


def _velocity(case, seed, fib, dtype):
    """A divergence-free channel flow around the fibers, from a stream
    function: the inflow's parabola and a few smooth waves, corrected near
    the fibers so that the stream function is constant on each of them (some
    relaxation sweeps of the Laplace equation; no flow crosses a fiber)."""
    nx, ny = case["nx"], case["ny"]
    nx_pad = (nx + 31) // 32 * 32
    u = torch.zeros((2, ny, nx_pad), dtype=dtype, device="cuda")
    if case.get("periodic") == 3:
        return u                          # the no-flow box
    rng = np.random.RandomState((seed + 77) % (1 << 31))
    waves = [(0.1 * U0 * ny / math.pi * (2 * rng.random_sample() - 1) / k,
              2 * math.pi * max(1, round(k * nx / (2 * ny))) / nx,
              2 * math.pi * rng.random_sample()) for k in range(1, 4)]

    def stream(x, y, np):
        y = (y + 0.5) / ny
        s = np.sin(math.pi * y) ** 2
        return U0 * ny * y * y * (2 - 4 / 3 * y) + s * sum(
            a * np.sin(kx * x + ph) for a, kx, ph in waves)

    x = torch.arange(nx, dtype=torch.float64, device="cuda")[None, :]
    y = torch.arange(ny, dtype=torch.float64, device="cuda")[:, None]
    psi = stream(x, y, torch)
    solid = np.zeros((ny, nx), bool)
    on = np.zeros((ny, nx), np.float32)
    for cx, cy, r in fib[:, :3]:
        box, inside = _disc(cx, cy, r, nx, ny)
        solid[box] |= inside
        on[box][inside] = stream(cx, cy, np)
    solid = torch.from_numpy(solid).cuda()
    # the correction, with its value kept on the fibers and 0 on the walls
    fixed = torch.where(solid, torch.from_numpy(on).cuda() - psi,
                        torch.zeros_like(psi)).float()
    f = torch.nn.functional.pad(fixed, (1, 1, 1, 1))
    mid = f[1:-1, 1:-1]
    for _ in range(60):
        mean = 0.25 * (f[1:-1, :-2] + f[1:-1, 2:] + f[:-2, 1:-1] +
                       f[2:, 1:-1])
        mid.copy_(torch.where(solid, fixed, mean))
    psi += mid
    u[0, 1:-1, :nx] = (0.5 * (psi[2:] - psi[:-2])).to(dtype)
    u[0, 0, :nx] = (0.5 * psi[1]).to(dtype)
    u[0, -1, :nx] = (0.5 * (2 / 3 * U0 * ny - psi[-2])).to(dtype)
    u[1, :, 1:nx - 1] = (-0.5 * (psi[:, 2:] - psi[:, :-2])).to(dtype)
    u[:, :, :nx].masked_fill_(solid, 0.0)
    return u


def _disc(cx, cy, r, nx, ny):
    """The box of lattice nodes around a fiber, and which are inside it."""
    x0, x1 = max(0, math.floor(cx - r)), min(nx - 1, math.ceil(cx + r))
    y0, y1 = max(0, math.floor(cy - r)), min(ny - 1, math.ceil(cy + r))
    dx = np.arange(x0, x1 + 1)[None, :] - cx
    dy = np.arange(y0, y1 + 1)[:, None] - cy
    return (slice(y0, y1 + 1), slice(x0, x1 + 1)), dx * dx + dy * dy <= r * r


def _rates(case, r):
    d = U0 * r / case["pe"]
    return 3.0 * d + 0.5, min(0.9, case["da"] * d / (r * r))


def _plane(case):
    # the adjoint's plane lies among the fibers, where a few hundred
    # iterations carry its sensitivities to them
    return int(0.62 * case["nx"]) if case["kind"] == "adjoint" else \
        case["nx"] - 3


def _instances(case):
    """The lattices of a batch: widths 16..64 and heights 8..16 times scale,
    Pe and Da over the sweep's range."""
    out = []
    for i in range(case["count"]):
        nx = case["scale"] * (16 + (i * 29) % 49)
        ny = case["scale"] * (8 + (i * 5) % 9)
        out.append(dict(kind="batch", nx=nx, ny=ny, ns=case["ns"],
                        prec=case["prec"], steps=case["steps"],
                        fibers=4 + (nx * ny) // 9000,
                        pe=10.0 ** (-0.2 + 2.0 * ((i * 5) % 8) / 7),
                        da=10.0 ** (-2.0 + 3.0 * ((i * 3) % 8) / 7)))
    return out


def _problem(case, seed):
    """Fiber table, tau and rate of one ADR lattice."""
    fib, r = _fiber_table(case, seed)
    tau, k = _rates(case, r)
    return fib, tau, k


def _flags(case):
    return (lbm.LBM_ADR_NODEWISE if case.get("nodewise") else 0) | \
        (lbm.LBM_ADR_INLET_ABB_ALL if case.get("abb") else 0)


def _c_in(case):
    return (1.0, 0.2, 0.1) if case.get("abb") else (1.0, 0.0, 0.0)


def _geometry(case, fib, k):
    geom = lbm.Geometry(case["nx"], case["ny"], fib, k, 0.8 * k)
    if case.get("periodic"):
        geom.set_periodic(case["periodic"])
    return geom.upload()


def _adr_parts(case, seed):
    fib, tau, k = _problem(case, seed)
    dtype = torch.float64 if case["prec"] == "f64" else torch.float32
    prm = lbm.adr_params(case["ns"], [tau, 1.1 * tau - 0.05, tau],
                         c_in=_c_in(case), precision=PREC[case["prec"]],
                         max_steps=case["steps"],
                         check_every=max(2, case["steps"]),
                         x_plane=_plane(case), flags=_flags(case),
                         neg_tol=-1.0)
    return _geometry(case, fib, k), prm, _velocity(case, seed, fib, dtype)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "flow":
        # other seeds: other fibers and an inflow within a few percent
        fib, _ = _fiber_table(case, seed)
        geom = lbm.Geometry(case["nx"], case["ny"], fib, 0.0, 0.0).upload()
        return dict(case=case, geom=geom, u0=_inflow(seed))
    if kind == "particles":
        fib, r = _fiber_table(case, seed)
        cap = int(1.3 * case["density"] * case["nx"] * case["ny"]) + 4096
        walk = lbm.RWPT(case["nx"], case["ny"], fib, 0.5, 0.4,
                        u=_velocity(case, seed, fib, torch.float64), D=0.1,
                        dt=0.5, delta=0.2, density=case["density"], seed=seed,
                        nspecies=case["ns"], capacity=cap)
        return dict(case=case, walk=walk)
    if kind == "batch":
        parts = [_adr_parts(c, seed + 1000 * i)
                 for i, c in enumerate(_instances(case))]
        return dict(case=case, batch=lbm.Batch(*(list(p) for p in
                                                 zip(*parts))))
    geom, prm, u = _adr_parts(case, seed)
    if kind == "solve":
        return dict(case=case, geom=geom, prm=prm, u=u)
    solver = lbm.ADRSolver(geom, prm, u)
    if kind == "adjoint":
        solver.init().run(_forward_steps(case))   # the state to differentiate
    return dict(case=case, solver=solver, nfibers=int(geom._fib.shape[0]))


def _inflow(seed):
    return U0 * (1.0 + 0.02 * math.sin(seed))


def _forward_steps(case):
    # enough for the sensitivities of both reactions to be there at the plane
    return max(20, min(300, case["nx"] // 4))


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _numbers(case, infos):
    """The reported numbers of the lattices solved, in the precision they were
    computed from.  In reduced precision the per-step residual is the rounding
    noise of the state, so only float64 returns it; without a flow the outflux
    is a difference of equal terms."""
    ns = case["ns"]
    kind = np.float64 if case["prec"] == "f64" else np.float32
    out = dict(mass=np.array([i["mass"][:ns] for i in infos], kind),
               steps=np.array([i["steps"] for i in infos]))
    if case.get("periodic") != 3:
        out["flux"] = np.array([i["flux"][:ns] for i in infos], kind)
    if case["prec"] == "f64":
        out["residual"] = np.array([i["residual"] for i in infos])
    return out


def run(state):
    case = state["case"]
    kind, n = case["kind"], case["steps"]
    if kind == "flow":
        u, info = lbm.lbm_flow_solve(state["geom"], TAU_FLOW, state["u0"], n,
                                     precision=PREC[case["prec"]])
        return dict(u=u, residual=info["residual"], steps=info["steps"])
    if kind == "solve":
        conc, info = lbm.lbm_adr_solve(state["geom"], state["prm"],
                                       state["u"])
        return dict(conc=conc, **_numbers(case, [info]))
    if kind == "run":
        info = state["solver"].init().run(n)
        return dict(conc=state["solver"].conc(), **_numbers(case, [info]))
    if kind == "adjoint":
        dkab, dkbc, dw, info = state["solver"].adjoint(
            n, nfibers=state["nfibers"])
        # the gradients as parameters of the lattice's precision
        kind = torch.float64 if case["prec"] == "f64" else torch.float32
        return dict(dkab=dkab.to(kind), dkbc=dkbc.to(kind), dw=dw.to(kind),
                    steps=info["steps"])
    if kind == "batch":
        b = state["batch"]
        infos = b.solve()
        return dict(conc=[b.conc(i) for i in range(b.count)],
                    **_numbers(case, infos))
    walk = state["walk"]
    info = walk.init().run(n)
    # the particles, in arrays of the walk's capacity
    fields = []
    for a in walk.particles():
        full = np.zeros(walk.capacity, np.float64 if a.dtype.kind == "f"
                        else np.int64)
        full[:a.size] = a
        fields.append(full)
    return dict(x=fields[0], y=fields[1], species=fields[2], ident=fields[3],
                out=np.array(info["out"]), alive=info["alive"])


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _lattice_work(c, kind):
    """One solve: the velocity, the link words and the final fields are read
    or written once; the populations are advanced step by step, each step
    reading and writing them once."""
    nodes, n = c["nx"] * c["ny"], c["steps"]
    size = {"f64": 8, "f32": 4, "f16dev": 2}[c["prec"]]
    field = 8 if c["prec"] == "f64" else 4
    ns = 1 if kind == "flow" else c["ns"]
    flops = nodes * n * (90 if kind == "flow" else 50 * ns)
    ref = 2 if c["prec"] == "f16dev" else 0
    byte = nodes * n * (2 * ns * (9 * size + ref) + 4 + 2 * field *
                        (kind != "flow"))
    return byte + nodes * field * (2 if kind == "flow" else ns), flops


def work(case):
    if case["kind"] == "batch":
        parts = [_lattice_work(c, "batch") for c in _instances(case)]
        return dict(bytes=sum(p[0] for p in parts),
                    flops=sum(p[1] for p in parts))
    if case["kind"] == "particles":
        n = case["density"] * case["nx"] * case["ny"]
        # x, y, id and species read and written each step
        return dict(bytes=2 * 28 * n * case["steps"],
                    flops=100 * n * case["steps"])
    byte, flops = _lattice_work(case, case["kind"])
    return dict(bytes=byte, flops=flops)


# ---------------------------------------------------------------------------
# the same results in plain float64
# ---------------------------------------------------------------------------
CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
W = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4


class _Lattice:
    """Masks of the links of one geometry, for pulls (source x - c_i) and
    gathers (x + c_i)."""

    def __init__(self, case, fib, k1, k2):
        nx, ny = case["nx"], case["ny"]
        per = case.get("periodic", 0)
        self.nx, self.ny, self.px, self.py = nx, ny, bool(per & 1), \
            bool(per & 2)
        solid = np.zeros((ny, nx), bool)
        kab, kbc = np.zeros((ny, nx)), np.zeros((ny, nx))
        owner = np.full((ny, nx), -1)
        for f, (cx, cy, r, cat, ang, weight) in enumerate(fib):
            box, new = _disc(cx, cy, r, nx, ny)
            new &= ~solid[box]
            solid[box] |= new
            dx = np.arange(box[1].start, box[1].stop)[None, :] - cx
            dy = np.arange(box[0].start, box[0].stop)[:, None] - cy
            first = dx * math.cos(ang) + dy * math.sin(ang) >= 0.0
            a = new & ((cat == 1) | ((cat == 3) & first))
            b = new & ((cat == 2) | ((cat == 3) & ~first))
            kab[box][a] = k1
            kbc[box][b] = k2
            if weight >= 0:
                kab[box][new] = weight * k1
                kbc[box][new] = (1 - weight) * k2
            owner[box][new] = f
        self.solid = torch.from_numpy(solid).cuda()
        self.kab = torch.from_numpy(kab).cuda()
        self.kbc = torch.from_numpy(kbc).cuda()
        self.owner = torch.from_numpy(owner).cuda()
        # bounce[i]: fluid nodes whose neighbour x + c_i is a wall or solid
        self.bounce, self.cat = [None] * 9, [None] * 9
        for i in range(1, 9):
            hit = self._from(self.solid, i)
            edge_x = torch.zeros_like(hit)
            if not self.px and CX[i]:
                edge_x[:, -1 if CX[i] > 0 else 0] = True
            if not self.py and CY[i]:
                hit[-1 if CY[i] > 0 else 0, :] = True
            hit &= ~edge_x
            self.bounce[i] = hit & ~self.solid
            # links into a fiber node: (flat fluid node, flat fiber node)
            link = hit & ~self.solid
            if not self.py and CY[i]:
                link[-1 if CY[i] > 0 else 0, :] = False
            yy, xx = torch.nonzero(link, as_tuple=True)
            self.cat[i] = (yy * nx + xx, ((yy + CY[i]) % ny) * nx +
                           (xx + CX[i]) % nx)

    @staticmethod
    def _from(a, i):
        """a at x + c_i."""
        return torch.roll(a, (-CY[i], -CX[i]), (-2, -1))


def _equilibrium(u, nx):
    ux, uy = u[0, :, :nx].double(), u[1, :, :nx].double()
    uu = ux * ux + uy * uy
    out = []
    for i in range(9):
        cu = CX[i] * ux + CY[i] * uy
        out.append(W[i] * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * uu))
    return out


def _pad(a):
    nx = a.shape[-1]
    out = torch.zeros(a.shape[:-1] + ((nx + 31) // 32 * 32,), dtype=a.dtype,
                      device=a.device)
    out[..., :nx] = a
    return out


def _exact_adr(case, fib, tau, k, u, steps):
    """(g* after the last step, C, C before, flux, lattice, E, omega)"""
    ns, nx, ny = case["ns"], case["nx"], case["ny"]
    lat = _Lattice(case, fib, k, 0.8 * k)
    E = _equilibrium(u, nx)
    om = [1.0 / t for t in (tau, 1.1 * tau - 0.05, tau)][:ns]
    cin = _c_in(case)
    fluid = (~lat.solid).double()
    g = [[(fluid if s == 0 else 0 * fluid) * E[i] for i in range(9)]
         for s in range(ns)]
    kab, kbc = lat.kab.view(-1), lat.kbc.view(-1)
    if case.get("nodewise"):
        cnt, sa, sb = (torch.zeros(nx * ny, dtype=torch.float64,
                                   device="cuda") for _ in range(3))
        for j in range(1, 9):
            x, n = lat.cat[j]
            on = (kab[n] != 0) | (kbc[n] != 0)
            cnt[x] += on.double()
            sa[x] += kab[n]
            sb[x] += kbc[n]
        cnt.clamp_(min=1)
        ka_node, kb_node = (sa / cnt).view(ny, nx), (sb / cnt).view(ny, nx)

    def react(g, C):
        for s in range(ns):
            for j in range(9):
                if case.get("nodewise"):
                    q = -ka_node * C[0] if s == 0 else (
                        ka_node * C[0] - (kb_node * C[1] if ns > 2 else 0)
                        if s == 1 else kb_node * C[1])
                    g[s][j] += W[j] * q * fluid
                elif j:
                    x, n = lat.cat[j]
                    ca = C[0].view(-1)[x]
                    cb = C[1].view(-1)[x] if ns > 1 else 0
                    q = -kab[n] * ca if s == 0 else (
                        kab[n] * ca - (kbc[n] * cb if ns > 2 else 0)
                        if s == 1 else kbc[n] * cb)
                    g[s][j].view(-1)[x] += W[j] * q

    C = [fluid] + [0 * fluid] * (ns - 1)
    react(g, C)                     # the start is collided as well
    for _ in range(steps):
        prev, C = C, []
        for s in range(ns):
            old = g[s]
            new = []
            last = sum(o[:, -1] for o in old) if not lat.px else None
            for i in range(9):
                if i == 0:
                    new.append(old[0].clone())
                    continue
                j = OPP[i]
                p = torch.where(lat.bounce[j], old[j], lat._from(old[i], j))
                if not lat.px and CX[i] > 0:
                    b = old[j][:, 0]
                    p[:, 0] = -b + 2 * W[i] * cin[s] \
                        if s == 0 or case.get("abb") else b
                elif not lat.px and CX[i] < 0:
                    p[:, -1] = -old[j][:, -1] + 2 * W[i] * last
                new.append(p)
            c = sum(new) * fluid
            C.append(c)
            for i in range(9):
                new[i].mul_(1 - om[s]).add_(om[s] * c * E[i]).mul_(fluid)
            g[s] = new
        react(g, C)
    xp = _plane(case)
    flux = [float(sum(CX[i] * g[s][i][:, xp].sum() for i in range(9))) / ny
            for s in range(ns)]
    return g, C, prev, flux, lat, E, om


def _exact_solution(case, seed):
    fib, tau, k = _problem(case, seed)
    dtype = torch.float64 if case["prec"] == "f64" else torch.float32
    u = _velocity(case, seed, fib, dtype)
    g, C, prev, flux, _, _, _ = _exact_adr(case, fib, tau, k, u,
                                           case["steps"])
    mass = [float(c.abs().sum()) for c in C]
    res = max(float((c - p).abs().sum()) / m if m > 0 else 0.0
              for c, p, m in zip(C, prev, mass))
    return dict(conc=_pad(torch.stack(C)),
                **_numbers(case, [dict(mass=mass, flux=flux, residual=res,
                                       steps=case["steps"])]))


def _exact_flow(case, seed):
    fib, _ = _fiber_table(case, seed)
    lat = _Lattice(case, fib, 0.0, 0.0)
    nx, ny, u0, om = case["nx"], case["ny"], _inflow(seed), 1.0 / TAU_FLOW
    y = torch.arange(ny, dtype=torch.float64, device="cuda")
    uin = 4 * u0 * (y + 0.5) * (ny - 0.5 - y) / ny ** 2
    fluid = (~lat.solid).double()

    def feq(i, rho, ux, uy, uu):
        cu = CX[i] * ux + CY[i] * uy
        return W[i] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * uu)

    ux0 = uin[:, None].expand(ny, nx)
    f = [feq(i, fluid, ux0, 0 * ux0, ux0 * ux0) for i in range(9)]
    ux = uy = None
    for _ in range(case["steps"]):
        r = sum(v[:, -1] for v in f)
        wx = sum(CX[i] * f[i][:, -1] for i in range(9)) / r
        wy = sum(CY[i] * f[i][:, -1] for i in range(9)) / r
        new = [f[0]]
        for i in range(1, 9):
            j = OPP[i]
            p = torch.where(lat.bounce[j], f[j], lat._from(f[i], j))
            if CX[i] > 0:
                p[:, 0] = f[j][:, 0] + 6 * W[i] * uin
            elif CX[i] < 0:
                cu = CX[i] * wx + CY[i] * wy
                p[:, -1] = -f[j][:, -1] + 2 * W[i] * (
                    1 + 4.5 * cu * cu - 1.5 * (wx * wx + wy * wy))
            new.append(p)
        rho = sum(new) + lat.solid.double()
        px, py = ux, uy
        ux = sum(CX[i] * new[i] for i in range(9)) / rho * fluid
        uy = sum(CY[i] * new[i] for i in range(9)) / rho * fluid
        uu = ux * ux + uy * uy
        f = [(v + om * (feq(i, rho, ux, uy, uu) - v)) * fluid
             for i, v in enumerate(new)]
    res = float((ux - px).abs().sum() + (uy - py).abs().sum()) / \
        float(ux.abs().sum() + uy.abs().sum())
    return dict(u=_pad(torch.stack([ux, uy])), residual=res, steps=None)


def _exact_adjoint(case, seed):
    fib, tau, k = _problem(case, seed)
    dtype = torch.float64 if case["prec"] == "f64" else torch.float32
    ns, nx, ny = case["ns"], case["nx"], case["ny"]
    _, C, _, flux, lat, E, om = _exact_adr(
        case, fib, tau, k, _velocity(case, seed, fib, dtype),
        _forward_steps(case))
    total = sum(flux)
    if ns == 2:
        dN = [-flux[1] / total ** 2, flux[0] / total ** 2]
    else:
        dN = [-flux[2] / total ** 2] * 2 + [(flux[0] + flux[1]) / total ** 2]
    fluid = (~lat.solid).double()
    kab, kbc, xp = lat.kab.view(-1), lat.kbc.view(-1), _plane(case)

    def gather(nu):
        out = []
        for s in range(ns):
            mu, extra = [nu[s][0].clone()], torch.zeros(
                ny, dtype=torch.float64, device="cuda")
            for i in range(1, 9):
                back = nu[s][OPP[i]]
                m = torch.where(lat.bounce[i], back, lat._from(nu[s][i], i))
                if CX[i] < 0:
                    m[:, 0] = -back[:, 0] if s == 0 else back[:, 0]
                elif CX[i] > 0:
                    m[:, -1] = -back[:, -1]
                    extra = extra + 2 * W[i] * back[:, -1]
                mu.append(m)
            for i in range(9):
                mu[i][:, -1] += extra
                mu[i][:, xp] += CX[i] * dN[s] / ny
            out.append(mu)
        return out

    nu = [[torch.zeros_like(fluid) for _ in range(9)] for _ in range(ns)]
    for _ in range(case["steps"]):
        mu = gather(nu)
        R = [torch.zeros_like(fluid) for _ in range(ns)]
        for j in range(1, 9):
            x, n = lat.cat[j]
            at = [mu[s][j].view(-1)[x] for s in range(ns)]
            R[0].view(-1)[x] += kab[n] * W[j] * (at[1] - at[0])
            if ns > 2:
                R[1].view(-1)[x] += kbc[n] * W[j] * (at[2] - at[1])
        nu = []
        for s in range(ns):
            lam = om[s] * sum(E[i] * mu[s][i] for i in range(9)) + R[s]
            nu.append([((1 - om[s]) * mu[s][i] + lam) * fluid
                       for i in range(9)])
    mu = gather(nu)
    dkab, dkbc = torch.zeros_like(kab), torch.zeros_like(kab)
    for j in range(1, 9):
        x, n = lat.cat[j]
        at = [mu[s][j].view(-1)[x] for s in range(ns)]
        dkab.index_add_(0, n, W[j] * C[0].view(-1)[x] * (at[1] - at[0]))
        if ns > 2:
            dkbc.index_add_(0, n, W[j] * C[1].view(-1)[x] * (at[2] - at[1]))
    own = lat.owner.view(-1)
    dw = torch.zeros(len(fib), dtype=torch.float64, device="cuda")
    on = own >= 0
    dw.index_add_(0, own[on], k * dkab[on] - 0.8 * k * dkbc[on])
    return dict(dkab=_pad(dkab.view(ny, nx)), dkbc=_pad(dkbc.view(ny, nx)),
                dw=dw, steps=None)


def exact(case, seed):
    kind = case["kind"]
    if kind == "flow":
        return _exact_flow(case, seed)
    if kind == "adjoint":
        return _exact_adjoint(case, seed)
    if kind == "batch":
        got = [_exact_solution(c, seed + 1000 * i)
               for i, c in enumerate(_instances(case))]
        return dict({key: np.concatenate([o[key] for o in got])
                     for key in got[0] if key != "conc"},
                    conc=[o["conc"] for o in got])
    if kind == "particles":
        return None        # a sequence of single IEEE operations: it is exact
    return _exact_solution(case, seed)
