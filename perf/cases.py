"""The work that a program built on this library has it do, as measurable cases.

A case is one call pattern: a chip (or a batch of chips) in some state, advanced by
n time steps through the public calls and read out into device arrays.  ``prepare``
builds the chip with ``Chip.from_problem`` / ``Chip.batch`` and gives it seeded fields
near a developed channel flow; ``run`` makes the calls; ``exact`` evaluates the same
steps in 64 bits with plain torch operations (written out below from the method: pull
streaming, bounce-back or the paper's walls, port completion, both BGK collisions).

Kinds of case:
  steps    Chip.step(n), then the four fields
  monitor  Chip.step_diagnostics(n): every step's totals, then the four fields
  scalar   Chip.scalar_step(n) on a stored velocity field, then the concentration
  batch    many chips in one handle: Chip.step(n), then the stacked fields
  gradient Chip.adjoint(n): objective and all derivatives, then the concentration
"""
import math

import numpy as np
import torch

from paper_1307_4703_gb300 import lbm, workloads as W

PRECISIONS = ("fp32", "fp16", "bf16")


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _chip(name, nx, ny, n, kind="steps", geometry="chip", precision="fp32", valves="held", paper_ports=False,
          walls=False, decay=0.0, ckpt=0, u_scale=1.0, chips=1):
    """geometry: "small" (the 256 x 128 chip's proportions, tau 0.8), "chip" (the 1024 x
    768 / 4096 x 2048 chips' proportions, tau 0.6) or "obstacles" (random solid cells,
    every kind of port, two valve words in turn)."""
    c = dict(kind=kind, nx=nx, ny=ny, n=n, geometry=geometry, precision=precision, valves=valves,
             paper_ports=paper_ports, walls=walls, decay=decay, ckpt=ckpt, u_scale=u_scale, chips=chips)
    return c if name is None else dict(c, name=name)


def listed():
    return [
        # the smallest call: a control loop that advances the 256 x 128 chip by a single
        # step and looks at the fields each time (launches and latency count)
        _chip("one-step-256x128", 256, 128, 1, geometry="small"),
        # the same chip between two looks
        _chip("steps-256x128", 256, 128, 100, geometry="small"),
        # the full-resolution chip of the paper's layout (1 um per cell), held valve state
        _chip("steps-1024x768", 1024, 768, 100),
        # the same chip run by a driver that records mass, compound and outlet fluxes of
        # every step
        _chip("monitor-1024x768", 1024, 768, 50, kind="monitor"),
        # a ragged porous layout: odd sizes, random obstacles, Zou-He and pressure ports on
        # both sides, another valve word every seven steps
        _chip("obstacles-1001x517", 1001, 517, 40, geometry="obstacles"),
        # the paper's own boundary conditions: equilibrium walls, rescaling pressure ports,
        # a decaying compound
        _chip("paper-1024x512", 1024, 512, 50, paper_ports=True, walls=True, decay=1e-4),
        # the largest chip, the throughput workload of the benchmark, in each storage type
        _chip("steps-4096x2048", 4096, 2048, 50),
        _chip("steps-4096x2048-fp16", 4096, 2048, 50, precision="fp16"),
        _chip("steps-4096x2048-bf16", 4096, 2048, 50, precision="bf16"),
        # the paper's workflow: stationary stored flow, the compound advanced alone
        _chip("scalar-4096x2048", 4096, 2048, 50, kind="scalar"),
        # screening many designs at once
        _chip("batch-64", 1024, 512, 20, kind="batch", chips=64, valves="toggle"),
        # gradient of a chamber objective with respect to tau_c, inlet speeds and inlet
        # concentrations: forward sweep, recomputation, reverse sweep
        _chip("gradient-1024x512", 1024, 512, 150, kind="gradient", ckpt=50),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: sizes over the logarithm of the range, odd ones among them."""
    kind = rng.choice(("steps", "steps", "steps", "steps", "monitor", "scalar", "batch", "gradient"))
    if kind == "batch":
        return _chip(None, 1024, 512, rng.randint(5, 20), kind="batch", chips=rng.randint(3, 63), valves="toggle")
    if kind == "gradient":
        nx = _log_int(rng, 150, 1024)
        return _chip(None, nx, max(48, int(nx * rng.uniform(0.4, 0.8))), rng.randint(20, 150), kind="gradient",
                     ckpt=rng.choice((1, 10, 25, 60)))
    nx = _log_int(rng, 150, 4000)
    ny = min(2047, max(40, int(nx * rng.uniform(0.4, 0.9))))
    n = rng.randint(1, 50)
    if kind == "scalar":
        return _chip(None, nx, ny, n, kind="scalar", paper_ports=rng.random() < 0.3,
                     decay=rng.choice((0.0, 0.0, 2e-4)), u_scale=rng.choice((1.0, 0.5)))
    if kind == "monitor":
        return _chip(None, nx, ny, n, kind="monitor", precision=rng.choice(PRECISIONS))
    if rng.random() < 0.25:
        return _chip(None, min(nx, 1500), min(ny, 900), n, geometry="obstacles", precision=rng.choice(PRECISIONS),
                     paper_ports=rng.random() < 0.3)
    paper = rng.random() < 0.25
    return _chip(None, nx, ny, n, geometry="small" if nx < 600 and not paper else "chip",
                 precision=rng.choice(PRECISIONS),
                 valves=rng.choice(("held", "toggle")), paper_ports=paper, walls=paper and rng.random() < 0.5,
                 decay=rng.choice((0.0, 0.0, 1e-4)))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _problem(case, seed):
    """The problem description (mask, ports, inlet values, valve words) and, for the
    obstacle layouts, their initial fields."""
    nx, ny = case["nx"], case["ny"]
    if case["geometry"] == "obstacles":
        p, init = W.random_case(seed, nx, ny, solid_frac=0.03, paper_ports=case["paper_ports"], decay=case["decay"])
        # a slow seepage flow (a porous layout holds back a fast one), outlets open in both words
        return dict(p, tau=0.8, tau_c=0.6, states=[7, 5], period=7, edge_u=0.1 * p["edge_u"]), init
    if case["geometry"] == "small":
        w = max(4, ny // 8)
        p = W.two_channel_chip(nx, ny, w, nx, max(8, nx // 4), 0.8, 0.55, 0.05, 500, 2000,
                               paper_ports=case["paper_ports"], decay=case["decay"])
    else:
        w = max(6, int(round(ny * 267 / 2048)))
        p = W.two_channel_chip(nx, ny, w, int(round(nx * 4000 / 4096)), max(8, int(round(nx * 800 / 4096))), 0.6, 0.51,
                               0.04, 2000, 50000, paper_ports=case["paper_ports"], decay=case["decay"])
    if case["walls"]:
        p["wall_scheme"] = lbm.LBM_WALL_EQUILIBRIUM
    if case["valves"] == "held":
        p["states"] = [1]
    return p, None


def _flow_fields(p, seed):
    """Fields near the developed flow of a two-channel chip, float32 (ny, nx): parabolic
    channel flow in the open channel, a weak one in the other, smooth seeded disturbances,
    and a compound front part of the way along the channels."""
    r = np.random.Generator(np.random.PCG64(seed))
    ny, nx = p["solid"].shape
    dev = "cuda"
    y = torch.arange(ny, device=dev, dtype=torch.float64)[:, None]
    x = torch.arange(nx, device=dev, dtype=torch.float64)[None, :]

    def wave(amplitude):
        out = 0.0
        for _ in range(3):
            a, b, c, d = r.uniform(-1, 1), r.integers(1, 6), r.integers(1, 6), r.uniform(0, 2 * np.pi)
            out = out + a * torch.sin(2 * np.pi * float(b) * x / nx + d) * torch.cos(2 * np.pi * float(c) * y / ny + a)
        return amplitude * out

    ux = torch.zeros((ny, nx), device=dev, dtype=torch.float64)
    for port in p["ports"]:
        if port["side"] != W.WEST:
            continue
        h = port["y1"] - port["y0"]
        s = torch.arange(h, device=dev, dtype=torch.float64)[:, None] + 0.5
        u = p["u_max"] * (r.uniform(0.8, 1.0) if (p["states"][0] >> port["channel"]) & 1 else r.uniform(0.0, 0.05))
        ux[port["y0"]:port["y1"], port["x"]:] = u * 4 * s * (h - s) / h ** 2
    front = nx * r.uniform(0.3, 0.7)
    c = 0.5 + 0.45 * torch.tanh((front - x) / (0.05 * nx)) * torch.cos(np.pi * (1 - y / ny)) + wave(0.01)
    fluid = torch.from_numpy((np.asarray(p["solid"]) == 0)).to(dev)
    fields = (1.0 + wave(1e-3), ux + wave(1e-3), wave(1e-3), c.clamp(0.0, 1.0))
    return [torch.where(fluid, f, (1.0 if k == 0 else 0.0)).to(torch.float32).cpu().numpy()
            for k, f in enumerate(fields)]


def _stored_flow(p, word):
    """The stationary flow of a valve word: every open channel carries its parabola from end
    to end, the rest is still."""
    ux = np.zeros(p["solid"].shape, np.float32)
    for port in p["ports"]:
        if port["side"] == W.WEST and (word >> port["channel"]) & 1:
            h = port["y1"] - port["y0"]
            east = next(q for q in p["ports"] if q["channel"] == port["channel"] and q["side"] == W.EAST)
            s = np.arange(h)[:, None] + 0.5
            ux[port["y0"]:port["y1"], port["x"]:east["x"] + 1] = p["u_max"] * 4 * s * (h - s) / h ** 2
    return ux, np.zeros_like(ux)


def _objective(p, seed):
    """The chamber's centre column against a linear profile, and the open channel four
    nodes from its inlet against a full one."""
    x0, x1, y0, y1 = p["chamber"]
    inlet = next(q for q in p["ports"] if q["side"] == W.WEST and (p["states"][0] >> q["channel"]) & 1)
    chamber, channel = np.arange(y0, y1), np.arange(inlet["y0"], inlet["y1"])
    oy = np.concatenate([chamber, channel])
    ox = np.concatenate([np.full(len(chamber), (x0 + x1) // 2), np.full(len(channel), inlet["x"] + 4)])
    target = np.concatenate([(chamber - y0) / max(1, y1 - y0 - 1), np.ones(len(channel))]).astype(np.float32)
    weight = np.random.Generator(np.random.PCG64(seed)).uniform(0.5, 1.5, len(oy)).astype(np.float32)
    return ox, oy, target, weight


def _batch_problems(case):
    probs = W.config_batch(case["chips"], seed=W.SEED + case["chips"])
    return probs


def _inputs(case, seed):
    """(problem or problems, initial fields as float32 arrays)."""
    if case["kind"] == "batch":
        probs = _batch_problems(case)
        nx = max(p["nx"] for p in probs)
        parts = [[], [], [], []]
        for k, p in enumerate(probs):
            f = _flow_fields(p, seed * 1000 + k)
            for q in range(4):
                rest = 1.0 if q == 0 else 0.0
                a = np.full((p["ny"] + (1 if k else 0), nx), rest, np.float32)  # one solid row between chips
                a[-p["ny"]:, :p["nx"]] = f[q]
                parts[q].append(a)
        return probs, [np.concatenate(a) for a in parts]
    p, init = _problem(case, seed)
    if init is not None:
        return p, [np.asarray(init[k], np.float32) for k in ("rho", "ux", "uy", "C")]
    if case["kind"] == "gradient":
        rows = np.flatnonzero(p["edge_C"][W.WEST] == 1.0)
        p["edge_C"][W.WEST, rows] = np.random.Generator(np.random.PCG64(seed)).uniform(0.8, 1.0, len(rows))
    return p, _flow_fields(p, seed)


def prepare(case, seed):
    prob, init = _inputs(case, seed)
    kw = dict(precision=case["precision"])
    if case["kind"] == "batch":
        chip = lbm.Chip.batch(prob, **kw)
        for k, p in enumerate(prob):
            chip.set_instance_schedule(k, p["period"], p["states"])
    else:
        chip = lbm.Chip.from_problem(prob, **kw)
        if len(prob["states"]) == 1:
            chip.set_valves(prob["states"][0])
        else:
            chip.set_valve_schedule(prob["period"], prob["states"])
    chip.init_equilibrium(*init)
    shape = (chip.ny, chip.nx)
    state = dict(case=case, chip=chip, C=torch.empty(shape, device="cuda"))
    if case["kind"] not in ("scalar", "gradient"):
        for k in ("rho", "ux", "uy"):
            state[k] = torch.empty(shape, device="cuda")
    if case["kind"] == "monitor":
        state["totals"] = torch.empty((case["n"], 4), device="cuda", dtype=torch.float64)
    if case["kind"] == "scalar":  # the stored stationary flow of each valve word
        for word in sorted(set(prob["states"])):
            chip.set_velocity_field(word, *_stored_flow(prob, word))
    if case["kind"] == "gradient":
        state["objective"] = _objective(prob, seed)
    return state


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    case, chip = state["case"], state["chip"]
    kind, n = case["kind"], case["n"]
    if kind == "gradient":
        ox, oy, target, weight = state["objective"]
        J, dtau, du, dc = chip.adjoint(n, ox, oy, target, weight, ckpt_every=case["ckpt"])
        chip.fields_device(C=state["C"])
        return dict(J=J, dtau_c=dtau, du_in=du, dC_in=dc, C=state["C"])
    if kind == "scalar":
        chip.scalar_step(n, case["u_scale"])
        chip.fields_device(C=state["C"])
        return dict(C=state["C"])
    if kind == "monitor":
        chip.step_diagnostics(n, state["totals"].data_ptr())
    else:
        chip.step(n)
    chip.fields_device(state["rho"], state["ux"], state["uy"], state["C"])
    out = {k: state[k] for k in ("rho", "ux", "uy", "C")}
    if kind == "monitor":
        out["totals"] = state["totals"]
    return out


def _fluid_nodes(case):
    if case["kind"] == "batch":
        probs = _batch_problems(case)
        nx = max(p["nx"] for p in probs)
        return sum(W.fluid_count(p) for p in probs), nx * (sum(p["ny"] for p in probs) + len(probs) - 1)
    p, _ = _problem(case, 1)
    return W.fluid_count(p), case["nx"] * case["ny"]


def work(case):
    """The state read once and written once (its neighbour masks too), the outputs written
    once; arithmetic per node and step: about 250 FP32 operations for the coupled step (60
    for the scalar alone, three coupled steps' worth for a gradient)."""
    fluid, cells = _fluid_nodes(case)
    elem = 4 if case["precision"] == "fp32" else 2
    kind, n = case["kind"], case["n"]
    planes, outputs, ops = (5, 1, 60) if kind == "scalar" else (14, 1, 750) if kind == "gradient" else (14, 4, 250)
    stored = 2 if kind == "scalar" else 0
    return {"bytes": fluid * (2 * planes * elem + stored * 4 + 1) + cells * outputs * 4, "flops": fluid * n * ops}


# ---------------------------------------------------------------------------
# the same steps in 64 bits, with plain torch operations
# ---------------------------------------------------------------------------
EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
WF = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4


def _moved(a, i):
    """a(x - e_i), wrapping at the edges (wrapped values are never used)."""
    return torch.roll(a, (EY[i], EX[i]), (-2, -1)) if i else a


def _feq(i, rho, ux, uy):
    eu = EX[i] * ux + EY[i] * uy
    return WF[i] * rho * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * (ux * ux + uy * uy))


class _Exact:
    def __init__(self, fluid, ports, edge_u, edge_c, omega_f, omega_g, w0, decay, walls):
        self.fluid, self.ports, self.edge_u, self.edge_c = fluid, ports, edge_u, edge_c
        self.omega_f, self.omega_g, self.decay, self.walls = omega_f, omega_g, decay, walls
        self.wg = (w0,) + ((1 - w0) / 4,) * 4
        self.cs2 = (1 - w0) / 2
        padded = torch.zeros((fluid.shape[0] + 2, fluid.shape[1] + 2), dtype=torch.bool, device=fluid.device)
        padded[1:-1, 1:-1] = fluid
        ny, nx = fluid.shape
        self.wall = [~padded[1 - EY[i]:1 - EY[i] + ny, 1 - EX[i]:1 - EX[i] + nx] for i in range(9)]

    def geq(self, i, c, ux, uy):
        return self.wg[i] * c * (1 + (EX[i] * ux + EY[i] * uy) / self.cs2)

    def start(self, rho, ux, uy, c):
        f = torch.stack([_feq(i, rho, ux, uy) for i in range(9)])
        g = torch.stack([self.geq(i, c, ux, uy) - self.wg[i] * self.decay * c for i in range(5)])
        return f, g

    @staticmethod
    def moments(f):
        rho = f.sum(0)
        jx = f[1] - f[3] + f[5] - f[6] + f[8] - f[7]
        jy = f[2] - f[4] + f[5] + f[6] - f[7] - f[8]
        return rho, jx, jy

    def wall_value(self, i, f):
        """The paper's wall: density extrapolated along e_i, a third of the next node's
        momentum."""
        rho, jx, jy = self.moments(f)
        o = OPP[i]
        r1, x1, y1 = (_moved(a, o) for a in (rho, jx, jy))        # at x + e_i
        r2 = _moved(r1, o)                                         # at x + 2 e_i
        no1, no2 = self.wall[o], _moved(self.wall[o], o)
        r = torch.where(no1, rho, torch.where(no2, r1, 2 * r1 - r2))
        r = torch.where(self.fluid, r, 1.0)
        jx, jy = torch.where(no1, 0.0, x1 / 3), torch.where(no1, 0.0, y1 / 3)
        return _feq(i, r, jx / r, jy / r)

    def pulled(self, f, g):
        F = [f[0]]
        for i in range(1, 9):
            F.append(torch.where(self.wall[i], self.wall_value(i, f) if self.walls else f[OPP[i]], _moved(f[i], i)))
        G = [g[0]] + [torch.where(self.wall[i], g[OPP[i]], _moved(g[i], i)) for i in range(1, 5)]
        return torch.stack(F), torch.stack(G)

    def complete(self, F, G, f, g, word, velocity=None):
        """Open ports, in place on F and G (F None: the scalar alone, with the stored flow)."""
        flux = []
        for port in self.ports:
            if not (word >> port["channel"]) & 1:
                continue
            west, kind = port["side"] == W.WEST, port["kind"]
            at = (slice(port["y0"], port["y1"]), port["x"])
            s = 1.0 if west else -1.0
            rows = slice(port["y0"], port["y1"])
            ia, iu, idn, oa, odn, oup = (1, 5, 8, 3, 7, 6) if west else (3, 6, 7, 1, 8, 5)
            cin = self.edge_c[port["side"], rows]
            ux = uy = None
            if F is not None:
                if kind in (W.VELOCITY, W.PRESSURE):
                    k = F[0][at] + F[2][at] + F[4][at] + 2 * (F[oa][at] + F[odn][at] + F[oup][at])
                    if kind == W.VELOCITY:
                        u = self.edge_u[port["side"], rows]
                        jx = k * u / (1 - s * u)
                    else:
                        jx = s * (port["rho"] - k)
                    half = 0.5 * (F[2][at] - F[4][at])
                    a, b, c = F[oa][at] + s * 2 / 3 * jx, F[odn][at] - half + s / 6 * jx, F[oup][at] + half + s / 6 * jx
                    F[(ia,) + at], F[(iu,) + at], F[(idn,) + at] = a, b, c
                else:
                    for i in (ia, iu, idn):
                        F[(i,) + at] = f[i][at]
                    gamma = port["rho"] / F[(slice(None),) + at].sum(0)
                    F[(slice(None),) + at] = F[(slice(None),) + at] * gamma
                rho, jx, jy = self.moments(F[(slice(None),) + at])
                ux, uy = jx / rho, jy / rho
            else:
                ux, uy = velocity[0][at], velocity[1][at]
            if kind == W.VELOCITY:
                G[(ia,) + at] = cin - (G[(slice(None),) + at].sum(0) - G[ia][at])
                continue
            G[(ia,) + at] = g[ia][at]
            if kind == W.INLET_RESCALE:
                total = G[(slice(None),) + at].sum(0)
                scaled = G[(slice(None),) + at] * (cin / torch.where(total > 0, total, 1.0))
                fresh = torch.stack([self.geq(i, cin, ux, uy) for i in range(5)])
                G[(slice(None),) + at] = torch.where(total > 0, scaled, fresh)
            else:
                flux.append((at, ux))
        return flux

    def collide_scalar(self, G, ux, uy):
        c = G.sum(0)
        out = [G[i] + self.omega_g * (self.geq(i, c, ux, uy) - G[i]) - self.wg[i] * self.decay * c for i in range(5)]
        return torch.stack(out), c

    def step(self, f, g, word, totals=None):
        F, G = self.pulled(f, g)
        flux = self.complete(F, G, f, g, word)
        rho, jx, jy = self.moments(F)
        rho = torch.where(self.fluid, rho, 1.0)
        ux, uy = torch.where(self.fluid, jx / rho, 0.0), torch.where(self.fluid, jy / rho, 0.0)
        f = torch.stack([F[i] + self.omega_f * (_feq(i, rho, ux, uy) - F[i]) for i in range(9)])
        g, c = self.collide_scalar(G, ux, uy)
        if totals is not None:
            q = sum(((jx[at]).sum() for at, _ in flux), torch.zeros((), device=f.device, dtype=f.dtype))
            qc = sum(((c[at] * ux[at]).sum() for at, _ in flux), torch.zeros((), device=f.device, dtype=f.dtype))
            totals.append(torch.stack([rho[self.fluid].sum(), c[self.fluid].sum(), q, qc]))
        return f, g

    def scalar_step(self, g, word, ux, uy):
        G = torch.stack([g[0]] + [torch.where(self.wall[i], g[OPP[i]], _moved(g[i], i)) for i in range(1, 5)])
        self.complete(None, G, None, g, word, velocity=(ux, uy))
        return self.collide_scalar(G, ux, uy)[0]

    def fields(self, f, g):
        rho, jx, jy = self.moments(f)
        zero = torch.zeros_like(rho)
        keep = lambda a: torch.where(self.fluid, a, zero)  # noqa: E731
        return dict(rho=keep(rho), ux=keep(jx / rho), uy=keep(jy / rho), C=keep(g.sum(0) / (1 - self.decay)))


def _t64(a):
    return torch.from_numpy(np.array(a, np.float64)).cuda()


def _exact_batch(case, seed):
    probs, init = _inputs(case, seed)
    ny, nx = init[0].shape
    fluid = torch.zeros((ny, nx), dtype=torch.bool, device="cuda")
    edge_u, edge_c = np.zeros((2, ny)), np.zeros((2, ny))
    tau, tau_c = np.ones((ny, 1)), np.ones((ny, 1))
    ports, row0 = [], 0
    for k, p in enumerate(probs):
        rows = slice(row0, row0 + p["ny"])
        fluid[rows, :p["nx"]] = torch.from_numpy(np.asarray(p["solid"]) == 0).cuda()
        edge_u[:, rows], edge_c[:, rows] = np.float32(p["edge_u"]), np.float32(p["edge_C"])
        tau[rows], tau_c[rows] = p["tau"], p["tau_c"]
        ports.append([dict(q, y0=q["y0"] + row0, y1=q["y1"] + row0) for q in p["ports"]])
        row0 += p["ny"] + 1
    e = _Exact(fluid, [], _t64(edge_u), _t64(edge_c), 1 / _t64(tau), 1 / _t64(tau_c), probs[0]["w0"], 0.0, False)
    f, g = e.start(*(_t64(a) for a in init))
    for t in range(case["n"]):
        e.ports = [dict(q, channel=0) for p, qs in zip(probs, ports) for q in qs
                   if (W.valve_word(p, t) >> q["channel"]) & 1]
        f, g = e.step(f, g, 1)
    return e.fields(f, g)


def exact(case, seed):
    if case["kind"] == "batch":
        return _exact_batch(case, seed)
    p, init = _inputs(case, seed)
    n = case["n"]
    gradient = case["kind"] == "gradient"
    omega_g = 1 / torch.tensor(p["tau_c"], dtype=torch.float64, device="cuda")
    edge_u, edge_c = _t64(np.float32(p["edge_u"])), _t64(np.float32(p["edge_C"]))
    e = _Exact(torch.from_numpy(np.asarray(p["solid"]) == 0).cuda(), p["ports"], edge_u, edge_c, 1 / p["tau"], omega_g,
               p["w0"], p.get("decay", 0.0), bool(p.get("wall_scheme", 0)))
    word = [W.valve_word(p, t) for t in range(n)]
    if case["kind"] == "scalar":
        f, g = e.start(*(_t64(a) for a in init))
        flow = {w: [_t64(a) for a in _stored_flow(p, w)] for w in set(word)}
        s = float(np.float32(case["u_scale"]))
        for t in range(n):
            ux, uy = flow[word[t]]
            g = e.scalar_step(g, word[t], s * ux, s * uy)
        return dict(C=e.fields(f, g)["C"])
    f, g = e.start(*(_t64(a) for a in init))
    if not gradient:
        totals = [] if case["kind"] == "monitor" else None
        for t in range(n):
            f, g = e.step(f, g, word[t], totals)
        out = e.fields(f, g)
        if totals is not None:
            out["totals"] = torch.stack(totals)
        return out
    # the gradient by autograd, a few steps recomputed at a time
    from torch.utils.checkpoint import checkpoint
    omega_g.requires_grad_(True)
    edge_u.requires_grad_(True)
    edge_c.requires_grad_(True)
    ox, oy, target, weight = _objective(p, seed)

    def some(f, g, wg, eu, ec, t0, t1):
        e.omega_g, e.edge_u, e.edge_c = wg, eu, ec
        for t in range(t0, t1):
            f, g = e.step(f, g, word[t])
        return f, g

    for t in range(0, n, 8):
        f, g = checkpoint(some, f, g, omega_g, edge_u, edge_c, t, min(n, t + 8), use_reentrant=False)
    c = g.sum(0)[torch.from_numpy(oy).cuda(), torch.from_numpy(ox).cuda()]
    J = (_t64(weight) * (c - _t64(target)) ** 2).sum()
    dw, du, dc = torch.autograd.grad(J, (omega_g, edge_u, edge_c))
    return dict(J=float(J), dtau_c=float(-dw / p["tau_c"] ** 2), du_in=du.cpu().numpy(), dC_in=dc.cpu().numpy(),
                C=e.fields(f.detach(), g.detach())["C"])
