"""Workloads of the regularized Particles-on-Demand library, each through its public calls.

A pass of a flow case is what a program does with a solver that it keeps: it sets primitive
fields that lie on the device, advances a number of steps and reads the conserved fields
back into its own device arrays.  The library hands fields over as doubles; a program that
runs FP32 populations keeps them as float32, so such a pass returns float32 fields.

``exact`` advances the same fields in FP64 with plain torch operations on populations, as the
paper states the scheme (arXiv 2203.05477, Sec. II.C, III.A and III.B).
"""
import itertools
import math

import numpy as np
import torch

import paper_2203_05477_gb300 as pond
from paper_2203_05477_gb300 import inputs

TAU = 1e-5
TRANSMISSIVE, PERIODIC, INFLOW = inputs.TRANSMISSIVE, inputs.PERIODIC, inputs.INFLOW


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # One short tube advanced a few steps, as inside a coupling or parameter loop: the time
        # is launches and latency.
        dict(name="tube_200_fp32", kind="tube", flow="riemann", precision="fp32", nx=200, steps=4, cfl=0.2),
        # The paper's shock-tube runs (400 cells, CFL 0.5, FP64): long, small and serial.
        dict(name="tube_400_fp64", kind="tube", flow="riemann", precision="fp64", nx=400, steps=256, cfl=0.5),
        # A 1D grid far larger than the caches (the size of the scheme comparison in bench.py).
        dict(name="tube_4m_fp32", kind="tube", flow="smooth", precision="fp32", nx=1 << 22, steps=16, cfl=0.3),
        # A parameter study: thousands of tubes of uneven length in one persistent launch.
        dict(name="batch_4096_fp32", kind="batch", precision="fp32", tubes=4096, len_min=200, len_max=8000,
             steps=100, cfl=0.2),
        # The headline benchmark: four-quadrant Riemann problem, FP32 populations.
        dict(name="quadrants_1024_fp32", kind="grid2", flow="quadrants", precision="fp32", nx=1024, ny=1024, steps=40,
             cfl=0.2, limiter="vanleer"),
        # The same problem in FP64 at the size of a convergence study.
        dict(name="quadrants_256_fp64", kind="grid2", flow="quadrants", precision="fp64", nx=256, ny=256, steps=8,
             cfl=0.2, limiter="vanleer"),
        # A shock hitting a perturbed interface: inflow and periodic sides, odd sizes, minmod.
        dict(name="interface_1001x253_fp32", kind="grid2", flow="interface", precision="fp32", nx=1001, ny=253, steps=24,
             cfl=0.2, limiter="minmod"),
        # The interface with the learned face-gauge predictor switched on.
        dict(name="interface_learned_fp32", kind="learned2", flow="interface", precision="fp32", nx=1024, ny=256,
             steps=24, cfl=0.2, limiter="vanleer"),
        # The semi-Lagrangian realization on a smooth periodic field.
        dict(name="sl_500_fp32", kind="sl2", flow="smooth", precision="fp32", nx=500, ny=500, steps=8, cfl=0.2),
        # Three dimensions: an explosion in a box, FP32, and a smaller FP64 one of odd sizes.
        dict(name="blast_64_fp32", kind="grid3", flow="blast", precision="fp32", nx=64, ny=64, nz=64, steps=8, cfl=0.3),
        dict(name="blast_25_fp64", kind="grid3", flow="blast", precision="fp64", nx=25, ny=23, nz=21, steps=4, cfl=0.3),
        # One gradient evaluation of the predictor network (training: forward and backward).
        dict(name="gradient_64k", kind="gradient", rows=65536),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["tube", "tube", "batch", "grid2", "grid2", "grid2", "learned2", "sl2", "grid3", "gradient"])
    precision = rng.choice(["fp32", "fp32", "fp64"])
    if kind == "tube":
        nx = log_int(100, 4_000_000 if precision == "fp32" else 200_000)
        steps = max(2, min(log_int(4, 300), 60_000_000 // nx if precision == "fp32" else 2_000_000 // nx))
        return dict(kind=kind, flow=rng.choice(["riemann", "smooth"]), precision=precision, nx=nx, steps=steps,
                    cfl=rng.choice([0.2, 0.3, 0.5]))
    if kind == "batch":
        tubes = log_int(8, 4096 if precision == "fp32" else 256)
        lo = log_int(100, 400)
        return dict(kind=kind, precision=precision, tubes=tubes, len_min=lo, len_max=lo * rng.randint(2, 20),
                    steps=rng.randint(10, 60 if precision == "fp32" else 20), cfl=0.2)
    if kind == "grid2":
        nx, ny = (log_int(24, 1024), log_int(24, 1024)) if precision == "fp32" else (log_int(24, 300), log_int(24, 200))
        flow = rng.choice(["quadrants", "interface"])
        return dict(kind=kind, flow=flow, precision=precision, nx=nx, ny=ny, steps=rng.randint(2, 32 if precision == "fp32" else 8),
                    cfl=0.2, limiter=rng.choice(["vanleer", "vanleer", "minmod"]))
    if kind == "learned2":
        return dict(kind=kind, flow="interface", precision="fp32", nx=log_int(64, 1024), ny=log_int(32, 300),
                    steps=rng.randint(4, 24), cfl=0.2, limiter="vanleer")
    if kind == "sl2":
        n = 600 if precision == "fp32" else 100
        return dict(kind=kind, flow="smooth", precision=precision, nx=log_int(24, n), ny=log_int(24, n),
                    steps=rng.randint(2, 8), cfl=0.2)
    if kind == "grid3":
        n = 64 if precision == "fp32" else 24
        return dict(kind=kind, flow=rng.choice(["blast", "smooth"]), precision=precision, nx=log_int(8, n),
                    ny=log_int(8, n), nz=log_int(8, n), steps=rng.randint(2, 8 if precision == "fp32" else 4), cfl=0.3)
    return dict(kind="gradient", rows=log_int(100, 65536))


# ------------------------------------------------------------------ inputs

def _axis(n, length=1.0, device="cpu"):
    return (torch.arange(n, dtype=torch.float64, device=device) + 0.5) * (length / n)


def _device():
    return torch.device("cuda") if torch.cuda.is_available() else torch.device("cpu")


def _pick(mask, a, b):
    two = torch.tensor([b, a], dtype=torch.float64, device=mask.device)
    return two[mask.long()]


def _smooth(rng, coords):
    """1 + a few random Fourier modes of the unit box, of relative amplitude 0.15 together."""
    f = 0.0
    for _ in range(3):
        phase = rng.uniform(0.0, 2.0 * math.pi)
        for c in coords:
            phase = phase + 2.0 * math.pi * int(rng.integers(0, 3)) * c
        f = f + rng.uniform(-0.05, 0.05) * torch.sin(phase + 2.0 * math.pi * coords[0])
    return 1.0 + f


def _flow(case, seed):
    """Grid and primitive fields [rho, u..., p] (x fastest, on the device) of a flow case."""
    rng = np.random.default_rng(seed)
    dev = _device()
    kind = case["kind"]
    if kind == "batch":
        # the lengths belong to the case, the states to the seed
        spread = np.random.default_rng(case["tubes"]).uniform(math.log(case["len_min"]), math.log(case["len_max"]), case["tubes"])
        lengths = np.rint(np.exp(spread)).astype(np.int64)
        gammas = np.where(rng.integers(0, 2, case["tubes"]) == 0, 1.4, 5.0 / 3.0)
        # two states a tube: densities and pressures within a factor of ten, colliding at up to
        # Mach 1.5 or receding: every tube stays physical and takes all its steps
        state = np.empty((case["tubes"], 2, 3))
        state[:, :, 0] = np.exp(rng.uniform(-1.15, 1.15, (case["tubes"], 2)))
        state[:, :, 2] = np.exp(rng.uniform(-1.15, 1.15, (case["tubes"], 2)))
        jump = rng.uniform(-0.5, 1.5, case["tubes"]) * np.sqrt(gammas * np.minimum(state[:, 0, 2] / state[:, 0, 0], state[:, 1, 2] / state[:, 1, 0]))
        state[:, 0, 1], state[:, 1, 1] = 0.5 * jump, -0.5 * jump
        ln = torch.from_numpy(lengths).to(dev)
        tube = torch.repeat_interleave(torch.arange(case["tubes"], device=dev), ln)
        first = torch.cumsum(ln, 0) - ln
        right = (2 * (torch.arange(tube.numel(), device=dev) - first[tube]) + 1 > ln[tube]).long()
        q = torch.from_numpy(state).to(dev)[tube, right]
        return dict(dim=1, lengths=lengths, gammas=gammas, tube=tube, first=first), [q[:, k].contiguous() for k in range(3)]
    dim = {"tube": 1, "grid2": 2, "learned2": 2, "sl2": 2, "grid3": 3}[kind]
    n = [case["nx"], case.get("ny", 1), case.get("nz", 1)][:dim]
    gamma, flow = 1.4, case["flow"]
    size = [4.0, 1.0] if flow == "interface" else [1.0] * dim
    bc, inflow = [TRANSMISSIVE] * (2 * dim), None
    axes = [_axis(n[a], size[a], dev) for a in range(dim)]
    coords = torch.meshgrid(*axes[::-1], indexing="ij")[::-1]   # x fastest
    if flow == "smooth":
        bc = [PERIODIC] * (2 * dim)
        mean = rng.uniform(-1.0, 1.0, dim)
        q = [_smooth(rng, coords)] + [float(mean[a]) + (_smooth(rng, coords) - 1.0) for a in range(dim)] + [_smooth(rng, coords)]
    elif flow == "riemann":
        # two states with densities and pressures up to a factor of ten apart
        rho, p = np.exp(rng.uniform(-1.15, 1.15, 2)), np.exp(rng.uniform(-1.15, 1.15, 2))
        u = rng.uniform(-0.5, 0.5, 2)
        left = coords[0] < 0.5
        q = [_pick(left, a, b) for a, b in (rho, u, p)]
    elif flow == "quadrants":
        # each quadrant: rho and p within a factor of ten, up to Mach 2 towards the centre
        rho, p = np.exp(rng.uniform(-1.15, 1.15, (2, 4)))
        speed = rng.uniform(0.0, 2.0, 4) * np.sqrt(gamma * p / rho)
        cx, cy = np.array([0.25, 0.75, 0.25, 0.75]), np.array([0.25, 0.25, 0.75, 0.75])
        th = np.arctan2(0.5 - cy, 0.5 - cx) + rng.uniform(-math.pi / 4, math.pi / 4, 4)
        state = torch.from_numpy(np.stack([rho, speed * np.cos(th), speed * np.sin(th), p], 1)).to(dev)
        which = (coords[0] > 0.5).long() + 2 * (coords[1] > 0.5).long()
        q = [state[:, k][which] for k in range(4)]
    elif flow == "interface":
        # a planar shock of Mach 1.5-2.2 moves towards a wavy interface to a heavier gas, all of it
        # drifting along the interface
        mach, atwood, modes, drift = rng.uniform(1.5, 2.2), rng.uniform(0.5, 0.7), int(rng.integers(2, 9)), rng.uniform(0.2, 0.5)
        p2 = (2.0 * gamma * mach * mach - (gamma - 1.0)) / (gamma + 1.0)
        rho2 = (gamma + 1.0) * mach * mach / ((gamma - 1.0) * mach * mach + 2.0)
        u2 = mach * math.sqrt(gamma) * (1.0 - 1.0 / rho2)
        post = coords[0] < 0.5
        heavy = coords[0] >= 1.0 + 0.05 * torch.sin(2.0 * math.pi * modes * coords[1])
        rho = torch.where(post, rho2, _pick(heavy, (1.0 + atwood) / (1.0 - atwood), 1.0))
        q = [rho, _pick(post, u2, 0.0), torch.full_like(rho, drift), _pick(post, p2, 1.0)]
        bc, inflow = [INFLOW, TRANSMISSIVE, PERIODIC, PERIODIC], [rho2, u2, drift, p2]
    else:   # "blast": a sphere of hot dense gas off the centre of the box
        centre = rng.uniform(0.4, 0.6, 3)
        inside = sum((coords[a] - float(centre[a])) ** 2 for a in range(3)) < float(rng.uniform(0.15, 0.3)) ** 2
        zero = torch.zeros_like(coords[0])
        q = [_pick(inside, 1.0, 0.125), zero + 0.3, zero - 0.2, zero + 0.1, _pick(inside, rng.uniform(0.8, 1.5), 0.1)]
    q = [f.reshape(-1).contiguous() for f in q]
    return dict(dim=dim, n=n, size=size, gamma=gamma, bc=bc, inflow=inflow), q


def _solver(case, grid):
    limiter = pond.POND_MINMOD if case.get("limiter") == "minmod" else pond.POND_VANLEER
    opts = dict(tau=TAU, cfl=case["cfl"], precision=case["precision"], limiter=limiter)
    if case["kind"] == "batch":
        return pond.BatchSolver(grid["lengths"], grid["gammas"], **opts)
    n, size = grid["n"], grid["size"]
    if grid["dim"] == 3:
        return pond.Solver3(inputs.Problem3(*n, 0.0, size[0], 0.0, size[1], 0.0, size[2], grid["gamma"], None, None, None, None,
                                            None, bc=tuple(grid["bc"])), **opts)
    ny, ly = (n[1], size[1]) if grid["dim"] == 2 else (1, 1.0)
    pb = inputs.Problem(grid["dim"], n[0], ny, 0.0, size[0], 0.0, ly, grid["gamma"], None, None, None, None,
                        bc=tuple(grid["bc"]) + (TRANSMISSIVE,) * (4 - len(grid["bc"])))
    if grid["inflow"]:
        pb.inflow[0] = grid["inflow"]
        pb.inflow_range[0] = (0, ny)
    return pond.Solver(pb, scheme="sl" if case["kind"] == "sl2" else "fv", **opts)


def _train(seed):
    """Parameters of the face-gauge predictor, trained on pairs of a small run of the same flow."""
    grid, q = _flow(dict(kind="grid2", flow="interface", nx=128, ny=32), seed + 1)
    s = _solver(dict(kind="grid2", cfl=0.2, precision="fp32"), grid)
    s.set_primitive(q[0], q[1], q[2], q[3])
    pairs = s.gauge_collect(32, cap=100_000, every=2)
    s.gauge_train(pairs, epochs=4, batch=4096, lr=2e-3)
    params = s.gauge_params()
    s.close()
    return params


def _network(case, seed):
    g = torch.Generator().manual_seed(seed)
    n = case["rows"]
    params = torch.cat([torch.randn(64 * 48, generator=g) * math.sqrt(2 / 48), torch.zeros(64),
                        torch.randn(64 * 64, generator=g) * math.sqrt(2 / 64), torch.zeros(64),
                        torch.randn(16 * 64, generator=g) * 0.1, torch.zeros(16)])
    x = torch.randn(n, pond.MLP_PAIR_STRIDE, generator=g)
    return params.to(_device()), x.to(_device())


def prepare(case, seed):
    if case["kind"] == "gradient":
        params, x = _network(case, seed)
        return dict(case=case, params=params, x=x)
    grid, q = _flow(case, seed)
    s = _solver(case, grid)
    if case["kind"] == "learned2":
        s.set_gauge_params(_train(seed))
        s.gauge_enable(True)
    outs = [torch.empty_like(f) for f in q]
    if grid["dim"] == 1:
        outs.insert(2, None)
    return dict(case=case, solver=s, fields=q, outs=outs)


# ------------------------------------------------------------------ one pass

def run(state):
    case = state["case"]
    if case["kind"] == "gradient":
        loss, grad = pond.mlp_gradient(state["params"], state["x"], state["x"])
        return {"loss": loss, "grad": grad}
    s, q = state["solver"], state["fields"]
    if s.D == 1:
        s.set_primitive(q[0], q[1], None, q[2])
    else:
        s.set_primitive(*q)
    s.step(case["steps"])
    s.moments_device(state["outs"])
    outs = [f for f in state["outs"] if f is not None]
    return [f.float() for f in outs] if case["precision"] == "fp32" else outs


def work(case):
    """Bytes: the fields in and out.  FLOPs: a face's stencil cells moved into its frame once a
    step, its populations reconstructed and summed, and the cell updates."""
    if case["kind"] == "gradient":
        macs = 48 * 64 + 64 * 64 + 64 * 16
        return {"bytes": case["rows"] * 4 * 51 + 2 * 4 * pond.MLP_PARAMS, "flops": case["rows"] * 6 * macs}
    if case["kind"] == "batch":
        mean = (case["len_max"] - case["len_min"]) / math.log(case["len_max"] / case["len_min"])
        cells, dim = case["tubes"] * mean, 1
    else:
        cells = case["nx"] * case.get("ny", 1) * case.get("nz", 1)
        dim = {"tube": 1, "grid3": 3}.get(case["kind"], 2)
    per_cell = {1: 450 + 250, 2: 2 * 2900 + 900, 3: 3 * 14000 + 3200}[dim]
    if case["kind"] == "sl2":
        per_cell = 12000   # 25 stencil nodes moved into the node's frame, 16 populations interpolated twice
    return {"bytes": cells * 8 * 2 * (dim + 2), "flops": cells * case["steps"] * per_cell}


# ------------------------------------------------------------------ the scheme in FP64

C4 = [-math.sqrt(3 + math.sqrt(6)), -math.sqrt(3 - math.sqrt(6)), math.sqrt(3 - math.sqrt(6)), math.sqrt(3 + math.sqrt(6))]
W4 = [(3 - math.sqrt(6)) / 12, (3 + math.sqrt(6)) / 12, (3 + math.sqrt(6)) / 12, (3 - math.sqrt(6)) / 12]


def _he(k, c):
    return (1.0, c, c * c - 1.0, c * c * c - 3.0 * c)[k]


class _Set:
    """Populations of one kind (f: order 3, g: order 2) on the D-dimensional lattice: Hermite
    coefficients by multi-index, and the matrices from and to populations over weights."""

    def __init__(self, dim, top, dev):
        self.dim = dim
        self.orders = [k for k in itertools.product(range(top + 1), repeat=dim) if sum(k) <= top]
        self.at = {k: i for i, k in enumerate(self.orders)}
        nodes = list(itertools.product(range(4), repeat=dim))
        self.nodes = torch.tensor(nodes, device=dev).T                    # [dim, Q]
        vals = [[math.prod(_he(a, C4[m]) for a, m in zip(k, q)) for k in self.orders] for q in nodes]
        fact = [math.prod(math.factorial(a) for a in k) for k in self.orders]
        w = [math.prod(W4[m] for m in q) for q in nodes]
        vals = torch.tensor(vals, dtype=torch.float64, device=dev)
        self.expand = vals / torch.tensor(fact, dtype=torch.float64, device=dev)        # [Q, K]
        self.moments = (vals * torch.tensor(w, dtype=torch.float64, device=dev)[:, None]).T.contiguous()   # [K, Q]

    def move(self, coef, T, du, Tn):
        """Coefficients in the frame (u, T) re-expressed in one of temperature Tn whose velocity
        is u - du (the regularized transformation: moments up to the order kept)."""
        s, e, rs = torch.sqrt(T / Tn), (T - Tn) / Tn, 1.0 / torch.sqrt(Tn)
        v = dict(zip(self.orders, coef))
        for a in range(self.dim):
            d = du[a] * rs
            t = [[None], [d, s], [e + d * d, 2 * s * d, s * s], [d * (3 * e + d * d), 3 * s * (e + d * d), 3 * s * s * d, s * s * s]]
            out = {}
            for k in self.orders:
                r = k[a]
                acc = v[k] if r == 0 else 0.0
                for p in range(r + 1 if r else 0):
                    acc = acc + t[r][p] * v[k[:a] + (p,) + k[a + 1:]]
                out[k] = acc
            v = out
        return torch.stack([v[k] for k in self.orders])

    def times_c(self, coef, axis):
        """Coefficients of c_axis times the populations, orders kept."""
        out = torch.zeros_like(coef)
        for k, i in self.at.items():
            up, down = k[:axis] + (k[axis] + 1,) + k[axis + 1:], k[:axis] + (k[axis] - 1,) + k[axis + 1:]
            if up in self.at:
                out[i] += coef[self.at[up]]
            if k[axis] > 0:
                out[i] += k[axis] * coef[self.at[down]]
        return out


def _limiter(kind, a, b):
    ab = a * b
    if kind == "minmod":
        return torch.where(ab > 0, torch.where(a.abs() < b.abs(), a, b), torch.zeros_like(a))
    return torch.where(ab > 0, 2 * ab / torch.where(ab > 0, a + b, torch.ones_like(a)), torch.zeros_like(a))


class _Exact:
    def __init__(self, case, grid, q):
        self.case, self.dim, self.dev = case, grid["dim"], q[0].device
        D, dev = self.dim, self.dev
        self.f, self.g = _Set(D, 3, dev), _Set(D, 2, dev)
        self.first = [tuple(int(a == b) for b in range(D)) for a in range(D)]
        self.second = [tuple(2 * int(a == b) for b in range(D)) for a in range(D)]
        self.tol = 1e-10 if case["precision"] == "fp64" else 1e-6
        self.N = N = q[0].numel()
        self.inflow, self.around, self.group = grid.get("inflow"), None, None
        if case["kind"] == "batch":
            ln = torch.from_numpy(grid["lengths"]).to(dev)
            self.group, self.groups = grid["tube"], len(grid["lengths"])
            cv = torch.from_numpy(1.0 / (grid["gammas"] - 1.0)).to(dev)
            self.dx = [(1.0 / ln.double())[self.group]]
            self.Cv = cv[self.group]
            ftube = torch.repeat_interleave(torch.arange(self.groups, device=dev), ln + 1)
            lo, hi = grid["first"][ftube], (grid["first"] + ln - 1)[ftube]
            face = torch.arange(ftube.numel(), device=dev) - (grid["first"][ftube] + ftube)   # within its tube
            cell = lambda o: torch.minimum(torch.maximum(lo + face + o, lo), hi)
            self.stencil = [[cell(o) for o in (-2, -1, 0, 1)]]
            self.fgroup, self.fdx, self.fCv = [ftube], [[(1.0 / ln.double())[ftube]]], [cv[ftube]]
            below = torch.arange(N, device=dev) + self.group
            self.sides = [(below, below + 1)]
            return
        n, bc = grid["n"], grid["bc"]
        self.dx = [grid["size"][a] / n[a] for a in range(D)]
        self.Cv = 1.0 / (grid["gamma"] - 1.0)
        strides = [1, n[0], n[0] * (n[1] if D > 1 else 1)]

        def index(coords):
            """Flat indices of cells, ghosts resolved (y before x); N stands for the inflow state."""
            out, flow = 0, None
            for a in reversed(range(D)):
                c = coords[a]
                if bc[2 * a] == PERIODIC:
                    r = c % n[a]
                else:
                    r = c.clamp(0, n[a] - 1)
                if a == 0 and bc[0] == INFLOW:
                    flow = c < 0
                out = out + r * strides[a]
            return (out if flow is None else torch.where(flow, N, out)).reshape(-1)

        def mesh(sizes):
            ar = [torch.arange(k, device=dev) for k in sizes]
            return list(torch.meshgrid(*ar[::-1], indexing="ij")[::-1])

        if case["kind"] == "sl2":
            i, j = mesh(n)
            self.around = [[index([i + b, j + a]) for b in range(-2, 3)] for a in range(-2, 3)]
            return
        self.stencil, self.sides = [], []
        for a in range(D):
            sizes = [n[b] + (b == a) for b in range(D)]
            c = mesh(sizes)
            shift = lambda on, b=None, ob=0: index([c[k] + (on if k == a else 0) + (ob if k == b else 0) for k in range(D)])
            slots = [shift(o) for o in (-2, -1, 0, 1)]
            for b in range(D):
                if b != a:
                    slots += [shift(-1, b, -1), shift(-1, b, 1), shift(0, b, -1), shift(0, b, 1)]
            self.stencil.append(slots)
            fs, cc = [1, sizes[0], sizes[0] * (sizes[1] if D > 1 else 1)], mesh(n)
            below = sum(cc[k] * fs[k] for k in range(D)).reshape(-1)
            self.sides.append((below, below + fs[a]))

    # ---- state

    def start(self, q):
        D = self.dim
        rho, self.U, p = q[0], torch.stack(q[1:1 + D]), q[1 + D]
        self.T = p / rho
        self.F = torch.zeros(len(self.f.orders), self.N, dtype=torch.float64, device=self.dev)
        self.G = torch.zeros(len(self.g.orders), self.N, dtype=torch.float64, device=self.dev)
        self.F[0], self.G[0] = rho, (self.Cv - 0.5 * D) * rho * self.T
        self.faces = []
        if self.around is None:
            for a in range(D):
                F, _, U, T = self.with_inflow(self.F, self.G)
                l, r = self.stencil[a][1], self.stencil[a][2]
                Cv = self.fCv[a] if self.group is not None else self.Cv
                E = lambda c: F[0][c] * (Cv * T[c] + 0.5 * (U[:, c] ** 2).sum(0))
                rm, em = 0.5 * (F[0][l] + F[0][r]), 0.5 * (E(l) + E(r))
                m = 0.5 * (F[0][l] * U[:, l] + F[0][r] * U[:, r])
                self.faces.append((m / rm, (em - 0.5 * (m * m).sum(0) / rm) / (Cv * rm)))
        self.time_step()

    def time_step(self):
        c = torch.sqrt(self.T) * C4[3]
        rate = torch.stack([(self.U[a].abs() + c) / self.dx[a] for a in range(self.dim)]).amax(0)
        if self.group is None:
            self.dt = self.case["cfl"] / rate.max()
        else:
            top = torch.zeros(self.groups, dtype=torch.float64, device=self.dev)
            self.dt = self.case["cfl"] / top.scatter_reduce(0, self.group, rate, "amax")

    def with_inflow(self, F, G):
        """Cell arrays with the inflow state appended (index N)."""
        if not self.inflow:
            return F, G, self.U, self.T
        rho, T = self.inflow[0], self.inflow[-1] / self.inflow[0]
        f, g = torch.zeros_like(F[:, :1]), torch.zeros_like(G[:, :1])
        f[0], g[0] = rho, (self.Cv - 0.5 * self.dim) * rho * T
        u = torch.tensor(self.inflow[1:-1], dtype=torch.float64, device=self.dev)[:, None]
        return torch.cat([F, f], 1), torch.cat([G, g], 1), torch.cat([self.U, u], 1), torch.cat([self.T, torch.full_like(self.T[:1], T)])

    def frame_of(self, Phi, Psi, T, Cv):
        """Density, velocity relative to the frame and temperature of moments in a frame; ok."""
        D = self.dim
        rho = Phi[0]
        du = torch.stack([torch.sqrt(T) * Phi[self.f.at[k]] / rho for k in self.first])
        k2 = (du * du).sum(0)
        tr = sum(Phi[self.f.at[k]] for k in self.second) + D * rho
        Tn = (0.5 * T * tr + Psi[0] - 0.5 * rho * k2) / (Cv * rho)
        return rho, du, Tn, (Tn > 0) & torch.isfinite(Tn) & torch.isfinite(rho) & torch.isfinite(du).all(0)

    def iterate(self, one_pass, U, T, pooled, Cv):
        """The corrector of every face (or node) from the frame (U, T) to convergence: the last
        valid pass's moments and frame and the frame its moments define."""
        n = T.numel()
        act = torch.arange(n, device=self.dev)
        U, T = U.clone(), T.clone()
        keep = [None] * 7
        restarted = torch.zeros(n, dtype=torch.bool, device=self.dev)
        for it in range(16):
            cv = Cv[act] if torch.is_tensor(Cv) else Cv
            Phi, Psi = one_pass(act, U[:, act], T[act])
            rho, du, Tn, ok = self.frame_of(Phi, Psi, T[act], cv)
            new = (Phi, Psi, U[:, act], T[act], rho, du, Tn)
            if it == 0:
                keep = [x.clone() for x in new]
            else:
                for k, x in zip(keep, new):
                    k[..., act[ok]] = x[..., ok]
            done = ok & ((Tn - T[act]).abs() <= self.tol * T[act]) & (du.abs() <= self.tol * torch.sqrt(T[act])).all(0)
            Un, Tm = U[:, act] + du, Tn
            again = ~ok & ~restarted[act]
            if bool(again.any()):
                pu, pt = pooled(act[again])
                Un[:, again], Tm = pu, Tm.clone()
                Tm[again] = pt
                restarted[act[again]] = True
            U[:, act], T[act] = Un, Tm
            act = act[~done & (ok | again)]
            if not act.numel():
                break
        return keep

    def pooled(self, F, U, T, slots, Cv):
        def of(act):
            ix = [s[act] for s in slots]
            cv = Cv[act] if torch.is_tensor(Cv) else Cv
            r = sum(F[0][i] for i in ix) / len(ix)
            m = sum(F[0][i] * U[:, i] for i in ix) / len(ix)
            e = sum(F[0][i] * (cv * T[i] + 0.5 * (U[:, i] ** 2).sum(0)) for i in ix) / len(ix)
            return m / r, (e - 0.5 * (m * m).sum(0) / r) / (cv * r)
        return of

    # ---- the finite-volume step (Sec. III.B)

    def step_fv(self):
        D, case = self.dim, self.case
        tube = self.group is not None
        dt = self.dt[self.group] if tube else self.dt
        h = 0.5 * dt
        eqF, eqG = self.F[0], (self.Cv - 0.5 * D) * self.F[0] * self.T
        cp, ce = (2 * TAU - h) / (2 * TAU + dt), 3 * h / (2 * TAU + dt)
        ca, cb = (2 * TAU - dt) / (2 * TAU + dt), 2 * dt / (2 * TAU + dt)
        Fa, Ga, U, T = self.with_inflow(self.F, self.G)
        A, B = cp * self.F, cp * self.G
        A[0] += ce * eqF
        B[0] += ce * eqG
        A, B, U, T = self.with_inflow(A, B)
        if self.inflow:   # phi-bar-plus of an equilibrium
            A[:, -1], B[:, -1] = (cp + ce) * Fa[:, -1], (cp + ce) * Ga[:, -1]
        H, K = ca * self.F, ca * self.G
        H[0] += cb * eqF
        K[0] += cb * eqG
        for a in range(D):
            slots = self.stencil[a]
            fdt = self.dt[self.fgroup[a]] if tube else self.dt
            fh, Cv = 0.5 * fdt, self.fCv[a] if tube else self.Cv
            fdx = self.fdx[a] if tube else self.dx
            tang = [b for b in range(D) if b != a]

            def one_pass(act, u, Tl):
                at = lambda x: x[act] if torch.is_tensor(x) and x.dim() else x
                hh = [at(fh / fdx[b]) for b in range(D)]
                v = torch.sqrt(Tl) * torch.tensor(C4, dtype=torch.float64, device=self.dev)[:, None]   # [4, faces] per axis, about u
                left4 = v + u[a] > 0
                left, offn = left4[self.f.nodes[a]], (torch.where(left4, 0.5, -0.5) - (v + u[a]) * hh[a])[self.f.nodes[a]]
                offt = [(-(v + u[b]) * hh[b])[self.f.nodes[b]] for b in tang]
                got = []
                for s, X in ((self.f, A), (self.g, B)):
                    p = [s.expand @ s.move(X[:, i[act]], T[i[act]], U[:, i[act]] - u, Tl) for i in slots]
                    pick = lambda l, r: torch.where(left, p[l], p[r])
                    up = pick(1, 2)
                    b = up + offn * _limiter(case.get("limiter"), up - pick(0, 1), pick(2, 3) - up)
                    for t in range(D - 1):
                        b = b + offt[t] * _limiter(case.get("limiter"), up - pick(4 + 4 * t, 6 + 4 * t), pick(5 + 4 * t, 7 + 4 * t) - up)
                    got.append(s.moments @ b)
                return got

            Phi, Psi, u0, T0, rho, du, Tn = self.iterate(one_pass, *self.faces[a], self.pooled(A, U, T, slots, Cv), Cv)
            wb, we = 2 * TAU / (2 * TAU + fh), fh / (2 * TAU + fh)
            Fo, Go = wb * self.f.move(Phi, T0, -du, Tn), wb * self.g.move(Psi, T0, -du, Tn)
            Fo[0] += we * rho
            Go[0] += we * (Cv - 0.5 * D) * rho * Tn
            uf = u0 + du
            self.faces[a] = (uf, Tn)
            for side, sign in zip(self.sides[a], (-1.0, 1.0)):
                scale = sign * dt / self.dx[a]
                for s, X, Y in ((self.f, Fo, H), (self.g, Go, K)):
                    m = s.move(X[:, side], Tn[side], uf[:, side] - self.U, self.T)
                    Y -= scale * (self.U[a] * m + torch.sqrt(self.T) * s.times_c(m, a))
        # the new co-moving frame and the projection into it
        rho, du, Tn, _ = self.frame_of(H, K, self.T, self.Cv)
        self.F, self.G = self.f.move(H, self.T, -du, Tn), self.g.move(K, self.T, -du, Tn)
        for k in self.first:
            self.F[self.f.at[k]] = 0.0
        self.U, self.T = self.U + du, Tn
        self.time_step()

    # ---- the semi-Lagrangian step on D2Q16 (Sec. III.A)

    def step_sl(self):
        dt, near = self.dt, self.around
        F, G, U, T = self.F, self.G, self.U, self.T

        def one_pass(act, u, Tl):
            c4 = torch.tensor(C4, dtype=torch.float64, device=self.dev)[:, None]
            d = [((torch.sqrt(Tl) * c4 + u[a]) * dt / self.dx[a])[self.f.nodes[a]] for a in range(2)]
            fwd = [x > 0 for x in d]
            th = [torch.where(w, 1.0 - x, -x) for w, x in zip(fwd, d)]
            wt = [[-t * (t - 1) * (t - 2) / 6, (t + 1) * (t - 1) * (t - 2) / 2, -(t + 1) * t * (t - 2) / 2, (t + 1) * t * (t - 1) / 6]
                  for t in th]
            got = []
            for s, X in ((self.f, F), (self.g, G)):
                moved = lambda i: s.move(X[:, i[act]], T[i[act]], U[:, i[act]] - u, Tl)
                own = moved(near[2][2])
                P = [[s.expand @ (moved(i) - own) for i in row] for row in near]
                v = [[torch.where(fwd[1], torch.where(fwd[0], P[a][b], P[a][b + 1]), torch.where(fwd[0], P[a + 1][b], P[a + 1][b + 1]))
                      for b in range(4)] for a in range(4)]
                p = sum(wt[1][a] * wt[0][b] * v[a][b] for a in range(4) for b in range(4))
                mid = torch.stack([v[1][1], v[1][2], v[2][1], v[2][2]])
                flat = (1 - th[1]) * ((1 - th[0]) * mid[0] + th[0] * mid[1]) + th[1] * ((1 - th[0]) * mid[2] + th[0] * mid[3])
                p = torch.where((p < mid.amin(0)) | (p > mid.amax(0)), flat, p)
                got.append(own + s.moments @ p)
            return got

        flat = [i for row in near for i in row]
        Phi, Psi, u0, T0, rho, du, Tn = self.iterate(one_pass, U, T, self.pooled(F, U, T, flat, self.Cv), self.Cv)
        beta2 = 2 * dt / (2 * TAU + dt)
        self.F, self.G = (1 - beta2) * self.f.move(Phi, T0, -du, Tn), (1 - beta2) * self.g.move(Psi, T0, -du, Tn)
        self.F[0] += beta2 * rho
        self.G[0] += beta2 * (self.Cv - 1.0) * rho * Tn
        for k in self.first:
            self.F[self.f.at[k]] = 0.0
        self.U, self.T = u0 + du, Tn
        self.time_step()

    def fields(self):
        rho = self.F[0]
        return [rho, *(rho * self.U), rho * (self.Cv * self.T + 0.5 * (self.U ** 2).sum(0))]


def exact(case, seed):
    if case["kind"] == "gradient":
        params, x = _network(case, seed)
        p = params.double().requires_grad_()
        w1, b1, w2, b2, w3, b3 = torch.split(p, [64 * 48, 64, 64 * 64, 64, 16 * 64, 16])
        h = torch.relu(x[:, :48].double() @ w1.view(64, 48).T + b1)
        h = torch.relu(h @ w2.view(64, 64).T + b2)
        out = (h @ w3.view(16, 64).T + b3)[:, :3]
        loss = torch.mean((out - x[:, 48:51].double()) ** 2)
        loss.backward()
        return {"loss": float(loss), "grad": p.grad}
    grid, q = _flow(case, seed)
    e = _Exact(case, grid, q)
    e.start(q)
    for _ in range(case["steps"]):
        if case["kind"] == "sl2":
            e.step_sl()
        else:
            e.step_fv()
    return e.fields()
