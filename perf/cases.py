"""Performance cases of the library's public entry points.

Each case is one call of a user's program: a lattice (or a batch of them)
that has been set up, ``steps`` iterations (``Lattice.iteration`` /
``Batch.iteration``, which ends with a thermo record unless the program asks
for records less often), and the state read from the caller-owned buffers.
Sizes and parameters are those of the repository's workloads (the paper's
channel, the porous medium, the Shan-Chen ring, the reactive channel, the
batch of uneven lattices) and ragged or smaller relatives of them; geometry
and initial fields come from the seed.  ``exact`` is a plain torch FP64
restatement of the method, independent of the package.
"""
import numpy as np
import torch

from paper_1202_0442_gb300 import lb2d, synth

NEVER = 1 << 30  # thermo interval of a program that asks for no records

EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
W = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
EX4, EY4 = (1, 0, -1, 0), (0, 1, 0, -1)
OPP4 = (2, 3, 0, 1)

DTYPE = {"fp32": torch.float32, "fp16": torch.float16, "bf16": torch.bfloat16}
POROSITY = 0.7
H_MAX = 2e-3  # bound on |f - w rho_ref| the FP16 runs are set up with


def listed():
    return [
        # the paper's first example: a small channel, a hundred iterations
        # between two thermo records; latency and launches are all of it
        {"name": "channel_64x32", "kind": "flow", "geometry": "channel", "nx": 64, "ny": 32, "steps": 100,
         "storage": "fp32", "precise": False, "velocity": False, "records": True},
        # the same script on the paper's 61 x 31 nodes, one iteration per
        # call with exact momentum pairs: the smallest call there is
        {"name": "channel_61x31_step", "kind": "flow", "geometry": "channel", "nx": 61, "ny": 31, "steps": 1,
         "storage": "fp32", "precise": True, "velocity": False, "records": False},
        # the headline lattice as a run executes it: an output interval of a
        # hundred iterations, then density and velocity to page-locked memory
        {"name": "porous_1024", "kind": "flow", "geometry": "porous", "nx": 1024, "ny": 1024, "steps": 100,
         "storage": "fp32", "precise": False, "velocity": True, "records": True},
        # the same lattice stepped by a driver that looks at every state
        {"name": "porous_1024_step", "kind": "flow", "geometry": "porous", "nx": 1024, "ny": 1024, "steps": 1,
         "storage": "fp32", "precise": False, "velocity": False, "records": False},
        # the profiling lattice, far beyond L2
        {"name": "porous_4096", "kind": "flow", "geometry": "porous", "nx": 4096, "ny": 4096, "steps": 20,
         "storage": "fp32", "precise": False, "velocity": False, "records": True},
        # 16-bit storage with stochastic rounding on odd sizes
        {"name": "porous_fp16_2003x1501", "kind": "flow", "geometry": "porous", "nx": 2003, "ny": 1501, "steps": 50,
         "storage": "fp16", "precise": False, "velocity": False, "records": True},
        # two components with interforce and adhesion (the Shan-Chen ring)
        {"name": "shan_chen_2048", "kind": "two", "nx": 2048, "ny": 2048, "steps": 10},
        # one component separating into vapour and liquid, odd sizes
        {"name": "vapour_777x500", "kind": "vapour", "nx": 777, "ny": 500, "steps": 10},
        # solute, surface reaction and growth: the paper's application
        {"name": "reactive_1024x512_q9", "kind": "reactive", "nx": 1024, "ny": 512, "q": 9, "steps": 200},
        # the paper's D2Q4 solute on a small ragged channel
        {"name": "reactive_333x190_q4", "kind": "reactive", "nx": 333, "ny": 190, "q": 4, "steps": 200},
        # 256 uneven lattices in one launch per iteration, as the benchmark
        # runs them (exact momentum pairs)
        {"name": "batch_256", "kind": "batch", "count": 256, "steps": 40, "storage": "fp32"},
        # a small sweep of lattices in 16-bit storage
        {"name": "batch_24_fp16", "kind": "batch", "count": 24, "steps": 40, "storage": "fp16"},
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["flow", "flow", "flow", "two", "vapour", "reactive", "batch"])
    if kind == "batch":
        return {"kind": kind, "count": _log(rng, 4, 256), "steps": rng.choice([20, 30, 40]),
                "storage": rng.choice(["fp32", "fp16", "bf16"])}
    if kind == "two":
        nx, ny = _log(rng, 64, 2048), _log(rng, 64, 2048)
        return {"kind": kind, "nx": nx, "ny": ny, "steps": rng.randint(1, 10)}
    if kind == "vapour":
        return {"kind": kind, "nx": _log(rng, 64, 1024), "ny": _log(rng, 64, 1024), "steps": rng.randint(1, 10)}
    if kind == "reactive":
        return {"kind": kind, "nx": _log(rng, 100, 1024), "ny": _log(rng, 70, 768), "q": rng.choice([4, 9]),
                "steps": _log(rng, 1, 200)}
    geometry = rng.choice(["channel", "porous", "porous"])
    nx = _log(rng, 24, 512) if geometry == "channel" else _log(rng, 64, 4096)
    ny = _log(rng, 12, 512) if geometry == "channel" else _log(rng, 64, 4096)
    steps = max(1, min(_log(rng, 1, 100), 20 * 4096 * 4096 // (nx * ny)))
    storage = rng.choice(["fp32", "fp32", "fp16", "bf16"])
    return {"kind": kind, "geometry": geometry, "nx": nx, "ny": ny, "steps": steps, "storage": storage,
            "precise": storage == "fp32" and rng.random() < 0.25, "velocity": rng.random() < 0.25,
            "records": rng.random() < 0.75}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------


def _device():
    return torch.device("cuda", 0) if torch.cuda.is_available() else torch.device("cpu")


def _discs(nx, ny, seed, cell, rmin, rmax, gap, x0, y0, share=1.0):
    """uint8 [ny][nx]: one disc of radius rmin..rmax per cell x cell square
    of the lattice inside x0 <= x < nx - x0, y0 <= y < ny - y0 (a share of
    the cells), jittered so that two discs stay ``gap`` nodes apart."""
    dev = _device()
    rng = np.random.default_rng(seed)
    mx, my = (nx - 2 * x0) // cell, (ny - 2 * y0) // cell
    m = torch.zeros((ny, nx), dtype=torch.uint8, device=dev)
    if mx < 1 or my < 1:
        return m.cpu().numpy()
    r = rng.integers(rmin, rmax + 1, (my, mx))
    room = np.maximum(cell // 2 - r - (gap + 1) // 2, 0)
    cx = cell // 2 + np.rint(room * rng.uniform(-1, 1, (my, mx))).astype(np.int64)
    cy = cell // 2 + np.rint(room * rng.uniform(-1, 1, (my, mx))).astype(np.int64)
    r = np.where(rng.random((my, mx)) < share, r, -1)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a).astype(np.int32)).to(dev)
    gx, gy, gr = t(cx), t(cy), t(r)
    k = torch.arange(cell, device=dev, dtype=torch.int32)
    dx2 = (k.view(1, 1, -1) - gx.unsqueeze(2)) ** 2            # [my, mx, cell]
    dy2 = (k.view(1, 1, -1) - gy.unsqueeze(2)) ** 2
    r2 = torch.where(gr < 0, -1, gr * gr)
    inside = (dy2.permute(0, 2, 1).unsqueeze(3) + dx2.unsqueeze(1)) <= r2.view(my, 1, mx, 1)
    m[y0:y0 + my * cell, x0:x0 + mx * cell] = inside.reshape(my * cell, mx * cell).to(torch.uint8)
    return m.cpu().numpy()


def _waves(nx, ny, rng, amplitude):
    """A smooth velocity field: a few periodic waves with random phases."""
    x, y = np.arange(nx) * (2 * np.pi / nx), np.arange(ny) * (2 * np.pi / ny)
    u = np.zeros((ny, nx))
    v = np.zeros((ny, nx))
    for k in (1, 2):
        a, b, c, d = rng.uniform(0, 2 * np.pi, 4)
        u += np.outer(np.sin(k * y + a), np.cos(k * x + b))
        v += np.outer(np.cos(k * y + c), np.sin(k * x + d))
    return amplitude / 2 * u, amplitude / 2 * v


def _flow(case, seed):
    nx, ny = case["nx"], case["ny"]
    rng = np.random.default_rng([seed, 11])
    if case["geometry"] == "channel":
        solid = np.zeros((ny, nx), np.uint8)
        solid[0, :] = solid[-1, :] = 1
        rho, ops, force, ref, tau = np.ones((ny, nx)), [], ((1e-6, 0.0),), 1.0, 1.0
    else:
        cell = min(54, max(10, min(nx, ny) // 3))
        big = cell * 24 // 54
        solid = _discs(nx, ny, [seed, 1], cell, max(1, big // 3), big, 2, 4, 0)
        rho = np.broadcast_to(np.linspace(1.001, 1.0, nx), (ny, nx))
        ops = [synth.Opening("xlo", 0, ny - 1, "inlet", [("dirichlet", 0.0, 1.001)]),
               synth.Opening("xhi", 0, ny - 1, "outlet", [("dirichlet", 0.0, 1.0)])]
        force, ref, tau = ((0.0, 0.0),), 1.0005, 0.8
    ux, uy = _waves(nx, ny, rng, 1e-3)
    return synth.Workload(name="flow", nx=nx, ny=ny, solid=solid, rho=[np.where(solid, 0.0, rho)], ux=ux, uy=uy,
                          tau=(tau,), aveforce=force, openings=ops, rho_ref=(ref,))


def _two(case, seed):
    nx, ny = case["nx"], case["ny"]
    rng = np.random.default_rng([seed, 12])
    n = min(nx, ny)
    s = n / 2048.0
    ri = int(round(600 * s))
    ro = max(int(round(604 * s)), ri + 2)
    y, x = np.mgrid[0:ny, 0:nx]
    d2 = (x - nx // 2) ** 2 + (y - ny // 2) ** 2
    solid = ((d2 >= ri * ri) & (d2 < ro * ro)).astype(np.uint8)
    ddx, ddy = (x - nx // 10 + nx // 2) % nx - nx // 2, (y - ny // 10 + ny // 2) % ny - ny // 2
    one = (d2 < ri * ri) | (ddx * ddx + ddy * ddy <= max(int(round(100 * s)), 3) ** 2)
    noise = lambda: 1.0 + rng.uniform(-0.01, 0.01, (ny, nx))
    rho = [np.where(solid, 0.0, np.where(one, 1.0, 0.03) * noise()),
           np.where(solid, 0.0, np.where(one, 0.03, 1.0) * noise())]
    return synth.Workload(name="two", nx=nx, ny=ny, solid=solid, rho=rho, tau=(1.0, 1.0), alpha=(4 / 9, 4 / 9),
                          aveforce=((0.0, 0.0),) * 2, aveacceleration=((0.0, 0.0),) * 2,
                          interforce=(0.9, 0.0, 0.0), adhesive=((0.3, 0.0, 0.0), (-0.3, 0.0, 0.0)),
                          rho_ref=(0.515, 0.515))


def _vapour(case, seed):
    nx, ny = case["nx"], case["ny"]
    rng = np.random.default_rng([seed, 13])
    return synth.Workload(name="vapour", nx=nx, ny=ny, solid=np.zeros((ny, nx), np.uint8),
                          rho=[200.0 + rng.uniform(0.0, 1.0, (ny, nx))], tau=(1.0,),
                          interforce=(-120.0, 4.0, 200.0), rho_ref=(200.0,))


REACTION = (1e-4, 0.0, 0.0, 1.0, 7)  # k_r, C_s, b0, b_max, growth seed


def _reactive(case, seed):
    """The reactive channel: pressure driven, solute entering with C = 1,
    deposits part of the way to b_max as in a run under way (so that surface
    nodes grow during the call)."""
    nx, ny, q = case["nx"], case["ny"], case["q"]
    rng = np.random.default_rng([seed, 14])
    cell = min(58, max(20, min(nx, ny) // 3))
    big = cell * 24 // 58
    solid = _discs(nx, ny, [seed, 2], cell, max(2, big // 3), big, 4, 5, 5, 0.4)
    solid[0, :] = solid[-1, :] = 1
    rho = np.broadcast_to(np.linspace(1.005, 1.0, nx), (ny, nx))
    ux, uy = _waves(nx, ny, rng, 1e-3)
    C = 1.0 - 0.5 * np.outer(np.ones(ny), np.linspace(0, 1, nx)) + 20 * ux
    ops = [synth.Opening("xlo", 1, ny - 2, "inlet", [("dirichlet", 0.0, 1.005)], solute=("dirichlet", 1.0)),
           synth.Opening("xhi", 1, ny - 2, "outlet", [("dirichlet", 0.0, 1.0)], solute=("adiabatic", 1.0))]
    w = synth.Workload(name="reactive", nx=nx, ny=ny, solid=solid, rho=[np.where(solid, 0.0, rho)], ux=ux, uy=uy,
                       tau=(0.9,), openings=ops, solute_q=q, taus=0.7, C=np.where(solid, 0.0, C),
                       reaction=REACTION, rho_ref=(1.0,))
    return w, np.where(solid, rng.random((ny, nx)), 0.0)


def _batch(case, seed):
    out = []
    for k in range(case["count"]):
        rng = np.random.default_rng([seed, 15, k])
        # sides of lattice k, whatever the seed
        nx, ny = (int(s) for s in np.random.default_rng([15, k]).choice(np.arange(64, 513, 32), 2))
        cell = 32
        # discs of this radius range cover 10 to 60 % of their cells
        cover = float(rng.uniform(0.1, 0.6))
        r = int(round(cell * (cover / np.pi) ** 0.5))
        y, x = np.mgrid[0:ny, 0:nx]
        cx, cy = rng.integers(10, 22, (2, ny // cell, nx // cell))
        rr = rng.integers(max(3, r - 2), r + 3, (ny // cell, nx // cell))
        solid = ((x % cell - cx[y // cell, x // cell]) ** 2 + (y % cell - cy[y // cell, x // cell]) ** 2
                 <= rr[y // cell, x // cell] ** 2).astype(np.uint8)
        ux, uy = _waves(nx, ny, rng, 1e-3)
        out.append(synth.Workload(name="batch", nx=nx, ny=ny, solid=solid, rho=[np.where(solid, 0.0, 1.0)],
                                  ux=ux, uy=uy, tau=(float(rng.uniform(0.6, 1.5)),), aveforce=((1e-6, 0.0),),
                                  rho_ref=(1.0,)))
    return out


def _pitch(nx):
    return (nx + 31) // 32 * 32


def _buffers(w, storage):
    """f0/f1 (and g0/g1) as the program's own tensors, in the documented
    [component][9][ny][pitch] layout."""
    dev = _device()
    shape = (w.ncomp, 9, w.ny, _pitch(w.nx))
    bind = {k: torch.zeros(shape, dtype=DTYPE[storage], device=dev) for k in ("f0", "f1")}
    if w.solute_q:
        for k in ("g0", "g1"):
            bind[k] = torch.zeros((w.solute_q,) + shape[2:], dtype=torch.float32, device=dev)
    return bind


def _options(storage, precise):
    return {"precise": precise} if storage == "fp32" else {"h_max": H_MAX, "rounding": "stochastic"}


def prepare(case, seed):
    kind, steps = case["kind"], case["steps"]
    if kind == "batch":
        ws = _batch(case, seed)
        dev = _device()
        at, total = [], 0
        for w in ws:
            at.append(total)
            total += -(-9 * w.ny * _pitch(w.nx) // 128) * 128  # 256-byte aligned
        f = [torch.zeros(total, dtype=DTYPE[case["storage"]], device=dev) for _ in range(2)]
        lats = []
        for w, a in zip(ws, at):
            n = 9 * w.ny * _pitch(w.nx)
            lats.append(lb2d.from_workload(w, case["storage"], bind={"f0": f[0][a:a + n], "f1": f[1][a:a + n]},
                                           thermo=NEVER, **_options(case["storage"], True)))
        batch = lb2d.Batch(lats)
        batch.autotune(None)
        return {"kind": kind, "steps": steps, "batch": batch, "first": lats[0], "f": f}
    b0 = None
    storage, precise, thermo = "fp32", False, 0
    if kind == "flow":
        w = _flow(case, seed)
        storage, precise = case["storage"], case["precise"]
        thermo = 0 if case["records"] else NEVER
    elif kind == "two":
        w = _two(case, seed)
    elif kind == "vapour":
        w = _vapour(case, seed)
    else:
        w, b0 = _reactive(case, seed)
    bind = _buffers(w, storage)
    lt = lb2d.from_workload(w, storage, bind=bind, thermo=thermo, **_options(storage, precise))
    if b0 is not None:
        lt.set_precipitate(b0)
    state = {"kind": kind, "steps": steps, "lt": lt, "bind": bind, "nx": w.nx}
    if case.get("velocity"):
        lt.output(steps)
        pin = torch.cuda.is_available()
        state["out"] = tuple(torch.zeros((w.ny, w.nx), pin_memory=pin) for _ in range(3))
    return state


def run(state):
    if state["kind"] == "batch":
        state["batch"].iteration(state["steps"])
        return {"f": state["f"][state["first"].current_buffer()]}
    lt, nx = state["lt"], state["nx"]
    lt.iteration(state["steps"])
    k = str(lt.current_buffer())
    out = {"f": state["bind"]["f" + k][..., :nx]}
    if "out" in state:
        out["rho"], out["ux"], out["uy"] = lt.velocity_f32(state["out"])
    if state["kind"] == "reactive":
        out["g"] = state["bind"]["g" + k][..., :nx]
        # the deposits grow by FP32 shares: the program keeps them as FP32
        out["b"] = lt.solute_state(g=False, Cf=False, b=True)[2].astype(np.float32)
        out["grown"] = lt.get_thermo()["flips"]
    return out


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------


def work(case):
    """Every population of every fluid node in once and out once (and the
    other outputs once); per fluid node and iteration some 110 operations for
    a component's moments, equilibrium and relaxation, 60 more for the
    interforce sums, 10 per solute mode."""
    kind, steps = case["kind"], case["steps"]
    if kind == "batch":
        nodes = case["count"] * 288 * 288 * 0.65
        size = 4 if case["storage"] == "fp32" else 2
        return {"bytes": 18 * size * nodes, "flops": 110 * nodes * steps}
    nodes = case["nx"] * case["ny"]
    if kind == "two":
        return {"bytes": 2 * 72 * nodes, "flops": 2 * 170 * nodes * steps}
    if kind == "vapour":
        return {"bytes": 72 * nodes, "flops": 170 * nodes * steps}
    if kind == "reactive":
        fluid, q = 0.9 * nodes, case["q"]
        return {"bytes": (72 + 8 * q) * fluid + 16 * (nodes - fluid), "flops": (110 + 10 * q) * fluid * steps}
    fluid = nodes * (POROSITY if case["geometry"] == "porous" else 1.0 - 2.0 / case["ny"])
    size = 4 if case["storage"] == "fp32" else 2
    return {"bytes": 18 * size * fluid + (12 * nodes if case["velocity"] else 0), "flops": 110 * fluid * steps}


# ---------------------------------------------------------------------------
# the method in 64 bits
# ---------------------------------------------------------------------------


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(_device())


def _roll(a, ex, ey):
    return torch.roll(a, (ey, ex), (0, 1)) if ex or ey else a


def _feq(rho, ux, uy):
    usq = 1.5 * (ux * ux + uy * uy)
    out = []
    for i in range(9):
        eu = EX[i] * ux + EY[i] * uy
        out.append(W[i] * rho * (1.0 + 3.0 * eu + 4.5 * eu * eu - usq))
    return out


class _Exact:
    def __init__(self, w):
        self.w = w
        self.solid = _t(w.solid != 0)
        self.sources()
        zero = torch.zeros((w.ny, w.nx), dtype=torch.float64, device=_device())
        self.u0 = [zero if a is None else _t(a) for a in (w.ux, w.uy)]
        self.f = []
        for rho in w.rho:
            fe = _feq(_t(np.asarray(rho, np.float64)), *self.u0)
            self.f.append([torch.where(self.solid, 0.0, x) for x in fe])
        self.force = None

    def sources(self):
        self.src = [_roll(self.solid, EX[i], EY[i]) for i in range(9)]

    def stream(self, f):
        return [f[0]] + [torch.where(self.src[i], f[OPP[i]], _roll(f[i], EX[i], EY[i])) for i in range(1, 9)]

    def openings(self, f, rho_in, rho_out, rows):
        c = [a[rows, 0] for a in f]
        a = rho_in - (c[0] + c[2] + c[4] + 2 * (c[3] + c[6] + c[7]))
        d = 0.5 * (c[2] - c[4])
        f1, f5, f8 = c[3] + 2 / 3 * a, c[7] - d + a / 6, c[6] + d + a / 6
        f[1][rows, 0], f[5][rows, 0], f[8][rows, 0] = f1, f5, f8
        c = [a[rows, -1] for a in f]
        a = (c[0] + c[2] + c[4] + 2 * (c[1] + c[5] + c[8])) - rho_out
        d = 0.5 * (c[4] - c[2])
        f3, f6, f7 = c[1] - 2 / 3 * a, c[8] + d - a / 6, c[5] - d - a / 6
        f[3][rows, -1], f[6][rows, -1], f[7][rows, -1] = f3, f6, f7

    def step(self):
        w = self.w
        fs, rho, jx, jy = [], [], [], []
        for f in self.f:
            f = self.stream(f)
            if w.openings:
                a, b = w.openings
                f = [x.clone() for x in f]
                self.openings(f, a.momentum[0][2], b.momentum[0][2], slice(a.a0, a.a1 + 1))
            fs.append(f)
            rho.append(sum(f[1:], f[0]))
            jx.append(f[1] - f[3] + f[5] - f[7] + f[8] - f[6])
            jy.append(f[2] - f[4] + f[5] - f[7] + f[6] - f[8])
        n = w.ncomp
        F = []
        for c in range(n):
            fx, fy = w.aveforce[c]
            F.append([fx, fy])
        if w.interforce is not None:
            G, psi0, rho0 = w.interforce
            psi = [torch.where(self.solid, 0.0, r if n == 2 else psi0 * torch.exp(-rho0 / r)) for r in rho]
            for c in range(n):
                p = psi[1 - c] if n == 2 else psi[0]
                for k, E in enumerate((EX, EY)):
                    s = sum(W[i] * E[i] * _roll(p, -EX[i], -EY[i]) for i in range(1, 9) if E[i])
                    F[c][k] = F[c][k] - G * psi[c] * s
        for c in range(n):
            if c < len(w.adhesive) and w.adhesive[c] is not None:
                s = self.solid.to(torch.float64)
                for k, E in enumerate((EX, EY)):
                    t = sum(W[i] * E[i] * _roll(s, -EX[i], -EY[i]) for i in range(1, 9) if E[i])
                    F[c][k] = F[c][k] - w.adhesive[c][0] * rho[c] * t
        tau = w.tau
        if n == 2:
            den = rho[0] / tau[0] + rho[1] / tau[1]
            up = [(j[0] / tau[0] + j[1] / tau[1]) / den for j in (jx, jy)]
            ueq = [[up[k] + tau[c] * F[c][k] / rho[c] for k in (0, 1)] for c in range(2)]
        else:
            ueq = [[(j[0] + tau[0] * F[0][k]) / rho[0] for k, j in enumerate((jx, jy))]]
        for c in range(n):
            fe = _feq(rho[c], *ueq[c])
            self.f[c] = [torch.where(self.solid, 0.0, a - (a - e) / tau[c]) for a, e in zip(fs[c], fe)]
        self.rho = torch.where(self.solid, 0.0, sum(rho[1:], rho[0]))
        self.u = [torch.where(self.solid, 0.0, sum(j[c] + 0.5 * F[c][k] for c in range(n)) / sum(rho[1:], rho[0]))
                  for k, j in enumerate((jx, jy))]

    def populations(self, scale=1.0):
        out = []
        for c, f in enumerate(self.f):
            ref = float(np.float32(self.w.rho_ref[c]))
            out.append(torch.stack([torch.where(self.solid, 0.0, (f[i] - W[i] * ref) * scale) for i in range(9)]))
        return torch.stack(out)


class _ExactReactive(_Exact):
    def __init__(self, w, b):
        super().__init__(w)
        self.q = w.solute_q
        self.ex, self.ey, self.opp, self.wt = (EX4, EY4, OPP4, (0.25,) * 4) if self.q == 4 else (EX, EY, OPP, W)
        self.g = [torch.where(self.solid, 0.0, a) for a in self.geq(_t(w.C), *self.u0)]
        self.b, self.t, self.kept = _t(b), 0, []

    def geq(self, C, ux, uy):
        k = 2.0 if self.q == 4 else 3.0
        return [self.wt[i] * C * (1.0 + k * (self.ex[i] * ux + self.ey[i] * uy)) for i in range(self.q)]

    def step(self):
        super().step()
        self.t += 1
        w, q = self.w, self.q
        before = self.g
        kr, Cs, b0, bmax, seed = w.reaction
        rows = slice(w.openings[0].a0, w.openings[0].a1 + 1)
        opening = torch.zeros_like(self.solid)
        opening[rows, 0] = opening[rows, -1] = True
        gt, links = [], []
        Cw = torch.zeros_like(self.b)
        nU = torch.zeros_like(self.b)
        for i in range(q):
            ex, ey, o = self.ex[i], self.ey[i], self.opp[i]
            cross = torch.zeros_like(self.solid)
            if ex > 0:
                cross[rows, 0] = True
            if ex < 0:
                cross[rows, -1] = True
            link = _roll(self.solid, ex, ey) & ~cross & ~self.solid
            if ex == 0 and ey == 0:
                link = torch.zeros_like(link)
            Ci = (2.0 * self.g[o] + kr * Cs) / (kr + 2.0 * self.wt[i])
            v = torch.where(link, -self.g[o] + 2.0 * self.wt[i] * Ci, _roll(self.g[i], ex, ey))
            gt.append(torch.where(cross | self.solid, 0.0, v))
            Cw = Cw + torch.where(link, Ci, 0.0)
            nU = nU + link
            links.append(link)
        into = [i for i in range(q) if self.ex[i] > 0]
        C1 = w.openings[0].solute[1]
        ws = sum(self.wt[i] for i in into)
        rest = sum(gt[i][rows, 0] for i in range(q) if i not in into)
        for i in into:
            gt[i][rows, 0] = torch.where(self.solid[rows, 0], 0.0, (C1 - rest) * self.wt[i] / ws)
        for i in range(q):
            if self.ex[i] < 0:
                gt[i][rows, -1] = gt[self.opp[i]][rows, -1]
        C = sum(gt[1:], gt[0])
        geq = self.geq(C, *self.u)
        g = [a - (a - e) / w.taus for a, e in zip(gt, geq)]
        some = nU > 0
        n1 = torch.where(some, nU, 1.0)
        dB = kr * (Cw / n1 - Cs)
        share = torch.where(some & (dB > 0), dB / n1, 0.0)
        self.g = [torch.where(self.solid, 0.0, g[i] - torch.where(links[i], share, 0.0)) for i in range(q)]
        # the solid node behind link i of fluid node x is x - e_i
        for i in range(q):
            self.b = self.b + _roll(torch.where(links[i], share, 0.0), -self.ex[i], -self.ey[i])
        hot = torch.nonzero(self.solid & (self.b > bmax)).cpu().tolist()
        if not hot:
            return
        free = (~self.solid & ~opening).cpu().numpy()
        flips = set()
        for y, x in hot:
            near = [((y + EY4[d]) % w.ny, (x + EX4[d]) % w.nx) for d in range(4)]
            near = [p for p in near if free[p]]
            if near:
                flips.add(near[_splitmix64(seed ^ (self.t * w.nx * w.ny + y * w.nx + x)) % len(near)])
                self.b[y, x] = 0.0
        for y, x in flips:
            # a node that grows solid is left as it is in both g buffers
            self.kept.append((y, x, self.t, [a[y, x].clone() for a in self.g], [a[y, x].clone() for a in before]))
            self.solid[y, x] = True
            self.b[y, x] = b0
            for a in self.f[0] + self.g:
                a[y, x] = 0.0
        self.sources()

    def solute(self):
        """The current g buffer."""
        g = torch.stack(self.g)
        for y, x, t, new, old in self.kept:
            g[:, y, x] = torch.stack(new if (self.t - t) % 2 == 0 else old)
        return g


def _splitmix64(x):
    m = (1 << 64) - 1
    z = (x + 0x9E3779B97F4A7C15) & m
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & m
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & m
    return z ^ (z >> 31)


def _scale(storage):
    return 2.0 ** int(np.floor(np.log2(16384.0 / H_MAX))) if storage == "fp16" else 1.0


def exact(case, seed):
    kind, steps = case["kind"], case["steps"]
    if kind == "batch":
        parts = []
        for w in _batch(case, seed):
            e = _Exact(w)
            for _ in range(steps):
                e.step()
            v = e.populations(_scale(case["storage"])).reshape(-1)
            parts.append(torch.nn.functional.pad(v, (0, -(-v.numel() // 128) * 128 - v.numel())))
        return {"f": torch.cat(parts)}
    if kind == "reactive":
        w, b = _reactive(case, seed)
        e = _ExactReactive(w, b)
    else:
        w = {"flow": _flow, "two": _two, "vapour": _vapour}[kind](case, seed)
        e = _Exact(w)
    for _ in range(steps):
        e.step()
    out = {"f": e.populations(_scale(case.get("storage", "fp32")))}
    if case.get("velocity"):
        out["rho"], out["ux"], out["uy"] = e.rho, e.u[0], e.u[1]
    if kind == "reactive":
        out["g"], out["b"], out["grown"] = e.solute(), e.b, None
    return out
