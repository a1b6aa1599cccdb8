"""The work that users of this framework have it do, as cases to be timed.

Four kinds, each through the public binding (paper_2103_02119_gb300.lbm):

- "flow": one lattice from initial fields on the GPU, `steps` time steps, the
  fields read out (with `monitor`, the diagnostics before that): channels with a
  body force, lid-driven cavities and decaying vortices, FP32 and FP64, both
  schemes, with and without solid obstacles.
- "readout": post-processing of a given state: set from distributions, then
  diagnostics, strain rates and stresses, and the distributions back.
- "batch": many uneven lattices advanced together by the batched solver, either a
  fixed number of steps with one residual check, or a run to a steady residual.
- "net": the warm-start network: parameter gradients of a batch, or predictions,
  prolonged to a finer grid when `factor` is above 1.

The state of an FP32 lattice carries FP32 accuracy, so a program keeps its fields
in FP32; those of an FP64 lattice, and what only reads a state out, stay FP64.
"""
import math

import numpy as np
import torch

from paper_2103_02119_gb300 import lbm
from paper_2103_02119_gb300 import workloads as W


def listed():
    return [
        # a channel of 32 x 32 cells in FP64: the smallest flow of the repository's
        # configurations, bound by latency; a short run as in a parameter scan
        dict(name="channel_f64_32x32", kind="flow", flow="channel", nx=32, ny=32, a=0.5, precision=64,
             scheme=0, coverage=0.0, steps=100, monitor=False),
        # a small masked cavity of odd sizes in FP32, watched while it runs
        dict(name="cavity_f32_61x53_solid", kind="flow", flow="cavity", nx=61, ny=53, a=0.7, precision=32,
             scheme=0, coverage=0.1, steps=200, monitor=True),
        # the size of the larger warm-start instances: above the smallest, far
        # below what fills the GPU
        dict(name="cavity_f32_256x256_solid", kind="flow", flow="cavity", nx=256, ny=256, a=0.75, precision=32,
             scheme=0, coverage=0.1, steps=100, monitor=True),
        # the periodic validation flow at its configured size
        dict(name="vortex_f32_2048x1024", kind="flow", flow="vortex", nx=2048, ny=1024, a=0.5, precision=32,
             scheme=0, coverage=0.0, steps=100, monitor=False),
        # the benchmark's cavity: the state is far larger than the L2
        dict(name="cavity_f32_2048x8192", kind="flow", flow="cavity", nx=2048, ny=8192, a=0.25, precision=32,
             scheme=0, coverage=0.0, steps=100, monitor=False),
        # a channel around obstacles, ragged sizes, body force
        dict(name="channel_f32_1543x3001_solid", kind="flow", flow="channel", nx=1543, ny=3001, a=0.4, precision=32,
             scheme=0, coverage=0.05, steps=50, monitor=False),
        # a cavity with the raw-moment scheme, which the stability studies compare with
        dict(name="cavity_f32_raw_1001x2003", kind="flow", flow="cavity", nx=1001, ny=2003, a=0.5, precision=32,
             scheme=1, coverage=0.0, steps=50, monitor=False),
        # accuracy runs: the periodic flow in FP64
        dict(name="vortex_f64_1024x1024", kind="flow", flow="vortex", nx=1024, ny=1024, a=0.5, precision=64,
             scheme=0, coverage=0.0, steps=20, monitor=False),
        # checkpoint and post-processing of an FP32 lattice with obstacles
        dict(name="readout_f32_2048x2047_solid", kind="readout", nx=2048, ny=2047, a=0.5, precision=32,
             coverage=0.02),
        # the sweep recipe: uneven channels and cavities around obstacles
        dict(name="batch_96_uneven", kind="batch", count=96, lo=64, hi=1024, relo=100.0, rehi=5000.0,
             coverage=0.1, steps=50, until=0.0),
        # small lattices to a steady residual, as when training states are made
        dict(name="batch_64_small_to_steady", kind="batch", count=64, lo=16, hi=32, relo=10.0, rehi=100.0,
             coverage=0.1, steps=1000, until=1e-8),
        # one mini-batch of the warm-start network's training
        dict(name="net_gradients_16x64x64", kind="net", levels=4, width=32, n=16, size=64, factor=0),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["flow"] * 6 + ["readout", "batch", "batch", "net"])
    if kind == "flow":
        precision = rng.choice([32, 32, 32, 64])
        most = 2048 * 8192 if precision == 32 else 1024 * 1024
        while True:
            nx, ny = log(16, 3000), log(16, 8192)
            if nx * ny <= most:
                break
        flow = rng.choice(["channel", "cavity", "vortex"])
        return dict(kind="flow", flow=flow, nx=nx, ny=ny, a=round(rng.uniform(0.25, 1.0), 3), precision=precision,
                    scheme=rng.choice([0, 0, 0, 1]),
                    coverage=0.0 if flow == "vortex" else rng.choice([0.0, 0.02, 0.1]),
                    steps=log(2, 100) if precision == 32 else log(2, 20), monitor=rng.random() < 0.4)
    if kind == "readout":
        return dict(kind="readout", nx=log(40, 2048), ny=log(40, 2048), a=round(rng.uniform(0.25, 1.0), 3),
                    precision=rng.choice([32, 32, 64]), coverage=rng.choice([0.0, 0.05]))
    if kind == "batch":
        if rng.random() < 0.5:
            return dict(kind="batch", count=rng.randint(8, 96), lo=64, hi=log(200, 1024), relo=100.0, rehi=5000.0,
                        coverage=0.1, steps=log(5, 50), until=0.0)
        return dict(kind="batch", count=rng.randint(8, 128), lo=16, hi=rng.randint(24, 64), relo=10.0, rehi=100.0,
                    coverage=0.1, steps=rng.randrange(200, 1001, 100), until=1e-8)
    size = rng.choice([16, 24, 32, 40, 48, 64])
    return dict(kind="net", levels=4, width=rng.choice([8, 16, 32]), n=rng.randint(1, 16), size=size,
                factor=rng.choice([0, 0, 1, 2, 4]))


def work(case):
    if case["kind"] == "flow":
        cells = case["nx"] * case["ny"]
        # rho and u in (FP64) and out; the collision of every cell and step
        return {"bytes": cells * (24 + 3 * case["precision"] // 8), "flops": cells * case["steps"] * 200}
    if case["kind"] == "readout":
        cells = case["nx"] * case["ny"]
        return {"bytes": cells * 8 * (9 + 6 + 9), "flops": cells * 200}
    if case["kind"] == "batch":
        cells = sum(w["nx"] * w["ny"] for w in _sweep(case, 0))
        return {"bytes": cells * (24 + 12), "flops": cells * case["steps"] * 200}
    flops, size = 0, case["size"]
    for cin, cout, level in _convs(case):
        flops += 2 * 9 * cin * cout * case["n"] * (size >> level) ** 2
    params = sum(9 * cin * cout + cout for cin, cout, _ in _convs(case))
    cells = case["n"] * size * size
    if case["factor"] == 0:  # forward, input gradient and weight gradient
        return {"bytes": cells * 29 + 8 * params, "flops": 3 * flops}
    return {"bytes": cells * (16 + 13 * case["factor"] ** 2) + 4 * params, "flops": flops}


# ------------------------------------------------------------------ inputs --

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _solid(nx, ny, rng, coverage, margin=2):
    """Rectangles of up to a quarter of the shorter side until they cover `coverage` of the cells, a fluid
    margin along the edges; holes without a fluid neighbour are filled."""
    m = np.zeros((ny, nx), np.uint8)
    side = max(2, min(nx, ny) // 4)
    left = coverage * nx * ny
    for _ in range(400):
        w, h = int(rng.integers(1, side + 1)), int(rng.integers(1, side + 1))
        x = int(rng.integers(margin, max(margin + 1, nx - margin - w)))
        y = int(rng.integers(margin, max(margin + 1, ny - margin - h)))
        box = m[y:min(y + h, ny - margin), x:min(x + w, nx - margin)]
        new = box.size - int(box.sum())
        if new > left:
            break
        box[:] = 1
        left -= new
    p = np.pad(m, 1, constant_values=1)
    around = np.ones((ny, nx), np.uint8)
    for dy in (0, 1, 2):
        for dx in (0, 1, 2):
            if (dx, dy) != (1, 1):
                around &= p[dy:dy + ny, dx:dx + nx]
    m |= around
    return m


def _smooth(nx, ny, rng, u_amp, rho_amp):
    """Smooth random rho, u_x, u_y: three Fourier modes each, on the GPU."""
    dev = _device()
    X = ((torch.arange(nx, dtype=torch.float64, device=dev) + 0.5) / nx)[None, :]
    Y = ((torch.arange(ny, dtype=torch.float64, device=dev) + 0.5) / ny)[:, None]
    out = []
    for base, amp in ((1.0, rho_amp), (0.0, u_amp), (0.0, u_amp)):
        f = torch.full((ny, nx), base, dtype=torch.float64, device=dev)
        for _ in range(3):
            kx, ky = (int(k) for k in rng.integers(-3, 4, 2))
            f += amp / 3 * float(rng.uniform(0.3, 1.0)) * torch.cos(2 * math.pi * (kx * X + ky * Y + float(rng.random())))
        out.append(f)
    return out


def _spec(case, seed):
    """Parameters, mask and initial fields of one flow."""
    rng = np.random.default_rng([1, seed])
    nx, ny, a = case["nx"], case["ny"], case["a"]
    cs2 = W.stable_cs2(a)
    U = min(0.05, 0.3 * math.sqrt(cs2))
    nu = cs2 * float(rng.uniform(0.2, 0.5))
    s = dict(nx=nx, ny=ny, a=a, cs2=cs2, omega=W.omega_for(nu, cs2), Fx=0.0, px=1, py=1,
             wall_u=((0.0, 0.0),) * 4, mask=None, scheme=case.get("scheme", 0))
    if case.get("flow") == "channel":
        s.update(py=0, Fx=8.0 * nu * U / (ny * a) ** 2)
    elif case.get("flow", "cavity") == "cavity":
        s.update(px=0, py=0, wall_u=((0.0, 0.0),) * 3 + ((U, 0.0),))
    if case["coverage"] > 0:
        s["mask"] = _solid(nx, ny, rng, case["coverage"])
    if case.get("flow") == "vortex":
        dev = _device()
        kx, ky = 2 * math.pi / nx, 2 * math.pi / (ny * a)
        p1, p2 = (2 * math.pi * float(v) for v in rng.random(2))
        X = ((torch.arange(nx, dtype=torch.float64, device=dev) + 0.5) * kx + p1)[None, :]
        Y = ((torch.arange(ny, dtype=torch.float64, device=dev) + 0.5) * a * ky + p2)[:, None]
        u0 = 0.5 * U
        s["fields"] = [1.0 + u0 * u0 / (4 * cs2) * (torch.cos(2 * X) + torch.cos(2 * Y)),
                       (u0 * torch.sin(X) * torch.cos(Y)).contiguous(),
                       (-u0 * kx / ky * torch.cos(X) * torch.sin(Y)).contiguous()]
    else:
        s["fields"] = _smooth(nx, ny, rng, 0.5 * U, 1e-3)
    return s


def _params(s, precision):
    return lbm.make_params(s["nx"], s["ny"], s["a"], s["cs2"], s["omega"], Fx=s["Fx"], precision=precision,
                           periodic_x=s["px"], periodic_y=s["py"], wall_u=s["wall_u"], scheme=s["scheme"])


def _lattice(s, precision):
    return lbm.Lattice(s["nx"], s["ny"], s["a"], s["cs2"], s["omega"], Fx=s["Fx"], precision=precision,
                       periodic_x=s["px"], periodic_y=s["py"], wall_u=s["wall_u"], mask=s["mask"],
                       stream=torch.cuda.current_stream(), scheme=s["scheme"])


def _distributions(s, seed):
    """Post-stream distributions of a flow: equilibrium populations with a part out of equilibrium."""
    rho, u, v = s["fields"]
    g = torch.Generator(device=rho.device)
    g.manual_seed(seed)
    f = _equilibrium(rho, u, v, s)
    f += 1e-4 * (torch.rand(f.shape, dtype=torch.float64, device=f.device, generator=g) - 0.5)
    if s["mask"] is not None:
        f *= torch.from_numpy(1.0 - s["mask"]).to(f.device)
    return f


def _sweep(case, seed):
    """Sizes (the same for every seed) and parameters of the lattices of a batch."""
    sizes = np.random.default_rng([2, case["count"], case["lo"], case["hi"]])
    rng = np.random.default_rng([3, seed])
    lo, hi = math.log(case["lo"]), math.log(case["hi"])
    out = []
    for k in range(case["count"]):
        nx, ny = (int(round(math.exp(sizes.uniform(lo, hi)))) for _ in range(2))
        a = float(rng.uniform(0.2, 1.0))
        cs2 = W.stable_cs2(a)
        Re = math.exp(rng.uniform(math.log(case["relo"]), math.log(case["rehi"])))
        nu = min(max(min(0.05, 0.3 * math.sqrt(cs2)) * nx / Re, 0.06 * cs2), 1.5 * cs2)
        U = min(0.05, 0.3 * math.sqrt(cs2), nu * Re / nx)
        s = dict(nx=nx, ny=ny, a=a, cs2=cs2, omega=W.omega_for(nu, cs2), Fx=0.0, px=k % 2, py=0,
                 wall_u=((0.0, 0.0),) * 4, scheme=0)
        if k % 2:
            s["Fx"] = 8.0 * nu * U / (ny * a) ** 2
        else:
            s["wall_u"] = ((0.0, 0.0),) * 3 + ((U, 0.0),)
        out.append(s)
    return out


def _batch_spec(case, seed):
    out = _sweep(case, seed)
    rng = np.random.default_rng([4, seed])
    for s in out:
        s["mask"] = _solid(s["nx"], s["ny"], rng, float(rng.uniform(0.0, case["coverage"])))
        if case["until"] == 0:
            s["fields"] = _smooth(s["nx"], s["ny"], rng, 0.01, 1e-3)
        else:  # from rest
            s["fields"] = [torch.full((s["ny"], s["nx"]), v, dtype=torch.float64, device=_device())
                           for v in (1.0, 0.0, 0.0)]
    return out


def _convs(case):
    """(cin, cout, level) of the network's convolutions in order."""
    L, ch = case["levels"], [case["width"] << i for i in range(case["levels"])]
    out, c = [], 4
    for i in range(L):
        out += [(c, ch[i], i), (ch[i], ch[i], i)]
        c = ch[i]
    for i in range(L - 2, -1, -1):
        out += [(ch[i + 1], ch[i], i), (ch[i], ch[i], i)]
    return out + [(ch[0], 3, 0)]


def _net_inputs(case, seed):
    """Input planes, targets, fluid flags (fine ones for predictions) and a trained-size parameter vector."""
    rng = np.random.default_rng([5, seed])
    n, size, f = case["n"], case["size"], max(1, case["factor"])
    fine = np.stack([_solid(size * f, size * f, rng, 0.08) for _ in range(n)])
    x = np.zeros((n, size, size, 4), np.float32)
    x[..., 0] = fine.reshape(n, size, f, size, f).mean(axis=(2, 4))
    x[..., 1:] = rng.uniform([0.5, 0.4, 0.6], [1.0, 0.8, 1.6], (n, 1, 1, 3))
    t = rng.standard_normal((n, 3, 4, 4))
    t = np.kron(t, np.ones((1, 1, size // 4, size // 4))).transpose(0, 2, 3, 1)
    fluid = (fine == 0).astype(np.uint8)
    p = [np.concatenate([(rng.standard_normal(9 * i * o) * math.sqrt(2.0 / (9 * i))), 0.02 * rng.standard_normal(o)])
         for i, o, _ in _convs(case)]
    return x, (0.3 * t).astype(np.float32), fluid, np.concatenate(p).astype(np.float32)


# ---------------------------------------------------------------- the pass --

def prepare(case, seed):
    dev = _device()
    if case["kind"] == "flow":
        s = _spec(case, seed)
        N = case["nx"] * case["ny"]
        return dict(case=case, N=N, lat=_lattice(s, case["precision"]), fields=s["fields"],
                    out=[torch.empty(case["ny"], case["nx"], dtype=torch.float64, device=dev) for _ in range(3)])
    if case["kind"] == "readout":
        s = _spec(case, seed)
        N = case["nx"] * case["ny"]
        return dict(case=case, N=N, lat=_lattice(s, case["precision"]), f=_distributions(s, seed),
                    stress=[torch.empty(case["ny"], case["nx"], dtype=torch.float64, device=dev) for _ in range(6)],
                    out=torch.empty(9, case["ny"], case["nx"], dtype=torch.float64, device=dev))
    if case["kind"] == "batch":
        spec = _batch_spec(case, seed)
        b = lbm.lbm_batch_create([_params(s, 32) for s in spec], [s["mask"] for s in spec], torch.cuda.current_stream())
        # the launch shapes that the autotuner finds for large and for small lattices
        lbm.lbm_batch_set_shape(b, *((64, 32) if case["hi"] > 128 else (32, 1)))
        sizes = [s["nx"] * s["ny"] for s in spec]
        flat = [torch.empty(sum(sizes), dtype=torch.float64, device=dev) for _ in range(3)]
        return dict(case=case, batch=_Owned(b, lbm.lbm_batch_destroy), sizes=sizes, fields=[s["fields"] for s in spec],
                    flat=flat, views=list(zip(*(t.split(sizes) for t in flat))))
    x, t, fluid, p = _net_inputs(case, seed)
    chans = [case["width"] << i for i in range(case["levels"])]
    nn = lbm.lbm_nn_create(chans, case["n"], case["size"], case["size"], seed=0, stream=torch.cuda.current_stream())
    lbm.lbm_nn_set_params(nn, p)
    return dict(case=case, nn=_Owned(nn, lbm.lbm_nn_destroy), x=x, t=t, fluid=fluid)


class _Owned:
    """A handle of the library, freed with its owner."""

    def __init__(self, h, free):
        self.h, self.free = h, free

    def __del__(self):
        self.free(self.h)


def run(state):
    case = state["case"]
    if case["kind"] == "flow":
        lat, N = state["lat"], state["N"]
        lat.init_fields(*state["fields"])
        if case["monitor"]:
            lat.diagnostics()
        lat.step(case["steps"])
        diag = lat.diagnostics()[1] if case["monitor"] else None
        lbm.lbm_moments(lat.h, N, *state["out"])
        if case["precision"] == 64:
            out = {"rho": state["out"][0], "ux": state["out"][1], "uy": state["out"][2]}
        else:
            out = {k: v.float() for k, v in zip(("rho", "ux", "uy"), state["out"])}
        if diag is not None:
            diag = diag if case["precision"] == 64 else diag.astype(np.float32)
            out.update(sums=diag[:4], monitor=diag[4:])
        return out
    if case["kind"] == "readout":
        lat, N = state["lat"], state["N"]
        lat.set_f(state["f"])
        diag = lat.diagnostics()[1]
        lbm.lbm_stress(lat.h, N, *state["stress"])
        lbm.lbm_get_f(lat.h, N, state["out"])
        return {"sums": diag[:4], "monitor": diag[4:], "stress": state["stress"], "f": state["out"]}
    if case["kind"] == "batch":
        b, n = state["batch"].h, case["count"]
        for k in range(n):
            lbm.lbm_batch_set_active(b, k, True)
            lbm.lbm_batch_init_fields(b, k, state["sizes"][k], *state["fields"][k])
        if case["until"] > 0:
            lbm.lbm_batch_run(b, n, case["until"], 100, case["steps"])
        else:
            lbm.lbm_batch_step(b, case["steps"])
            lbm.lbm_batch_residuals(b, n)
        for k in range(n):
            lbm.lbm_batch_moments(b, k, state["sizes"][k], *state["views"][k])
        return {k: v.float() for k, v in zip(("rho", "ux", "uy"), state["flat"])}
    nn = state["nn"].h
    if case["factor"] == 0:
        loss, grads = lbm.lbm_nn_gradients(nn, state["x"], state["t"], state["fluid"])
        return {"loss": np.float32(loss), "grads": grads}
    y = lbm.lbm_nn_forward(nn, state["x"])
    if case["factor"] > 1:
        y = lbm.lbm_nn_prolong(nn, y, case["factor"], state["fluid"])
    return {"y": y}


# ------------------------------------------------------- the same in 64 bits --

EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)


def _factors(u, e, cs2, h):
    """The three-velocity equilibrium factor along one axis with spacing h."""
    q = (cs2 + u * u) / (h * h)
    return 1.0 - q if e == 0 else 0.5 * (q + e * u / h)


def _equilibrium(rho, u, v, s):
    return torch.stack([rho * _factors(u, EX[i], s["cs2"], 1.0) * _factors(v, EY[i], s["cs2"], s["a"])
                        for i in range(9)])


def _neighbour(t, dx, dy):
    """t at (x + dx, y + dy), periodic."""
    return torch.roll(t, (-dy, -dx), (-2, -1))


class _Exact:
    """One lattice in 64 bits, written from the scheme's equations."""

    def __init__(self, s):
        self.s = s
        dev = s["fields"][0].device
        ny, nx = s["ny"], s["nx"]
        self.solid = (torch.zeros(ny, nx, dtype=torch.bool, device=dev) if s["mask"] is None
                      else torch.from_numpy(s["mask"] != 0).to(dev))
        walls = torch.ones(ny + 2, nx + 2, dtype=torch.bool, device=dev)
        walls[1:-1, 1:-1] = self.solid
        if s["px"]:
            walls[1:-1, 0], walls[1:-1, -1] = self.solid[:, -1], self.solid[:, 0]
        if s["py"]:
            walls[0, :], walls[-1, :] = walls[-2, :].clone(), walls[1, :].clone()
        self.walls = walls
        # whether the cell that population i comes from is a wall or solid
        self.blocked = [walls[1 - EY[i]:1 - EY[i] + ny, 1 - EX[i]:1 - EX[i] + nx] for i in range(9)]
        self.f = None

    def start(self):
        self.f = list(_equilibrium(*self.s["fields"], self.s))

    def macro(self, f):
        s = self.s
        rho = sum(f)
        jx = (f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7])
        jy = s["a"] * ((f[2] - f[4]) + (f[5] - f[8]) + (f[6] - f[7]))
        rho = torch.where(self.solid, torch.ones_like(rho), rho)
        return rho, (jx + 0.5 * s["Fx"]) / rho, jy / rho

    def raw(self, f):
        """sum f ex^p ey^q for p, q = 0 .. 2."""
        a = self.s["a"]
        R = [[None] * 3 for _ in range(3)]
        for q in range(3):
            col = []
            for z, p, m in ((0, 2, 4), (1, 5, 8), (3, 6, 7)):
                col.append(f[z] + f[p] + f[m] if q == 0 else a * (f[p] - f[m]) if q == 1 else a * a * (f[p] + f[m]))
            R[0][q], R[1][q], R[2][q] = col[0] + col[1] + col[2], col[1] - col[2], col[1] + col[2]
        return R

    def gradient(self, rho):
        a = self.s["a"]
        east = torch.where(self.blocked[3], rho, _neighbour(rho, 1, 0))
        west = torch.where(self.blocked[1], rho, _neighbour(rho, -1, 0))
        north = torch.where(self.blocked[4], rho, _neighbour(rho, 0, 1))
        south = torch.where(self.blocked[2], rho, _neighbour(rho, 0, -1))
        return 0.5 * (east - west), (north - south) / (2 * a)

    def strain(self, rho, u, v, n3, n4):
        """d_x u_x and d_y u_y from the second-order moments out of equilibrium."""
        s = self.s
        cs2, a2, w3, w4 = s["cs2"], s["a"] ** 2, s["omega"][3], s["omega"][4]
        dx, dy = self.gradient(rho)
        gx, gy = 0.5 * (1 - 3 * cs2) * u * dx, 0.5 * (a2 - 3 * cs2) * v * dy
        b1 = rho * (-2 * cs2 / w3 - 0.5 * (1 - 3 * cs2) + 1.5 * u * u)
        b2 = rho * (-2 * cs2 / w3 - 0.5 * (a2 - 3 * cs2) + 1.5 * v * v)
        c1 = rho * (-2 * cs2 / w4 - 0.5 * (1 - 3 * cs2) + 1.5 * u * u)
        c2 = rho * (2 * cs2 / w4 + 0.5 * (a2 - 3 * cs2) - 1.5 * v * v)
        r3, r4 = n3 + gx + gy, n4 + gx - gy
        det = b1 * c2 - b2 * c1
        return (c2 * r3 - b2 * r4) / det, (b1 * r4 - c1 * r3) / det, dx, dy

    def collide(self, f):
        s = self.s
        cs2, a, a2, w, Fx = s["cs2"], s["a"], s["a"] ** 2, s["omega"], s["Fx"]
        rho, u, v = self.macro(f)
        R = self.raw(f)
        central = s["scheme"] == 0
        U, V = (u, v) if central else (0.0 * u, 0.0 * v)
        # moments about (U, V): shift along y, then along x
        K = [[None] * 3 for _ in range(3)]
        for p in range(3):
            K[p] = [R[p][0], R[p][1] - V * R[p][0], R[p][2] - 2 * V * R[p][1] + V * V * R[p][0]]
        K = [[K[0][q], K[1][q] - U * K[0][q], K[2][q] - 2 * U * K[1][q] + U * U * K[0][q]] for q in range(3)]  # K[q][p]
        e20, e02 = (cs2, cs2) if central else (cs2 + u * u, cs2 + v * v)
        du, dv = (0.0, 0.0) if central else (u, v)
        n20, n02 = K[0][2] - rho * e20, K[2][0] - rho * e02
        n11, n21, n12 = K[1][1] - rho * du * dv, K[1][2] - rho * e20 * dv, K[2][1] - rho * du * e02
        n22 = K[2][2] - rho * e20 * e02
        # strain rates take the raw moments out of equilibrium (Eq. 34-35)
        uF = u * Fx if central else 0.0
        dxu, dyv, dx, dy = self.strain(rho, u, v, n20 + n02 - uF, n20 - n02 - uF)
        px = (1 - 3 * cs2) * (u * dx + rho * dxu) - 3 * rho * dxu * u * u
        py = (a2 - 3 * cs2) * (v * dy + rho * dyv) - 3 * rho * dyv * v * v
        half = [1 - 0.5 * r for r in w]
        src = 0.0 if central else 2 * u * Fx
        d3 = half[3] * (px + py + src) - w[3] * (n20 + n02)
        d4 = half[4] * (px - py + src) - w[4] * (n20 - n02)
        D = {(1, 0): Fx, (2, 0): 0.5 * (d3 + d4), (0, 2): 0.5 * (d3 - d4), (1, 1): -w[5] * n11, (2, 1): -w[6] * n21,
             (1, 2): -w[7] * n12, (2, 2): -w[8] * n22}
        if not central:
            D[1, 1] = D[1, 1] + half[5] * Fx * v
            D[2, 1] = D[2, 1] + half[6] * 2 * Fx * u * v
            D[1, 2] = D[1, 2] + half[7] * Fx * v * v
            D[2, 2] = D[2, 2] + half[8] * 2 * Fx * u * v * v
        g = [[D.get((p, q), 0.0) for q in range(3)] for p in range(3)]
        # back to moments about 0, then to populations, axis by axis
        g = [[g[p][0], g[p][1] + V * g[p][0], g[p][2] + 2 * V * g[p][1] + V * V * g[p][0]] for p in range(3)]
        g = [g[0], [g[1][q] + U * g[0][q] for q in range(3)],
             [g[2][q] + 2 * U * g[1][q] + U * U * g[0][q] for q in range(3)]]
        cols = {0: [g[0][q] - g[2][q] for q in range(3)], 1: [0.5 * (g[2][q] + g[1][q]) for q in range(3)],
                -1: [0.5 * (g[2][q] - g[1][q]) for q in range(3)]}
        out = []
        for i in range(9):
            m0, m1, m2 = cols[EX[i]]
            add = m0 - m2 / a2 if EY[i] == 0 else 0.5 * (m2 / a2 + EY[i] * m1 / a)
            out.append(f[i] + add)
        return out, rho

    def moving(self, f, rho):
        s = self.s
        ny, nx = s["ny"], s["nx"]
        for i in range(1, 9):
            for wall, (Ux, Uy) in enumerate(s["wall_u"]):
                if Ux == 0 and Uy == 0:
                    continue
                if (wall in (2, 3) and s["py"]) or (wall in (0, 1) and s["px"]):
                    continue
                if (EY[i], EY[i], EX[i], EX[i])[3 - wall] != (-1, 1, -1, 1)[wall]:
                    continue
                row = {0: (slice(None), 0), 1: (slice(None), nx - 1), 2: (0, slice(None)), 3: (ny - 1, slice(None))}[wall]
                r = rho[row]
                cx, cy = (torch.as_tensor(Ux, dtype=r.dtype, device=r.device), torch.as_tensor(Uy, dtype=r.dtype, device=r.device))
                odd = [_factors(cx, k * EX[i], s["cs2"], 1.0) * _factors(cy, k * EY[i], s["cs2"], s["a"]) for k in (1, -1)]
                f[i][row] -= r * (odd[0] - odd[1])

    def step(self):
        out, rho = self.collide(self.f)
        self.moving(out, rho)
        self.f = [torch.where(self.blocked[i], out[OPP[i]], _neighbour(out[i], -EX[i], -EY[i])) for i in range(9)]

    def fields(self):
        rho, u, v = self.macro(self.f)
        z = torch.zeros_like(rho)
        return [torch.where(self.solid, z, t) for t in (rho, u, v)]

    def sums(self):
        rho, u, v = self.fields()
        return [float(t.sum()) for t in (rho, rho * u, rho * v, 0.5 * rho * (u * u + v * v))]

    def stress(self):
        s = self.s
        f = self.f
        rho, u, v = self.macro(f)
        R = self.raw(f)
        n20, n02 = R[2][0] - rho * (s["cs2"] + u * u), R[0][2] - rho * (s["cs2"] + v * v)
        exx, eyy, _, _ = self.strain(rho, u, v, n20 + n02, n20 - n02)
        exy = -(R[1][1] - rho * u * v) * s["omega"][5] / (rho * s["cs2"])
        z3, z4, z5 = (s["cs2"] * (1 / s["omega"][k] - 0.5) for k in (3, 4, 5))
        div = exx + eyy
        out = [exx, eyy, exy, rho * (z4 * (2 * exx - div) + z3 * div), rho * (z4 * (2 * eyy - div) + z3 * div), rho * z5 * exy]
        return [torch.where(self.solid, torch.zeros_like(t), t) for t in out]


def _net_forward(case, x, p):
    """The network on x (n, h, w, 4) in 64 bits, before the output stage."""
    F = torch.nn.functional
    k, layers = 0, []
    for i, o, _ in _convs(case):
        w = p[k:k + 9 * i * o].reshape(3, 3, i, o).permute(3, 2, 0, 1)
        layers.append((w, p[k + 9 * i * o:k + 9 * i * o + o]))
        k += 9 * i * o + o
    layers = iter(layers)

    def conv(t):
        return F.conv2d(t, *next(layers), padding=1)

    t, skips, L = x.permute(0, 3, 1, 2), [], case["levels"]
    for i in range(L):
        t = conv(conv(t).relu()).relu()
        skips.append(t)
        t = F.avg_pool2d(t, 2) if i < L - 1 else t
    for i in range(L - 2, -1, -1):
        t = conv(F.interpolate(t, scale_factor=2, mode="nearest")).relu()
        t = conv(t + skips[i]).relu()
    return conv(t)


def _output_stage(y, fluid):
    """(n, 3, h, w), fluid (n, 1, h, w): smoothing over the fluid cells, then the staggered parts taken out."""
    y = y * fluid
    k = torch.tensor([0.25, 0.5, 0.25], dtype=y.dtype, device=y.device)
    y = torch.nn.functional.conv2d(y, (k[:, None] * k[None, :]).expand(3, 1, 3, 3), padding=1, groups=3) * fluid
    h, w = y.shape[-2:]
    sx = (1.0 - 2.0 * (torch.arange(w, device=y.device) % 2)).to(y.dtype)[None, None, :]
    sy = (1.0 - 2.0 * (torch.arange(h, device=y.device) % 2)).to(y.dtype)[None, :, None]
    fl = fluid[:, 0]
    count = fl.sum(dim=(1, 2), keepdim=True).clamp(min=1.0)
    u, v = y[:, 1], y[:, 2]
    u = u - fl * sx * (u * fl * sx).sum(dim=(1, 2), keepdim=True) / count
    v = v - fl * sy * (v * fl * sy).sum(dim=(1, 2), keepdim=True) / count
    return torch.stack([y[:, 0], u, v], dim=1)


def exact(case, seed):
    if case["kind"] == "flow":
        e = _Exact(_spec(case, seed))
        e.start()
        for _ in range(case["steps"]):
            e.step()
        out = dict(zip(("rho", "ux", "uy"), e.fields()))
        if case["monitor"]:
            out.update(sums=np.array(e.sums()), monitor=None)
        return out
    if case["kind"] == "readout":
        s = _spec(case, seed)
        e = _Exact(s)
        e.f = list(_distributions(s, seed))
        return {"sums": np.array(e.sums()), "monitor": None, "stress": e.stress(), "f": torch.stack(e.f)}
    if case["kind"] == "batch":
        if case["until"] > 0 or case["count"] * case["steps"] > 5000:
            return None  # lattices leave the run one by one; a minute and more here
        flat = [[], [], []]
        for s in _batch_spec(case, seed):
            e = _Exact(s)
            e.start()
            for _ in range(case["steps"]):
                e.step()
            for k, t in enumerate(e.fields()):
                flat[k].append(t.reshape(-1))
        return dict(zip(("rho", "ux", "uy"), (torch.cat(t) for t in flat)))
    x, t, fluid, p = _net_inputs(case, seed)
    dev = _device()
    x64 = torch.from_numpy(x).to(dev, torch.float64)
    p64 = torch.from_numpy(p).to(dev, torch.float64).requires_grad_(case["factor"] == 0)
    y = _output_stage(_net_forward(case, x64, p64), (x64[..., 0] < 0.5).double()[:, None])
    if case["factor"] == 0:
        fl = torch.from_numpy(fluid).to(dev, torch.float64)[:, None]
        d = (y - torch.from_numpy(t).to(dev, torch.float64).permute(0, 3, 1, 2)) * fl
        loss = (d * d).sum() / (3.0 * fl.sum())
        grads, = torch.autograd.grad(loss, p64)
        return {"loss": np.float64(loss.item()), "grads": grads}
    if case["factor"] > 1:
        fine = torch.from_numpy(fluid).to(dev, torch.float64)[:, None]
        y = torch.nn.functional.interpolate(y, scale_factor=case["factor"], mode="bilinear", align_corners=False)
        y = _output_stage(y, fine)
    return {"y": y.permute(0, 2, 3, 1).contiguous()}
