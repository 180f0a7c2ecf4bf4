"""What is measured: the work that users of this framework have it do, through its public entry points.

The listed cases cover every form of the framework (single handles, the precision form, ragged batches, time slices,
multilevel iterations, the adjoint), both ionic models, every kind of conductivity and both stencils, from a 500-node
cable to 4.2 million nodes.  `draw` gives more cases of the same families with other sizes.  A pass starts from a saved
state in mid-wave (the state a run is resumed from) and takes the case's time steps; the outputs are the whole state.

`exact` is the same method in 64-bit torch, written from the paper and sharing no code with the framework: Lagrange
integrals by Gauss-Legendre quadrature, solves by dense cosine transforms or CG, gradients by torch's autograd.
"""
import math

import numpy as np
import torch

import paper_2405_19994_gb300 as P
from paper_2405_19994_gb300 import esdc as E
from paper_2405_19994_gb300 import inputs as I

SIGMA, CHI, CM = 0.17, 140.0, 0.01
V_REST = {"hh": -75.0, "syn19": -83.4}


def listed():
    return [
        # The 32x32 sheet of the tests and of `bench.py --form sheet`: a user's first run, a debugging run, a
        # parameter scan.  Four steps of a time loop; launches and latency are what it costs.
        dict(name="sheet32", kind="sweep", model="hh", cond="scalar", order=2, precision="fp64", nx=32, ny=32, nz=1,
             h=0.25, M=3, K=4, dt=0.025, steps=4),
        # The paper's one-dimensional domain (100 mm, 0.2 mm cells) at high order: convergence studies in time.
        dict(name="cable500", kind="sweep", model="hh", cond="scalar", order=2, precision="fp64", nx=500, ny=1, nz=1,
             h=0.2, M=6, K=8, dt=0.05, steps=2),
        # A small sheet of odd sides: meshes come from a tissue's outline, not from powers of two.
        dict(name="sheet_odd", kind="sweep", model="hh", cond="scalar", order=2, precision="fp64", nx=101, ny=75, nz=1,
             h=0.25, M=3, K=4, dt=0.025, steps=2),
        # The paper's two-dimensional experiments: 100 mm square, 0.4 mm cells, fourth-order differences, the
        # 19-state model, M = 6.
        dict(name="sheet_order4", kind="sweep", model="syn19", cond="scalar", order=4, precision="fp64", nx=256, ny=256,
             nz=1, h=0.4, M=6, K=6, dt=0.05, steps=1),
        # The headline slab of `python bench.py`: production runs of a 3D tissue.
        dict(name="slab_syn19", kind="sweep", model="syn19", cond="scalar", order=2, precision="fp64", nx=128, ny=128,
             nz=32, h=0.2, M=4, K=6, dt=0.05, steps=1),
        # The same kind of tissue with sides that are not powers of two (the iterative solves).
        dict(name="slab_odd", kind="sweep", model="syn19", cond="scalar", order=2, precision="fp64", nx=90, ny=75,
             nz=19, h=0.2, M=4, K=6, dt=0.05, steps=1),
        # Ventricular slab with fibres rotating through the depth, 4.2 million nodes, FP64: the largest production mesh.
        dict(name="aniso_fp64", kind="sweep", model="hh", cond="layers", order=2, precision="fp64", nx=256, ny=256,
             nz=64, h=0.2, M=4, K=6, dt=0.05, steps=1),
        # The precision form on such a slab.
        dict(name="aniso_mixed", kind="sweep", model="hh", cond="layers", order=2, precision="mixed", nx=128, ny=128,
             nz=64, h=0.2, M=4, K=6, dt=0.05, steps=1),
        # A training step of a conductivity fit: forward run, loss, adjoint gradients of the field, g_Na and g_K.
        dict(name="adjoint256", kind="adjoint", model="hh", nx=256, ny=256, h=0.25, M=3, K=4, dt=0.025, steps=6, sens=64),
        # The ragged batch of `bench.py --form batch`: 64 tissues of 64..512 nodes a side (parameter studies).
        dict(name="batch64", kind="batch", model="hh", n=64, lo=64, hi=512, h=0.25, M=3, K=4, dt=0.025, steps=1),
        # Parallel-in-time Q^par over 16 slices.
        dict(name="qpar16", kind="qpar", model="hh", n=16, nx=256, ny=256, h=0.25, M=3, iters=4, dt=0.025),
        # Two-level Algorithm HSDC over 8 slices.
        dict(name="hsdc8", kind="hsdc", model="hh", n=8, nx=128, ny=128, h=0.25, M=3, M2=2, iters=2, dt=0.025),
    ]


def _logint(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def _side(rng, lo, hi):
    """A side length: a power of two half of the time, any number (odd ones among them) otherwise."""
    if rng.random() < 0.5:
        return 1 << rng.randint(int(math.ceil(math.log2(lo))), int(math.floor(math.log2(hi))))
    return _logint(rng, lo, hi)


def draw(rng):
    kind = rng.choice(["sheet", "sheet", "cable", "slab", "slab", "slab", "adjoint", "batch", "qpar", "hsdc"])
    if kind in ("sheet", "cable", "slab"):
        model = rng.choice(["hh", "syn19"])
        c = dict(kind="sweep", model=model, cond="scalar", order=2, precision="fp64")
        if kind == "cable":
            c.update(nx=_side(rng, 33, 8192), ny=1, nz=1, h=0.2, order=rng.choice([2, 4]))
        elif kind == "sheet":
            c.update(nx=_side(rng, 12, 512), ny=_side(rng, 12, 512), nz=1, h=rng.choice([0.2, 0.25, 0.4]))
            c["cond"] = rng.choice(["scalar", "scalar", "field"])
            if c["cond"] == "scalar":
                c["order"] = rng.choice([2, 2, 4])
        else:
            top = 200 if model == "hh" else 96
            c.update(nx=_side(rng, 16, top), ny=_side(rng, 16, top), nz=_side(rng, 4, 48), h=0.2)
            c["cond"] = rng.choice(["scalar", "scalar", "layers"])
            c["precision"] = rng.choice(["fp64", "fp64", "mixed"])
        # M = 2..6 and K <= 2M - 1 as in the convergence studies; dt of the workloads
        M = rng.choice([2, 3, 4, 4, 6])
        c.update(M=M, K=rng.choice([M, M + 2]), dt=rng.choice([0.025, 0.05]) if model == "syn19" else 0.025,
                 steps=rng.choice([1, 2, 4]) if kind != "slab" else 1)
        return c
    if kind == "adjoint":
        return dict(kind="adjoint", model="hh", nx=_side(rng, 16, 256), ny=_side(rng, 16, 256), h=0.25, M=3, K=4, dt=0.025,
                    steps=rng.randint(2, 6), sens=rng.choice([16, 64]))
    if kind == "batch":
        lo = rng.choice([12, 32, 64])
        return dict(kind="batch", model="hh", n=_logint(rng, 4, 64), lo=lo, hi=lo * rng.choice([2, 4]), h=0.25, M=3, K=4,
                    dt=0.025, steps=rng.choice([1, 2]))
    if kind == "qpar":
        return dict(kind="qpar", model="hh", n=rng.choice([4, 8, 16]), nx=_side(rng, 32, 256), ny=_side(rng, 32, 256),
                    h=0.25, M=rng.choice([2, 3, 4]), iters=rng.choice([2, 4]), dt=0.025)
    return dict(kind="hsdc", model="hh", n=rng.choice([4, 8]), nx=_side(rng, 24, 128), ny=_side(rng, 24, 128), h=0.25,
                M=rng.choice([3, 3, 4]), M2=2, iters=2, dt=0.025)


# ------------------------------------------------------------------------------------------------ inputs
def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _params(model):
    return I.hh1952_params() if model == "hh" else I.syn19_params()


def _state(model, nx, ny, nz, seed):
    """A state in mid-wave [n_state, N]: a travelling front and its tail around a random centre, potentials between
    rest and the plateau with smooth 0.5 mV variations, gates at the steady state of the potential that passed a little
    earlier, auxiliaries near theirs."""
    g = torch.Generator().manual_seed(int(seed))
    u = torch.rand(64, generator=g, dtype=torch.float64).tolist()
    dev, f = _device(), torch.float64
    x = (torch.arange(nx, device=dev, dtype=f) / max(nx, 8)).view(1, 1, nx)
    y = (torch.arange(ny, device=dev, dtype=f) / max(nx, 8)).view(1, ny, 1)
    z = (torch.arange(nz, device=dev, dtype=f) / max(nx, 8)).view(nz, 1, 1)
    r = ((x - 0.2 * u[0]) ** 2 + (0.6 * (y - u[1])) ** 2 + (0.6 * (z - u[2])) ** 2).sqrt()
    wob = sum(torch.cos(6.0 * (k + 1) * (u[3 + k] * x + u[8 + k] * y + u[13 + k] * z) + 6.28 * u[18 + k]) for k in range(5))
    front, tail, w, wt = 0.35 + 0.4 * u[23], 0.12 * u[24], max(0.03, 2.5 / max(nx, 8)), max(0.08, 5.0 / max(nx, 8))
    rest = V_REST[model]
    top = 100.0 if model == "hh" else 95.0

    def wave(shift):
        return torch.sigmoid((front - shift - r) / w) * (0.15 + 0.85 * torch.sigmoid((r - tail + shift) / wt))

    V = (rest + top * wave(0.0) + 0.5 * wob).reshape(-1)
    Vl = (rest + top * wave(0.01) + 0.5 * wob).reshape(-1)
    mod = _Model(model, dev)
    lam, b = mod.gates(Vl)
    gates = -b / lam
    if model == "hh":
        return torch.cat([V[None], gates]).contiguous()
    g6 = gates[5]
    a = torch.stack([1 - g6, g6, 1 - g6, gates[3] * gates[4], gates[3] * gates[4], gates[3] * gates[4]])
    a = a * (0.9 + 0.1 * torch.sigmoid(wob).reshape(-1))
    return torch.cat([V[None], a, gates]).contiguous()


def _stimulus(nx, ny, nz, seed):
    """One box of 8 x 8 (x all) nodes switched on throughout the first step's interval."""
    rng = np.random.default_rng(int(seed))
    px, py = min(8, nx), min(8, ny)
    x0, y0 = int(rng.integers(0, nx - px + 1)), int(rng.integers(0, ny - py + 1))
    return dict(boxes=np.array([[x0, x0 + px, y0, y0 + py, 0, nz]], np.int32), amp=np.array([0.5]), t_on=np.array([0.0]),
                t_off=np.array([1.0]))


T0 = 0.4


def _workload(c, seed, nx, ny, nz, sigma=SIGMA):
    layers = I.fibre_layers(nz) if c.get("cond") == "layers" else None
    field = None
    if c.get("cond") == "field" or c["kind"] == "adjoint":
        field = I.lognormal_field(nx, ny, nz, seed=int(seed) % 1000003)
    return I.Workload(name="case", dim=3 if nz > 1 else (2 if ny > 1 else 1), nx=nx, ny=ny, nz=nz, h=c["h"],
                      model=I.MODEL_HH1952 if c["model"] == "hh" else I.MODEL_SYN19, params=_params(c["model"]),
                      V0=V_REST[c["model"]], M=c["M"], K=c.get("K", 1), dt=c["dt"], T=1.0, sigma=sigma, layers=layers,
                      sigma_field=field, order=c.get("order", 2), **_stimulus(nx, ny, nz, seed))


def _tissues(c, seed):
    rng = np.random.default_rng(int(seed) + 7)
    # the sides belong to the case (a batch is laid out once); conductivities, stimuli and states to the seed
    sides = np.random.default_rng(c["n"] * 1009 + c["lo"] * 31 + c["hi"]).integers(c["lo"], c["hi"] + 1, size=(c["n"], 2))
    return [_workload(c, seed * 131 + k, int(sides[k][0]), int(sides[k][1]), 1, sigma=float(rng.uniform(0.05, 0.3)))
            for k in range(c["n"])]


def _sensors(c, seed):
    rng = np.random.default_rng(int(seed) + 3)
    return np.sort(rng.choice(c["nx"] * c["ny"], size=min(c["sens"], c["nx"] * c["ny"]), replace=False)).astype(np.int32)


def _target(c, seed):
    g = torch.Generator().manual_seed(int(seed) + 5)
    return -60.0 + 20.0 * torch.rand((c["steps"], min(c["sens"], c["nx"] * c["ny"])), generator=g, dtype=torch.float64)


def prepare(case, seed):
    c = case
    if c["kind"] == "sweep":
        wl = _workload(c, seed, c["nx"], c["ny"], c["nz"])
        s = P.Solver.from_workload(wl, M_max=wl.M, precision=c["precision"])
        y0 = s.new_state()
        y0[:, : s.n_nodes] = _state(c["model"], c["nx"], c["ny"], c["nz"], seed)
        return dict(case=c, solver=s, y0=y0, y=s.new_state())
    if c["kind"] == "adjoint":
        wl = _workload(c, seed, c["nx"], c["ny"], 1)
        s = P.Solver.from_workload(wl, M_max=wl.M)
        y0 = s.new_state()
        y0[:, : s.n_nodes] = _state("hh", c["nx"], c["ny"], 1, seed)
        return dict(case=c, solver=s, y0=y0, sigma=torch.from_numpy(wl.sigma_field).cuda(),
                    sens=torch.from_numpy(_sensors(c, seed)).cuda(), target=_target(c, seed).cuda())
    if c["kind"] == "batch":
        wls = _tissues(c, seed)
        b = P.Batch.from_workloads(wls, M_max=c["M"])
        y0 = b.new_state()
        b.init_state(y0, wls[0].V0)
        for k, w in enumerate(wls):
            b.tissue(y0, k)[:] = _state(c["model"], w.nx, w.ny, 1, seed * 131 + k)
        return dict(case=c, batch=b, y0=y0, y=b.new_state())
    # time slices: P copies of one sheet
    wl = _workload(c, seed, c["nx"], c["ny"], 1)
    b = P.Batch.from_workloads([wl] * c["n"], M_max=c["M"])
    y_in = b.new_state()
    b.init_state(y_in, wl.V0)
    b.tissue(y_in, 0)[:] = _state(c["model"], c["nx"], c["ny"], 1, seed)
    st = dict(case=c, batch=b, y_in=y_in, y_out=b.new_state())
    if c["kind"] == "hsdc":
        st["coarse"] = [P.Batch.from_workloads([wl], M_max=c["M2"]) for _ in range(c["n"])]
    return st


def run(state):
    c = state["case"]
    if c["kind"] == "sweep":
        s, y = state["solver"], state["y"]
        y.copy_(state["y0"])
        for n in range(c["steps"]):
            s.sweep(y, T0 + n * c["dt"], c["dt"], c["M"], c["K"])
        return {"V": y[0, : s.n_nodes], "w": y[1:, : s.n_nodes]}
    if c["kind"] == "adjoint":
        s = state["solver"]
        sig = state["sigma"].clone().requires_grad_(True)
        gna = torch.tensor(1.2, dtype=torch.float64, requires_grad=True)
        gk = torch.tensor(0.36, dtype=torch.float64, requires_grad=True)
        tr = E.sensor_traces(s, sig, gna, gk, state["y0"], T0, c["dt"], c["M"], c["K"], c["steps"], state["sens"])
        (0.5 * (tr - state["target"]).square().sum()).backward()
        return {"traces": tr.detach(), "sigma": sig.grad, "gna": gna.grad, "gk": gk.grad}
    b = state["batch"]
    if c["kind"] == "batch":
        y = state["y"]
        y.copy_(state["y0"])
        for n in range(c["steps"]):
            b.sweep(y, T0 + n * c["dt"], c["dt"], c["M"], c["K"])
        cols = [b.tissue(y, k) for k in range(b.n)]
        return {"V": [t[0] for t in cols[:20]], "w": [t[1:] for t in cols[:20]], "all": y}
    if c["kind"] == "qpar":
        b.qpar(state["y_in"], state["y_out"], T0, c["dt"], c["M"], c["iters"])
    else:
        E.hsdc2(b, state["coarse"], state["y_in"], state["y_out"], T0, c["dt"], c["M"], c["M2"], c["iters"])
    cols = [b.tissue(state["y_out"], k) for k in range(b.n)]
    return {"V": [t[0] for t in cols], "w": [t[1:] for t in cols]}


def work(case):
    """The state in and out once per pass; FP64 operations: per node, sweep and collocation node one ionic evaluation,
    the M-term quadrature of every state and a diffusion solve of about 30 operations."""
    c = case
    ns, ionic = (4, 40) if c["model"] == "hh" else (19, 180)
    M, K, steps = c["M"], c.get("K", 1), c.get("steps", 1)
    if c["kind"] == "batch":
        sides = np.random.default_rng(c["n"] * 1009 + c["lo"] * 31 + c["hi"]).integers(c["lo"], c["hi"] + 1, size=(c["n"], 2))
        n = int((sides[:, 0] * sides[:, 1]).sum())
    else:
        n = c["nx"] * c["ny"] * c.get("nz", 1)
    per = K * M * (ionic + 2 * M * ns + 30) * steps
    if c["kind"] == "adjoint":
        return dict(bytes=8.0 * n * (ns + 2), flops=4.0 * n * per)
    if c["kind"] == "qpar":
        n, per = n * c["n"], c["iters"] * M * (ionic + 2 * M * ns + 30)
    if c["kind"] == "hsdc":
        m2 = c["M2"]
        n, per = n * c["n"], c["iters"] * (2 * M * (ionic + 2 * M * ns) + M * 30 + 2 * m2 * (ionic + 2 * m2 * ns) + m2 * 30)
    return dict(bytes=16.0 * n * ns, flops=1.0 * n * per)


# ------------------------------------------------------------------------------------------------ 64-bit reference
class _Model:
    """Currents and gate functions of the two ionic models (plain formulas)."""

    def __init__(self, model, dev, gna=None, gk=None):
        p = torch.from_numpy(_params(model)).to(dev)
        self.hh, self.p, self.na = model == "hh", p, 0 if model == "hh" else 6
        self.gna, self.gk = (gna if gna is not None else p[0]), (gk if gk is not None else p[1])

    @staticmethod
    def _xe(x):
        small = x.abs() < 0.05
        xs = torch.where(small, torch.ones_like(x), x)
        s = torch.where(small, x, torch.zeros_like(x))
        return torch.where(small, 1 - s / 2 + s**2 / 12 - s**4 / 720 + s**6 / 30240, xs / torch.expm1(xs))

    def gates(self, V):
        """Lambda and b = -Lambda w_inf, [gates, N]."""
        p = self.p
        if self.hh:
            v = V - p[6]
            al = torch.stack([self._xe((25 - v) / 10), 0.07 * torch.exp(-v / 20), 0.1 * self._xe((10 - v) / 10)])
            be = torch.stack([4 * torch.exp(-v / 18), 1 / (torch.exp((30 - v) / 10) + 1), 0.125 * torch.exp(-v / 80)])
            return -(al + be), al
        g = p[:72].view(12, 6, 1)
        winf = 1 / (1 + torch.exp((g[:, 0] - V) / g[:, 1]))
        lam = -g[:, 2] * torch.exp(g[:, 3] / (1 + torch.exp((g[:, 4] - V) / g[:, 5])))
        return lam, -lam * winf

    def currents(self, u):
        """-I_ion [N] and the auxiliaries' derivatives [na, N]."""
        p, V = self.p, u[0]
        if self.hh:
            m, h, n = u[1], u[2], u[3]
            return -(self.gna * m**3 * h * (V - p[3]) + self.gk * n**4 * (V - p[4]) + p[2] * (V - p[5])), u[1:1]
        a, g, c, tau = u[1:7], u[7:], p[72:82], p[82:88]
        mi = -(c[0] * g[0] * g[1] * g[2] * a[0] * (V - c[1]) + c[2] * g[3] * g[4] * a[2] * (V - c[3])
               + c[4] * a[1] * (1 + c[9] * a[5]) * (V - c[5]) + c[6] * g[6] * g[7] * (V - c[5])
               + c[7] / 4 * (g[8] + g[9] + g[10] + g[11]) * (V - c[8]))
        src = torch.stack([1 - g[5], g[5], 1 - g[5], g[3] * g[4], a[3], a[4]])
        return mi, (src - a) / tau[:, None]


def _radau(M):
    if M == 1:
        return np.array([1.0])
    c = np.zeros(M + 1)
    c[M], c[M - 1] = 1.0, -1.0
    x = np.sort(np.real(np.polynomial.legendre.legroots(c)))
    d = np.polynomial.legendre.legder(c)
    for _ in range(3):
        x = x - np.polynomial.legendre.legval(x, c) / np.polynomial.legendre.legval(x, d)
    x[-1] = 1.0
    return (x + 1) / 2


def _lagrange(c, s):
    """l_j(s) for the nodes c, as an array [len(c), len(s)]."""
    return np.array([np.prod([(s - c[k]) / (c[j] - c[k]) for k in range(len(c)) if k != j], axis=0) * np.ones_like(s)
                     for j in range(len(c))])


def _aij(z, M, zmax):
    """a_ij(z) = c_i int_0^1 e^{(1-s) c_i z} l_j(c_i s) ds, [M, M, *z.shape]: 20-point Gauss-Legendre on panels graded
    towards s = 1, where e^{(1-s) c_i z} lives."""
    c = _radau(M)
    cut = [0.0] + [2.0**-k for k in range(max(0, int(math.ceil(math.log2(max(zmax, 1.0))))), -1, -1)]
    gx, gw = np.polynomial.legendre.leggauss(20)
    r = np.concatenate([(b - a) / 2 * gx + (a + b) / 2 for a, b in zip(cut, cut[1:])])
    w = np.concatenate([(b - a) / 2 * gw for a, b in zip(cut, cut[1:])])
    rows = []
    for i in range(M):
        l = _lagrange(c, c[i] * (1 - r)) * w * c[i]
        acc = [0.0] * M
        for q in range(len(r)):
            e = torch.exp((r[q] * c[i]) * z)
            acc = [acc[j] + float(l[j, q]) * e for j in range(M)]
        rows.append(torch.stack(acc))
    return torch.stack(rows)


class _Box:
    """The mesh of one tissue: A v and the solve of (I - g A) x = b, with A the Laplacian times sigma of any kind."""

    def __init__(self, wl, dev, field=None):
        self.n = (wl.nz, wl.ny, wl.nx)
        self.ih2, self.order, self.dev = 1.0 / wl.h**2, wl.order, dev
        self.lay = None if wl.layers is None else {k: torch.from_numpy(v).to(dev).view(-1, 1, 1) for k, v in wl.layers.items()}
        self.field = field if field is not None else (None if wl.sigma_field is None else
                                                      torch.from_numpy(wl.sigma_field).to(dev))
        self.sigma = wl.sigma
        if self.lay is None and self.field is None:
            self.U, self.mu = [], 0.0
            for a, n in enumerate(self.n):
                k = np.arange(n)
                U = np.cos(np.pi * (np.outer(k, 2 * k + 1) % (4 * n)) / (2 * n))     # k (2i + 1) reduced exactly
                U = U * np.where(k == 0, np.sqrt(1 / n), np.sqrt(2 / n))[:, None]
                t = np.pi * k / n
                mu = -4 * np.sin(t / 2) ** 2 if self.order == 2 else (32 * np.cos(t) - 2 * np.cos(2 * t) - 30) / 12
                sh = [1, 1, 1]
                sh[a] = n
                self.U.append(torch.from_numpy(U).to(dev))
                self.mu = self.mu + torch.from_numpy(mu * self.ih2 * self.sigma).to(dev).view(sh)

    def A(self, v, field=None):
        v = v.view(self.n)
        out = torch.zeros_like(v)
        if self.field is not None:
            s = (self.field if field is None else field).view(self.n)
            for a in range(3):
                if self.n[a] > 1:
                    lo, hi = [slice(None)] * 3, [slice(None)] * 3
                    lo[a], hi[a] = slice(0, -1), slice(1, None)
                    f = (s[tuple(lo)] + s[tuple(hi)]) / 2 * (v[tuple(hi)] - v[tuple(lo)])
                    out = out + torch.nn.functional.pad(f, self._pad(a, 0, 1))
                    out = out - torch.nn.functional.pad(f, self._pad(a, 1, 0))
            return (out * self.ih2).reshape(-1)
        if self.lay is not None:
            L = self.lay
            dx, dy = v[:, :, 1:] - v[:, :, :-1], v[:, 1:, :] - v[:, :-1, :]
            out[:, :, :-1] += L["sxx"] * dx
            out[:, :, 1:] -= L["sxx"] * dx
            out[:, :-1, :] += L["syy"] * dy
            out[:, 1:, :] -= L["syy"] * dy
            if self.n[0] > 1:
                dz = (L["szz"][1:] + L["szz"][:-1]) / 2 * (v[1:] - v[:-1])
                out[:-1] += dz
                out[1:] -= dz
            cd = L["sxy"] / 2
            e, f = cd * (v[:, 1:, 1:] - v[:, :-1, :-1]), cd * (v[:, :-1, 1:] - v[:, 1:, :-1])
            out[:, :-1, :-1] += e
            out[:, 1:, 1:] -= e
            out[:, 1:, :-1] -= f
            out[:, :-1, 1:] += f
            return (out * self.ih2).reshape(-1)
        for a in range(3):
            n = self.n[a]
            if n == 1:
                continue
            w = {1: 1.0} if self.order == 2 else {1: 16 / 12, 2: -1 / 12}
            i = torch.arange(n, device=self.dev)
            for k, cf in w.items():
                for s in (-k, k):
                    j = i + s
                    while bool(((j < 0) | (j >= n)).any()):
                        j = torch.where(j < 0, -j - 1, torch.where(j >= n, 2 * n - 1 - j, j))
                    out += cf * (v.index_select(a, j) - v)
        return (out * (self.ih2 * self.sigma)).reshape(-1)

    @staticmethod
    def _pad(a, lo, hi):
        p = [0] * 6
        p[2 * (2 - a)], p[2 * (2 - a) + 1] = lo, hi
        return p

    def solve(self, g, b, x0=None):
        if self.lay is None and self.field is None:
            v = b.view(self.n)
            v = torch.einsum("kz,zyx->kyx", self.U[0], v)
            v = torch.einsum("ky,zyx->zkx", self.U[1], v)
            v = torch.einsum("kx,zyx->zyk", self.U[2], v) / (1 - g * self.mu)
            v = torch.einsum("kz,kyx->zyx", self.U[0], v)
            v = torch.einsum("ky,zkx->zyx", self.U[1], v)
            return torch.einsum("kx,zyk->zyx", self.U[2], v).reshape(-1)
        x = b.clone() if x0 is None else x0.clone()
        for _ in range(2):                                # restarted once: the second residual is the true one
            r = b - (x - g * self.A(x))
            p, rr = r.clone(), r.dot(r)
            stop = 1e-33 * b.dot(b)
            for _ in range(200):
                if bool(rr <= stop):
                    break
                q = p - g * self.A(p)
                al = rr / p.dot(q)
                x, r = x + al * p, r - al * q
                rn = r.dot(r)
                p, rr = r + (rn / rr) * p, rn
        return x


class _SolveField(torch.autograd.Function):
    """x = (I - g A(field))^{-1} b with its derivatives in b and the field."""

    @staticmethod
    def forward(ctx, b, field, box, g):
        x = box.solve(g, b)
        ctx.save_for_backward(x, field)
        ctx.box, ctx.g = box, g
        return x

    @staticmethod
    def backward(ctx, gx):
        x, field = ctx.saved_tensors
        lam = ctx.box.solve(ctx.g, gx.contiguous())
        with torch.enable_grad():
            f = field.detach().requires_grad_(True)
            (gf,) = torch.autograd.grad((lam * ctx.box.A(x, f)).sum() * ctx.g, f)
        return lam, gf, None, None


class _Ref:
    """One tissue's step: sweeps of the recursive form from a given iterate, and the collocation residual."""

    def __init__(self, c, wl, dev, M, field=None, gna=None, gk=None):
        self.M, self.dt, self.dev, self.wl = M, wl.dt, dev, wl
        self.mod = _Model(c["model"], dev, gna, gk)
        self.box = _Box(wl, dev, None if field is None else field.detach())
        self.field = field
        self.D = 1.0 / (wl.chi * wl.Cm)
        self.c = np.concatenate([[0.0], _radau(M)])
        st = torch.zeros((wl.nz, wl.ny, wl.nx), dtype=torch.float64, device=dev)
        for bx, a in zip(wl.boxes, wl.amp):
            st[bx[4]:bx[5], bx[2]:bx[3], bx[0]:bx[1]] += float(a)
        self.stim = st.reshape(-1)
        self.a0 = _aij(torch.zeros(1, dtype=torch.float64), M, 1.0)[..., 0].tolist()

    def fI(self, V):
        return self.D * self.box.A(V, self.field)

    def fE(self, u, t):
        mi, ha = self.mod.currents(u)
        on = 1.0 if self.wl.t_on[0] <= t < self.wl.t_off[0] else 0.0
        return (mi + on * self.stim) / self.wl.Cm, ha

    def setup(self, yn):
        na = self.mod.na
        lam, _ = self.mod.gates(yn[0])
        z = self.dt * lam
        zmax = float(-z.detach().min())
        N = yn.shape[1]
        if z.requires_grad:
            a = _aij(z, self.M, zmax)
        else:                                             # in pieces: the quadrature keeps M^2 copies of z
            a = torch.empty((self.M, self.M) + tuple(z.shape), dtype=torch.float64, device=self.dev)
            for lo in range(0, N, 1 << 19):
                a[..., lo:lo + (1 << 19)] = _aij(z[:, lo:lo + (1 << 19)].contiguous(), self.M, zmax)
        self.lam, self.a, self.yn, self.na = lam, a, yn, na

    def phi(self, i):
        x = (self.c[i] - self.c[i - 1]) * self.dt * self.lam
        return torch.expm1(x) / x

    def G(self, u, t, fi):
        e, ha = self.fE(u, t)
        lam, b = self.mod.gates(u[0])
        w = u[1 + self.na:]
        return e, torch.cat([(fi + e)[None], ha, lam * w + b + self.lam * (self.yn[1 + self.na:] - w)])

    def quad(self, i, Gs):
        """dt sum_j (a_ij - a_{i-1,j}) G_j."""
        na, out = self.na, 0.0
        lo, hi = [], []
        for j in range(self.M):
            s0 = self.a0[i - 1][j] - (self.a0[i - 2][j] if i > 1 else 0.0)
            s = self.a[i - 1, j] - (self.a[i - 2, j] if i > 1 else 0.0)
            lo.append(s0 * Gs[j][:1 + na])
            hi.append(s * Gs[j][1 + na:])
        return self.dt * torch.cat([sum(lo), sum(hi)]) + out

    def evaluate(self, Y, t):
        fi = [self.fI(y[0]) for y in Y]
        return fi, [self.G(y, t + self.c[j + 1] * self.dt, fi[j])[1] for j, y in enumerate(Y)]

    def sweep(self, Y, t, tau=None):
        M, dt, na = self.M, self.dt, self.na
        fi, Gs = self.evaluate(Y, t)
        new, prev, prevG = [], self.yn, None
        for i in range(1, M + 1):
            d = self.c[i] - self.c[i - 1]
            rhs = prev + self.quad(i, Gs)
            if tau is not None:
                rhs = rhs + tau[i - 1] - (tau[i - 2] if i > 1 else 0.0)
            add = [-fi[i - 1], None, None]
            if i > 1:
                e, Gn = self.G(prev, t + self.c[i - 1] * dt, self.fI(prev[0]))
                dG = Gn - Gs[i - 2]
                add = [-fi[i - 1] + e - (Gs[i - 2][0] - fi[i - 2]), dG[1:1 + na], self.phi(i) * dG[1 + na:]]
            V = rhs[0] + dt * d * add[0]
            w = rhs[1:] if i == 1 else rhs[1:] + dt * d * torch.cat([add[1], add[2]])
            g = dt * d * self.D
            if self.field is not None and (V.requires_grad or self.field.requires_grad):
                V = _SolveField.apply(V, self.field, self.box, g)
            else:
                V = self.box.solve(g, V, Y[i - 1][0].detach())
            prev = torch.cat([V[None], w])
            new.append(prev)
        return new

    def residual(self, Y, t, tau=None):
        _, Gs = self.evaluate(Y, t)
        out, acc = [], self.yn
        for i in range(1, self.M + 1):
            acc = acc + self.quad(i, Gs)
            out.append(acc - Y[i - 1] + (tau[i - 1] if tau is not None else 0.0))
        return out

    def step(self, yn, t, K):
        self.setup(yn)
        Y = [yn] * self.M
        for _ in range(K):
            Y = self.sweep(Y, t)
        return Y[-1]


def _interp(W, Y):
    return [sum(float(W[i][j]) * Y[j] for j in range(len(Y))) for i in range(len(W))]


def exact(case, seed):
    c, dev = case, _device()
    if c["kind"] == "sweep":
        wl = _workload(c, seed, c["nx"], c["ny"], c["nz"])
        ref, y = _Ref(c, wl, dev, c["M"]), _state(c["model"], c["nx"], c["ny"], c["nz"], seed)
        for n in range(c["steps"]):
            y = ref.step(y, T0 + n * c["dt"], c["K"])
        return {"V": y[0], "w": y[1:]}
    if c["kind"] == "adjoint":
        wl = _workload(c, seed, c["nx"], c["ny"], 1)
        sig = torch.from_numpy(wl.sigma_field).to(dev).requires_grad_(True)
        gna = torch.tensor(1.2, dtype=torch.float64, requires_grad=True)
        gk = torch.tensor(0.36, dtype=torch.float64, requires_grad=True)
        ref = _Ref(c, wl, dev, c["M"], sig, gna.to(dev), gk.to(dev))
        y, sens, tr = _state("hh", c["nx"], c["ny"], 1, seed), torch.from_numpy(_sensors(c, seed)).long().to(dev), []
        for n in range(c["steps"]):
            y = ref.step(y, T0 + n * c["dt"], c["K"])
            tr.append(y[0][sens])
        tr = torch.stack(tr)
        (0.5 * (tr - _target(c, seed).to(dev)).square().sum()).backward()
        return {"traces": tr.detach(), "sigma": sig.grad, "gna": gna.grad, "gk": gk.grad}
    if c["kind"] == "batch":
        out = []
        for k, wl in enumerate(_tissues(c, seed)[:20]):
            ref, y = _Ref(c, wl, dev, c["M"]), _state(c["model"], wl.nx, wl.ny, 1, seed * 131 + k)
            for n in range(c["steps"]):
                y = ref.step(y, T0 + n * c["dt"], c["K"])
            out.append(y)
        return {"V": [y[0] for y in out], "w": [y[1:] for y in out], "all": None}
    # time slices: every slice starts from y0; an iteration sweeps each from the end value of the one before it
    wl = _workload(c, seed, c["nx"], c["ny"], 1)
    y0, n, dt, M = _state(c["model"], c["nx"], c["ny"], 1, seed), c["n"], c["dt"], c["M"]
    ref = _Ref(c, wl, dev, M)
    Z = [[y0] * M for _ in range(n)]

    def qpar(Z, taus):
        ends = [y0] + [z[-1] for z in Z[:-1]]
        new = []
        for p in range(n):
            ref.setup(ends[p])
            new.append(ref.sweep(Z[p], T0 + p * dt, taus[p] if taus else None))
        return new

    if c["kind"] == "qpar":
        for _ in range(c["iters"]):
            Z = qpar(Z, None)
    else:
        M2 = c["M2"]
        crs = _Ref(c, wl, dev, M2)
        cf, cc = _radau(M), _radau(M2)
        down, up = _lagrange(cf, cc).T, _lagrange(cc, cf).T          # [M2][M], [M][M2]
        start = [y0] * n                                              # the values that the iterates were swept from
        for _ in range(c["iters"]):
            coarse, taus = [], []
            for p in range(n):
                ref.setup(start[p])
                rf = _interp(down, ref.residual(Z[p], T0 + p * dt))
                sz = _interp(down, Z[p])
                crs.setup(start[p])
                rc = crs.residual(sz, T0 + p * dt)
                taus.append([a - b for a, b in zip(rf, rc)])
                coarse.append(sz)
            y, delta = y0, []
            for p in range(n):                                        # the coarse level, one slice after another
                crs.setup(y)
                z2 = crs.sweep(coarse[p], T0 + p * dt, taus[p])
                delta.append(_interp(up, [a - b for a, b in zip(z2, coarse[p])]))
                y = z2[-1]
            Z = [[a + b for a, b in zip(Z[p], delta[p])] for p in range(n)]
            start = [y0] + [z[-1] for z in Z[:-1]]
            Z = qpar(Z, None)
    return {"V": [z[-1][0] for z in Z], "w": [z[-1][1:] for z in Z]}
