"""What a user of this package runs, as measurable cases.

A lattice case is one short simulation through ``Lattice``: initial fields in device memory, a
number of time steps, macroscopic fields (and diagnostics) out.  The set-ups are the ones of the
paper this package implements: static and oscillating droplets in periodic boxes (Sec. III.A and
III.B), Rayleigh-Taylor between walls (Sec. III.C), liquid jets with a nozzle inlet and a convective
outflow (Sec. IV), and a batch of small jets as the regime-map sweep advances them.  The surrogate
cases are the network's batch inference and its training loop.

``exact`` recomputes a case in FP64 with plain torch: per-node collision by a dense 27 x 27 moment
matrix, streaming by scattering every population to its target, nothing shared with the package.
"""
import math

import numpy as np
import torch

import paper_1705_03141_gb300 as pkg

PERIODIC, NOSLIP, FREESLIP, INFLOW, OUTFLOW = range(5)
# bytes per node of the stored populations (two colours in FP64 / FP32; 4 bytes per direction packed;
# 2 bytes per direction and a 16-byte colour record compact)
POP_BYTES = {"f64": 432, "f32": 216, "f16": 108, "bf16": 108, "c16": 72, "cbf16": 72}
# storage of the relaxation rates: slot of each of the 27 moments, and the rates quoted in Sec. II
SLOT = [1, 1, 1, 1, 5, 6, 6, 8, 8, 8, 11, 11, 11, 14, 14, 14, 17, 18, 19, 19, 21, 21, 21, 24, 24, 24, 27]
SUGA = {1: 0.0, 5: 1.5, 11: 1.5, 14: 1.83, 17: 1.4, 18: 1.61, 19: 1.98, 21: 1.98, 24: 1.74, 27: 1.74}
N_IN, WIDTH, DEPTH, N_POS, N_CLS = 5, 256, 4, 64, 4  # the surrogate network
LR = 1e-3


def _box(name, kind, nx, ny, nz, storage, steps, samples=1, D=0.0):
    return dict(name=name, kind=kind, nx=nx, ny=ny, nz=nz, storage=storage, steps=steps, samples=samples, D=float(D))


def listed():
    return [
        # the smallest box: the static droplet of the FP64 mode that is compared with the oracle
        _box("droplet 32 f64", "droplet", 32, 32, 32, "f64", 96),
        # the oscillating drop of Table II, its shape sampled every ten steps: short runs between reads
        _box("droplet 41 f64 sampled", "droplet", 41, 41, 41, "f64", 60, samples=6),
        # the oscillating drop at 64^3 in FP32
        _box("droplet 64 f32", "droplet", 64, 64, 64, "f32", 192),
        # the static drops of Table I (85^3, rows that fill no whole 32-node block)
        _box("droplet 85 f32", "droplet", 85, 85, 85, "f32", 96),
        # Rayleigh-Taylor between no-slip walls, periodic sides, packed half storage
        _box("rayleigh-taylor 64 f16", "rt", 64, 64, 256, "f16", 96),
        # the jet of Sec. IV at the main benchmark's size, in each storage a user picks for it
        _box("jet 128 f32", "jet", 128, 128, 512, "f32", 48, D=16),
        _box("jet 128 f16", "jet", 128, 128, 512, "f16", 48, D=16),
        _box("jet 128 c16", "jet", 128, 128, 512, "c16", 48, D=16),
        # the paper's own jets (Table IV): 8D x 8D x 20D at D = 25
        _box("jet 200 f32", "jet", 200, 200, 500, "f32", 32, D=25),
        # regime-map sweep: jets of uneven size advanced by one batch, each jet's leading edge read
        dict(name="sweep 6 jets f16", kind="sweep", jets=6, storage="f16", steps=64, pick=2024),
        # the surrogate: batch inference, and minibatch training on host arrays
        dict(name="surrogate forward 4096", kind="forward", batch=4096),
        dict(name="surrogate train 64", kind="train", batch=64, steps=24),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["droplet", "droplet", "rt", "jet", "jet", "jet", "sweep", "forward", "train", "grad"])
    if what == "droplet":
        storage = rng.choice(["f64", "f32", "f32", "f16", "bf16", "c16", "cbf16"])
        n = [_log(rng, 17, 48 if storage == "f64" else 140) for _ in range(3)]
        return _strip(_box("", what, *n, storage, rng.choice([10, 16, 31, 48, 64]), samples=rng.choice([1, 1, 2])))
    if what == "rt":
        w = _log(rng, 16, 110)
        return _strip(_box("", what, w, w, 4 * w, rng.choice(["f32", "f16", "bf16", "c16"]), rng.choice([16, 31, 48])))
    if what == "jet":
        D = rng.uniform(6.0, 18.0)
        nx, ny = int(rng.uniform(5.0, 8.0) * D), int(rng.uniform(5.0, 8.0) * D)
        return _strip(_box("", what, nx, ny, int(rng.uniform(14.0, 30.0) * D), rng.choice(["f32", "f32", "f16", "f16", "bf16", "c16", "cbf16"]),
                           rng.choice([10, 16, 31, 48]), D=D))
    if what == "sweep":
        return dict(kind=what, jets=rng.randint(2, 8), storage=rng.choice(["f16", "f16", "f32", "c16"]), steps=rng.choice([16, 31, 64]),
                    pick=rng.randrange(1, 10 ** 6))
    if what == "forward":
        return dict(kind=what, batch=_log(rng, 1, 4096))
    if what == "train":
        return dict(kind=what, batch=_log(rng, 16, 512), steps=rng.choice([8, 16, 24]))
    return dict(kind=what, batch=_log(rng, 8, 4096))


def _strip(case):
    return {k: v for k, v in case.items() if k != "name"}


# ---------------------------------------------------------------------------
# set-ups

def _params(kind, shape, D, seed):
    """Lattice parameters of a set-up (Sec. III.A/B droplets, III.C Rayleigh-Taylor, IV.A jet)."""
    nx, ny, nz = shape
    rates = [SUGA.get(k, 1.0) for k in SLOT]
    p = dict(rho_r0=1.0, rho_b0=1.0, nu_r=0.01, nu_b=0.01, A=0.01, beta=0.7, s=rates, g=(0.0, 0.0, 0.0), force_mode=0,
             bc=(PERIODIC,) * 6, inflow=None, seed=int(seed))
    if kind == "droplet":
        p.update(rho_r0=1.5, nu_r=3.333e-3, nu_b=3.333e-3)
    elif kind == "rt":
        g = 1e-5
        nu = math.sqrt(nx * g) * nx / 512.0
        p.update(rho_r0=3.0, nu_r=nu, nu_b=nu, A=0.0, g=(0.0, 0.0, -g), force_mode=1,
                 bc=(PERIODIC, PERIODIC, PERIODIC, PERIODIC, NOSLIP, NOSLIP))
    else:
        gamma, nu_c, nu_j, u = 1.2, 1.8e-4, 5.4e-4, 0.1
        p.update(rho_b0=1.0 / gamma, nu_r=nu_j, nu_b=nu_c, A=0.005, g=(0.0, 0.0, u * u / (8.5 * D)), force_mode=2,
                 bc=(FREESLIP, FREESLIP, FREESLIP, FREESLIP, INFLOW, OUTFLOW),
                 inflow=dict(xc=0.5 * (nx - 1), yc=0.5 * (ny - 1), D=D, u_j0=u, noise_frac=0.01))
    return p


def _sweep_jets(case):
    """The jets of a regime-map sweep: uneven boxes, nozzles and groups (Re, Oh) drawn log-uniformly (Sec. IV.C)."""
    rng = np.random.default_rng(int(case["pick"]))
    jets = []
    for k in range(int(case["jets"])):
        n, D = int(rng.choice([64, 80, 96])), float(rng.integers(8, 13))
        Re, Oh = 10.0 ** rng.uniform(1.0, 3.4), 10.0 ** rng.uniform(-3.0, 0.0)
        gamma, eta = rng.uniform(1.1, 1.5), rng.uniform(1.0, 5.0)
        nu_j = min(0.1 * D / Re, 0.015)
        u = Re * nu_j / D
        p = _params("jet", (n, n, 4 * n), D, k)
        tau = 1.5 * (nu_j + nu_j / eta) + 0.5
        p.update(rho_b0=1.0 / gamma, nu_r=nu_j, nu_b=nu_j / eta, A=min(9.0 * u * u * D / (Re * Oh) ** 2 / (4.0 * tau), 0.02),
                 g=(0.0, 0.0, u * u / (8.5 * D)))
        p["inflow"]["u_j0"] = u
        jets.append(((n, n, 4 * n), D, p))
    return jets


def _fields(kind, shape, D, p, seed):
    """(rho_r, rho_b, u) on the GPU in FP64: tanh interfaces of width 4 (Sec. III), a smooth random velocity."""
    nx, ny, nz = shape
    g = torch.Generator().manual_seed(int(seed))
    r = lambda *s: torch.rand(*s, generator=g, dtype=torch.float64)  # noqa: E731
    dev = dict(dtype=torch.float64, device="cuda")
    x = torch.arange(nx, **dev)[None, None, :]
    y = torch.arange(ny, **dev)[None, :, None]
    z = torch.arange(nz, **dev)[:, None, None]
    jet = kind == "jet"
    if kind == "droplet":
        c = [0.5 * (n - 1) + float(d) for n, d in zip(shape, 2.0 * r(3) - 1.0)]
        ax = [0.25 * min(shape) * (0.9 + 0.3 * float(d)) for d in r(3)]
        R = (ax[0] * ax[1] * ax[2]) ** (1.0 / 3.0)
        dist = (torch.sqrt(((x - c[0]) / ax[0]) ** 2 + ((y - c[1]) / ax[1]) ** 2 + ((z - c[2]) / ax[2]) ** 2) - 1.0) * R
        amp = 0.01
    elif kind == "rt":
        ph = 6.283185307179586 * r(2)
        h = 0.05 * nx * (torch.cos(2 * math.pi * x / nx + float(ph[0])) + torch.cos(2 * math.pi * y / ny + float(ph[1])))
        dist = -(z - (0.5 * nz + h))
        amp = 0.005
    else:  # a jet that has come half way: a column with surface waves and a round head
        xc, yc = 0.5 * (nx - 1), 0.5 * (ny - 1)
        rad = torch.sqrt((x - xc) ** 2 + (y - yc) ** 2)
        wave = torch.zeros(nz, 1, 1, **dev)
        for k in range(3):
            wave = wave + 0.05 * torch.sin(2 * math.pi * (k + 1.0 + float(r(1))) * z / (6.0 * D) + 6.283 * float(r(1)))
        top = (0.45 + 0.1 * float(r(1))) * nz
        col = rad - 0.5 * D * (1.0 + wave)
        head = torch.sqrt(rad ** 2 + (z - top).clamp(min=0.0) ** 2) - 0.8 * D
        dist = torch.minimum(torch.where(z <= top, col, torch.full_like(col, 1e3)), torch.where(z >= top - D, head, torch.full_like(head, 1e3)))
        amp = 0.02 * p["inflow"]["u_j0"]
    phase = 0.5 * (1.0 - torch.tanh(0.5 * dist)).expand(nz, ny, nx)
    u = torch.zeros(3, nz, ny, nx, **dev)
    for c in range(3):
        for _ in range(2):
            k = torch.randint(1, 4, (3,), generator=g)
            ph = 6.283185307179586 * r(3)
            u[c] += 0.5 * amp * (torch.sin(2 * math.pi * int(k[0]) * x / nx + float(ph[0])) * torch.sin(2 * math.pi * int(k[1]) * y / ny + float(ph[1])) *
                                 torch.sin(2 * math.pi * int(k[2]) * z / nz + float(ph[2])))
    if jet:
        u[2] += p["inflow"]["u_j0"] * phase
    return (p["rho_r0"] * phase).contiguous(), (p["rho_b0"] * (1.0 - phase)).contiguous(), u


def _jets(case, seed):
    """[(shape, params, fields)] of a lattice case."""
    if case["kind"] == "sweep":
        out = []
        for k, (shape, D, p) in enumerate(_sweep_jets(case)):
            p["seed"] = int(seed) * 1000 + k
            out.append((shape, p, _fields("jet", shape, D, p, int(seed) * 1000 + k)))
        return out
    shape = (case["nx"], case["ny"], case["nz"])
    p = _params(case["kind"], shape, case["D"], seed)
    return [(shape, p, _fields(case["kind"], shape, case["D"], p, seed))]


def _net_inputs(case, seed):
    rng = np.random.default_rng(int(seed))
    n, steps = int(case["batch"]), int(case.get("steps", 1))
    x = rng.uniform(-1.0, 1.0, (steps, n, N_IN)).astype(np.float32)
    ramp = np.linspace(0.0, 1.0, N_POS, dtype=np.float32)
    target = (ramp * (0.8 + 0.4 * x[..., :1]) + 0.05 * np.sin(3.0 * x[..., 1:2])).astype(np.float32)
    label = np.clip(np.floor((x[..., 2] + 1.0) * 2.0), 0, N_CLS - 1).astype(np.int32)
    flat = []
    for a, b in zip([N_IN] + [WIDTH] * DEPTH, [WIDTH] * DEPTH + [N_POS + N_CLS]):
        flat += [rng.uniform(-1.0, 1.0, a * b) / math.sqrt(a), rng.uniform(-1.0, 1.0, b) / math.sqrt(a)]
    return x, target, label, np.concatenate(flat).astype(np.float32)


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("forward", "train", "grad"):
        x, target, label, params = _net_inputs(case, seed)
        net = pkg.Mlp(n_in=N_IN, width=WIDTH, depth=DEPTH, n_pos=N_POS, n_cls=N_CLS, max_batch=max(4096, case["batch"]))
        net.set_params(params)
        state = dict(case=case, net=net, x=x, target=target, label=label, params=params)
        if kind == "forward":  # queries already on the device, the answer buffer reused
            state["x"] = torch.from_numpy(x[0]).cuda()
            state["y"] = torch.empty((case["batch"], N_POS + N_CLS), dtype=torch.float32, device="cuda")
        return state
    boxes = []
    for shape, p, fields in _jets(case, seed):
        lat = pkg.Lattice(shape, p, storage=case["storage"])
        nx, ny, nz = shape
        out = tuple(torch.empty(s, dtype=torch.float64, device="cuda") for s in ((nz, ny, nx), (nz, ny, nx), (3, nz, ny, nx)))
        boxes.append((lat, fields, out))
    state = dict(case=case, boxes=boxes)
    if kind == "sweep":
        for lat, fields, _ in boxes:
            lat.init_fields(*fields)
            lat.step(1)  # a batch takes compact storage after its first step
        state["batch"] = pkg.Batch([b[0] for b in boxes])
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "forward":
        return state["net"].forward(state["x"], out=state["y"])
    if kind == "train":
        net, losses = state["net"], []
        net.set_params(state["params"])
        for x, target, label in zip(state["x"], state["target"], state["label"]):
            losses.append(net.train_step(x, target, label, lr=LR, w_pos=1.0, w_cls=0.2))
        return np.array(losses), net.get_params()
    if kind == "grad":
        return state["net"].loss_grad(state["x"][0], state["target"][0], state["label"][0], w_pos=1.0, w_cls=0.2)
    if kind == "sweep":
        for lat, fields, _ in state["boxes"]:
            lat.init_fields(*fields)
            lat.step(1)
        state["batch"].step(case["steps"])
        state["batch"].synchronize()
        return [(lat.macro(out), _diag(lat)) for lat, _, out in state["boxes"]]
    lat, fields, out = state["boxes"][0]
    lat.init_fields(*fields)
    each, got = case["steps"] // case["samples"], []
    for k in range(case["samples"]):
        lat.step(each)
        if case["samples"] > 1:
            got.append(_diag(lat))
    return lat.macro(out), got


def _diag(lat):
    d = lat.diag()
    return [d["mass_r"], d["mass_b"], d["z_le"]]


def _nodes(case):
    if case["kind"] == "sweep":
        return sum(s[0] * s[1] * s[2] for s, _, _ in _sweep_jets(case))
    return case["nx"] * case["ny"] * case["nz"]


def work(case):
    """Bytes: every step reads and writes the populations once; the initial fields are read and the
    macroscopic fields written once (FP64); a sample reads the populations.  The collision, the gradients
    and the recolouring of a node take about 900 operations.  Network: the weights, the inputs and the
    outputs once (FP32 parameters and moments read and written by a training step)."""
    kind = case["kind"]
    weights = N_IN * WIDTH + (DEPTH - 1) * WIDTH * WIDTH + WIDTH * (N_POS + N_CLS)
    if kind == "forward":
        return {"bytes": 2 * weights + 4 * case["batch"] * (N_IN + N_POS + N_CLS), "flops": 2 * weights * case["batch"]}
    if kind in ("train", "grad"):
        n = case.get("steps", 1)
        return {"bytes": n * (4 * weights * (7 if kind == "train" else 2) + 4 * case["batch"] * (N_IN + N_POS + 1)), "flops": n * 6 * weights * case["batch"]}
    pop, nodes, samples = POP_BYTES[case["storage"]], _nodes(case), case.get("samples", 1)
    steps = case["steps"] + (1 if kind == "sweep" else 0)
    return {"bytes": nodes * (2 * pop * steps + 40 + pop + samples * pop + 40), "flops": nodes * 900.0 * steps}


def tolerance(case):
    """Relative 2-norm error of each output: about four times what the listed cases and the drawn ones of
    their kind show against ``exact`` (FP64 7.5e-14, FP32 3.2e-5, packed half 4.7e-3, compact half 2.0e-3;
    bfloat16, three bits shorter, eight times half's; network outputs 6.8e-4, gradients 5.6e-4, trained
    parameters 1.9e-3).  The velocity, small against the rounding of the populations, sets the number."""
    kind = case["kind"]
    if kind in ("forward", "grad"):
        return {"rel": 3e-3}
    if kind == "train":
        return {"rel": 8e-3}
    return {"rel": {"f64": 3e-13, "f32": 1.3e-4, "f16": 2e-2, "bf16": 1.5e-1, "c16": 8e-3, "cbf16": 6e-2}[case["storage"]]}


# ---------------------------------------------------------------------------
# the same in FP64, in plain torch

_C = [(x, y, z) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)]
_W1 = {-1: 1.0 / 6.0, 0: 2.0 / 3.0, 1: 1.0 / 6.0}
_W = [_W1[a] * _W1[b] * _W1[c] for a, b, c in _C]


def _moment_rows():
    """The 27 moment polynomials of Eq. (momentSet) on the velocities (rows) in the order of SLOT."""
    x, y, z = (np.array([c[a] for c in _C], dtype=np.float64) for a in range(3))
    x2, y2, z2 = x * x, y * y, z * z
    s2, s4, s6 = x2 + y2 + z2, x2 * y2 + y2 * z2 + z2 * x2, x2 * y2 * z2
    return np.stack([
        np.ones(27), x, y, z, s2 - 2, 3 * x2 - s2, y2 - z2, x * y, y * z, z * x,
        3 * x * (y2 + z2) - 4 * x, 3 * y * (x2 + z2) - 4 * y, 3 * z * (x2 + y2) - 4 * z,
        x * (9 * y2 * z2 - 6 * (y2 + z2) + 4), y * (9 * x2 * z2 - 6 * (x2 + z2) + 4), z * (9 * x2 * y2 - 6 * (x2 + y2) + 4),
        3 * s4 + 4 * (1 - s2), 27 * s6 - 18 * s4 + 12 * s2 - 8,
        2 * (y2 + z2) + 3 * (x2 * y2 + x2 * z2) - 4 * x2 - 6 * y2 * z2, 2 * (z2 - y2) + 3 * (x2 * y2 - x2 * z2),
        x * y * (3 * z2 - 2), y * z * (3 * x2 - 2), z * x * (3 * y2 - 2),
        x * (y2 - z2), y * (z2 - x2), z * (x2 - y2), x * y * z])


def _splitmix(h):
    h = (h + np.uint64(0x9E3779B97F4A7C15))
    h = (h ^ (h >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    h = (h ^ (h >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return h ^ (h >> np.uint64(31))


class _Exact:
    """One box in FP64: total populations per colour [2][27][nz][ny][nx], one scatter per direction."""

    def __init__(self, shape, p, fields, device):
        self.shape, self.p, self.t = shape, p, 0
        nx, ny, nz = shape
        self.dev = dict(dtype=torch.float64, device=device)
        rr, rb, u = (v.to(device) for v in fields)
        self.ab = 8.0 / 27.0
        self.ar = 1.0 - (1.0 - self.ab) * p["rho_b0"] / p["rho_r0"]
        M = _moment_rows()
        self.M, self.Mi = torch.tensor(M, **self.dev), torch.tensor(np.linalg.inv(M), **self.dev)
        self.n = nx * ny * nz
        uu = [u[a].reshape(-1) for a in range(3)]
        self.f = torch.stack([self._feq(rr.reshape(-1), uu, self.ar), self._feq(rb.reshape(-1), uu, self.ab)])
        self.inlet = None
        if p["inflow"]:
            i = p["inflow"]
            yy, xx = np.meshgrid(np.arange(ny), np.arange(nx), indexing="ij")
            node = np.flatnonzero(((xx - i["xc"]) ** 2 + (yy - i["yc"]) ** 2 < (0.5 * i["D"]) ** 2).reshape(-1))
            self.inlet_np, self.inlet = node, torch.from_numpy(node).to(device)
        self.plane = nx * ny
        self.top = self.f[:, :, -self.plane:].clone()
        axis = [torch.arange(n, device=device) for n in shape]
        self.pos = [axis[0][None, None, :], axis[1][None, :, None], axis[2][:, None, None]]

    def _feq(self, rho, u, alpha):
        uu = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
        out = torch.empty((27,) + tuple(rho.shape), **self.dev)
        for i, c in enumerate(_C):
            cu = c[0] * u[0] + c[1] * u[1] + c[2] * u[2]
            vphi = alpha if c == (0, 0, 0) else 27.0 / 19.0 * (1.0 - alpha) * _W[i]
            out[i] = rho * (vphi + _W[i] * (3.0 * cu + 4.5 * cu * cu - 1.5 * uu))
        return out

    def _gradient(self, v):
        """3 sum_i w_i v(x + c_i) c_i: wrapped on periodic faces, clamped (a mirror ghost) on the others."""
        nx, ny, nz = self.shape
        v = v.view(nz, ny, nx)
        for a, n, dim in ((0, nx, 2), (1, ny, 1), (2, nz, 0)):
            lo = n - 1 if self.p["bc"][2 * a] == PERIODIC else 0
            hi = 0 if self.p["bc"][2 * a] == PERIODIC else n - 1
            v = torch.cat([v.narrow(dim, lo, 1), v, v.narrow(dim, hi, 1)], dim)
        smooth = lambda w, d: (w.narrow(d, 0, w.shape[d] - 2) + 4.0 * w.narrow(d, 1, w.shape[d] - 2) + w.narrow(d, 2, w.shape[d] - 2)) / 6.0  # noqa: E731
        diff = lambda w, d: 0.5 * (w.narrow(d, 2, w.shape[d] - 2) - w.narrow(d, 0, w.shape[d] - 2))  # noqa: E731
        gx = smooth(smooth(diff(v, 2), 1), 0)
        gy = smooth(smooth(diff(v, 1), 2), 0)
        gz = smooth(smooth(diff(v, 0), 2), 1)
        return [w.reshape(-1) for w in (gx, gy, gz)]

    def _force(self, rho):
        m, g = self.p["force_mode"], self.p["g"]
        if m == 0:
            return [0.0, 0.0, 0.0]
        ref = 0.5 * (self.p["rho_r0"] + self.p["rho_b0"]) if m == 1 else self.p["rho_b0"]
        return [(rho - ref) * g[a] for a in range(3)]

    def macro(self):
        r, b = self.f[0].sum(0), self.f[1].sum(0)
        rho = r + b
        F = self._force(rho)
        u = []
        for a in range(3):
            j = 0.5 * F[a]
            for i, c in enumerate(_C):
                if c[a]:
                    j = j + c[a] * (self.f[0, i] + self.f[1, i])
            u.append(j / rho)
        nx, ny, nz = self.shape
        return r.view(nz, ny, nx), b.view(nz, ny, nx), torch.stack(u).view(3, nz, ny, nx)

    def diag(self):
        r, b, _ = self.macro()
        phi = (r - b) / (r + b)
        z = torch.arange(self.shape[2], **self.dev)[:, None, None].expand_as(phi).clone()
        nxt = phi[1:]
        cross = (phi[:-1] > 0) & (nxt <= 0)
        z[:-1] = torch.where(cross, z[:-1] + phi[:-1] / (phi[:-1] - nxt), z[:-1])
        le = torch.where(phi > 0, z, torch.full_like(z, -1.0)).max()
        return [float(r.sum()), float(b.sum()), float(le)]

    def step(self):
        p, nx, ny, nz = self.p, *self.shape
        r, b = self.f[0].sum(0), self.f[1].sum(0)
        if self.inlet is not None:
            r[self.inlet], b[self.inlet] = p["rho_r0"], 0.0
        rho = r + b
        phi = (r - b) / rho
        gphi, grho = self._gradient(phi), self._gradient(rho)
        f = self.f[0] + self.f[1]
        F = self._force(rho)
        u = [(sum(c[a] * f[i] for i, c in enumerate(_C) if c[a]) + 0.5 * F[a]) / rho for a in range(3)]
        nu = 0.5 * (1.0 + phi) * p["nu_r"] + 0.5 * (1.0 - phi) * p["nu_b"]
        shear = 1.0 / (3.0 * nu + 0.5)
        ug = sum(u[a] * grho[a] for a in range(3))
        uF = sum(u[a] * F[a] for a in range(3))
        h = f - self._feq(r, u, self.ar) - self._feq(b, u, self.ab)
        force = torch.empty_like(f)
        for i, c in enumerate(_C):
            cg = sum(c[a] * grho[a] for a in range(3))
            cu = sum(c[a] * u[a] for a in range(3))
            cF = sum(c[a] * F[a] for a in range(3))
            h[i] -= nu * (-3.0 * ug if c == (0, 0, 0) else 9.0 * _W[i] * cu * cg)  # Eq. (Phi), the colours summed
            force[i] = _W[i] * (3.0 * (cF - uF) + 9.0 * cu * cF)
        # f* = f - M^-1 K M (f - feq) + M^-1 (I - K/2) M F' + perturbation; the rows of the shear slots per node
        m = self.M @ h + 0.5 * (self.M @ force)
        for j, k in enumerate(SLOT):
            m[j] *= shear if k in (6, 8) else (0.0 if k == 1 else p["s"][j])
        f = f - self.Mi @ m + force
        del h, force, m
        g2 = gphi[0] ** 2 + gphi[1] ** 2 + gphi[2] ** 2
        on = g2 > 1e-24
        inv = torch.where(on, 1.0 / torch.sqrt(torch.where(on, g2, torch.ones_like(g2))), torch.zeros_like(g2))
        nrm = [g * inv for g in gphi]
        ag = p["A"] * g2 * inv
        abar = 0.5 * (1.0 + phi) * self.ar + 0.5 * (1.0 - phi) * self.ab
        coef = p["beta"] * r * b / rho * (27.0 / 19.0) * (1.0 - abar)
        new = torch.zeros_like(self.f)
        for i, c in enumerate(_C):
            cn = sum(c[a] * nrm[a] for a in range(3))
            length = math.sqrt(c[0] ** 2 + c[1] ** 2 + c[2] ** 2)
            f[i] += ag * (_W[i] * cn * cn - (-10.0 / 27.0 if length == 0 else _W[i]))  # ag = 0 where there is no normal
            red = r / rho * f[i] + (coef * _W[i] * cn / length if length else 0.0)
            blue = f[i] - red
            if self.inlet is not None:
                red[self.inlet], blue[self.inlet] = self._inlet(i), 0.0
            dst, keep = self._target(c)
            for k, v in ((0, red), (1, blue)):
                flat = new[k].view(-1)
                if keep is None:
                    flat[dst] = v
                else:
                    flat[dst[keep]] = v[keep]
        self.f = new
        if p["bc"][5] == OUTFLOW:
            below = new[:, :, -2 * self.plane:-self.plane]
            tot = below.sum(0)
            rho = tot.sum(0)
            mz = sum(c[2] * tot[i] for i, c in enumerate(_C) if c[2])
            lam = ((mz + 0.5 * self._force(rho)[2]) / rho).clamp(min=0.0)
            self.top = (self.top + lam * below) / (1.0 + lam)
            new[:, :, -self.plane:] = self.top
        self.t += 1

    def _inlet(self, i):
        p, q = self.p, self.p["inflow"]
        u = []
        for a in range(3):
            with np.errstate(over="ignore"):
                h = _splitmix(np.full(1, p["seed"], dtype=np.uint64))
                h = _splitmix(h ^ np.uint64(self.t))
                h = _splitmix(_splitmix(h ^ self.inlet_np.astype(np.uint64)) ^ np.uint64(a))
            xi = (h >> np.uint64(11)).astype(np.float64) * 2.0 ** -53 * 2.0 - 1.0
            u.append((q["u_j0"] if a == 2 else 0.0) + q["u_j0"] * q["noise_frac"] * xi)
        c = _C[i]
        cu, uu = c[0] * u[0] + c[1] * u[1] + c[2] * u[2], u[0] ** 2 + u[1] ** 2 + u[2] ** 2
        vphi = self.ar if c == (0, 0, 0) else 27.0 / 19.0 * (1.0 - self.ar) * _W[i]
        return torch.tensor(p["rho_r0"] * (vphi + _W[i] * (3.0 * cu + 4.5 * cu * cu - 1.5 * uu)), **self.dev)

    def _target(self, c):
        """Flat index (direction * nodes + node) where what leaves each node along c arrives; None, or the
        nodes from which it stays in the box (not through the outflow)."""
        nx, ny, nz = self.shape
        full = (nz, ny, nx)
        at, cc, bounce, leave = [], [], torch.zeros(full, dtype=torch.bool, device=self.dev["device"]), None
        for a, n in enumerate(self.shape):
            q, ca = self.pos[a] + c[a], torch.full_like(self.pos[a], c[a])
            outside = (q < 0) | (q >= n)
            kind = self.p["bc"][2 * a + (1 if c[a] > 0 else 0)]
            if kind == PERIODIC:
                q = q % n
            elif c[a]:
                if kind == NOSLIP:
                    bounce = bounce | outside
                elif kind == OUTFLOW:
                    leave = outside.expand(full).reshape(-1)
                else:
                    ca = torch.where(outside, -ca, ca)
                q = torch.where(outside, self.pos[a], q)
            at.append(q)
            cc.append(ca)
        node = at[0] + nx * (at[1] + ny * at[2])
        own = self.pos[0] + nx * (self.pos[1] + ny * self.pos[2])
        j = (cc[0] + 1) + 3 * (cc[1] + 1) + 9 * (cc[2] + 1)
        opp = (1 - c[0]) + 3 * (1 - c[1]) + 9 * (1 - c[2])
        dst = torch.where(bounce, opp * self.n + own, j * self.n + node).reshape(-1)
        return dst, (None if leave is None else ~leave)


def _exact_net(case, seed):
    x, target, label, flat = (torch.from_numpy(v) for v in _net_inputs(case, seed))
    sizes, ps, o = list(zip([N_IN] + [WIDTH] * DEPTH, [WIDTH] * DEPTH + [N_POS + N_CLS])), [], 0
    for a, b in sizes:
        ps += [flat[o:o + a * b].double().view(b, a).clone().requires_grad_(True), flat[o + a * b:o + a * b + b].double().clone().requires_grad_(True)]
        o += a * b + b

    def net(v):
        h = v.double()
        for k in range(0, len(ps), 2):
            h = h @ ps[k].t() + ps[k + 1]
            if k + 2 < len(ps):
                h = h * torch.sigmoid(h)
        return h

    def loss(k):
        y = net(x[k])
        ce = torch.nn.functional.cross_entropy(y[:, N_POS:], label[k].long())
        return ((y[:, :N_POS] - target[k].double()) ** 2).mean() + 0.2 * ce

    if case["kind"] == "forward":
        with torch.no_grad():
            return net(x[0])
    if case["kind"] == "grad":
        v = loss(0)
        v.backward()
        return float(v.detach()), torch.cat([q.grad.reshape(-1) for q in ps])
    opt = torch.optim.Adam(ps, lr=LR, betas=(0.9, 0.999), eps=1e-8)
    losses = []
    for k in range(int(case["steps"])):
        opt.zero_grad()
        v = loss(k)
        v.backward()
        losses.append(float(v.detach()))
        opt.step()
    return np.array(losses), torch.cat([q.detach().reshape(-1) for q in ps])


def exact(case, seed, device="cuda"):
    if case["kind"] in ("forward", "train", "grad"):
        return _exact_net(case, seed)
    if _nodes(case) * case["steps"] > 48 * 128 * 128 * 512:  # more than about 20 seconds
        return None
    out = []
    for shape, p, fields in _jets(case, seed):
        box = _Exact(shape, p, fields, device)
        del fields
        got = []
        each = case["steps"] // case.get("samples", 1)
        for k in range(each * case.get("samples", 1) + (1 if case["kind"] == "sweep" else 0)):
            box.step()
            if case.get("samples", 1) > 1 and (k + 1) % each == 0:
                got.append(box.diag())
        out.append((box.macro(), box.diag()) if case["kind"] == "sweep" else (box.macro(), got))
    return out if case["kind"] == "sweep" else out[0]
