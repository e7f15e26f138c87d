"""The work a user of this library has it do, as timed cases through its public entry points.

Most cases advance a plasma: MIXED32 and FP64 particles, shape orders 1 to 3, periodic
boxes and the walled, fed shock, one simulation or a batch, the implicit and the explicit
field update, both gather readings and the three initial guesses of the solve. The others
are what surrounds a run: loading it from host arrays, its diagnostics, the training of the
learned initial guess and the stand-alone field solve. Sizes are those of the benchmark's
workloads, the parameter scan and the experiments, or lie between them.

Inputs are made on the GPU from the seed alone: the drifting pair plasma of inputs.py (the
same recipe, drawn by torch) in smooth seeded fields, so that gather, push, deposit and
solve all have something to do in the first step already.
"""
import math

import numpy as np
import torch

import paper_1412_2480_gb300 as pic
from paper_1412_2480_gb300 import inputs

PI = math.pi
SKIN_DEPTH = 10.0  # c / omega_pe in cells, as in every configuration of the repository

# What a "step" case may leave out, and what it then is (pic_params_default's values, mostly).
STEP = {"kind": "step", "precision": "mixed32", "order": 2, "cfl": 1.0, "theta": 0.5, "gamma0": 20.0,
        "u_th": 1e-3, "ppc": 16, "rtol": 1e-10, "walls": False, "fill": 1.0, "sigma_b": 0.0,
        "explicit": False, "nodal": False, "warm": "zero", "amplitude": 0.02, "colocated": True, "steps": 1}


def listed():
    return [
        # the first configuration (64 x 64, order 1, 8 per cell): the smallest run, all
        # latency and launches; twenty steps between two looks at the fields
        dict(STEP, name="step_64x64", nx=64, ny=64, order=1, ppc=8, steps=20),
        # the theta scan of experiments.py: a hot, dense plasma on a small grid, thousands
        # of steps at a loose solver tolerance
        dict(STEP, name="step_128x128_hot", nx=128, ny=128, ppc=100, gamma0=100.0, u_th=0.1, theta=0.501,
             rtol=1e-8, steps=5),
        # the production size and the benchmark's default workload: 67 million particles
        dict(STEP, name="step_2048x512", nx=2048, ny=512, ppc=32, gamma0=40.0),
        # the shock at its full configured size: third order, magnetised beam, walls, injector
        dict(STEP, name="shock_8192x512_order3", nx=8192, ny=512, order=3, gamma0=40.0, theta=0.501,
             walls=True, fill=0.5, sigma_b=0.1),
        # the Sec. 4 shock of experiments.py (5650 x 990, 50 per cell) at a quarter of its
        # size per direction: both sides ragged, unmagnetised, CFL 1/2
        dict(STEP, name="shock_1413x247", nx=1413, ny=247, ppc=50, gamma0=100.0, u_th=0.05, theta=0.501,
             cfl=0.5, walls=True, fill=0.6),
        # the parameter scan: uneven simulations of every order in one handle (the first
        # twelve rows of its table), two steps per call
        {"name": "scan_12", "kind": "scan", "first": 0, "count": 12, "steps": 2},
        # the plain FP64 form, the library's default precision, with the particles read back
        dict(STEP, name="fp64_256x128", nx=256, ny=128, precision="fp64", steps=2),
        # the learned initial guess on the grid it is configured for
        dict(STEP, name="learned_1024x256", nx=1024, ny=256, order=1, ppc=8, warm="learned", steps=2),
        # a run as it begins: fields and particles from host arrays, a first (explicit)
        # step, fields and species densities back to the host
        {"name": "setup_512x256", "kind": "setup", "nx": 512, "ny": 256, "ppc": 8, "order": 2, "cfl": 0.5,
         "gamma0": 20.0, "u_th": 1e-3, "explicit": True, "amplitude": 0.02},
        # what a run looks at between its steps: spectrum of B_z, densities, conservation
        {"name": "diagnostics_1024x256", "kind": "diagnostics", "nx": 1024, "ny": 256, "ppc": 16, "order": 2,
         "gamma0": 40.0, "u_th": 1e-3, "amplitude": 0.02},
        # one step of the training of the learned guess: the batch that warmstart.train takes
        {"name": "cnn_train_8x64x64", "kind": "train", "nimg": 8, "nx": 64, "ny": 64},
        # the stand-alone field solve at its largest grid
        {"name": "field_solve_256x256", "kind": "solve", "nx": 256, "ny": 256, "cfl": 1.0, "theta": 0.5},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, lo, hi):
    """A grid of lo to hi cells: multiples of 16, 4 and 2, and odd sides."""
    cells, aspect = _log_int(rng, lo, hi), math.exp(rng.uniform(0.0, math.log(8.0)))
    m = rng.choice((16, 4, 2, 1))
    nx = max(16, int(math.sqrt(cells * aspect)) // m * m)
    ny = max(16, int(math.sqrt(cells / aspect)) // rng.choice((m, 1)))
    return nx, max(16, ny if cells // nx < 16 else cells // nx)


def draw(rng):
    kind = rng.choices(("step", "scan", "setup", "diagnostics", "train", "solve"), (12, 2, 2, 2, 2, 2))[0]
    if kind == "scan":
        return {"kind": "scan", "first": rng.randrange(0, 36), "count": rng.randint(2, 12), "steps": rng.randint(1, 4)}
    if kind == "train":
        n = rng.choice((32, 64, 96, 128))
        return {"kind": "train", "nimg": rng.randint(1, 16), "nx": n, "ny": rng.choice((32, 64, 96, 128))}
    if kind == "solve":
        nx, ny = _grid(rng, 256, 60000)
        return {"kind": "solve", "nx": nx, "ny": ny, "cfl": rng.choice(inputs.SCAN_CFL), "theta": rng.choice(inputs.SCAN_THETA)}
    if kind == "setup":
        nx, ny = _grid(rng, 4096, 400000)
        return {"kind": "setup", "nx": nx, "ny": ny, "ppc": rng.randint(2, 12), "order": rng.randint(1, 3),
                "cfl": rng.choice((0.5, 0.7)), "gamma0": 20.0, "u_th": rng.choice((1e-3, 0.1)),
                "explicit": rng.random() < 0.5, "amplitude": 0.02}
    if kind == "diagnostics":
        nx, ny = _grid(rng, 4096, 400000)
        return {"kind": "diagnostics", "nx": nx, "ny": ny, "ppc": rng.randint(2, 24), "order": rng.randint(1, 3),
                "gamma0": 40.0, "u_th": rng.choice((1e-3, 0.1)), "amplitude": 0.02}
    fp64 = rng.random() < 0.25
    nx, ny = _grid(rng, 4096, 120000 if fp64 else 1500000)
    ppc = min(_log_int(rng, 4, 100), max(2, (3000000 if fp64 else 30000000) // (2 * nx * ny)))
    walls = rng.random() < 0.25
    explicit = not walls and rng.random() < 0.2
    # (the walled box is fed at the end of each step: one step per call, as its own loop
    # over the injector's schedule takes them)
    c = dict(STEP, nx=nx, ny=ny, ppc=ppc, precision="fp64" if fp64 else "mixed32", order=rng.randint(1, 3),
             cfl=rng.choice((0.5, 0.6, 0.7)) if explicit else rng.choice(inputs.SCAN_CFL),
             theta=rng.choice((0.5, 0.501, 0.55, 0.6, 0.75)), gamma0=rng.choice((20.0, 40.0, 100.0)),
             u_th=rng.choice((1e-3, 0.05, 0.1)), walls=walls, explicit=explicit,
             nodal=not walls and rng.random() < 0.2,
             steps=1 if walls or nx * ny * ppc > 500000 else rng.randint(1, 10))
    if walls:
        c.update(fill=round(rng.uniform(0.4, 0.8), 2), sigma_b=rng.choice((0.0, 0.1)))
    elif not fp64 and not explicit and rng.random() < 0.3:
        c["warm"] = "previous"
    return c


# ---- inputs ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _smooth(nx, ny, n, amplitude, g, modes=4):
    """n smooth fields (n, ny, nx): a few random Fourier modes each."""
    i = torch.arange(nx, dtype=torch.float64, device="cuda") * (2 * PI / nx)
    j = torch.arange(ny, dtype=torch.float64, device="cuda") * (2 * PI / ny)
    out = torch.zeros(n, ny, nx, dtype=torch.float64, device="cuda")
    k = torch.randint(-4, 5, (n, modes, 2), generator=g, device="cuda").double()
    a = torch.randn(n, modes, generator=g, dtype=torch.float64, device="cuda") * amplitude
    ph = torch.rand(n, modes, generator=g, dtype=torch.float64, device="cuda") * 2 * PI
    for c in range(n):
        for m in range(modes):
            out[c] += a[c, m] * torch.cos((k[c, m, 0] * i)[None, :] + (k[c, m, 1] * j)[:, None] + ph[c, m])
    return out


def _plasma(nx, ny, ppc, gamma0, u_th, g, sign=1.0, colocated=True):
    """Two species (5, n) [x, y, ux, uy, uz] of pairs drifting along x, cell by cell: co-located
    at the start of a run, each species at its own places later on."""
    n = nx * ny * ppc
    cell = torch.arange(nx * ny, device="cuda").repeat_interleave(ppc)
    x = (cell % nx) + torch.rand(n, generator=g, dtype=torch.float64, device="cuda")
    y = torch.div(cell, nx, rounding_mode="floor") + torch.rand(n, generator=g, dtype=torch.float64, device="cuda")
    beta = math.sqrt(1.0 - 1.0 / gamma0 ** 2)
    species = []
    for s in range(2):
        if s and not colocated:
            x = torch.floor(x) + torch.rand(n, generator=g, dtype=torch.float64, device="cuda")
            y = torch.floor(y) + torch.rand(n, generator=g, dtype=torch.float64, device="cuda")
        u = torch.randn(3, n, generator=g, dtype=torch.float64, device="cuda") * u_th
        ux = sign * gamma0 * (u[0] + beta * torch.sqrt(1.0 + (u * u).sum(0)))
        species.append(torch.stack((x, y, ux, u[1], u[2])))
    return species


def _fields(c, g):
    F = _smooth(c["nx"], c["ny"], 6, c["amplitude"], g)
    if c.get("walls"):
        if c["sigma_b"] > 0:  # the magnetised beam: uniform Bz and its motional Ey
            b0 = c["gamma0"] / SKIN_DEPTH * math.sqrt(2.0 * c["sigma_b"])
            F[5] += b0
            F[1] -= math.sqrt(1.0 - 1.0 / c["gamma0"] ** 2) * b0
        F[1:4, :, 0] = 0.0  # a conductor's wall nodes
    return F


def _box(c, seed):
    """Fields (6, ny, nx) and species of one simulation."""
    g = _gen(seed)
    F = _fields(c, g)
    filled = int(c["nx"] * c.get("fill", 1.0))
    return F, _plasma(filled, c["ny"], c["ppc"], c["gamma0"], c["u_th"], g, -1.0 if c["walls"] else 1.0,
                      c["colocated"])


def _scan_rows(c):
    rows = inputs.scan_table(48)[c["first"]: c["first"] + c["count"]]
    return [dict(STEP, nx=r["nx"], ny=r["ny"], order=r["order"], cfl=r["cfl"], theta=r["theta"], gamma0=r["gamma0"],
                 ppc=r["ppc"], u_th=r["u_th"], steps=c["steps"]) for r in rows]


def _params(c):
    flags = (pic.PIC_EXPLICIT if c["explicit"] else 0) | (pic.PIC_GATHER_NODAL if c["nodal"] else 0)
    warm = {"zero": pic.PIC_WS_ZERO, "previous": pic.PIC_WS_PREV, "learned": pic.PIC_WS_LEARNED}[c["warm"]]
    return pic.pic_params_default(
        nx=c["nx"], ny=c["ny"], cfl=c["cfl"], theta=c["theta"], shape_order=c["order"], gamma0=c["gamma0"],
        ppc=c["ppc"], precision=pic.PIC_FP64 if c["precision"] == "fp64" else pic.PIC_MIXED32, cg_rtol=c["rtol"],
        warm_start=warm, flags=flags, bc_x=pic.PIC_BC_WALLS if c["walls"] else pic.PIC_BC_PERIODIC,
        inject_x0=float(int(c["nx"] * c["fill"])) if c["walls"] else -1.0, u_th=c["u_th"], seed=105)


def _network(cfl, theta):
    """Parameters of a network that applies the first five terms of the Neumann series of
    A^-1 (each layer carries b and the partial sum), as a trained one comes close to."""
    cx = (theta * cfl) ** 2
    c0 = 1.0 + 4.0 * cx
    p, o = [], 0
    for layer, (cin, cout) in enumerate(((3, 32), (32, 32), (32, 32), (32, 3))):
        W = np.zeros((cout, 9, cin), dtype=np.float32)
        for k in range(3):
            s = k if layer == 0 else 3 + k    # the partial sum's channel in the input
            to = k if layer == 3 else 3 + k   # ... and in the output
            scale = 1.0 / c0 if layer == 3 else 1.0
            if layer < 3:
                W[k, 4, k] = 1.0
            W[to, 4, k] += scale
            for tap in (1, 3, 5, 7):
                W[to, tap, s] += scale * cx / c0
        p += [W.ravel(), np.zeros(cout, dtype=np.float32)]
    return np.concatenate(p)


class _Sim:
    """A handle, what the calls on it need, and the buffers the fields are read into."""

    def __init__(self, rows):
        self.rows, self.net, self.h = rows, None, None
        prm = [_params(c) for c in rows]
        self.h = pic.pic_init(prm[0]) if len(prm) == 1 else pic.pic_init_batch(prm)
        self.out = [torch.empty(9, c["nx"] * c["ny"], dtype=torch.float64, device="cuda") for c in rows]

    def load(self, k, F, species):
        pic.pic_select(self.h, k)
        torch.cuda.synchronize()
        for comp in range(6):
            pic.pic_set_fields(self.h, comp, F[comp].reshape(-1))
        for s, d in enumerate(species):
            pic.pic_load_particles(self.h, s, *(d[a] for a in range(5)))

    def __del__(self):
        if self.h:
            pic.pic_free(self.h)
        if self.net:
            pic.pic_cnn_free(self.net)


class _Net:
    def __init__(self, params):
        self.c = pic.pic_cnn_create()
        pic.pic_cnn_set_params(self.c, params)

    def __del__(self):
        pic.pic_cnn_free(self.c)


def _full(c):
    """The setup and diagnostics cases as a step case's dict."""
    return dict(STEP, colocated=c["kind"] != "diagnostics", **{k: v for k, v in c.items() if k not in ("kind", "name")})


def _solve_inputs(c, seed):
    g = _gen(seed)
    nx, ny = c["nx"], c["ny"]
    F = _smooth(nx, ny, 6, 0.05, g) + 0.005 * torch.randn(6, ny, nx, generator=g, dtype=torch.float64, device="cuda")
    J = 1e-3 * torch.randn(3, ny, nx, generator=g, dtype=torch.float64, device="cuda")
    return F, J


def _train_inputs(c, seed):
    """A batch of (b, dB) / rms(b) pairs of Eq. (7) at CFL 1, theta 1/2, as host arrays."""
    rng = np.random.Generator(np.random.Philox(int(seed)))
    b = rng.standard_normal((c["nimg"], 3, c["ny"], c["nx"]))
    k = np.fft.fftfreq(c["nx"]) ** 2 + np.fft.fftfreq(c["ny"])[:, None] ** 2
    b = np.fft.ifft2(np.fft.fft2(b) / (1.0 + 40.0 * k)).real  # currents of extended particles
    b /= np.sqrt((b * b).mean(axis=(1, 2, 3), keepdims=True))
    lam = 1.0 + 0.25 * (4.0 - 2.0 * np.cos(2 * PI * np.fft.fftfreq(c["nx"])) - 2.0 * np.cos(2 * PI * np.fft.fftfreq(c["ny"]))[:, None])
    x = np.fft.ifft2(np.fft.fft2(b) / lam).real
    return b.astype(np.float32), x.astype(np.float32)


def _train_params(seed):
    """Weights a tenth of the way into a training: the series network and noise."""
    rng = np.random.Generator(np.random.Philox(int(seed) + 1))
    return (_network(1.0, 0.5) + 0.03 * rng.standard_normal(pic.PIC_CNN_NPARAMS)).astype(np.float32)


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("step", "scan"):
        rows = [case] if kind == "step" else _scan_rows(case)
        sim = _Sim(rows)
        for k, c in enumerate(rows):
            sim.load(k, *_box(c, seed * 64 + k))
        if rows[0]["warm"] == "learned":
            sim.net = pic.pic_cnn_create()
            pic.pic_cnn_set_params(sim.net, _network(case["cfl"], case["theta"]))
            pic.pic_set_cnn(sim.h, sim.net)
        if rows[0]["precision"] == "fp64":
            sim.particles = [torch.empty(5, pic.pic_particle_count(sim.h, s), dtype=torch.float64, device="cuda")
                             for s in range(2)]
        return {"kind": "step", "sim": sim, "steps": case["steps"]}
    if kind == "setup":
        F, species = _box(_full(case), seed * 64)
        return {"kind": kind, "sim": _Sim([_full(case)]), "F": [f.reshape(-1).cpu().numpy() for f in F],
                "species": [[a.cpu().numpy() for a in d] for d in species]}
    if kind == "diagnostics":
        sim = _Sim([_full(case)])
        sim.load(0, *_box(_full(case), seed * 64))
        return {"kind": kind, "sim": sim}
    if kind == "train":
        return {"kind": kind, "net": _Net(_train_params(seed)), "pairs": _train_inputs(case, seed)}
    F, J = _solve_inputs(case, seed)
    return {"kind": kind, "case": dict(case), "F": F.reshape(-1), "J": J.reshape(-1), "dB": torch.empty_like(J).reshape(-1)}


# ---- one pass -------------------------------------------------------------------------

def run(state):
    kind = state["kind"]
    if kind == "step":
        return _run_step(state["sim"], state["steps"])
    if kind == "setup":
        return _run_setup(state)
    if kind == "diagnostics":
        return _run_diagnostics(state["sim"])
    if kind == "train":
        net = state["net"].c
        loss = pic.pic_cnn_train_step(net, *state["pairs"], lr=2e-3)
        return {"loss": loss, "params": pic.pic_cnn_get_params(net)}
    c = state["case"]
    pic.pic_field_solve_noalloc(c["nx"], c["ny"], 1.0, 1.0, c["cfl"], c["theta"], 1e-10, 200, state["F"], state["J"],
                                state["dB"])
    return {"dB": state["dB"]}


def _run_step(sim, steps):
    """Advance, then read E, B and J of every simulation, and FP64 particles, whose order is
    the caller's. MIXED32 keeps its particles in an order of its own that differs between
    runs; every one of them is in J, its momentum in that of the next step."""
    pic.pic_step(sim.h, steps)
    counts = []
    for k in range(len(sim.rows)):
        if len(sim.rows) > 1:
            pic.pic_select(sim.h, k)
        for which in range(9):
            pic.pic_fields(sim.h, which, sim.out[k][which])
        counts += [pic.pic_particle_count(sim.h, s) for s in range(2)]
    got = {"fields": [o[:6] for o in sim.out], "currents": [o[6:] for o in sim.out], "counts": np.array(counts)}
    if hasattr(sim, "particles"):
        if sim.particles[0].shape[1] != counts[0]:  # the injector adds pairs
            sim.particles = [torch.empty(5, n, dtype=torch.float64, device="cuda") for n in counts]
        order_kept = not sim.rows[0]["walls"]
        got["particles"] = [pic.pic_particles(sim.h, s, sim.particles[s]) for s in range(2)] if order_kept else []
    return got


def _run_setup(state):
    sim, c = state["sim"], state["sim"].rows[0]
    for comp in range(6):
        pic.pic_set_fields(sim.h, comp, state["F"][comp])
    for s, d in enumerate(state["species"]):
        pic.pic_load_particles(sim.h, s, *d)
    pic.pic_step(sim.h, 1)
    read = lambda which: pic.fields_numpy(sim.h, which, c["nx"], c["ny"])  # noqa: E731
    return {"fields": np.stack([read(k) for k in range(6)]), "currents": np.stack([read(6 + k) for k in range(3)]),
            "density": np.stack([read(pic.PIC_DENSITY_P), read(pic.PIC_DENSITY_E)])}


def _run_diagnostics(sim):
    c = sim.rows[0]
    cons = pic.pic_conservation(sim.h)
    read = lambda which: pic.fields_numpy(sim.h, which, c["nx"], c["ny"])  # noqa: E731
    return {"spectrum": pic.pic_spectrum(sim.h, pic.PIC_BZ, c["nx"], c["ny"]), "rho": read(pic.PIC_RHO),
            "density": np.stack([read(pic.PIC_DENSITY_P), read(pic.PIC_DENSITY_E)]),
            "momentum": np.array(cons["momentum"]), "gauss": np.array([cons["gauss_max"], cons["gauss_rms"]])}


# ---- what a pass cannot do without ------------------------------------------------------

def _step_work(c):
    """Per particle: its state in and out; per cell: E and B in and out, J and, for the
    implicit update, dB out; and what is read back. Operations of every step: 6 components
    gathered, the push, the deposit, the field update."""
    n, cells, p = 2 * int(c["nx"] * c["fill"]) * c["ny"] * c["ppc"], c["nx"] * c["ny"], c["order"]
    value = 80 if c["precision"] == "fp64" else 48
    flops = 6 * 2 * (p + 1) * (p + 2) + 4 * 8 * (p + 1) + 100 + 3 * 3 * (p + 2) ** 2
    field = 60 if c["explicit"] else 400
    reread = 9 * 8 * 2 * cells + (2 * 40 * n * 2 if c["precision"] == "fp64" and not c["walls"] else 0)
    return {"bytes": value * n + (96 + 24 + (0 if c["explicit"] else 24)) * cells + reread,
            "flops": c["steps"] * (flops * n + field * cells)}


def work(case):
    kind = case["kind"]
    if kind == "step":
        return _step_work(case)
    if kind == "scan":
        w = [_step_work(c) for c in _scan_rows(case)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    n = case["nx"] * case["ny"]
    if kind == "setup":
        c = _full(case)
        w = _step_work(c)
        return {"bytes": w["bytes"] + (40 + 24) * 2 * n * c["ppc"] + 48 * n + 16 * n, "flops": w["flops"]}
    if kind == "diagnostics":  # the particles three times (their momenta once), FFT, grids
        return {"bytes": (3 * 12 + 12) * 2 * n * case["ppc"] + 8 * n * 8, "flops": 5 * n * math.log2(n) + 2 * n * case["ppc"] * 3 * 30}
    if kind == "train":
        px = case["nimg"] * n
        macs = 9 * (3 * 32 + 2 * 32 * 32 + 32 * 3)
        return {"bytes": 24 * px + 5 * 4 * pic.PIC_CNN_NPARAMS, "flops": 2 * macs * px * 3}
    return {"bytes": (9 + 3) * 8 * n, "flops": 3 * 12 * 20 * n}


# ---- the same results in 64 bits, in plain torch -------------------------------------------

def _spline(order, d):
    d = d.abs()
    if order == 1:
        return (1.0 - d).clamp(min=0.0)
    if order == 2:
        return torch.where(d < 0.5, 0.75 - d * d, 0.5 * (1.5 - d).clamp(min=0.0) ** 2)
    return torch.where(d < 1.0, (4.0 - 6.0 * d * d + 3.0 * d ** 3) / 6.0, (2.0 - d).clamp(min=0.0) ** 3 / 6.0)


def _nodes(order, X, width):
    """First node and weights of the `width` nodes from it."""
    b = torch.floor(X - 0.5 * (order - 1))
    k = torch.arange(width, dtype=torch.float64, device=X.device)
    return b, _spline(order, X[:, None] - b[:, None] - k)


def _image(i, nx, half, odd, walls):
    """Stored column and sign of node i: periodic, or the images at two walls."""
    if not walls:
        return i % nx, None
    if half:
        s = torch.where((i < 0) | (i >= nx), -1.0, 1.0).double()
        col = torch.where(i < 0, -i - 1, torch.where(i >= nx, 2 * nx - i - 1, i))
    else:
        s = torch.where((i < 0) | (i > nx), -1.0, 1.0).double()
        col = torch.where(i < 0, -i, torch.where(i > nx, 2 * nx - i, i))
        s = torch.where((col == nx) | (odd & (col == 0)), 0.0, s)
        col = torch.where(col >= nx, 0, col)
    return col, s if odd else s.abs()


HALF = ((True, False), (False, True), (False, False), (False, True), (True, False), (True, True))  # Ex .. Bz in x, y


class _Exact:
    def __init__(self, c, seed):
        self.c = c
        self.nx, self.ny, self.dt, self.theta = c["nx"], c["ny"], c["cfl"], 1.0 if c["explicit"] else c["theta"]
        self.F, self.species = _box(c, seed)
        self.w = c["gamma0"] / SKIN_DEPTH ** 2 / (4 * PI * c["ppc"])
        self.J = None

    # neighbours: the last axis is x; `odd`: a quantity on the integer-x lattice
    def east(self, v, odd):
        e = torch.roll(v, -1, 1)
        if self.c["walls"]:
            e[:, -1] = 0.0 if odd else v[:, -1]
        return e

    def west(self, v, odd):
        w = torch.roll(v, 1, 1)
        if self.c["walls"]:
            w[:, 0] = -v[:, 1] if odd else v[:, 0]
        return w

    def curl_E(self, V, J=False):
        x, y, z = V[0], V[1].clone(), V[2].clone()
        if self.c["walls"]:
            y[:, 0] = z[:, 0] = 0.0
        n = lambda v: torch.roll(v, -1, 0)  # noqa: E731
        return torch.stack((n(z) - z, -(self.east(z, True) - z), self.east(y, True) - y - (n(x) - x)))

    def curl_B(self, V):
        x, y, z = V
        s = lambda v: torch.roll(v, 1, 0)  # noqa: E731
        return torch.stack((z - s(z), -(z - self.west(z, False)), y - self.west(y, False) - (x - s(x))))

    def laplacian(self, V):
        return torch.stack([self.east(v, k == 0) + self.west(v, k == 0) + torch.roll(v, 1, 0) + torch.roll(v, -1, 0) - 4 * v
                            for k, v in enumerate(V)])

    def invert(self, b):
        """(1 - (theta dt)^2 Lap) x = b by Fourier transforms, of the images' extension at walls."""
        out = []
        for k, v in enumerate(b):
            if self.c["walls"]:
                if k == 0:
                    z = torch.zeros_like(v[:, :1])
                    v = torch.cat((z, v[:, 1:], z, -v[:, 1:].flip(1)), 1)
                else:
                    v = torch.cat((v, v.flip(1)), 1)
            kx = torch.fft.fftfreq(v.shape[1], dtype=torch.float64, device=v.device) * 2 * PI
            ky = torch.fft.fftfreq(v.shape[0], dtype=torch.float64, device=v.device) * 2 * PI
            lam = 1.0 + (self.theta * self.dt) ** 2 * (4.0 - 2 * torch.cos(kx)[None, :] - 2 * torch.cos(ky)[:, None])
            out.append(torch.fft.ifft2(torch.fft.fft2(v) / lam).real[:, : self.nx])
        return torch.stack(out)

    def gathered(self):
        """The fields the particles see, and their lattices."""
        F = self.F
        if not self.c["nodal"]:
            return F, HALF
        w, s = (lambda v: torch.roll(v, 1, 1)), (lambda v: torch.roll(v, 1, 0))
        ax, ay = (lambda v: 0.5 * (v + w(v))), (lambda v: 0.5 * (v + s(v)))
        return torch.stack((ax(F[0]), ay(F[1]), F[2], ay(F[3]), ax(F[4]), ax(ay(F[5])))), ((False, False),) * 6

    def push(self):
        c, nx, ny, P, dt, walls = self.c, self.nx, self.ny, self.c["order"], self.dt, self.c["walls"]
        J = torch.zeros(3, nx * ny, dtype=torch.float64, device="cuda")
        G, lattice = self.gathered()
        G = G.reshape(6, -1)
        for s, q in enumerate((1.0, -1.0)):
            S = self.species[s]
            n = S.shape[1]
            new = torch.empty_like(S)
            stride = max(1, n // (1 << 20))  # neighbours in a chunk lie in different cells
            for first in range(stride):
                at = slice(first, n, stride)
                X, Y, u = S[0, at], S[1, at], S[2:, at]
                f = []
                for comp in range(6):
                    hx, hy = lattice[comp]
                    bx, wx = _nodes(P, X - 0.5 if hx else X, P + 1)
                    by, wy = _nodes(P, Y - 0.5 if hy else Y, P + 1)
                    k = torch.arange(P + 1, device="cuda")
                    col, sg = _image(bx.long()[:, None] + k, nx, hx, not hx, walls)
                    wx = wx if sg is None else wx * sg
                    row = (by.long()[:, None] + k) % ny
                    v = G[comp][(row[:, :, None] * nx + col[:, None, :])]
                    f.append(((v * wx[:, None, :]).sum(2) * wy).sum(1))
                E, B = torch.stack(f[:3]), torch.stack(f[3:])
                h = 0.5 * q * dt
                um = u + h * E
                t = h * B / torch.sqrt(1 + (um * um).sum(0))
                up = um + torch.linalg.cross(um, t, dim=0)
                up = um + torch.linalg.cross(up, 2 * t / (1 + (t * t).sum(0)), dim=0) + h * E
                v = up / torch.sqrt(1 + (up * up).sum(0))
                X1, Y1 = X + dt * v[0], Y + dt * v[1]
                self.deposit(J, q * self.w, X, Y, X1, Y1, v[2])
                ux = up[0]
                if walls:
                    ux = torch.where((X1 < 0) | (X1 >= nx), -ux, ux)
                    X1 = torch.where(X1 < 0, -X1, torch.where(X1 >= nx, 2.0 * nx - X1, X1))
                else:
                    X1 = X1 % nx
                new[0, at], new[1, at], new[2, at], new[3, at], new[4, at] = X1, Y1 % ny, ux, up[1], up[2]
            self.species[s] = new
        self.J = J.reshape(3, ny, nx)

    def deposit(self, J, q, X0, Y0, X1, Y1, vz):
        """Density decomposition (Esirkepov 2001) on the window of both shapes."""
        nx, ny, P, dt, walls = self.nx, self.ny, self.c["order"], self.dt, self.c["walls"]
        k = torch.arange(P + 2, device="cuda")

        def shapes(a0, a1):
            o = torch.minimum(torch.floor(a0 - 0.5 * (P - 1)), torch.floor(a1 - 0.5 * (P - 1)))
            node = o[:, None] + k
            s0 = _spline(P, a0[:, None] - node)
            return node.long(), s0, _spline(P, a1[:, None] - node) - s0

        ix, S0x, Dx = shapes(X0, X1)
        iy, S0y, Dy = shapes(Y0, Y1)
        row = (iy % ny)[:, :, None] * nx
        wx = -(q / dt) * (S0y + 0.5 * Dy)[:, :, None] * torch.cumsum(Dx, 1)[:, None, :]
        wy = -(q / dt) * torch.cumsum(Dy, 1)[:, :, None] * (S0x + 0.5 * Dx)[:, None, :]
        wz = q * vz[:, None, None] * (S0y[:, :, None] * (S0x + 0.5 * Dx)[:, None, :]
                                      + Dy[:, :, None] * (0.5 * S0x + Dx / 3.0)[:, None, :])
        for comp, value in enumerate((wx, wy, wz)):
            col, sg = _image(ix, nx, comp == 0, comp == 0, walls)
            if sg is not None:
                value = value * sg[:, None, :]
            J[comp].index_add_(0, (row + col[:, None, :]).reshape(-1), value.reshape(-1))

    def step(self):
        dt, th = self.dt, self.theta
        self.push()
        E, B, J = self.F[:3], self.F[3:], self.J
        if self.c["explicit"]:
            half = B - 0.5 * dt * self.curl_E(E)
            E = E + dt * self.curl_B(half) - 4 * PI * dt * J
            if self.c["walls"]:
                E[1:, :, 0] = 0.0
            B = half - 0.5 * dt * self.curl_E(E)
        else:
            x = self.invert(th * dt * dt * (self.laplacian(B) + 4 * PI * self.curl_E(J)) - dt * self.curl_E(E))
            E = E + dt * self.curl_B(B + th * x) - 4 * PI * dt * J
            if self.c["walls"]:
                E[1:, :, 0] = 0.0
            B = B + x
        self.F = torch.cat((E, B))

    def density(self, s):
        c, P = self.c, self.c["order"]
        out = torch.zeros(self.nx * self.ny, dtype=torch.float64, device="cuda")
        bx, wx = _nodes(P, self.species[s][0], P + 1)
        by, wy = _nodes(P, self.species[s][1], P + 1)
        k = torch.arange(P + 1, device="cuda")
        at = ((by.long()[:, None] + k) % self.ny)[:, :, None] * self.nx + ((bx.long()[:, None] + k) % self.nx)[:, None, :]
        out.index_add_(0, at.reshape(-1), (wy[:, :, None] * wx[:, None, :]).reshape(-1))
        return out.reshape(self.ny, self.nx)


def _exact_train(case, seed):
    """Loss and weights after the first Adam step, by automatic differentiation."""
    b, x = (torch.from_numpy(a).double().cuda() for a in _train_inputs(case, seed))
    p = torch.from_numpy(_train_params(seed)).double().cuda().requires_grad_(True)
    y, o = b, 0
    for cin, cout in ((3, 32), (32, 32), (32, 32), (32, 3)):
        W = p[o: o + cout * 9 * cin].reshape(cout, 3, 3, cin).permute(0, 3, 1, 2)
        y = torch.nn.functional.conv2d(torch.nn.functional.pad(y, (1, 1, 1, 1), mode="circular"), W,
                                       p[o + cout * 9 * cin: o + cout * 9 * cin + cout])
        o += cout * 9 * cin + cout
    loss = ((y - x) ** 2).mean()
    loss.backward()
    g = p.grad
    return {"loss": float(loss), "params": (p - 2e-3 * g / (g.abs() + 1e-8)).detach()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "solve":
        F, J = _solve_inputs(case, seed)
        e = _Exact.__new__(_Exact)
        e.c, e.nx, e.ny, e.dt, e.theta = {"walls": False}, case["nx"], case["ny"], case["cfl"], case["theta"]
        b = e.theta * e.dt ** 2 * (e.laplacian(F[3:]) + 4 * PI * e.curl_E(J)) - e.dt * e.curl_E(F[:3])
        return {"dB": e.invert(b).reshape(-1)}
    rows = _scan_rows(case) if kind == "scan" else [case] if kind == "step" else [_full(case)]
    sims = [_Exact(c, seed * 64 + k) for k, c in enumerate(rows)]
    if kind == "diagnostics":
        e = sims[0]
        dens = torch.stack([e.density(s) for s in range(2)])
        rho = e.w * (dens[0] - dens[1])
        r = e.F[0] - torch.roll(e.F[0], 1, 1) + e.F[1] - torch.roll(e.F[1], 1, 0) - 4 * PI * rho
        mom = e.w * sum(s[2:].sum(1) for s in e.species)
        return {"spectrum": torch.fft.fft2(e.F[5]).abs() / (e.nx * e.ny), "rho": rho, "density": dens,
                "momentum": mom, "gauss": torch.stack((r.abs().max(), (r * r).mean().sqrt()))}
    for e in sims:
        for _ in range(e.c["steps"]):
            e.step()
    if kind == "setup":
        e = sims[0]
        return {"fields": e.F, "currents": e.J, "density": torch.stack([e.density(s) for s in range(2)])}
    got = {"fields": [e.F.reshape(6, -1) for e in sims], "currents": [e.J.reshape(3, -1) for e in sims], "counts": None}
    if rows[0]["precision"] == "fp64":
        got["particles"] = [None, None] if rows[0]["walls"] else [s for s in sims[0].species]
    return got
