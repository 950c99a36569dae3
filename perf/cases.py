"""Performance cases of the LBIBCell framework: what its users run, through the
Python binding of the public C interface, over the sizes they run it at.

Kinds of case
  tissue    one tissue advanced by `steps` coupled steps and read back: cells
            on a jittered grid (or a hexagonal packing with walls), springs,
            pressure, morphogen sources; optionally growing under the area
            controller
  loop      the host-driven loop of a cell-biology model: every step uploads
            the cells' pressures and reads positions and areas back beside
            the next step
  turing    the Schnakenberg system on a static cellular domain, the receptor
            confined by the membranes' no-flux closure
  ensemble  many independent tissues advanced together
  steady    batched steady morphogen solves on static tissues
  operator  the learned warm start: Adam steps on a minibatch, then the
            prediction for held-out tissues
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_1503_06726_gb300 import lbib


def listed():
    return [
        # one cell in a small box, full precision: a single-cell study or a
        # parameter fit, where launches and latency are all there is
        dict(name="cell_64_fp64", kind="tissue", nx=64, ny=64, precision="fp64", walls=False,
             species=1, pitch=64.0, vertices=64, growth=False, steps=40,
             dump="all"),
        # a biology model on the host drives a small tissue step by step
        dict(name="loop_500x380_fp32", kind="loop", nx=500, ny=380, precision="fp32",
             walls=True, species=2, pitch=51.2, vertices=100, growth=False,
             steps=40),
        # the ordinary tissue: channel walls, 400 cells, two reacting species
        dict(name="tissue_1024_fp32", kind="tissue", nx=1024, ny=1024, precision="fp32",
             walls=True, species=2, pitch=51.2, vertices=100, growth=False,
             steps=400, dump="all"),
        # the same tissue growing: area controller, pressure nodes
        dict(name="growth_1024_fp32", kind="tissue", nx=1024, ny=1024, precision="fp32",
             walls=True, species=2, pitch=51.2, vertices=100, growth=True,
             steps=200, dump="shape"),
        # a large tissue: about 10,000 cells, the working set far above the L2
        dict(name="tissue_4096_fp32", kind="tissue", nx=4096, ny=4096, precision="fp32",
             walls=False, species=1, pitch=40.96, vertices=64, growth=False,
             steps=250, dump="shape"),
        # half-precision storage: the same kind of tissue, more of it per byte
        dict(name="tissue_2600x2200_fp16", kind="tissue", nx=2600, ny=2200, precision="fp16",
             walls=False, species=1, pitch=40.96, vertices=64, growth=False,
             steps=300, dump="shape"),
        # a reference run in full precision, sides that divide by nothing
        dict(name="tissue_1237x811_fp64", kind="tissue", nx=1237, ny=811, precision="fp64",
             walls=False, species=1, pitch=41.0, vertices=64, growth=False,
             steps=100, dump="all"),
        # a parameter study: many tissues of different size and stiffness
        dict(name="ensemble_30", kind="ensemble", tissues=30, side_min=128, side_max=1024,
             steps=200),
        # Turing patterns on a static cellular domain
        dict(name="turing_1024", kind="turing", n=1024, steps=400),
        # one steady morphogen profile, as a warm-start user asks for it
        dict(name="steady_256_one", kind="steady", nx=256, ny=256, batch=1),
        # steady profiles of many tissues: the training pairs of the operator
        dict(name="steady_256_batch96", kind="steady", nx=256, ny=256, batch=96),
        # training the neural operator and predicting held-out tissues
        dict(name="operator_256_batch16", kind="operator", n=256, batch=16, steps=4),
    ]


def draw(rng):
    def size(lo, hi):  # spread over the logarithm, odd values as likely as even ones
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["tissue"] * 6 + ["loop", "turing", "ensemble", "steady", "steady",
                       "operator"])
    if kind in ("tissue", "loop"):
        precision = rng.choice(["fp32", "fp32", "fp16", "fp64"]) if kind == "tissue" else "fp32"
        growth = kind == "tissue" and precision == "fp32" and rng.random() < 0.3
        top = {"fp32": 3000, "fp16": 3000, "fp64": 1100}[precision]
        if kind == "loop":
            top = 1024
        if growth:
            top = 1200
        nx, ny = size(64, top), size(64, top)
        c = dict(kind=kind, nx=nx, ny=ny, precision=precision, walls=rng.random() < 0.5,
                 species=rng.choice([0, 1, 1, 2, 3]), pitch=round(rng.uniform(38.0, 56.0), 2),
                 vertices=rng.choice([32, 48, 64, 64, 100, 100, 140]), growth=growth,
                 steps=rng.randint(10, 60))
        if kind == "tissue":
            c["dump"] = rng.choice(["all", "shape"])
        return c
    if kind == "turing":
        return dict(kind=kind, n=size(100, 1100), steps=rng.randint(10, 200))
    if kind == "ensemble":
        return dict(kind=kind, tissues=rng.randint(2, 30), side_min=size(64, 200),
                    side_max=size(220, 1000), steps=rng.randint(10, 100))
    if kind == "steady":
        return dict(kind=kind, nx=size(96, 300), ny=size(96, 300), batch=size(1, 48))
    return dict(kind=kind, n=rng.choice([64, 128, 192, 256]), batch=rng.randint(1, 16),
                steps=rng.randint(1, 4))


# --------------------------------------------------------------- the inputs
class Params:
    """The fields of the C parameter block, with the configurations' defaults."""

    def __init__(self, nx, ny, walls=False, tau=1.0, species=0):
        self.nx, self.ny, self.bc_y, self.tau, self.rho0 = nx, ny, int(walls), tau, 1.0
        self.n_species = species
        self.D, self.decay, self.src_rate = [0.0] * 4, [0.0] * 4, [0.0] * 4
        self.react = [[0.0] * 4 for _ in range(4)]
        self.mass_sources = self.pressure_nodes = 0
        self.reaction = self.noflux = 0


class Cells:
    def __init__(self, centres, radii, vertices, k, pressure, src, rng, jitter=0.0):
        a = 2.0 * np.pi * np.arange(vertices) / vertices
        ring = np.stack([np.cos(a), np.sin(a)], axis=1)
        xy = centres[:, None, :] + radii[:, None, None] * ring[None]
        if jitter:
            xy = xy + rng.uniform(-jitter, jitter, size=xy.shape)
        C = len(centres)
        edge = np.roll(xy, -1, axis=1) - xy
        self.n_cells, self.n_vertices, self.per_cell = C, C * vertices, vertices
        self.cell_off = (np.arange(C + 1) * vertices).astype(np.int32)
        self.rest_len = np.hypot(edge[..., 0], edge[..., 1]).reshape(-1)
        self.xy = np.ascontiguousarray(xy.reshape(-1, 2))
        self.k_spring = np.full(C * vertices, float(k))
        self.pressure = np.full(C, float(pressure))
        self.src_flag = np.asarray(src, np.uint8)
        self.radii = radii


def _sources(rng, C, fraction):
    src = np.zeros(C, np.uint8)
    src[rng.choice(C, size=max(1, int(round(fraction * C))), replace=False)] = 1
    return src


def _grid(nx, ny, pitch):
    gx, gy = max(1, int(nx / pitch)), max(1, int(ny / pitch))
    sx, sy = nx / gx, ny / gy
    X, Y = np.meshgrid((np.arange(gx) + 0.5) * sx, (np.arange(gy) + 0.5) * sy)
    return np.stack([X.ravel(), Y.ravel()], axis=1), min(sx, sy)


def _tissue(case, seed):
    """(parameters, cells, initial morphogens, mass-source data) of a tissue."""
    rng = np.random.Generator(np.random.PCG64(seed))
    nx, ny, S = case["nx"], case["ny"], case["species"]
    P = Params(nx, ny, case["walls"], 0.8 if case["walls"] else 0.6, S)
    if S == 1:
        P.D[0], P.decay[0], P.src_rate[0] = 0.1, 1e-3, 1e-3
    elif S >= 2:
        P.D[0], P.D[1], P.src_rate[0] = 0.05, 0.1, 1e-3
        P.react[0][0], P.react[0][1] = 0.05, -0.1
        P.react[1][0], P.react[1][1] = 0.1, -0.15
        if S == 3:
            P.D[2], P.decay[2] = 0.15, 1e-3
    centres, step = _grid(nx, ny, case["pitch"])
    C = len(centres)
    r = 0.39 * step if case["walls"] else min(15.0, 0.37 * step)
    slack = 0.02 * step if case["walls"] else 0.1 * step
    centres = centres + rng.uniform(-slack, slack, size=centres.shape)
    radii = r * (1.0 + rng.uniform(-0.1, 0.1, size=C))
    T = Cells(centres, radii, case["vertices"], 0.02 if case["walls"] else 0.01, 1e-3,
              _sources(rng, C, 0.1), rng, jitter=0.02 * r)
    phi0 = None
    if S:  # a smooth morphogen profile, another one for every species and seed
        x = 2 * np.pi * np.arange(nx) / nx
        y = 2 * np.pi * np.arange(ny) / ny
        ph = rng.uniform(0, 2 * np.pi, size=(S, 2))
        phi0 = [0.02 * (s + 1) * (1.2 + np.cos(x + ph[s, 0])[None, :] *
                                  np.cos(y + ph[s, 1])[:, None]) for s in range(S)]
    mass = None
    if case["growth"]:
        P.mass_sources, P.mass_alpha = 1, 1e-6
        P.pressure_nodes, P.pressure_rho = 1, 1.0
        n, rows = case["vertices"], max(1, int(ny / case["pitch"]))
        mask = np.zeros((ny, nx), np.uint8)
        mask[(np.arange(rows) * ny) // rows] = 1  # drainage between the rows of cells
        mass = dict(rate=np.zeros(C), area=1.1 * 0.5 * n * radii ** 2 * math.sin(2 * math.pi / n),
                    mask=mask)
    return P, T, phi0, mass


def _voronoi(nx, ny, pitch, rng):
    """Label of the nearest centre of a jittered periodic grid, per node."""
    gx, gy = max(2, int(round(nx / pitch))), max(2, int(round(ny / pitch)))
    sx, sy = nx / gx, ny / gy
    cx = (np.arange(gx)[None, :] + 0.5) * sx + rng.uniform(-sx / 4, sx / 4, size=(gy, gx))
    cy = (np.arange(gy)[:, None] + 0.5) * sy + rng.uniform(-sy / 4, sy / 4, size=(gy, gx))
    X, Y = np.meshgrid(np.arange(nx, dtype=np.float64), np.arange(ny, dtype=np.float64))
    ci, cj = (X // sx).astype(np.int64), (Y // sy).astype(np.int64)
    best, lab = np.full((ny, nx), np.inf), np.zeros((ny, nx), np.int32)
    for dj in (-1, 0, 1):
        for di in (-1, 0, 1):
            i2, j2 = (ci + di) % gx, (cj + dj) % gy
            dx, dy = X - cx[j2, i2], Y - cy[j2, i2]
            d2 = (dx - nx * np.round(dx / nx)) ** 2 + (dy - ny * np.round(dy / ny)) ** 2
            m = d2 < best
            best[m] = d2[m]
            lab[m] = (j2 * gx + i2)[m]
    return lab


def _turing(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    n = case["n"]
    P = Params(n, n, False, 1.0, 2)
    P.D[0], P.D[1] = 0.05, 0.4
    P.reaction, P.schnak, P.noflux = 1, [0.02, 0.1, 0.9], 1
    phi0 = [1.0 + 0.05 * rng.uniform(-1, 1, size=(n, n)),
            0.9 * (1.0 + 0.05 * rng.uniform(-1, 1, size=(n, n)))]
    return P, _voronoi(n, n, 51.2, rng), phi0


def _ensemble(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    # the sides are spread evenly over the logarithm, so that every seed has
    # the same amount of work; stiffness, viscosity and cells are the seed's
    n = case["tissues"]
    side = np.exp(np.linspace(math.log(case["side_min"]), math.log(case["side_max"]), n))
    out = []
    for t in range(n):
        s = int(round(side[t]))
        P = Params(s, s, False, float(rng.uniform(0.6, 1.2)), 1)
        P.D[0], P.decay[0], P.src_rate[0] = 0.1, 1e-3, 1e-3
        centres, step = _grid(s, s, 40.0)
        C = len(centres)
        T = Cells(centres + rng.uniform(-2, 2, size=centres.shape), np.full(C, 15.0), 64,
                  float(rng.uniform(0.005, 0.05)), 1e-3, _sources(rng, C, 0.1), rng, jitter=0.3)
        out.append((P, T))
    return out


def _static_tissues(n, ny, nx, seed):
    """Static tissues of 30 - 80 cells of 32 vertices: cells, D, decay, rate."""
    rng = np.random.Generator(np.random.PCG64(seed))
    tissues, D, decay = [], np.empty(n), np.empty(n)
    for t in range(n):
        want = int(rng.integers(30, 81))
        a = math.sqrt(nx * ny / want)
        centres, step = _grid(nx, ny, min(a, nx / 2, ny / 2))
        C = len(centres)
        r = 0.42 * step
        centres = centres + rng.uniform(-0.05 * r, 0.05 * r, size=centres.shape)
        tissues.append(Cells(centres, r * (1 + rng.uniform(-0.1, 0.1, size=C)), 32, 0.0, 0.0,
                             _sources(rng, C, rng.uniform(0.05, 0.2)), rng))
        D[t] = rng.uniform(0.05, 0.2)
        # the tissues of a batch come sorted by decay, so they end together
        decay[t] = 10.0 ** (-2.6 + 0.6 * (t + rng.uniform(0.2, 0.8)) / n)
    return tissues, D, decay, np.full(n, 1e-3)


def _layers():
    ch, out, prev = (32, 48, 64, 96, 128, 192), [], 4
    for c in ch:
        out += [(prev, c), (c, c)]
        prev = c
    for level in range(4, -1, -1):
        out += [(ch[level] + ch[level + 1], ch[level]), (ch[level], ch[level])]
    return out + [(32, 1)]


def _operator_weights(rng):
    layers, flat = _layers(), []
    for i, (ci, co) in enumerate(layers):
        std = math.sqrt(2.0 / (9 * ci)) * (0.1 if i == len(layers) - 1 else 1.0)
        flat += [rng.normal(0.0, std, size=9 * ci * co), np.zeros(co)]
    return np.concatenate(flat).astype(np.float32)


def _target(src, decay, rate):
    """A smooth profile around the sources, in the size of the solved ones."""
    y = F.avg_pool2d(src[:, None].double(), 31, 1, 15)[:, 0] * 1.5
    return y * torch.as_tensor(rate / decay, device=src.device)[:, None, None]


# ------------------------------------------------------------- what is timed
PRECISION = {"fp64": lbib.LBIB_FP64, "fp32": lbib.LBIB_FP32, "fp16": lbib.LBIB_FP16}
ALL = lbib.LBIB_RHO | lbib.LBIB_U | lbib.LBIB_PHI | lbib.LBIB_X | lbib.LBIB_AREA
SHAPE = lbib.LBIB_PHI | lbib.LBIB_X | lbib.LBIB_AREA


def _labels(tissues, ny, nx):
    """(cell mask, source map) of static tissues, uint8 (n, ny, nx)."""
    mask = torch.empty((len(tissues), ny, nx), dtype=torch.uint8, device="cuda")
    src = torch.empty_like(mask)
    for i, T in enumerate(tissues):
        ids, sources = lbib.label_cells(nx, ny, 0, T)
        mask[i].copy_(ids > 0)
        src[i].copy_(sources)
    return mask, src


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("tissue", "loop"):
        P, T, phi0, mass = _tissue(case, seed)
        sim = lbib.Simulation(P, PRECISION[case["precision"]], T.n_vertices, T.n_cells)
        sim.set_cells(T)
        for s in range(case["species"]):
            sim.set_species(s, phi0[s])
        if mass:
            sim.set_mass_sources(mass["rate"], mass["area"])
            sim.set_pressure_nodes(mass["mask"])
        st = dict(case=case, sim=sim)
        if kind == "loop":  # the model's host side: its pressures, pinned read buffers
            wave = np.linspace(0, 2 * np.pi, T.n_cells)
            st["pressure"] = [1e-3 * (1 + 0.2 * np.sin(wave + 0.3 * t + seed % 7))
                              for t in range(case["steps"])]
            st["xy"] = [torch.empty((T.n_vertices, 2), dtype=torch.float64, pin_memory=True)
                        for _ in range(2)]
            st["area"] = [torch.empty(T.n_cells, dtype=torch.float64, pin_memory=True)
                          for _ in range(2)]
        return st
    if kind == "turing":
        P, domains, phi0 = _turing(case, seed)
        sim = lbib.Simulation(P, lbib.LBIB_FP32)
        sim.set_domains(domains)
        for s in range(2):
            sim.set_species(s, phi0[s])
        return dict(case=case, sim=sim)
    if kind == "ensemble":
        every = _ensemble(case, seed)
        ens = lbib.Ensemble([p for p, _ in every], [t for _, t in every])
        return dict(case=case, ens=ens)
    if kind == "steady":
        tissues, D, decay, rate = _static_tissues(case["batch"], case["ny"], case["nx"], seed)
        _, src = _labels(tissues, case["ny"], case["nx"])
        return dict(case=case, src=src, D=D, decay=decay, rate=rate)
    n, B = case["n"], case["batch"]
    tissues, D, decay, rate = _static_tissues(2 * B, n, n, seed)
    order = np.random.Generator(np.random.PCG64(seed + 1)).permutation(2 * B)
    tissues, D, decay = [tissues[i] for i in order], D[order], decay[order]
    mask, src = _labels(tissues, n, n)
    net = lbib.NeuralOperator(B, n, n)
    net.set_params(_operator_weights(np.random.Generator(np.random.PCG64(seed))))
    phi = _target(src[:B], decay[:B], rate[:B]).float().contiguous()
    return dict(case=case, net=net, mask=mask, src=src, D=D, decay=decay, rate=rate, phi=phi)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "tissue":
        sim = state["sim"]
        sim.step(case["steps"])
        return sim.fields(ALL if case["dump"] == "all" else SHAPE)
    if kind == "loop":
        sim, shape = state["sim"], lbib.LBIB_X | lbib.LBIB_AREA
        for t in range(case["steps"]):
            sim.set_cell_params(pressure=state["pressure"][t])
            sim.advance(1)
            if t:
                lbib.lbib_wait_readback(sim.ctx)
            lbib.lbib_get_cells_async(sim.ctx, shape, state["xy"][t % 2].data_ptr(),
                                      state["area"][t % 2].data_ptr())
        lbib.lbib_wait_readback(sim.ctx)
        last = (case["steps"] - 1) % 2
        return dict(xy=state["xy"][last], area=state["area"][last])
    if kind == "turing":
        sim = state["sim"]
        sim.step(case["steps"])
        return sim.fields(lbib.LBIB_PHI)
    if kind == "ensemble":
        ens = state["ens"]
        ens.step(case["steps"])
        ens.status()
        return [ens.fields(t, lbib.LBIB_PHI | lbib.LBIB_X) for t in range(case["tissues"])]
    if kind == "steady":
        phi, steps, resid = lbib.steady_solve(state["src"], state["D"], state["decay"],
                                              state["rate"])
        return dict(phi=phi, steps=steps, resid=resid)
    net, B = state["net"], case["batch"]
    mask, src, D, decay, rate = (state[k] for k in ("mask", "src", "D", "decay", "rate"))
    loss = [net.train_step(mask[:B], src[:B], D[:B], decay[:B], rate[:B], state["phi"], lr=1e-4)
            for _ in range(case["steps"])]
    phi = net.forward(mask[B:], src[B:], D[B:], decay[B:], rate[B:])
    return dict(loss=np.array(loss), params=net.get_params(), phi=phi)


def work(case):
    """Populations read and written once per step and node (operator: every
    layer's weights and activations once), outputs written once."""
    kind = case["kind"]
    if kind in ("tissue", "loop"):
        N, S, steps = case["nx"] * case["ny"], case["species"], case["steps"]
        b = {"fp64": 8, "fp32": 4, "fp16": 2}[case["precision"]]
        C = len(_grid(case["nx"], case["ny"], case["pitch"])[0])
        V = C * case["vertices"]
        out = V * 16 + C * 8
        if kind == "loop":
            out = steps * (V * 16 + C * 16)
        elif case["dump"] == "all":
            out += 8 * (3 + S) * N
        else:
            out += 8 * S * N
        return {"bytes": steps * (2 * b * (9 + 5 * S) * N + 64 * V) + out,
                "flops": steps * (N * (150 + 40 * S) + 400 * V)}
    if kind == "turing":
        N = case["n"] ** 2
        return {"bytes": case["steps"] * 152 * N + 16 * N, "flops": case["steps"] * 240 * N}
    if kind == "ensemble":
        side = np.exp(np.linspace(math.log(case["side_min"]), math.log(case["side_max"]),
                                  case["tissues"]))
        N = float((side ** 2).sum())
        return {"bytes": case["steps"] * (112 + 64 * 64 / 1600) * N + 8 * N,
                "flops": case["steps"] * (190 + 400 * 64 / 1600) * N}
    if kind == "steady":  # about the steps that a mean decay of the range takes
        N, steps = case["nx"] * case["ny"] * case["batch"], 1500
        return {"bytes": 40 * N * steps, "flops": 30 * N * steps}
    n, B, steps = case["n"], case["batch"], case["steps"]
    level = [0, 0, 1, 1, 2, 2, 3, 3, 4, 4, 5, 5, 4, 4, 3, 3, 2, 2, 1, 1, 0, 0, 0]
    flops = bytes_ = 0.0
    for (ci, co), lv in zip(_layers(), level):
        px = B * (n >> lv) ** 2
        flops += 2.0 * 9 * ci * co * px * (3 * steps + 1)
        bytes_ += (2.0 * px * (ci + co) + 18.0 * ci * co) * (3 * steps + 1)
    return {"bytes": bytes_ + 2.1e6 * 28 * steps, "flops": flops}


# ------------------------------------------------ the same in 64 bits (torch)
CX, CY = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
W9 = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
W5 = (1 / 3,) + (1 / 6,) * 4


def _pull(P, f):
    """The populations arriving at every node; walls bounce back half-way."""
    g = torch.empty_like(f)
    for q in range(f.shape[0]):
        g[q] = torch.roll(f[q], (CY[q], CX[q]), (0, 1))
        if P.bc_y and CY[q]:
            row = 0 if CY[q] > 0 else -1
            g[q, row] = f[OPP[q], row]
    return g


def _inside(poly, nx, ny, walls):
    """Nodes inside each polygon of (C, n, 2), by the crossing rule half-open
    in y: (C, H, W) truth values and their node indices (-1 outside walls)."""
    lo = torch.floor(poly.amin(1))
    size = (torch.ceil(poly.amax(1)) - lo).amax(0).long() + 1
    W, H = int(size[0]), int(size[1])
    xs = lo[:, 0, None] + torch.arange(W, device=poly.device)
    ys = lo[:, 1, None] + torch.arange(H, device=poly.device)
    A, B = poly, torch.roll(poly, -1, 1)
    inside = torch.zeros((len(poly), H, W), dtype=torch.bool, device=poly.device)
    step = max(1, int(2e8 // (len(poly) * H * W)))
    for e in range(0, poly.shape[1], step):
        ax, ay, bx, by = (v[:, e:e + step, None] for v in (A[..., 0], A[..., 1], B[..., 0],
                                                           B[..., 1]))
        y = ys[:, None, :]
        cross = (ay <= y) != (by <= y)
        xc = torch.where(cross, ax + (y - ay) * (bx - ax) / (by - ay), -math.inf)
        inside ^= ((xs[:, None, None, :] < xc[..., None]).sum(1) & 1).bool()
    yi, xi = ys.long(), xs.long() % nx
    bad = (yi < 0) | (yi >= ny) if walls else torch.zeros_like(yi, dtype=torch.bool)
    node = (yi % ny)[:, :, None] * nx + xi[:, None, :]
    return inside & ~bad[:, :, None], node


class Reference:
    """The coupled step of one tissue in double precision."""

    def __init__(self, P, T=None, phi0=None, mass=None, domains=None):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.P, self.T, self.mass = P, T, mass
        dd = dict(dtype=torch.float64, device=dev)
        w = torch.tensor(W9, **dd)[:, None, None]
        # deviations from the rest state keep the sums exact
        self.f = (w * 0).expand(9, P.ny, P.nx).clone()
        self.g = [torch.tensor(W5, **dd)[:, None, None] * torch.as_tensor(p, **dd)
                  for p in (phi0 or [])]
        self.dev = dev
        if T is not None:
            self.X = torch.as_tensor(T.xy, **dd)
            self.L0, self.k = torch.as_tensor(T.rest_len, **dd), torch.as_tensor(T.k_spring, **dd)
            self.p = torch.as_tensor(T.pressure, **dd)
            self.bits = torch.as_tensor(T.src_flag, device=dev) > 0
        if mass:
            self.pmask = torch.as_tensor(mass["mask"], device=dev) > 0
            self.target, self.rate = torch.as_tensor(mass["area"], **dd), torch.as_tensor(
                mass["rate"], **dd)
        if domains is not None:
            dom = torch.as_tensor(domains, device=dev)
            at = [torch.roll(dom, (CY[q], CX[q]), (0, 1)) == dom for q in range(5)]
            ahead = [torch.roll(dom, (-CY[q], -CX[q]), (0, 1)) == dom for q in range(5)]
            two = [torch.roll(dom, (-2 * CY[q], -2 * CX[q]), (0, 1)) == dom for q in range(5)]
            self.dom = [(~at[q], ahead[q], two[q]) for q in range(5)]
            g = self.g[0]
            self.mom = (g.sum(0), g[1] - g[3], g[2] - g[4])

    def areas(self):
        n = self.T.per_cell
        Q = self.X.view(-1, n, 2)
        Q = Q - Q[:, :1]
        R = torch.roll(Q, -1, 1)
        return 0.5 * (Q[..., 0] * R[..., 1] - R[..., 0] * Q[..., 1]).sum(1)

    def vertex_forces(self):
        P, n = self.P, self.T.per_cell
        Q = self.X.view(-1, n, 2)
        e = torch.roll(Q, -1, 1) - Q
        L = torch.sqrt((e * e).sum(-1))
        s = (self.k.view(-1, n) * (L - self.L0.view(-1, n)) / L)[..., None] * e
        Fv = s - torch.roll(s, 1, 1)
        nb = torch.roll(Q, -1, 1) - torch.roll(Q, 1, 1)
        Fv = Fv + 0.5 * self.p[:, None, None] * torch.stack([nb[..., 1], -nb[..., 0]], -1)
        Fv = Fv.reshape(-1, 2)
        return Fv

    def stencil(self):
        P, X = self.P, self.X
        base = torch.floor(X) - 1
        o = torch.arange(4, device=self.dev)
        node = base[:, :, None] + o
        w = 0.25 * (1 + torch.cos(0.5 * math.pi * (node - X[:, :, None])))
        node = node.long()
        wx, wy = w[:, 0], w[:, 1]
        if P.bc_y:
            wy = torch.where((node[:, 1] >= 0) & (node[:, 1] < P.ny), wy, 0.0)
        idx = (node[:, 1] % P.ny)[:, :, None] * P.nx + (node[:, 0] % P.nx)[:, None, :]
        return idx.reshape(len(X), 16), (wy[:, :, None] * wx[:, None, :]).reshape(len(X), 16)

    def step(self, last):
        P, N, shape = self.P, self.P.nx * self.P.ny, (self.P.ny, self.P.nx)
        Fx = Fy = 0.0
        src = Sm = None
        if self.T is not None:
            Q = self.X.view(-1, self.T.per_cell, 2)
            if self.mass:
                inside, node = _inside(Q, P.nx, P.ny, P.bc_y)
                C = len(Q)
                lab = torch.full((N,), C, dtype=torch.long, device=self.dev)
                which = torch.arange(C, device=self.dev)[:, None, None].expand_as(node)
                lab.scatter_reduce_(0, node[inside], which[inside], "amin")
                Sc = torch.cat([self.rate + P.mass_alpha * (self.target - self.areas()),
                                torch.zeros(1, dtype=torch.float64, device=self.dev)])
                Sm = Sc[lab].view(shape)
            if P.n_species:
                inside, node = _inside(Q[self.bits], P.nx, P.ny, P.bc_y)
                src = torch.zeros(N, dtype=torch.bool, device=self.dev)
                src[node[inside]] = True
                src = src.view(shape)
            Fv = self.vertex_forces()
            idx, w = self.stencil()
            Fg = torch.zeros((2, N), dtype=torch.float64, device=self.dev)
            for a in range(2):
                Fg[a].index_add_(0, idx.reshape(-1), (w * Fv[:, a, None]).reshape(-1))
            Fx, Fy = Fg[0].view(shape), Fg[1].view(shape)
        d = _pull(P, self.f)
        if self.mass:
            gam = torch.where(self.pmask, P.pressure_rho / (P.rho0 + d.sum(0)), 1.0)
            for q in range(9):
                d[q] = gam * d[q] + (gam - 1.0) * W9[q] * P.rho0
        dr = d.sum(0)
        rho = P.rho0 + dr
        ux = (d[1] - d[3] + d[5] - d[6] - d[7] + d[8] + 0.5 * Fx) / rho
        uy = (d[2] - d[4] + d[5] + d[6] - d[7] - d[8] + 0.5 * Fy) / rho
        om, pref = 1.0 / P.tau, 1.0 - 0.5 / P.tau
        usq = 1.5 * (ux * ux + uy * uy)
        uF = ux * Fx + uy * Fy
        for q in range(9):
            cu = CX[q] * ux + CY[q] * uy
            cF = CX[q] * Fx + CY[q] * Fy
            eq = W9[q] * (dr + rho * (3 * cu + 4.5 * cu * cu - usq))
            d[q] += om * (eq - d[q]) + pref * W9[q] * (3 * (cF - uF) + 9 * cu * cF)
            if Sm is not None:
                d[q] += W9[q] * Sm
        self.f = d
        g = [_pull(P, s) for s in self.g]
        if P.noflux:
            ph0, jx, jy = self.mom
            for q in range(1, 5):
                miss, one, two = self.dom[q]
                y1, y2 = (-CY[q], -CX[q]), (-2 * CY[q], -2 * CX[q])
                p1, p2 = torch.roll(ph0, y1, (0, 1)), torch.roll(ph0, y2, (0, 1))
                j1 = torch.roll(CX[q] * jx + CY[q] * jy, y1, (0, 1))
                val = torch.where(one, torch.where(two, 2 * p1 - p2, p1) + j1, ph0)
                g[0][q] = torch.where(miss, W5[q] * val, g[0][q])
            self.mom = (g[0].sum(0), g[0][1] - g[0][3], g[0][2] - g[0][4])
        phi = [s.sum(0) for s in g]
        for s in range(P.n_species):
            if P.reaction and s < 2:
                r2l = phi[0] * phi[0] * phi[1]
                gam, a, b = P.schnak
                R = gam * (a - phi[0] + r2l) if s == 0 else gam * (b - r2l)
            else:
                R = -P.decay[s] * phi[s]
                for b in range(P.n_species):
                    if P.react[s][b]:
                        R = R + P.react[s][b] * phi[b]
            if src is not None and s == 0 and P.src_rate[0]:
                R = R + P.src_rate[0] * src.double()
            for q in range(5):
                eq = phi[s] * W5[q] * (1 + 3 * (CX[q] * ux + CY[q] * uy))
                g[s][q] += (eq - g[s][q]) / (3 * P.D[s] + 0.5) + W5[q] * R
        self.g = g
        if self.T is not None:
            U = [(w * u.reshape(-1)[idx]).sum(1) for u in (ux, uy)]
            self.X = self.X + torch.stack(U, 1)
        if last:
            self.out = dict(rho=rho, ux=ux, uy=uy, phi=torch.stack(phi) if phi else None)

    def run(self, steps, which):
        for t in range(steps):
            self.step(t == steps - 1)
        out = dict(self.out)
        if self.T is not None:
            out["xy"], out["area"] = self.X, self.areas()
        return {k: out[k] for k in which if out.get(k) is not None}


def _steady_exact(src, D, decay, rate, tol=1e-6, every=16, most=200000):
    """Relaxation of every tissue until its own residual meets tol."""
    def col(v):
        return torch.as_tensor(v, dtype=torch.float64, device=src.device)[:, None, None]

    B = len(src)
    out = torch.zeros(src.shape, dtype=torch.float64, device=src.device)
    left = torch.arange(B, device=src.device)
    Q = (src > 0).double() * col(rate)
    om, dec = 1.0 / (3 * col(D) + 0.5), col(decay)
    g = torch.zeros((5,) + tuple(src.shape), dtype=torch.float64, device=src.device)
    for n in range(1, most + 1):
        g = torch.stack([torch.roll(g[q], (CY[q], CX[q]), (1, 2)) for q in range(5)])
        phi = g.sum(0)
        R = Q - dec * phi
        for q in range(5):
            g[q] += om * (phi * W5[q] - g[q]) + W5[q] * R
        if n % every == 0:
            new = torch.stack([torch.roll(g[q], (CY[q], CX[q]), (1, 2)) for q in range(5)]).sum(0)
            r = (new - phi).abs().amax((1, 2)) / new.abs().amax((1, 2))
            done = r <= tol
            if bool(done.any()):
                out[left[done]] = new[done]
                keep = ~done
                left, Q, om, dec, g = left[keep], Q[keep], om[keep], dec[keep], g[:, keep]
                if not len(left):
                    break
    return out


def _unet(params, mask, src, D, decay):
    def col(v):
        return torch.as_tensor(v, dtype=torch.float64, device=mask.device)[:, None, None, None]

    x = torch.cat([mask[:, None].double(), src[:, None].double(),
                   ((col(D) - 0.125) / 0.075).expand(-1, 1, *mask.shape[1:]),
                   (torch.log10(col(decay)) + 3).expand(-1, 1, *mask.shape[1:])], 1)
    layers, at, o = _layers(), [], 0
    for ci, co in layers:
        w = params[o:o + 9 * ci * co].view(3, 3, ci, co).permute(3, 2, 0, 1)
        o += 9 * ci * co
        at.append((w, params[o:o + co]))
        o += co

    def conv(i, h, relu=True):
        h = F.conv2d(h, at[i][0], at[i][1], padding=1)
        return F.relu(h) if relu else h

    h, skips, i = x, [], 0
    for level in range(6):
        if level:
            h = F.avg_pool2d(h, 2)
        h = conv(i + 1, conv(i, h))
        i += 2
        skips.append(h)
    for level in range(4, -1, -1):
        up = h.repeat_interleave(2, 2).repeat_interleave(2, 3)
        h = conv(i + 1, conv(i, torch.cat([skips[level], up], 1)))
        i += 2
    return conv(i, h, False)[:, 0]


def exact(case, seed):
    kind = case["kind"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if kind in ("tissue", "loop"):
        P, T, phi0, mass = _tissue(case, seed)
        R = Reference(P, T, phi0, mass)
        if kind == "tissue":
            shape = ["phi", "xy", "area"]
            return R.run(case["steps"],
                         shape if case["dump"] == "shape" else ["rho", "ux", "uy"] + shape)
        wave = np.linspace(0, 2 * np.pi, T.n_cells)
        for t in range(case["steps"]):
            p = 1e-3 * (1 + 0.2 * np.sin(wave + 0.3 * t + seed % 7))
            R.p = torch.as_tensor(p, device=R.dev)
            R.step(t == case["steps"] - 1)
        return dict(xy=R.X, area=R.areas())
    if kind == "turing":
        P, domains, phi0 = _turing(case, seed)
        return Reference(P, None, phi0, None, domains).run(case["steps"], ["phi"])
    if kind == "ensemble":
        return [Reference(P, T, [np.zeros((P.ny, P.nx))]).run(case["steps"], ["phi", "xy"])
                for P, T in _ensemble(case, seed)]
    if kind == "steady":
        tissues, D, decay, rate = _static_tissues(case["batch"], case["ny"], case["nx"], seed)
        src = torch.stack([_source_map(T, case["ny"], case["nx"], dev)[1] for T in tissues])
        return dict(phi=_steady_exact(src, D, decay, rate), steps=None, resid=None)
    n, B = case["n"], case["batch"]
    tissues, D, decay, rate = _static_tissues(2 * B, n, n, seed)
    order = np.random.Generator(np.random.PCG64(seed + 1)).permutation(2 * B)
    D, decay = D[order], decay[order]
    maps = [_source_map(tissues[i], n, n, dev) for i in order]
    mask, src = torch.stack([m for m, _ in maps]), torch.stack([s for _, s in maps])
    w = torch.as_tensor(_operator_weights(np.random.Generator(np.random.PCG64(seed))),
                        dtype=torch.float64, device=dev).requires_grad_()
    scale = torch.as_tensor(rate / decay, device=dev)[:, None, None]
    y = _target(src[:B], decay[:B], rate[:B]).float().double() / scale[:B]
    adam = torch.optim.Adam([w], lr=1e-4)
    losses = []
    for _ in range(case["steps"]):
        adam.zero_grad()
        loss = ((_unet(w, mask[:B], src[:B], D[:B], decay[:B]) - y) ** 2).mean()
        loss.backward()
        adam.step()
        losses.append(float(loss.detach()))
    with torch.no_grad():
        phi = _unet(w, mask[B:], src[B:], D[B:], decay[B:]) * scale[B:]
    return dict(loss=np.array(losses), params=w.detach(), phi=phi)


def _source_map(T, ny, nx, dev):
    """(cell mask, source map) of one static tissue."""
    maps = []
    for bits in (np.ones(T.n_cells, bool), T.src_flag > 0):
        poly = torch.as_tensor(T.xy.reshape(T.n_cells, -1, 2)[bits], device=dev)
        inside, node = _inside(poly, nx, ny, 0)
        m = torch.zeros(ny * nx, dtype=torch.uint8, device=dev)
        m[node[inside]] = 1
        maps.append(m.view(ny, nx))
    return maps
