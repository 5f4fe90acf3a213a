"""Performance cases of the framework's public entry points.

Two families, as in the configurations, tests and benchmark of this repository:

* the source iteration of the discrete-velocity solver (``dvm.Solver``): 2D and 3D porous media, one
  problem or a batch, FP64 and FP32, from a 24^3 medium where latency and launches count to the 128^3
  rock with 4096 velocities, with the wall, lateral and model options;
* the warm-start network (``warmstart.UNet``): inference and a training step.

``exact`` computes the same results in 64 bits with plain torch: the upwind sweep as a loop over the
hyperplanes of constant oriented coordinate sum, all octants and problems at once, and the network as
27 shifted matrix products per convolution with autograd.
"""
import itertools
import math

import numpy as np
import torch

from paper_1712_01132_gb300 import dvm, inputs, warmstart


# ------------------------------------------------------------------------------------ the cases

def _solver(name, **kw):
    case = {"kind": "solver", "geometry": "discs", "n1": 64, "n2": 64, "n3": 1, "problems": 1, "porosity": 0.5, "kn": 0.1,
            "nv": 16, "precision": "fp32", "lateral": "periodic", "order": 2, "iters": 100, "graph": False,
            "specular": 0.0, "tau": False, "shakhov": 0.0, "es": 0.0, "sub1": 1, "sub2": 1, "sub3": 1,
            "new": False, "warm": False}
    case.update(kw)
    if name:
        case["name"] = name
    return case


def _unet(name, **kw):
    case = {"kind": "unet", "train": False, "nz": 64, "ny": 64, "nx": 64, "levels": 4, "base": 32}
    case.update(kw)
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # the unit cell of the plain method in the library's default precision: one check interval
        _solver("cell_32_fp64", geometry="cell", n1=32, n2=32, porosity=0.7, precision="fp64"),
        # the level-3 carpet of the paper's first table, specular lateral faces, 8^2 velocities, FP64
        _solver("carpet_540_fp64", geometry="carpet", n1=540, n2=540, porosity=0.70233, nv=8, lateral="specular",
                precision="fp64", iters=20),
        # the random medium at four Knudsen numbers as one batched context
        _solver("kn_sweep_512", geometry="discs", n1=512, n2=512, problems=4, kn=0.0, nv=32, iters=20),
        # many packings of uneven sides, each at its own Knudsen number, iterated through the graph
        _solver("disc_batch_16", geometry="disc_batch", n1=64, n2=512, problems=16, porosity=0.55, kn=0.0, nv=24,
                iters=20, graph=True),
        # a small 3D medium as in parameter scans, one check interval through the graph
        _solver("rock_24", geometry="rock", n1=24, n2=24, n3=24, kn=0.3, nv=8, graph=True),
        # the size on which the warm-start network's training runs are made
        _solver("rock_64", geometry="rock", n1=64, n2=64, n3=64, porosity=0.35, kn=0.5, nv=16, iters=10),
        # the largest configuration: 128^3 rock, 4096 velocities
        _solver("rock_128", geometry="rock", n1=128, n2=128, n3=128, porosity=0.35, kn=0.5, nv=16, iters=5),
        # the quadrant of the cubic sphere array at half the paper's resolution, FP64, specular faces
        _solver("spheres_100_fp64", geometry="spheres", n1=100, n2=50, n3=50, porosity=0.75, nv=8, precision="fp64",
                lateral="specular", iters=10),
        # the Shakhov model (temperature term, Pr = 2/3), uneven sides
        _solver("shakhov_45", geometry="rock", n1=45, n2=48, n3=43, porosity=0.35, kn=0.2, nv=12, tau=True,
                shakhov=2.0 / 3.0, iters=10),
        # one new geometry from start to answer: context, warm start, one check interval, host readouts
        _solver("new_rock_48", geometry="rock", n1=48, n2=48, n3=48, porosity=0.35, kn=0.5, nv=8, new=True, warm=True),
        # the network's prediction for a 128^3 rock
        _unet("unet_predict_128", nz=128, ny=128, nx=128),
        # one training step on a 64^3 rock: forward, loss, backward, Adam
        _unet("unet_train_64", train=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


_MOST_UPDATES = 1.4e10   # cell-velocity updates of one pass of a drawn FP32 case (below rock_128's)


def draw(rng):
    kind = rng.choice(["2d", "2d", "batch", "3d", "3d", "model", "new", "predict", "train"])
    if kind in ("predict", "train"):
        levels = rng.randint(2, 4)
        m = 2 ** (levels - 1)
        top = 128 if kind == "predict" else 64
        side = [max(1, rng.randint(16, top) // m) * m for _ in range(3)]
        return _unet(None, train=kind == "train", nz=side[0], ny=side[1], nx=side[2], levels=levels,
                     base=rng.choice([8, 16, 24, 32]))
    kn = 10.0 ** rng.uniform(-2.0, 1.0)
    prec = rng.choice(["fp32", "fp32", "fp64"])
    lat = rng.choice(["periodic", "specular"])
    graph = rng.random() < 0.5
    if kind in ("2d", "batch"):
        nv = 2 * rng.randint(4, 16 if prec == "fp32" else 12)
        if kind == "batch":
            case = _solver(None, geometry="disc_batch", n1=_log_int(rng, 33, 64), n2=_log_int(rng, 128, 400),
                           problems=rng.randint(2, 16), porosity=0.55, kn=0.0, nv=nv, precision=prec, lateral=lat)
        else:
            case = _solver(None, n1=_log_int(rng, 32, 512), n2=_log_int(rng, 32, 512), porosity=rng.uniform(0.45, 0.7),
                           kn=kn, nv=nv, precision=prec, lateral=lat)
            option = rng.random()
            if option < 0.2:
                case["specular"] = rng.uniform(0.1, 0.9)
            elif option < 0.35:
                case.update(sub1=rng.randint(1, 3), sub2=rng.randint(1, 4))
            elif option < 0.45:
                case["order"] = 1
    else:
        case = _solver(None, geometry="rock", n1=_log_int(rng, 16, 96), n2=_log_int(rng, 16, 96), n3=_log_int(rng, 16, 96),
                       porosity=rng.uniform(0.3, 0.6), kn=max(kn, 0.05), nv=2 * rng.randint(3, 8), precision=prec, lateral=lat)
        if kind == "model":
            case["tau"] = True
            model = rng.choice(["tau", "shakhov", "es"])
            if model != "tau":
                case[model] = rng.choice([2.0 / 3.0, 0.7, 0.8])
        elif kind == "new":
            case.update(new=True, warm=rng.random() < 0.5)
        else:
            option = rng.random()
            if option < 0.2:
                case["specular"] = rng.uniform(0.1, 0.9)
            elif option < 0.35:
                case.update(sub1=rng.randint(1, 2), sub2=rng.randint(1, 2), sub3=rng.randint(1, 3))
            elif option < 0.45:
                case["order"] = 1
    case["graph"] = graph and not case["new"]
    # FP64 runs at about a thirtieth of the FP32 rate on this hardware
    per_iter = _updates(case) * (30.0 if case["precision"] == "fp64" else 1.0)
    case["iters"] = int(max(1, min(100, _MOST_UPDATES / 4 / per_iter)))
    return case


# ----------------------------------------------------------------------------- work and tolerance

def _cells(case):
    if case["geometry"] == "disc_batch":
        return case["problems"] * (0.5 * (case["n1"] + case["n2"])) ** 2
    return float(case["problems"] * case["n1"] * case["n2"] * case["n3"])


def _dims(case):
    return 3 if case["geometry"] in ("rock", "spheres") else 2


def _updates(case):
    """Cell-velocity updates of one iteration (fluid cells x velocities)."""
    return _cells(case) * case["porosity"] * case["nv"] ** _dims(case)


def _layers(case):
    return warmstart.layer_shapes(case["levels"], case["base"], 3, 4)


def _layer_levels(case):
    L = case["levels"]
    return [l for l in range(L) for _ in range(2)] + [l for l in reversed(range(L - 1)) for _ in range(2)] + [0]


def work(case):
    if case["kind"] == "unet":
        vox = case["nz"] * case["ny"] * case["nx"]
        macs = sum(27.0 * ci * co * vox / 8 ** l for (ci, co), l in zip(_layers(case), _layer_levels(case)))
        weights = sum(27 * ci * co + co for ci, co in _layers(case))
        if not case["train"]:
            return {"flops": 2.0 * macs, "bytes": 4.0 * (7 * vox + weights)}
        # weight and data gradients cost as much as the forward; the data gradient of the first layer is not needed
        first = 27.0 * 3 * case["base"] * vox
        # features, targets and mask read, prediction written; weights and two moments read and written, gradients written
        return {"flops": 2.0 * (3.0 * macs - first), "bytes": 4.0 * (12 * vox + 7 * weights)}
    d = _dims(case)
    size = 8 if case["precision"] == "fp64" else 4
    # source, upwind terms of d axes, reciprocal, quadrature of d + 1 moments (plus the models' terms)
    extra = (1 if case["tau"] else 0) + (3 if case["shakhov"] else 0) + (6 if case["es"] else 0)
    flops = (2 * d + 6 * d + 1 + 2 * (d + 1) + 4 * extra) * _updates(case)
    # the moments and wall terms of the previous iteration read, the octants' moment partials written
    per_cell = 2 + (3 * d + 1 + 2 ** d * (d + 1 + extra)) * size
    return {"flops": flops * case["iters"], "bytes": per_cell * _cells(case) * case["iters"]}


def tolerance(case):
    if case["kind"] == "unet":
        # BF16 operands: activations or gradients that round the other way travel through the layers
        return {"rel": 2e-2, "max": 0.9} if case["train"] else {"rel": 1e-2, "max": 0.5}
    if case["precision"] == "fp64":
        return {"rel": 1e-10, "max": 1e-8}
    # FP32 sums of up to 4096 velocities.  The velocity and temperature are what is left of O(1) octant sums that
    # nearly cancel: against the 64-bit results usually 1e-7 to 2e-5, at worst 1.5e-4 over the declared ranges
    return {"rel": 4e-4, "max": 1.6e-2}


# ------------------------------------------------------------------------------------ the inputs

def _discs(n1, n2, porosity, seed):
    """A disc packing that percolates: seeds without an x1 path are skipped."""
    small = min(n1, n2)
    for attempt in range(100):
        mask = inputs.random_discs(n1, n2, seed=seed + attempt, rmin=min(6.0, small / 8), rmax=min(20.0, small / 4),
                                   solid_fraction=1.0 - porosity)
        if not mask.all():
            break
    return mask


def _problems(case, seed):
    """(masks, Knudsen numbers) of a solver case."""
    rng = np.random.default_rng(100003 * seed + 17)
    geo = case["geometry"]
    if geo == "disc_batch":
        # sides and porosities belong to the case, the packings and Knudsen numbers to the seed
        sizes = np.random.default_rng(case["problems"] * 1000003 + case["n1"] * 1009 + case["n2"])
        masks, kns = [], []
        for b in range(case["problems"]):
            n1, n2 = (int(sizes.integers(case["n1"], case["n2"] + 1)) for _ in range(2))
            masks.append(_discs(n1, n2, float(sizes.uniform(0.4, 0.7)), 1000 * seed + 100 * b))
            kns.append(float(10.0 ** rng.uniform(-2.0, 1.0)))
        return masks, kns
    if geo == "cell":
        mask = inputs.cylinder_cell(case["n1"], case["porosity"])
    elif geo == "carpet":
        mask = inputs.sierpinski_carpet(case["n1"], 3)
    elif geo == "spheres":
        mask = inputs.sphere_quadrant(case["n1"], case["n2"], case["n3"], case["porosity"])
    elif geo == "discs":
        mask = _discs(case["n1"], case["n2"], case["porosity"], 1000 * seed)
    else:
        n = max(case["n1"], case["n2"], case["n3"])
        for attempt in range(100):
            mask = inputs.gaussian_rock(n, seed=1000 * seed + attempt, corr_len=max(2.0, n / 16), porosity=case["porosity"])
            mask = mask[:case["n3"], :case["n2"], :case["n1"]]
            if not mask.all() and mask.any():
                break
    if case["kn"] > 0.0:
        kns = case["kn"] * 10.0 ** rng.uniform(-0.1, 0.1, case["problems"])
    else:
        kns = 10.0 ** (np.linspace(-2.0, 1.0, case["problems"]) + rng.uniform(-0.1, 0.1, case["problems"]))
    return [np.ascontiguousarray(mask)] * case["problems"], [float(k) for k in kns]


def _start_fields(mask, seed):
    """A smooth start density and velocity of the size a prediction has (paper variables)."""
    rng = np.random.default_rng(7919 * seed + 3)
    n1 = mask.shape[-1]
    x1 = np.broadcast_to(np.arange(n1) / n1, mask.shape)
    wave = np.sin(2 * math.pi * (x1 + rng.uniform()))
    rho0 = (0.05 * wave - x1) * ~mask
    u0 = np.stack([(a + 0.3 * a * wave) * ~mask for a in rng.uniform(0.01, 0.03, mask.ndim)])
    return rho0, u0


def _options(case):
    return dict(precision=case["precision"], lateral=case["lateral"], stencil_order=case["order"], check_interval=case["iters"],
                use_graph=case["graph"], specular_fraction=case["specular"], temperature_term=case["tau"],
                shakhov_prandtl=case["shakhov"], es_prandtl=case["es"], subdomains=(case["sub1"], case["sub2"], case["sub3"]))


def _unet_inputs(case, seed):
    """(features, targets, fluid mask, weights, biases) on the GPU, FP32."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    g = torch.Generator(device="cpu").manual_seed(1000003 * seed + 11)
    shape = (case["nz"], case["ny"], case["nx"])
    z, y, x = (torch.arange(n, dtype=torch.float32, device=dev) / n * (2 * math.pi) for n in shape)
    ph = (2 * math.pi * torch.rand(16, generator=g)).tolist()
    # a smooth periodic field of a few waves: solid where it is positive, a distance-like channel from its value
    f = sum((torch.sin(a * z + ph[a])[:, None, None] * torch.cos((4 - a) * y + ph[4 + a])[None, :, None] *
             torch.sin((a + 1) * x + ph[8 + a])[None, None, :]) for a in range(4)) + 0.2
    solid = (f > 0).float()
    feat = torch.stack([solid, (4.0 * f).clamp(-2.0, 2.0), torch.full(shape, math.log10(0.5 * shape[2]), device=dev)])
    flow = torch.stack([f, torch.cos(f), torch.sin(2 * f), torch.cos(f + ph[13])])
    target = flow * (1.0 - solid)
    wts, bias = [], []
    for i, (ci, co) in enumerate(_layers(case)):
        std = math.sqrt(2.0 / (27 * ci))
        wts.append((torch.randn(co, ci, 27, generator=g) * std))
        bias.append(torch.randn(co, generator=g) * 0.05)
    return feat.contiguous(), target.contiguous(), (1.0 - solid).reshape(-1).contiguous(), wts, bias


def prepare(case, seed):
    if case["kind"] == "unet":
        feat, target, mask, wts, bias = _unet_inputs(case, seed)
        net = warmstart.UNet(levels=case["levels"], base=case["base"], seed=0)
        net.load_state({"w": [w.numpy() for w in wts], "b": [b.numpy() for b in bias]})
        return {"case": case, "net": net, "x": feat, "t": target, "mask": mask}
    masks, kns = _problems(case, seed)
    v, w = dvm.dvm_gh_velocity_grid(masks[0].ndim, case["nv"])
    st = {"case": case, "masks": masks, "kns": kns, "v": v, "w": w}
    st["fluid"] = [(~m).astype(np.float64) for m in masks]
    if not case["new"]:
        st["fluid"] = [torch.from_numpy(f).cuda() for f in st["fluid"]]
    if case["warm"]:
        st["start"] = [_start_fields(m, seed) for m in masks]
    if not case["new"]:
        # a graph needs a stream of its own
        st["stream"] = torch.cuda.Stream() if case["graph"] else torch.cuda.current_stream()
        with torch.cuda.stream(st["stream"]):
            st["solver"] = dvm.Solver(masks if len(masks) > 1 else masks[0], kns, v, w, **_options(case))
    return st


def _level(rho, fluid):
    """The density without its mean over the fluid: the problem fixes it only up to a constant."""
    return rho - fluid * (rho.sum() / fluid.sum())


def run(st):
    case = st["case"]
    if case["kind"] == "unet":
        net = st["net"]
        if not case["train"]:
            y = net.forward(st["x"])
            return {"y": y}
        net.zero_grad()
        y = net.forward(st["x"])
        loss, dy = net.loss_and_grad(y, st["t"], st["mask"])
        net.backward(dy)
        net.step(lr=1e-3)
        return {"loss": loss, "y": y, "dw": net.dw, "db": net.db, "w": net.w, "b": net.b}
    if case["new"]:
        s = dvm.Solver(st["masks"] if len(st["masks"]) > 1 else st["masks"][0], st["kns"], st["v"], st["w"], **_options(case))
        for b, (rho0, u0) in enumerate(st.get("start", [])):
            s.set_initial(rho0, u0, prob=b)
        s.iterate(case["iters"], 0.0)
        mom = [s.moments(b) for b in range(s.nprob)]
        k = np.array([s.permeability(b)[0] for b in range(s.nprob)])
        s.close()
        return {"rho": [_level(m[0], f) for m, f in zip(mom, st["fluid"])], "u": [m[1] for m in mom], "k": k}
    s = st["solver"]
    with torch.cuda.stream(st["stream"]):
        s.iterate(case["iters"], 0.0)
        rho, u = [], []
        for b, m in enumerate(st["masks"]):
            r = torch.empty(m.shape, dtype=torch.float64, device="cuda")
            q = torch.empty((m.ndim,) + m.shape, dtype=torch.float64, device="cuda")
            s.moments_device(b, r.data_ptr(), q.data_ptr())
            rho.append(_level(r, st["fluid"][b]))
            u.append(q)
        out = {"rho": rho, "u": u, "k": np.array([s.permeability(b)[0] for b in range(s.nprob)])}
    if case["tau"]:
        out["tau"] = s.temperature(0)
    return out


# ------------------------------------------------------------------------ the results in 64 bits

def _half_range_gauss(m):
    """Nodes and weights of the m-point rule for int_0^inf exp(-x^2) g(x) dx, weights normalised so
    that the mirrored rule has sum 1: Stieltjes' procedure on a fine Gauss-Legendre rule."""
    t, wt = np.polynomial.legendre.leggauss(300)
    edges = np.linspace(0.0, 14.0, 29)
    x = np.concatenate([0.5 * (b - a) * t + 0.5 * (a + b) for a, b in zip(edges[:-1], edges[1:])])
    q = np.concatenate([0.5 * (b - a) * wt for a, b in zip(edges[:-1], edges[1:])]) * np.exp(-x * x)
    alpha, beta = np.zeros(m), np.zeros(m)
    pm, p = np.zeros_like(x), np.full_like(x, 1.0 / math.sqrt(q.sum()))
    for j in range(m):
        alpha[j] = (q * x * p * p).sum()
        r = (x - alpha[j]) * p - (beta[j - 1] * pm if j else 0.0)
        beta[j] = math.sqrt((q * r * r).sum())
        pm, p = p, r / beta[j]
    val, vec = np.linalg.eigh(np.diag(alpha) + np.diag(beta[:-1], 1) + np.diag(beta[:-1], -1))
    wts = vec[0] ** 2
    return val, wts / (2.0 * wts.sum())


class _Reference:
    """The source iteration in 64 bits.  A row is (octant, fluid point); rows are stored in the order
    of their hyperplane (oriented coordinate sum) over all problems, lanes are the velocities of an
    octant ordered alike, so that lane l of octant o ^ (1 << j) is lane l of octant o reflected along
    axis j.  The unknown is h' = h + x1 (the pressure jump is then a source term)."""

    def __init__(self, case, masks, kns, start=None):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.dev, self.masks, self.kns, d = dev, masks, kns, masks[0].ndim
        self.d, self.case = d, case
        c, cw = _half_range_gauss(case["nv"] // 2)
        lanes = list(itertools.product(range(len(c)), repeat=d))
        self.av = torch.tensor([[c[i] for i in l] for l in lanes], dtype=torch.float64, device=dev)   # |v|
        self.W = torch.tensor([math.prod(cw[i] for i in l) for l in lanes], dtype=torch.float64, device=dev)
        NO = 2 ** d
        spec, order = case["specular"], case["order"]
        subs = [case["sub1"], case["sub2"], case["sub3"]][:d]
        parts = []
        base = 0
        self.slices = []
        for b, (mask, kn) in enumerate(zip(masks, kns)):
            n = mask.shape[::-1]                                  # extents along x1, x2, x3
            fl = torch.from_numpy(~mask).to(dev)
            nf = int(fl.sum())
            fid = torch.full(mask.shape, -1, dtype=torch.int64, device=dev)
            fid[fl] = torch.arange(nf, device=dev)
            pos = fl.nonzero().flip(1)                            # [nf, d], x1 first
            nu = math.sqrt(math.pi) / (2.0 * kn) * (case["es"] if case["es"] else 1.0)
            x1 = pos[:, 0].double() / n[0]
            for o in range(NO):
                sgn = [-1 if (o >> j) & 1 else 1 for j in range(d)]
                plane = sum(pos[:, j] if sgn[j] > 0 else n[j] - 1 - pos[:, j] for j in range(d))
                row = {"plane": plane, "prob": torch.full_like(plane, b), "oct": torch.full_like(plane, o), "x1": x1,
                       "nu": torch.full_like(x1, nu), "idx": n[0] * torch.ones_like(x1),
                       "point": torch.arange(nf, device=dev)}
                for j in range(d):
                    solid, far, old = [], [], []
                    for step in (1, 2):
                        q = pos.clone()
                        q[:, j] -= sgn[j] * step
                        out = (q[:, j] < 0) | (q[:, j] >= n[j])
                        oo = torch.full_like(plane, o)
                        if j == 0 or case["lateral"] == "periodic":
                            crossed = torch.zeros_like(out)       # not swept yet: still the previous value
                            q[:, j] %= n[j]
                        else:
                            crossed = out
                            q[:, j] = torch.where(q[:, j] < 0, -1 - q[:, j], torch.where(q[:, j] >= n[j], 2 * n[j] - 1 - q[:, j], q[:, j]))
                            oo = torch.where(out, torch.full_like(oo, o ^ (1 << j)), oo)
                        if subs[j] > 1:
                            crossed = crossed | ((q[:, j] * subs[j]) // n[j] != (pos[:, j] * subs[j]) // n[j])
                        f = fid[tuple(q[:, k] for k in reversed(range(d)))]
                        solid.append(f < 0)
                        far.append(torch.where(f < 0, torch.full_like(f, base), base + oo * nf + f))
                        old.append(crossed)
                    wall = solid[0]
                    first = ~wall & solid[1] if order == 2 else ~wall
                    second = ~(wall | first)
                    row["K1%d" % j] = torch.where(second, 2.0, torch.where(first, 1.0, 0.0)).double()
                    row["K2%d" % j] = torch.where(second, -0.5, 0.0).double()
                    row["C0%d" % j] = torch.where(second, 1.5, 1.0).double()
                    row["wall%d" % j] = wall.double()
                    row["i1%d" % j], row["i2%d" % j] = far
                    row["o1%d" % j], row["o2%d" % j] = old
                    row["mir%d" % j] = base + (o ^ (1 << j)) * nf + row["point"]
                parts.append(row)
            self.slices.append((base, nf, fl, x1, nu, n))
            base += NO * nf
        rows = {k: torch.cat([p[k] for p in parts]) for k in parts[0]}
        del parts
        order_ = torch.argsort(rows["plane"], stable=True)
        where = torch.empty_like(order_)
        where[order_] = torch.arange(len(order_), device=dev)    # natural row -> stored row
        self.where, self.order = where, order_
        self.rows = {k: (where[v[order_]] if k[:2] in ("i1", "i2", "mi") else v[order_]) for k, v in rows.items()}
        counts = torch.bincount(self.rows["plane"]).tolist()
        self.cuts = [0] + list(itertools.accumulate(counts))
        self.sgn = torch.stack([1.0 - 2.0 * ((self.rows["oct"] >> j) & 1).double() for j in range(d)])
        self.keep = spec > 0.0 or bool(any(self.rows["o%d%d" % (s, j)].any() for s in (1, 2) for j in range(d)))
        R = self.rows
        if start is None:
            self.H = R["x1"][:, None].expand(-1, len(self.W)).contiguous()
        else:
            self.H = torch.empty(len(order_), len(self.W), dtype=torch.float64, device=dev)
            for (rho0, u0), (b0, nf, fl, x1, nu, n) in zip(start, self.slices):
                r0 = torch.from_numpy(rho0).to(dev)[fl] + x1
                uu = [torch.from_numpy(u0[j]).to(dev)[fl] for j in range(d)]
                for o in range(NO):
                    st = self.where[b0 + o * nf:b0 + (o + 1) * nf]
                    h = r0[:, None].expand(-1, len(self.W)).clone()
                    for j in range(d):
                        h += 2.0 * uu[j][:, None] * ((-1.0 if (o >> j) & 1 else 1.0) * self.av[:, j])
                    self.H[st] = h

    def moments(self):
        """Per problem: (rho', u, tau, wall numerators [d][2], model moments), each on the fluid points."""
        d, NO, case = self.d, 2 ** self.d, self.case
        vv = (self.av ** 2).sum(1)
        cols = [self.W] + [self.W * self.av[:, j] for j in range(d)] + [self.W * vv]
        cols += [self.W * self.av[:, j] * (vv - 2.5) for j in range(d)]
        pairs = [(i, j) for i in range(d) for j in range(i, d)]
        cols += [self.W * self.av[:, i] * self.av[:, j] for i, j in pairs]
        M = (self.H @ torch.stack(cols, 1))[self.where]
        out = []
        for b0, nf, fl, x1, nu, n in self.slices:
            m = M[b0:b0 + NO * nf].reshape(NO, nf, -1)
            s = [torch.tensor([-1.0 if (o >> j) & 1 else 1.0 for o in range(NO)], dtype=torch.float64, device=self.dev)[:, None] for j in range(d)]
            rho = m[:, :, 0].sum(0)
            u = [(s[j] * m[:, :, 1 + j]).sum(0) for j in range(d)]
            num = [[(m[:, :, 1 + j] * (s[j] == sig)).sum(0) for sig in (-1.0, 1.0)] for j in range(d)]
            sw2 = float((self.W * vv).sum()) * NO
            tau = 2.0 / 3.0 * m[:, :, 1 + d].sum(0) - rho + x1 * (1.0 - 2.0 / 3.0 * sw2)
            flux = [(s[j] * m[:, :, 2 + d + j]).sum(0) for j in range(d)]
            stress = {}
            if case["es"]:
                e3 = m[:, :, 1 + d].sum(0) / 3.0
                for c, (i, j) in enumerate(pairs):
                    p = (s[i] * s[j] * m[:, :, 2 + 2 * d + c]).sum(0) - (e3 if i == j else 0.0)
                    grid = NO * (self.W * (self.av[:, i] ** 2 - vv / 3.0)).sum() if i == j else 0.0
                    stress[i, j] = 2.0 * (p - x1 * grid)
            out.append((rho, u, tau, num, flux, stress))
        return out

    def iterate(self, iters):
        d, NO, case, R = self.d, 2 ** self.d, self.case, self.rows
        vv = (self.av ** 2).sum(1)
        one = torch.ones_like(self.W)
        basis = [one] + [self.av[:, j] for j in range(d)] + [vv - 1.5] + [self.av[:, j] * (vv - 2.5) for j in range(d)]
        pairs = [(i, j) for i in range(d) for j in range(i, d)]
        basis += [self.av[:, i] * self.av[:, j] for i, j in pairs]
        B = torch.stack(basis)
        den = torch.stack([R["nu"]] + [R["C0%d" % j] * R["idx"] for j in range(d)], 1)
        dwall = [NO / 2 * float((self.W * self.av[:, j]).sum()) for j in range(d)]
        alpha = 1.0 - case["specular"]
        for _ in range(iters):
            mom = self.moments()

            def rows_of(vals):     # per-problem point values -> stored rows
                return torch.cat([v.repeat(NO) for v in vals])[self.order]
            S = torch.zeros(len(self.order), len(basis), dtype=torch.float64, device=self.dev)
            S[:, 0] = R["nu"] * rows_of([m[0] for m in mom])
            for j in range(d):
                S[:, 1 + j] = self.sgn[j] * (2.0 * R["nu"] * rows_of([m[1][j] for m in mom]) + (1.0 if j == 0 else 0.0))
                # wall value of the upstream face (side -s_j), source form
                lo, hi = (rows_of([m[3][j][s] for m in mom]) for s in (0, 1))
                E = alpha * torch.where(self.sgn[j] > 0, lo, hi) / dwall[j] - (self.sgn[j] / R["idx"] if j == 0 else 0.0)
                S[:, 1 + j] += R["wall%d" % j] * E * R["idx"]
            if case["tau"]:
                S[:, 1 + d] = R["nu"] * rows_of([m[2] for m in mom])
            if case["shakhov"]:
                for j in range(d):
                    S[:, 2 + d + j] = 0.8 * (1.0 - case["shakhov"]) * R["nu"] * self.sgn[j] * rows_of([m[4][j] for m in mom])
            if case["es"]:
                for c, (i, j) in enumerate(pairs):
                    f = (1.0 - 1.0 / case["es"]) * (1.0 if i == j else 2.0)
                    S[:, 2 + 2 * d + c] = f * R["nu"] * self.sgn[i] * self.sgn[j] * rows_of([m[5][i, j] for m in mom])
            old = self.H.clone() if self.keep else None
            for a, b in zip(self.cuts[:-1], self.cuts[1:]):
                num = S[a:b] @ B
                for j in range(d):
                    K1, K2, i1, i2 = (R[k + str(j)][a:b] for k in ("K1", "K2", "i1", "i2"))
                    h1, h2 = self.H[i1], self.H[i2]
                    if old is not None:
                        h1 = torch.where(R["o1%d" % j][a:b, None], old[i1], h1)
                        h2 = torch.where(R["o2%d" % j][a:b, None], old[i2], h2)
                    t = K1[:, None] * h1 + K2[:, None] * h2
                    if case["specular"]:
                        t += (case["specular"] * R["wall%d" % j][a:b])[:, None] * old[R["mir%d" % j][a:b]]
                    num += (R["idx"][a:b, None] * self.av[:, j]) * t
                self.H[a:b] = num / (den[a:b] @ B[:1 + d])

    def results(self):
        rho, u, tau, k = [], [], [], []
        for mask, kn, (b0, nf, fl, x1, nu, n), m in zip(self.masks, self.kns, self.slices, self.moments()):
            def field(vals):
                f = torch.zeros(mask.shape, dtype=torch.float64, device=self.dev)
                f[fl] = vals
                return f
            rho.append(field(m[0] - x1 - (m[0] - x1).mean()))
            u.append(torch.stack([field(c) for c in m[1]]))
            tau.append(field(m[2]))
            k.append(2.0 / math.sqrt(math.pi) * kn * float(m[1][0].sum()) / mask.size)
        out = {"rho": rho, "u": u, "k": np.array(k)}
        if self.case["tau"]:
            out["tau"] = tau[0]
        return out


def _conv(x, w, b):
    """3 x 3 x 3 convolution with periodic padding: x [ci][z][y][x], w [co][ci][27]."""
    y = b[:, None, None, None].expand(-1, *x.shape[1:])
    for k, (dz, dy, dx) in enumerate(itertools.product((-1, 0, 1), repeat=3)):
        y = y + (w[:, :, k] @ torch.roll(x, (-dz, -dy, -dx), (1, 2, 3)).reshape(x.shape[0], -1)).reshape(-1, *x.shape[1:])
    return y


def _unet_exact(case, seed):
    feat, target, mask, wts, bias = _unet_inputs(case, seed)
    dev, L = feat.device, case["levels"]
    # the network computes with the BF16 roundings of its FP32 weights
    w = [t.to(dev).bfloat16().double().requires_grad_(case["train"]) for t in wts]
    b = [t.to(dev).bfloat16().double().requires_grad_(case["train"]) for t in bias]
    h, p, kept = feat.double(), 0, []
    for l in range(L):
        for _ in range(2):
            h, p = torch.relu(_conv(h, w[p], b[p])), p + 1
        if l < L - 1:
            kept.append(h)
            h = torch.nn.functional.avg_pool3d(h[None], 2)[0]
    for l in reversed(range(L - 1)):
        up = h.repeat_interleave(2, 1).repeat_interleave(2, 2).repeat_interleave(2, 3)
        h = torch.cat([kept[l], up])
        for _ in range(2):
            h, p = torch.relu(_conv(h, w[p], b[p])), p + 1
    y = _conv(h, w[p], b[p])
    if not case["train"]:
        return {"y": y}
    m = mask.double().reshape(y.shape[1:])
    loss = ((m * (y - target.double())) ** 2).sum() / (4 * float(mask.sum()))
    loss.backward()
    # Adam's first step from zero moments: w - lr g / (|g| + eps)
    step = [[q.double().to(dev) - 1e-3 * t.grad / (t.grad.abs() + 1e-8) for q, t in zip(old, new)] for old, new in ((wts, w), (bias, b))]
    return {"loss": float(loss), "y": y.detach(), "dw": [t.grad for t in w], "db": [t.grad for t in b], "w": step[0], "b": step[1]}


def exact(case, seed):
    if case["kind"] == "unet":
        return _unet_exact(case, seed)
    masks, kns = _problems(case, seed)
    ref = _Reference(case, masks, kns, [_start_fields(m, seed) for m in masks] if case["warm"] else None)
    ref.iterate(case["iters"])
    out = ref.results()
    if case["new"]:
        out.pop("tau", None)
    return out
