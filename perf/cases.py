"""Performance cases: the work a user has the library do, through its public entry points.

Every path a program calls per time step (or per training step) is here, over the range it is used in:
  volume    u and grad u at every leaf node (VolumePotential), plain FP64 and split precision, from the
            64-leaf box to the 10.5M-node adaptive star, p 4..16, both kernels;
  batch     many independent trees replayed as one CUDA graph (vp_batch_*);
  layer     the double-layer velocity at every volume node with its near-boundary correction;
  boundary  GMRES on the boundary integral equation and the velocity at interior points;
  forward   inference of the warm-start network, and  grad  its loss and parameter gradient;
  periodic  the periodic modified Stokes solution by FFT (PeriodicStokes);
  sisdc     time steps of the Navier-Stokes equations on the periodic box (SISDC).

A case's numbers fix sizes and geometry; the seed of prepare() draws the field values. Trees are kept
between inputs of one case, as a time-stepping program keeps them; tables, plans and handles are made
in prepare().
"""
import functools
import math

import numpy as np
import torch

import paper_1908_07392_gb300 as V
from paper_1908_07392_gb300 import inputs as I

TWO_PI = 2.0 * math.pi


def listed():
    return [
        # the smallest call: 4,096 nodes, where launches and latency count; plain FP64 and split precision
        {"name": "volume_small_fp64", "path": "volume", "kernel": "mhelmholtz", "alpha": 10.0, "p": 8,
         "precision": "fp64", "tree": "uniform", "size": 3, "geometry": 1},
        {"name": "volume_small_split", "path": "volume", "kernel": "mhelmholtz", "alpha": 10.0, "p": 8,
         "precision": "split", "tree": "uniform", "size": 3, "geometry": 1},
        # a resolved adaptive tree in plain FP64: the form users take when they want 1e-10
        {"name": "volume_adaptive_fp64", "path": "volume", "kernel": "mbiharmonic", "alpha": 30.0, "p": 16,
         "precision": "fp64", "tree": "resolved", "size": 7, "geometry": 2},
        # an ordinary tree of the batched distribution evaluated alone (p that is no power of two)
        {"name": "volume_ordinary_split", "path": "volume", "kernel": "mhelmholtz", "alpha": 137.0, "p": 12,
         "precision": "split", "tree": "gauss", "size": 150000, "geometry": 3},
        # the largest: the 10.5M-node star, split precision (the benchmark's headline workload)
        {"name": "volume_star_split", "path": "volume", "kernel": "mbiharmonic", "alpha": 300.0, "p": 16,
         "precision": "split", "tree": "star", "size": 10, "geometry": 2},
        # many uneven trees in one graph
        {"name": "batch_split", "path": "batch", "trees": 4, "nodes_min": 10000, "nodes_max": 500000,
         "precision": "split", "geometry": 4},
        # the velocity u^H of a coupled step at all 4.19M nodes, with the near-boundary correction
        {"name": "layer_coupled_step", "path": "layer", "alpha": 316.0, "p": 16, "depth": 7, "panels": 256},
        # the boundary solve of a coupled step: 8,192 unknowns, cold start
        {"name": "boundary_solve", "path": "boundary", "alpha": 316.0, "panels": 256, "targets": 2000},
        # warm start: inference for one step, and a training step's gradient
        {"name": "warmstart_forward", "path": "forward", "batch": 1, "in_ch": 10, "width": 64, "layers": 4,
         "kernel_size": 9, "nodes": 4096},
        {"name": "warmstart_grad", "path": "grad", "batch": 32, "in_ch": 10, "width": 64, "layers": 4,
         "kernel_size": 9, "nodes": 4096},
        # the periodic solution on the largest grid, and a fourth-order time step on an ordinary one
        {"name": "periodic_4096", "path": "periodic", "n": 4096, "alpha": 316.0, "side": 3.0},
        {"name": "sisdc_order4_512", "path": "sisdc", "n": 512, "order": 4, "re": 100.0, "dt": 0.005, "steps": 1},
    ]


def draw(rng):
    def log_uniform(a, b):
        return math.exp(rng.uniform(math.log(a), math.log(b)))

    path = rng.choice(["volume", "volume", "volume", "batch", "layer", "boundary", "forward", "grad", "periodic",
                       "sisdc"])
    geometry = rng.randrange(10, 10000)
    if path == "volume":
        tree = rng.choice(["uniform", "gauss", "gauss", "resolved", "star"])
        precision = rng.choice(["fp64", "split", "split"])
        fp64 = precision == "fp64"
        p = rng.choice([4, 6, 8, 11, 12, 16])
        size = {"uniform": rng.randrange(2, 6 if fp64 else 7), "gauss": round(log_uniform(1e4, 2e5 if fp64 else 5e5)),
                "resolved": rng.randrange(4, 7 if fp64 else 8), "star": rng.randrange(5, 7 if fp64 else 9)}[tree]
        return {"path": path, "kernel": rng.choice(["mhelmholtz", "mbiharmonic"]),
                "alpha": round(log_uniform(10.0, 1000.0), 3), "p": 16 if tree in ("star", "resolved") else p,
                "precision": precision, "tree": tree, "size": size, "geometry": geometry}
    if path == "batch":
        return {"path": path, "trees": rng.randrange(2, 5), "nodes_min": 10000,
                "nodes_max": round(log_uniform(2e4, 4e5)), "precision": "split", "geometry": geometry}
    if path == "layer":
        return {"path": path, "alpha": round(log_uniform(30.0, 400.0), 3), "p": rng.choice([8, 12, 16]),
                "depth": rng.randrange(4, 8), "panels": rng.randrange(64, 257)}
    if path == "boundary":
        return {"path": path, "alpha": round(log_uniform(30.0, 400.0), 3), "panels": rng.randrange(64, 321),
                "targets": rng.randrange(100, 4000)}
    if path in ("forward", "grad"):
        nodes = 16 * rng.randrange(64, 257)
        return {"path": path, "batch": rng.randrange(1, 33), "in_ch": rng.choice([8, 10, 12, 20]),
                "width": rng.choice([16, 32, 48, 64]), "layers": rng.randrange(2, 5),
                "kernel_size": rng.choice([1, 3, 5, 9]), "nodes": nodes}
    if path == "periodic":
        return {"path": path, "n": 1 << rng.randrange(5, 13), "alpha": round(log_uniform(10.0, 1000.0), 3),
                "side": rng.choice([3.0, TWO_PI])}
    return {"path": path, "n": 1 << rng.randrange(6, 11), "order": rng.randrange(1, 5),
            "re": round(log_uniform(10.0, 1000.0), 3), "dt": 0.005, "steps": rng.randrange(1, 3)}


# ------------------------------------------------------------------------------------------- geometry

def _balanced(leaves_by_level, side):
    """The coarsest 2:1-balanced refinement of a leaf set given as {level: int64 array of ix + iy 2^32}."""
    top = max(leaves_by_level)
    ix = {l: k & 0xFFFFFFFF for l, k in leaves_by_level.items()}
    iy = {l: k >> 32 for l, k in leaves_by_level.items()}
    internal = [np.zeros(0, np.int64) for _ in range(top + 2)]
    for l in range(top, 0, -1):
        keys = []
        if l in ix:
            keys.append((ix[l] >> 1) | (iy[l] >> 1) << 32)
        bx, by = internal[l] & 0xFFFFFFFF, internal[l] >> 32
        for dx in (-1, 0, 1):        # all neighbours of an internal box exist, so their parents are internal
            for dy in (-1, 0, 1):
                x, y = bx + dx, by + dy
                ok = (x >= 0) & (y >= 0) & (x < 1 << l) & (y < 1 << l)
                keys.append((x[ok] >> 1) | (y[ok] >> 1) << 32)
        internal[l - 1] = np.unique(np.concatenate(keys))
    lv, xs, ys = [], [], []
    for l in range(0, top + 1):
        if l == 0:
            boxes = np.zeros(1, np.int64)
        else:
            bx, by = internal[l - 1] & 0xFFFFFFFF, internal[l - 1] >> 32
            boxes = np.concatenate([(2 * bx + a) | (2 * by + b) << 32 for b in (0, 1) for a in (0, 1)])
        boxes = np.setdiff1d(boxes, internal[l])
        lv.append(np.full(boxes.size, l, np.int32))
        xs.append((boxes & 0xFFFFFFFF).astype(np.int32))
        ys.append((boxes >> 32).astype(np.int32))
    return I.Tree(0.0, 0.0, side, np.concatenate(lv), np.concatenate(xs), np.concatenate(ys))


def _refined(fn, p, side, tol, depth):
    """Leaves split until the leaf's Legendre tail is below tol of the largest value, then balanced."""
    t = (I.gl_nodes(p)[0] + 1.0) / 2.0
    y, x = np.divmod(np.arange(16, dtype=np.int64), 4)
    leaves, scale = {}, 0.0
    for l in range(2, depth + 1):
        h = side / 2.0 ** l
        keep = np.ones(x.size, bool)
        if l < depth:
            px = torch.from_numpy(-side / 2 + (x[:, None] + t) * h).cuda()
            py = torch.from_numpy(-side / 2 + (y[:, None] + t) * h).cuda()
            F = fn(px[:, None, :], py[:, :, None]).expand(-1, p, p).cpu().numpy()
            scale = max(scale, float(np.abs(F).max()))
            keep = I.legendre_tail(F, p) <= tol * scale
        leaves[l] = x[keep] | y[keep] << 32
        x, y = x[~keep], y[~keep]
        x, y = (np.concatenate([2 * x + a for a in (0, 1) for _ in (0, 1)]),
                np.concatenate([2 * y + b for _ in (0, 1) for b in (0, 1)]))
        if not x.size:
            break
    return _balanced({l: k for l, k in leaves.items() if k.size}, side)


@functools.lru_cache(maxsize=None)
def _gaussians(geometry, uniform):
    """Centres and widths of a Gaussian-sum source."""
    rng = np.random.default_rng(geometry)
    n = 3 if uniform else int(rng.integers(3, 11))
    box = 0.5 if uniform else 0.6
    return rng.uniform(-box, box, (n, 2)), rng.uniform(*((0.1, 0.3) if uniform else (0.02, 0.2)), n)


@functools.lru_cache(maxsize=None)
def _tree(kind, size, p, geometry):
    if kind == "uniform":
        return I.uniform_tree(size, side=2.0)
    if kind == "star":
        return _refined(_field("star", geometry, 0), p, 3.0, 1e-11, size)
    if kind == "resolved":
        return _refined(_field("resolved", geometry, 0), p, 2.0, 1e-11, size)
    # "gauss": leaves nearest to the Gaussian centres split first until the tree has `size` nodes
    c, w = _gaussians(geometry, False)
    tree, target = I.uniform_tree(2, side=2.0), max(16, size // (p * p))
    while tree.n_leaves < target:
        x0, y0, h = tree.leaf_boxes()
        d = np.hypot(x0[:, None] + h[:, None] / 2 - c[:, 0], y0[:, None] + h[:, None] / 2 - c[:, 1]) / w
        order = np.argsort(-h / (1.0 + d.min(axis=1)), kind="stable")
        split = np.zeros(tree.n_leaves, bool)
        split[order[:(target - tree.n_leaves) // 3 + 1]] = True
        leaves = {}
        for l in range(2, tree.max_level + 2):
            at, up = (tree.level == l) & ~split, (tree.level == l - 1) & split
            x = np.concatenate([tree.ix[at]] + [2 * tree.ix[up] + a for a in (0, 1) for _ in (0, 1)])
            y = np.concatenate([tree.iy[at]] + [2 * tree.iy[up] + b for _ in (0, 1) for b in (0, 1)])
            if x.size:
                leaves[l] = x.astype(np.int64) | y.astype(np.int64) << 32
        tree = _balanced(leaves, 2.0)
    return tree


# --------------------------------------------------------------------------------------------- fields

def _amplitudes(geometry, seed, n):
    return np.random.default_rng((geometry, seed)).uniform(-1.0, 1.0, n)


def _field(kind, geometry, seed):
    """The source as a function of torch coordinates: a Gaussian sum, or the smooth star-shaped field."""
    if kind == "star":
        rng = np.random.default_rng(geometry)
        phase, th = rng.uniform(0.0, TWO_PI), rng.uniform(0.0, TWO_PI, 20)
        r = np.sqrt(rng.uniform(0.0, 1.0, 20)) * 0.8 * (1.0 + 0.3 * np.cos(5 * th + phase))
        c, w = np.stack([r * np.cos(th), r * np.sin(th)], axis=1), rng.uniform(0.01, 0.05, 20)
    else:
        c, w = _gaussians(geometry, kind == "uniform")
    a = _amplitudes(geometry, seed, len(w) + 1)

    def fn(X, Y):
        out = torch.zeros_like(X + Y)
        for k in range(len(w)):
            out += a[k] * torch.exp(-((X - c[k, 0]) ** 2 + (Y - c[k, 1]) ** 2) / w[k] ** 2)
        if kind == "star":
            s = (torch.hypot(X, Y) - (1.0 + 0.3 * torch.cos(5 * torch.atan2(Y, X) + phase))) / 0.05
            lo, hi = torch.clamp(s, 0.0, 1.0), torch.clamp(1.0 - s, 0.0, 1.0)
            pa, pb = torch.exp(-1.0 / hi), torch.exp(-1.0 / lo)      # exp(-1/0) = 0
            out = pa / (pa + pb) * (out + torch.cos(2 * X + a[-1]) * torch.sin(3 * Y) + 0.5)
        return out
    return fn


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _random(g, *shape, dtype=torch.float64):
    return torch.randn(*shape, generator=g, dtype=dtype, device="cuda")


def _modes(g, n, side, count=6):
    """Smooth periodic scalar field(s): `count` random low modes on an n x n grid ([row y][column x])."""
    x = torch.arange(n, dtype=torch.float64, device="cuda") * (TWO_PI / n)
    out = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    k = torch.randint(1, 9, (2, count), generator=g, device="cuda")
    a, ph = _random(g, count), _random(g, count)
    for q in range(count):
        out += a[q] * torch.sin(k[0, q] * x + ph[q])[None, :] * torch.cos(k[1, q] * x - ph[q])[:, None]
    return out


def _flow(case, seed):
    """A divergence-free velocity on [0, 2 pi)^2 from four interacting modes, its gradient and Laplacian."""
    n, rng = case["n"], np.random.default_rng(seed)
    x = torch.arange(n, dtype=torch.float64, device="cuda") * (TWO_PI / n)
    Y, X = torch.meshgrid(x, x, indexing="ij")
    u = torch.zeros(2, n, n, dtype=torch.float64, device="cuda")
    g = torch.zeros(2, 2, n, n, dtype=torch.float64, device="cuda")
    lap = torch.zeros_like(u)
    for kx, ky, amp, _ in I.INTERACTING_MODES:
        a, th = amp * rng.uniform(0.5, 1.0), kx * X + ky * Y + rng.uniform(0.0, TWO_PI)
        s, c = torch.sin(th), torch.cos(th)
        for comp, d in ((0, -a * ky), (1, a * kx)):
            u[comp] += d * s
            g[comp, 0] += d * kx * c
            g[comp, 1] += d * ky * c
            lap[comp] -= d * (kx * kx + ky * ky) * s
    return u, g, lap


def _stokeslets(alpha, src, f, xy):
    """Velocity of modified Stokes stokeslets at src [K, 2] with strengths f [K, 2] at points xy [2, M],
    for alpha r of a few and more (closed forms)."""
    u = torch.zeros(2, xy.shape[1], dtype=torch.float64, device=xy.device)
    for s, q in zip(src, f):
        rx, ry = xy[0] - s[0], xy[1] - s[1]
        z = alpha * torch.hypot(rx, ry)
        k0, k1 = torch.special.modified_bessel_k0(z), torch.special.modified_bessel_k1(z)
        s1 = (z * z * k0 + z * k1 - 1.0) / (TWO_PI * z * z)
        s2 = -(z * z * k0 + 2.0 * z * k1 - 2.0) / (TWO_PI * z ** 4) * alpha * alpha
        dot = s2 * (rx * q[0] + ry * q[1])
        u += torch.stack([s1 * q[0] + dot * rx, s1 * q[1] + dot * ry])
    return u


def _exterior_forcing(seed):
    """Five stokeslets on circles outside the star (radius 1.6 to 2.1)."""
    rng = np.random.default_rng(seed)
    th, r = rng.uniform(0.0, TWO_PI, 5), rng.uniform(1.6, 2.1, 5)
    return np.stack([r * np.cos(th), r * np.sin(th)], axis=1), rng.uniform(-1.0, 1.0, (5, 2))


def _interior_points(case, seed):
    rng = np.random.default_rng((case["panels"], seed))
    th, r = rng.uniform(0.0, TWO_PI, case["targets"]), 0.5 * np.sqrt(rng.uniform(0.0, 1.0, case["targets"]))
    return torch.from_numpy(np.stack([r * np.cos(th), r * np.sin(th)])).cuda()


def _net_sizes(case):
    return [case["in_ch"]] + [case["width"]] * (case["layers"] - 1) + [2]


def _net_data(case, seed):
    """Parameters (layer by layer: weights [out][in][k], bias), inputs and targets of the network, FP32."""
    g, c, k = _generator(seed), _net_sizes(case), case["kernel_size"]
    parts = []
    for l in range(case["layers"]):
        bound = 1.0 / math.sqrt(c[l] * k)
        parts.append((2 * torch.rand(c[l + 1] * c[l] * k + c[l + 1], generator=g, device="cuda") - 1) * bound)
    n, b = case["nodes"], case["batch"]
    th = torch.arange(n, device="cuda") * (TWO_PI / n)
    freq, ph = torch.randint(1, 30, (b, c[0], 1), generator=g, device="cuda"), _random(g, b, c[0], 1, dtype=torch.float32)
    x = torch.sin(freq * th + ph) + 0.1 * _random(g, b, c[0], n, dtype=torch.float32)
    t = torch.cos(freq[:, :2] * th - ph[:, :2])
    return torch.cat(parts), x.contiguous(), t.contiguous()


# ------------------------------------------------------------------------------------------- the cases

class _Held:
    """Library handles of a state, freed in order with it."""

    def __init__(self, *free):
        self.free = free

    def __del__(self):
        for f in self.free:
            f()


KERNELS = {"mhelmholtz": V.VP_KERNEL_MHELMHOLTZ, "mbiharmonic": V.VP_KERNEL_MBIHARMONIC}
PRECISIONS = {"fp64": V.VP_PREC_FP64, "split": V.VP_PREC_SPLIT}


def _volume(case, seed):
    tree = _tree(case["tree"], case["size"], case["p"], case["geometry"])
    vp = V.VolumePotential(KERNELS[case["kernel"]], case["alpha"], case["p"], tree,
                           precision=PRECISIONS[case["precision"]])
    xy = vp.nodes()
    f = _field(case["tree"], case["geometry"], seed)(xy[0], xy[1])
    u, g = torch.empty_like(f), torch.empty_like(xy)
    if case["precision"] == "split":
        V.vp_autotune(vp.tree, f, u, g)
    return vp, f, u, g


def _batch_members(case):
    """The trees of a batch: node counts log-uniform, alpha log-uniform in [10, 1000], p of {8, 12, 16}."""
    rng = np.random.default_rng(case["geometry"])
    for k in range(case["trees"]):
        nodes = int(np.exp(rng.uniform(np.log(case["nodes_min"]), np.log(case["nodes_max"]))))
        alpha, p = float(np.exp(rng.uniform(np.log(10.0), np.log(1000.0)))), int(rng.choice([8, 12, 16]))
        yield {"kernel": "mhelmholtz", "alpha": alpha, "p": p, "precision": case["precision"], "tree": "gauss",
               "size": nodes, "geometry": case["geometry"] + 1000 * (k + 1)}


def prepare(case, seed):
    path = case["path"]
    if path == "volume":
        return {"path": path, "args": _volume(case, seed)}
    if path == "batch":
        vps, f, u, g = zip(*[_volume(m, seed) for m in _batch_members(case)])
        batch = V.vp_batch_create([v.tree for v in vps], f, u, g)
        held = _Held(lambda: V.vp_batch_free(batch), lambda: [v.close() for v in vps])
        return {"path": path, "batch": batch, "u": u, "g": g, "f": f, "held": held}
    if path == "layer":
        phase = 0.4
        b = V.BIE(case["alpha"], phase=phase, n_panels=case["panels"], max_krylov=1)
        nodes = b.nodes.clone()
        b.close()
        tree = I.uniform_tree(case["depth"], side=3.0)
        vp = V.VolumePotential(V.VP_KERNEL_MBIHARMONIC, case["alpha"], case["p"], tree, precision=V.VP_PREC_SPLIT)
        layer = V.vp_layer_create(vp.tree, nodes[:5].cpu().numpy())
        held = _Held(lambda: V.vp_layer_free(layer), vp.close)
        V.vp_layer_near_star(layer, 1.0, 0.3, 5, phase, case["panels"])
        g = _generator(seed)
        k, a, ph = torch.arange(1, 9, device="cuda")[:, None], _random(g, 2, 8, 1), _random(g, 2, 8, 1)
        mu = (a * torch.sin(k * nodes[6] + ph)).sum(1).t().contiguous()
        return {"path": path, "layer": layer, "mu": mu, "held": held,
                "u": torch.empty(2, vp.N, dtype=torch.float64, device="cuda")}
    if path == "boundary":
        b = V.BIE(case["alpha"], phase=0.4, n_panels=case["panels"], max_krylov=60)
        src, f = _exterior_forcing(seed)
        g = _stokeslets(case["alpha"], src, f, b.nodes[:2]).t().reshape(-1).contiguous()
        return {"path": path, "bie": b, "g": g, "xy": _interior_points(case, seed)}
    if path in ("forward", "grad"):
        net = V.WarmStartNet(in_ch=case["in_ch"], width=case["width"], out_ch=2, n_layers=case["layers"],
                             ksize=case["kernel_size"], n=case["nodes"], max_batch=case["batch"])
        params, x, t = _net_data(case, seed)
        net.set_params(params)
        return {"path": path, "net": net, "x": x, "t": t}
    if path == "periodic":
        plan = V.PeriodicStokes(case["alpha"], case["n"], case["side"])
        g = _generator(seed)
        F = torch.stack([_modes(g, case["n"], case["side"]) for _ in range(2)])
        n = case["n"]
        return {"path": path, "plan": plan, "F": F, "u": torch.empty_like(F), "held": _Held(plan.close),
                "g": torch.empty(2, 2, n, n, dtype=torch.float64, device="cuda")}
    sd = V.SISDC(case["re"], case["dt"], case["order"], case["n"], TWO_PI)
    u, g, lap = _flow(case, seed)
    return {"path": path, "sisdc": sd, "steps": case["steps"], "start": (u, g, lap), "held": _Held(sd.close),
            "u": torch.empty_like(u), "g": torch.empty_like(g)}


def run(state):
    path = state["path"]
    if path == "volume":
        vp, f, u, g = state["args"]
        return vp(f, u, g)
    if path == "batch":
        V.vp_batch_run(state["batch"])
        return list(state["u"]) + list(state["g"])
    if path == "layer":
        V.vp_layer_eval(state["layer"], state["mu"], state["u"])
        return state["u"]
    if path == "boundary":
        mu, _, _ = state["bie"].solve(state["g"], tol=1e-11)
        return mu, state["bie"].eval(mu, state["xy"])
    if path == "forward":
        return state["net"].forward(state["x"])
    if path == "grad":
        return state["net"].grad(state["x"], state["t"])
    if path == "periodic":
        return state["plan"](state["F"], state["u"], state["g"])
    state["sisdc"].set(*state["start"])
    state["sisdc"].step(state["steps"])
    return state["sisdc"].get(state["u"], state["g"])


def _volume_work(case):
    """Inputs and outputs once, and the contractions of the method: near tables (about nine adjacent
    leaves), leaf sources to coefficients and back, and 27 translations per box and channel."""
    leaves, n, c = _tree(case["tree"], case["size"], case["p"], case["geometry"]).n_leaves, case["p"] ** 2, 81
    ch = 2 if case["kernel"] == "mbiharmonic" else 1
    flops = leaves * (9 * 6.0 * n * n + 8.0 * n * ch * c) + leaves * 4 / 3 * 27 * 2.0 * c * c * ch
    return {"bytes": 32.0 * leaves * n, "flops": flops}


def work(case):
    path = case["path"]
    if path == "volume":
        return _volume_work(case)
    if path == "batch":
        each = [_volume_work(m) for m in _batch_members(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    if path == "layer":   # two outputs per node; one local expansion to the nodes of each leaf, 27 translations per box
        leaves, n, c = 4 ** case["depth"], case["p"] ** 2, 81
        flops = 2 * leaves * (2.0 * n * 2 * c)
        return {"bytes": 16.0 * leaves * n + 32.0 * case["panels"] * 16, "flops": flops}
    if path == "boundary":   # the dense matrix is read once per Krylov step (about 18) and for two residuals
        n = 32 * case["panels"]
        return {"bytes": 20 * 8.0 * n * n, "flops": 20 * 2.0 * n * n}
    if path in ("forward", "grad"):
        c = _net_sizes(case)
        macs = sum(a * b for a, b in zip(c, c[1:])) * case["kernel_size"] * case["nodes"] * case["batch"]
        io = 4.0 * case["batch"] * case["nodes"] * (case["in_ch"] + 2)
        first = c[0] * c[1] * case["kernel_size"] * case["nodes"] * case["batch"]  # no gradient of the input
        return {"bytes": io, "flops": 2.0 * macs if path == "forward" else 2.0 * (3 * macs - first)}
    n2 = float(case["n"]) ** 2
    fft = 4 * 10 * n2 * math.log2(case["n"])   # four complex 2-D transforms
    if path == "periodic":
        return {"bytes": 64.0 * n2, "flops": fft}
    k = case["order"]
    solves = case["steps"] * (1 if k == 1 else k * k - k)
    return {"bytes": 8 * 14.0 * n2, "flops": solves * fft}


# ------------------------------------------------------------------------- the results in 64 bits, by torch

def _nodes(tree, p):
    x, y = I.node_coords(tree, p)
    return torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()


def _line(x, c, w, t, half):
    """Heat kernel at time t applied along one axis to exp(-(s - c)^2 / w^2) on [-half, half], and its
    derivative."""
    var = 4.0 * t + w * w
    sig2 = 1.0 / (1.0 / (4.0 * t) + 1.0 / (w * w))
    sig, mu = sig2 ** 0.5, (x / (4.0 * t) + c / (w * w)) * sig2
    lo, hi = (half + mu) / sig, (half - mu) / sig
    e = torch.exp(-(x - c) ** 2 / var)
    v = 0.5 * w / var ** 0.5 * e * (torch.erf(hi) + torch.erf(lo))
    edge = w / var ** 0.5 * e / math.sqrt(math.pi) * sig / (4.0 * t) * (torch.exp(-lo * lo) - torch.exp(-hi * hi))
    return v, -2.0 * (x - c) / var * v + edge


def _volume_exact(case, seed):
    """The potential of the Gaussian sum on the box, K0(alpha r) = int exp(-alpha^2 t - r^2 / 4t) / 2t dt
    and likewise log r, by the trapezoidal rule in log t. (The library integrates the leaf
    interpolants: on unresolved trees the two differ by the interpolation error.)"""
    if case["tree"] == "star":
        return None       # no closed form of the blended field's potential
    tree = _tree(case["tree"], case["size"], case["p"], case["geometry"])
    X, Y = _nodes(tree, case["p"])
    if X.numel() > 3_000_000:
        return None       # over 20 seconds
    c, w = _gaussians(case["geometry"], case["tree"] == "uniform")
    a = torch.from_numpy(_amplitudes(case["geometry"], seed, len(w) + 1)[:-1]).cuda()[:, None]
    cx, cy, w = (torch.from_numpy(np.ascontiguousarray(v)).cuda()[:, None] for v in (c[:, 0], c[:, 1], w))
    al2, half, h, two = case["alpha"] ** 2, tree.side / 2, 0.25, case["kernel"] == "mbiharmonic"
    mass = (a * (math.pi / 4) * w * w * (torch.erf((half - cx) / w) + torch.erf((half + cx) / w))
            * (torch.erf((half - cy) / w) + torch.erf((half + cy) / w))).sum()
    u, g = torch.zeros_like(X), torch.zeros(2, X.numel(), dtype=torch.float64, device="cuda")
    s, end = math.log(1e-17 / al2), math.log(1e17 if two else 45.0 / al2)
    while s < end:
        t = math.exp(s)
        factor = math.expm1(-al2 * t) / al2 if two else math.exp(-al2 * t)
        for at in range(0, X.numel(), 1 << 18):
            q = slice(at, at + (1 << 18))
            vx, dx = _line(X[q], cx, w, t, half)
            vy, dy = _line(Y[q], cy, w, t, half)
            uq = factor * (a * vx * vy).sum(0)
            if two:
                uq = uq + mass * math.exp(-0.25 / t) / (4.0 * math.pi * t * al2)
            u[q] += h * t * uq
            g[0, q] += h * t * factor * (a * dx * vy).sum(0)
            g[1, q] += h * t * factor * (a * vx * dy).sum(0)
        s += h
    return u, g


def _solve_periodic(alpha, side, F):
    """Velocity and gradient of (alpha^2 - Laplacian) u + grad p = F, div u = 0 on the periodic grid."""
    n = F.shape[-1]
    k = TWO_PI / side * torch.fft.fftfreq(n, d=1.0 / n, dtype=torch.float64, device=F.device)
    kd = k.clone()
    kd[n // 2] = 0.0
    KX, KY, DX, DY = k[None, :], k[:, None], kd[None, :], kd[:, None]
    K2 = KX ** 2 + KY ** 2
    den = torch.where(K2 > 0, 1.0 / (K2 * (alpha ** 2 + K2)), torch.zeros_like(K2))
    zero = torch.where(K2 > 0, 0.0, 1.0 / alpha ** 2)
    fx, fy = torch.fft.fft2(F[0]), torch.fft.fft2(F[1])
    cross = KX * KY * den
    cross[n // 2, :] = 0.0
    cross[:, n // 2] = 0.0
    cross[n // 2, n // 2] = KX[0, n // 2] * KY[n // 2, 0] * den[n // 2, n // 2]
    uh = ((KY ** 2 * den + zero) * fx - cross * fy, (KX ** 2 * den + zero) * fy - cross * fx)
    u = torch.stack([torch.fft.ifft2(v).real for v in uh])
    g = torch.stack([torch.stack([torch.fft.ifft2(1j * d * v).real for d in (DX, DY)]) for v in uh])
    return u, g


def _sisdc_exact(case, seed):
    u, g, lap = _flow(case, seed)
    re, K = case["re"], case["order"]
    p = max(1, K - 1)
    al2 = re / (case["dt"] / p)
    wts = np.zeros((p, p + 1))
    for j in range(p + 1):
        others = np.delete(np.arange(p + 1.0), j)
        ci = np.polyint(np.poly(others) / np.prod(j - others))
        wts[:, j] = [np.polyval(ci, m + 1.0) - np.polyval(ci, float(m)) for m in range(p)]

    def advect(u, g):
        return torch.stack([u[0] * g[a, 0] + u[1] * g[a, 1] for a in range(2)])

    def solve(F):
        un, gn = _solve_periodic(math.sqrt(al2), TWO_PI, F)
        return un, gn, al2 * un - F

    for _ in range(case["steps"]):
        U = [(u, g, lap)]
        for m in range(p):
            U.append(solve(al2 * U[m][0] - re * advect(U[m][0], U[m][1])))
        for _ in range(K - 1):
            N = [advect(v[0], v[1]) for v in U]
            W = [(u, g, lap)]
            for m in range(p):
                q = sum(wts[m, j] * (U[j][2] - re * N[j]) for j in range(p + 1))
                W.append(solve(al2 * W[m][0] - re * (advect(W[m][0], W[m][1]) - N[m]) - U[m + 1][2] + q))
            U = W
        u, g, lap = U[p]
    return u, g


def _net_exact(case, seed):
    params, x, t = _net_data(case, seed)
    params, x, t = params.double().requires_grad_(case["path"] == "grad"), x.double(), t.double()
    c, k = _net_sizes(case), case["kernel_size"]
    at = 0
    for l in range(case["layers"]):
        W = params[at:at + c[l + 1] * c[l] * k].view(c[l + 1], c[l] * k)
        at += W.numel()
        b = params[at:at + c[l + 1]]
        at += c[l + 1]
        cols = torch.stack([torch.roll(x, k // 2 - q, dims=2) for q in range(k)], dim=2)
        x = torch.matmul(W, cols.reshape(x.shape[0], c[l] * k, -1)) + b[:, None]
        if l < case["layers"] - 1:
            x = torch.relu(x)
    if case["path"] == "forward":
        return x
    loss = ((x - t) ** 2).mean()
    loss.backward()
    return params.grad, float(loss.detach())


def exact(case, seed):
    path = case["path"]
    if path == "volume":
        return _volume_exact(case, seed)
    if path == "batch":
        u, g = zip(*[_volume_exact(m, seed) for m in _batch_members(case)])
        return list(u) + list(g)
    if path == "layer":
        return None       # adaptive quadrature of every (node, panel) pair: over 20 seconds
    if path == "boundary":   # no closed form of the density; inside the star the velocity is the stokeslets'
        return None, _stokeslets(case["alpha"], *_exterior_forcing(seed), _interior_points(case, seed))
    if path in ("forward", "grad"):
        return _net_exact(case, seed)
    if path == "periodic":
        g = _generator(seed)
        F = torch.stack([_modes(g, case["n"], case["side"]) for _ in range(2)])
        return _solve_periodic(case["alpha"], case["side"], F)
    return _sisdc_exact(case, seed)
