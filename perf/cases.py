"""Performance cases: what a user of the ray-shooting library has it do.

Every case goes through the public binding (paper_2204_10871_gb300.irs): single
maps by the brute force and by the interpolated method, a band of lattice rows,
several maps in one call, deflections of chosen rays, and the learned far
field's network (forward, and the gradient of a training step).  Sizes are
those of the benchmark's workloads and side studies and of the tests.

Fields of a case, by "kind":
  map, noalloc   kappa_star, kappa_s, gamma; source region (cx, cy, sx, sy);
                 nx x ny pixels; nav rays per unlensed pixel; n lenses of mass
                 shape `shape`; plane "rect" / "circle"; method; cell_mult,
                 variant
  rows           the same, and `rows` lattice rows across the middle
  rays           the same, and `k` rays drawn in the plane's central quarter
  batch          `maps` uneven maps (drawn from `config`, at most max_rays rays
                 each) at one cell_mult and variant
  mlp-forward, mlp-grad   `k` points
"""
import math

import numpy as np
import torch

from paper_2204_10871_gb300 import irs, lensgen

METHODS = {"brute": irs.IRS_BRUTE, "interp": irs.IRS_INTERP}
PLANES = {"rect": irs.IRS_PLANE_RECT, "circle": irs.IRS_PLANE_CIRCLE}
SERIES_TERMS = {0: 6, 16: 4}  # level-2 terms of the ray-pass variants used here
NET_PARAMS = 13000
NET_FLOPS = 2 * (3 * 64 * 64 + 64 * 8)  # one point's forward products
EXACT_PAIRS = 1.0e11  # pair terms that the FP64 sum below gets through in a few seconds


def _map(name, method, kappas, src, npix, nav, n, shape="uniform", plane="rect", cell_mult=0.0, variant=0, **more):
    c = {"name": name, "kind": "map", "method": method, "kappa_star": kappas[0], "kappa_s": kappas[1],
         "gamma": kappas[2], "cx": src[0], "cy": src[1], "sx": src[2], "sy": src[3], "nx": npix[0], "ny": npix[1],
         "nav": nav, "n": n, "shape": shape, "plane": plane, "cell_mult": cell_mult, "variant": variant}
    c.update(more)
    return c


def listed():
    paper_mid = ((0.45, 0.0, 0.45), (0.0, 0.0, 20.0, 20.0), (2000, 2000), 100.0, 100000, "salpeter")
    return [
        # the smallest whole map: a first look at a parameter set, or one step
        # of a fit that makes thousands of maps; launches and latency count
        _map("brute-64", "brute", (0.3, 0.0, 0.3), (0.0, 0.0, 5.0, 5.0), (64, 64), 4.0, 40, "equal"),
        # few lenses, where the brute force is the method of choice
        _map("brute-128", "brute", (0.3, 0.0, 0.3), (0.0, 0.0, 5.0, 5.0), (128, 128), 25.0, 150, "equal"),
        # a band of the mid-size workload by the brute force: the reference
        # that interpolated maps are judged by, and chunked or sharded sweeps
        _map("brute-band", "brute", *paper_mid, kind="rows", rows=64),
        # a small map by the interpolated method at its default settings
        _map("interp-128", "interp", (0.3, 0.0, 0.3), (0.0, 0.0, 5.0, 5.0), (128, 128), 25.0, 150, "equal"),
        # a small survey map, at the settings of the many-map workload
        _map("interp-500", "interp", (0.3, 0.0, 0.25), (0.0, 0.0, 10.0, 10.0), (500, 500), 16.0, 10000,
             cell_mult=0.7, variant=16),
        # circular lens plane about an off-centre source region, odd map sides,
        # default settings
        _map("interp-circle", "interp", (0.35, 0.1, 0.25), (1.5, -0.7, 10.0, 7.2), (701, 505), 20.0, 50000,
             plane="circle"),
        # the mid-size production map, at the autotuned setting
        _map("paper-mid", "interp", *paper_mid, cell_mult=0.573, variant=16),
        # the high-resolution map (1e6 lenses, 1e8 pixels), autotuned setting
        _map("high-res", "interp", (0.35, 0.15, 0.4), (0.0, 0.0, 25.0, 25.0), (10000, 10000), 40.0, 1000000,
             cell_mult=0.72, variant=16),
        # a survey's uneven maps in one call (one replayed graph)
        {"name": "batch-24", "kind": "batch", "maps": 24, "config": 4, "max_rays": 1.0e9, "cell_mult": 0.7,
         "variant": 16},
        # deflections of chosen rays: the protective-border study's statistics
        _map("rays-50000", "brute", (0.4, 0.0, 0.0), (0.0, 0.0, 155.5, 155.5), (64, 64), 64.0, 10000, "equal",
             kind="rays", k=50000),
        # the learned far field: coefficients at every level-1 cell of a map ...
        {"name": "net-cells", "kind": "mlp-forward", "k": 300000},
        # ... and the gradient of one training batch
        {"name": "net-grad", "kind": "mlp-grad", "k": 4096},
    ]


# ------------------------------------------------------------------ drawing
def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _kappas(rng):
    """Convergences and shear of the many-map workload, away from the singular
    mean lens map."""
    while True:
        ks = rng.uniform(0.1, 0.6)
        kss = ks * rng.choice([0.0, 0.43, 1.5])
        g = rng.uniform(0.1, 0.6)
        if min(abs(1 - ks - kss - g), abs(1 - ks - kss + g)) >= 0.15:
            return ks, kss, g


def _draw_map(rng, method, work_max, pix, lenses, rays_max):
    while True:
        sx, sy = rng.uniform(3.0, 20.0), rng.uniform(3.0, 20.0)
        nx = max(24, int(_log(rng, *pix)))
        ny = max(24, min(pix[1], int(nx * sy / sx) + rng.randint(-3, 3)))
        centre = (rng.choice([0.0, rng.uniform(-2, 2)]), rng.choice([0.0, rng.uniform(-2, 2)]))
        c = _map("", method, _kappas(rng), centre + (sx, sy), (nx, ny), rng.uniform(4.0, 100.0),
                 int(_log(rng, *lenses)),
                 rng.choice(["equal", "uniform", "salpeter"]), rng.choice(["rect", "rect", "rect", "circle"]))
        del c["name"]
        s = _size(c)
        if method == "interp":
            c["cell_mult"], c["variant"] = rng.choice([(0.0, 0), (0.7, 16), (0.573, 16), (0.72, 16)])
            if c["plane"] == "circle" and s["r"] ** 2 / _cell(c, s) ** 2 > 2.0e6:
                continue
            if 2 * max(s["ix"], s["iy"], 2 * s["r"]) / _cell(c, s) > 9000:  # a grid that the transforms hold
                continue
        if s["nrx"] * s["nry"] <= rays_max and work(c)["flops"] <= work_max:
            return c


def draw(rng):
    kind = rng.choice(["brute", "brute", "noalloc", "rows", "interp", "interp", "interp", "interp", "rows-interp",
                       "batch", "rays", "mlp-forward", "mlp-grad"])
    if kind in ("mlp-forward", "mlp-grad"):
        top = 300000 if kind == "mlp-forward" else 16384
        return {"kind": kind, "k": int(_log(rng, 64, top))}
    if kind == "batch":
        return {"kind": "batch", "maps": rng.randint(2, 24), "config": rng.randint(10, 10 ** 6),
                "max_rays": _log(rng, 3.0e8, 1.0e9), "cell_mult": 0.7, "variant": 16}
    if kind in ("interp", "rows-interp"):
        c = _draw_map(rng, "interp", 2.0e12, (64, 2500), (60, 200000), 2.0e10)
        if kind == "rows-interp":
            c["kind"], c["rows"] = "rows", max(1, int(_size(c)["nry"] * rng.uniform(0.05, 0.6)))
        return c
    if kind == "rows":
        c = _draw_map(rng, "brute", 1.0e18, (200, 1500), (3000, 50000), 2.0e9)
        c["kind"] = "rows"
        c["rows"] = max(1, min(int(_size(c)["nry"]), int(_log(rng, 1, 300)), int(5.0e11 / (_size(c)["nrx"] * c["n"]))))
        return c
    if kind == "rays":
        c = _draw_map(rng, "brute", 1.0e18, (64, 600), (100, 10000), 1.0e9)
        c["kind"], c["k"] = "rays", int(_log(rng, 100, 50000))
        return c
    c = _draw_map(rng, "brute", 4.0e12, (32, 400), (20, 5000), 8.0e7)
    c["kind"] = "noalloc" if kind == "noalloc" else "map"
    return c


# ------------------------------------------------------------------ sizes
def _size(c):
    """The plane of a case: the protective border 10 sqrt(kappa_*), sides
    (S + 2 P) / |1 - kappa -+ gamma| in whole rays, its centre."""
    kap = c["kappa_star"] + c["kappa_s"]
    l1, l2 = 1.0 - kap - c["gamma"], 1.0 - kap + c["gamma"]
    P = 10.0 * math.sqrt(c["kappa_star"])
    dx = math.sqrt(c["sx"] / c["nx"] * (c["sy"] / c["ny"]) / c["nav"])
    nrx = max(1, math.ceil((c["sx"] + 2.0 * P) / abs(l1) / dx - 1e-9))
    nry = max(1, math.ceil((c["sy"] + 2.0 * P) / abs(l2) / dx - 1e-9))
    ix, iy = nrx * dx, nry * dx
    return {"dx": dx, "nrx": nrx, "nry": nry, "ix": ix, "iy": iy, "cx": c["cx"] / l1, "cy": c["cy"] / l2,
            "r": 0.5 * math.hypot(ix, iy)}


def _cell(c, s):
    rule = min(math.sqrt(s["ix"] * s["iy"] / max(1, c["n"])), min(s["ix"], s["iy"]) / 10.0)
    return s["dx"] * min(1024, max(4, math.ceil(rule * (c["cell_mult"] or 1.0) / s["dx"] - 1e-9)))


def _configs(c):
    """The uneven maps of a batch: 500^2 ... 2000^2 pixels over 10 ... 20
    theta_E, 1e3 ... 1e5 lenses, 16 ... 100 rays per pixel."""
    rng = np.random.Generator(np.random.PCG64(c["config"]))
    out = []
    while len(out) < c["maps"]:
        ks, frac, g = rng.uniform(0.1, 0.6), float(rng.choice([0.0, 0.3, 0.6])), rng.uniform(0.1, 0.6)
        kss = ks * frac / (1.0 - frac)
        S, npix, nav = rng.uniform(10.0, 20.0), int(rng.integers(500, 2001)), rng.uniform(16.0, 100.0)
        n = int(round(10 ** rng.uniform(3.0, 5.0)))
        if min(abs(1 - ks - kss - g), abs(1 - ks - kss + g)) < 0.15:
            continue
        m = _map("", "interp", (ks, kss, g), (0.0, 0.0, S, S), (npix, npix), nav, n, "uniform",
                 cell_mult=c["cell_mult"], variant=c["variant"])
        s = _size(m)
        if s["nrx"] * s["nry"] <= c["max_rays"]:
            out.append(m)
    return out


def work(case):
    c = case
    if c["kind"] == "mlp-forward":
        return {"bytes": c["k"] * (8 + 32) + 4 * NET_PARAMS, "flops": c["k"] * NET_FLOPS}
    if c["kind"] == "mlp-grad":
        return {"bytes": c["k"] * (8 + 32) + 8 * NET_PARAMS, "flops": 3 * c["k"] * NET_FLOPS}
    if c["kind"] == "batch":
        each = [work(m) for m in _configs(c)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    s = _size(c)
    lens = 24 * c["n"]
    if c["kind"] == "rays":  # index in, position and pixel out
        return {"bytes": lens + c["k"] * (8 + 16 + 8), "flops": 10 * c["k"] * c["n"]}
    rays = s["nrx"] * (c["rows"] if c["kind"] == "rows" else s["nry"])
    out = c["nx"] * c["ny"] * (4 if c["kind"] == "rows" else 8)
    if c["method"] == "brute":
        return {"bytes": lens + out, "flops": 10 * rays * c["n"]}
    # interpolated: the 3 x 3 cells' lenses per ray, the level-2 series, and
    # the smooth terms and pixel
    area = math.pi * s["r"] ** 2 if c["plane"] == "circle" else s["ix"] * s["iy"]
    near = min(c["n"], 9.0 * c["n"] * _cell(c, s) ** 2 / area)
    return {"bytes": lens + out, "flops": rays * (10.0 * near + 8.0 * (SERIES_TERMS[c["variant"]] - 1) + 20.0)}


# ------------------------------------------------------------------ inputs
def _params(c):
    src = (c["cx"] - c["sx"] / 2, c["cx"] + c["sx"] / 2, c["cy"] - c["sy"] / 2, c["cy"] + c["sy"] / 2)
    return irs.make_params(c["kappa_star"], c["kappa_s"], c["gamma"], src, (c["nx"], c["ny"]), c["nav"],
                           n_star=c["n"], plane=PLANES[c["plane"]], method=METHODS[c["method"]],
                           cell_mult=c["cell_mult"], kernel_variant=c["variant"])


def _lenses(c, seed):
    """Lenses uniform over the lens plane, rescaled to the case's kappa_*, on
    the host (numpy's seeded generator)."""
    s = _size(c)
    circle = c["plane"] == "circle"
    edge = 1.0 - 1e-12  # inside the plane whatever the last bit of its corners
    hx, hy = 0.5 * s["ix"] * edge, 0.5 * s["iy"] * edge
    box = (s["cx"] - hx, s["cx"] + hx, s["cy"] - hy, s["cy"] + hy)
    area = math.pi * s["r"] ** 2 if circle else s["ix"] * s["iy"]
    return lensgen.lens_field(c["n"], None if circle else box, shape=c["shape"], seed=seed,
                              total_mass=c["kappa_star"] * area / math.pi,
                              disc=(s["cx"], s["cy"], s["r"] * edge) if circle else None)


def _ray_idx(c, seed):
    s = _size(c)
    rng = np.random.Generator(np.random.PCG64(seed + 7))
    i = rng.integers(s["nrx"] // 4, 3 * s["nrx"] // 4 + 1, c["k"])
    j = rng.integers(s["nry"] // 4, 3 * s["nry"] // 4 + 1, c["k"])
    return j * s["nrx"] + i


def _net(c, seed):
    """A network at the spread of a trained one, points over the plane, targets
    of unit variance."""
    rng = np.random.Generator(np.random.PCG64(seed))
    theta = rng.uniform(-0.125, 0.125, NET_PARAMS)
    for lo, hi in ((4096, 4160), (8256, 8320), (12416, 12480), (12992, 13000)):
        theta[lo:hi] = 0.02 * rng.standard_normal(hi - lo)  # biases
    freq = 2.0 * rng.standard_normal((32, 2))
    x = rng.uniform(-1.0, 1.0, (c["k"], 2))
    t = rng.standard_normal((c["k"], 8))
    return [np.ascontiguousarray(v, dtype=np.float32) for v in (theta, freq, x, t)]


def _one(c, seed):
    xy, m = _lenses(c, seed)
    shape = (c["ny"], c["nx"])
    st = {"xy": torch.from_numpy(xy).cuda(), "m": torch.from_numpy(m).cuda(), "params": _params(c)}
    if c["kind"] != "noalloc":
        st["plan"] = irs.Plan(st["params"])
    if c["kind"] != "rays":
        st["counts"] = torch.zeros(shape, dtype=torch.uint32, device="cuda")
    if c["kind"] in ("map", "noalloc"):
        st["mag"] = torch.zeros(shape, dtype=torch.float32, device="cuda")
    return st


def prepare(case, seed):
    c = case
    if c["kind"].startswith("mlp"):
        theta, freq, x, t = _net(c, seed)
        # the learned field's test configuration; the network does not depend on it
        plan = irs.Plan(irs.make_params(0.4, 0.1, 0.35, (-2.0, 2.0, -2.0, 2.0), 64, 16.0, method=irs.IRS_MLP))
        irs.irs_mlp_params(plan.handle, theta, freq)
        return {"case": c, "plan": plan, "x": torch.from_numpy(x).cuda(), "t": torch.from_numpy(t).cuda()}
    if c["kind"] == "batch":
        return {"case": c, "maps": [_one(m, seed * 100 + k) for k, m in enumerate(_configs(c))]}
    st = _one(c, seed)
    st["case"] = c
    if c["kind"] == "rays":
        st["idx"] = torch.from_numpy(_ray_idx(c, seed)).cuda()
        st["beta"] = torch.zeros((c["k"], 2), dtype=torch.float64, device="cuda")
        st["pixel"] = torch.zeros(c["k"], dtype=torch.int64, device="cuda")
    if c["kind"] == "rows":
        r0 = (st["plan"].info.n_rays_y - c["rows"]) // 2
        if c["method"] == "brute":
            r0 = r0 // 64 * 64  # a whole row of tiles, as sweeps in pieces take them
        st["band"] = (r0, r0 + c["rows"])
    return st


def run(state):
    c = state["case"]
    if c["kind"] == "mlp-forward":
        return {"y": irs.irs_mlp_forward(state["plan"].handle, state["x"])}
    if c["kind"] == "mlp-grad":
        grad, loss = irs.irs_mlp_grad(state["plan"].handle, state["x"], state["t"])
        return {"grad": grad, "loss": loss}
    if c["kind"] == "batch":
        ms = state["maps"]
        irs.irs_make_maps_batched([s["plan"].handle for s in ms], [s["xy"] for s in ms], [s["m"] for s in ms],
                                  [s["counts"] for s in ms], [s["mag"] for s in ms])
        return [{"counts": s["counts"].view(torch.int32), "mag": s["mag"]} for s in ms]
    if c["kind"] == "rays":
        irs.irs_shoot_rays(state["plan"].handle, state["xy"], state["m"], state["idx"], state["beta"], state["pixel"])
        return {"beta": state["beta"], "pixel": state["pixel"]}
    counts = state["counts"]
    if c["kind"] == "rows":
        counts.zero_()
        irs.irs_make_map_rows(state["plan"].handle, state["xy"], state["m"], *state["band"], counts)
        return {"counts": counts.view(torch.int32)}
    if c["kind"] == "noalloc":
        irs.irs_make_map_brute_noalloc(state["params"], state["xy"], state["m"], counts, state["mag"])
    else:
        irs.irs_make_map(state["plan"].handle, state["xy"], state["m"], counts, state["mag"])
    return {"counts": counts.view(torch.int32), "mag": state["mag"]}


# ------------------------------------------------------------------ 64 bits
def _beta64(c, s, xy, m, z):
    """Source positions of the image-plane points z (complex128): every lens
    summed, the smooth terms, and the sheet in closed form."""
    area = math.pi * s["r"] ** 2 if c["plane"] == "circle" else s["ix"] * s["iy"]
    ks = math.pi * float(m.sum()) / area
    acc = torch.zeros_like(z)
    step = max(1, int(3.0e8 / z.numel()))
    for k in range(0, m.numel(), step):
        dx = z.real[:, None] - xy[None, k:k + step, 0]
        dy = z.imag[:, None] - xy[None, k:k + step, 1]
        w = m[None, k:k + step] / (dx * dx + dy * dy)
        acc += torch.complex((w * dx).sum(1), -(w * dy).sum(1))
    out = (1.0 - c["kappa_s"]) * z.conj() - c["gamma"] * z - acc
    if c["plane"] == "circle":
        return (out - ks * complex(s["cx"], -s["cy"])).conj()
    a1, a2 = s["cx"] - s["ix"] / 2, s["cx"] + s["ix"] / 2
    b1, b2 = s["cy"] - s["iy"] / 2, s["cy"] + s["iy"] / 2
    out = out + ks * (z - 2.0 * a2)
    for x, y, sign in ((a1, b1, 1.0), (a2, b1, -1.0), (a1, b2, -1.0), (a2, b2, 1.0)):
        w = z - complex(x, y)
        out = out - 1j * (sign * ks / math.pi) * w * torch.log(w)
    return out.conj()


def _mag64(c, seed):
    s = _size(c)
    rays = s["nrx"] * s["nry"]
    if rays * max(1, c["n"]) > EXACT_PAIRS:
        return None
    xy, m = (torch.from_numpy(v).cuda() for v in _lenses(c, seed))
    counts = torch.zeros(c["nx"] * c["ny"], dtype=torch.float64, device="cuda")
    step = 1 << 21
    for f in range(0, rays, step):
        idx = torch.arange(f, min(rays, f + step), device="cuda")
        z = torch.complex(s["cx"] - s["ix"] / 2 + ((idx % s["nrx"]).double() + 0.5) * s["dx"],
                          s["cy"] - s["iy"] / 2 + ((idx // s["nrx"]).double() + 0.5) * s["dx"])
        b = _beta64(c, s, xy, m, z)
        px = torch.floor((b.real - (c["cx"] - c["sx"] / 2)) / (c["sx"] / c["nx"]))
        py = torch.floor((b.imag - (c["cy"] - c["sy"] / 2)) / (c["sy"] / c["ny"]))
        ok = (px >= 0) & (px < c["nx"]) & (py >= 0) & (py < c["ny"])
        counts += torch.bincount((py[ok] * c["nx"] + px[ok]).long(), minlength=counts.numel()).double()
    return (counts * (s["dx"] ** 2 / (c["sx"] / c["nx"] * (c["sy"] / c["ny"])))).reshape(c["ny"], c["nx"])


def _net64(c, seed, backward):
    theta, freq, x, t = (torch.from_numpy(v).cuda().double() for v in _net(c, seed))
    theta.requires_grad_(backward)
    at, layers = 0, []
    for rows in (64, 64, 64, 8):
        W = theta[at:at + rows * 64].reshape(rows, 64)
        at += rows * 64
        layers.append((W, theta[at:at + rows]))
        at += rows
    a = math.pi * (x @ freq.T)
    h = torch.cat([torch.sin(a), torch.cos(a)], 1)
    for W, b in layers[:3]:
        h = torch.tanh(h @ W.T + b)
    y = h @ layers[3][0].T + layers[3][1]
    if not backward:
        return {"y": y}
    loss = (y - t).square().sum()
    (loss / t.numel()).backward()
    return {"grad": theta.grad, "loss": loss.detach().reshape(1)}


def exact(case, seed):
    c = case
    if c["kind"].startswith("mlp"):
        return _net64(c, seed, c["kind"] == "mlp-grad")
    if c["kind"] in ("map", "noalloc"):
        mag = _mag64(c, seed)
        return None if mag is None else {"counts": None, "mag": mag}
    if c["kind"] == "rays":
        s = _size(c)
        xy, m = (torch.from_numpy(v).cuda() for v in _lenses(c, seed))
        idx = torch.from_numpy(_ray_idx(c, seed)).cuda()
        z = torch.complex(s["cx"] - s["ix"] / 2 + ((idx % s["nrx"]).double() + 0.5) * s["dx"],
                          s["cy"] - s["iy"] / 2 + ((idx // s["nrx"]).double() + 0.5) * s["dx"])
        b = torch.cat([_beta64(c, s, xy, m, p) for p in z.split(1 << 14)])
        return {"beta": torch.view_as_real(b.resolve_conj()), "pixel": None}
    return None  # bands and batches: whole counts, or too many pair terms
