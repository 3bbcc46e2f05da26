"""The calls of this framework whose time matters, with the inputs they meet in use.

A program that uses the framework builds a model of one or more imaging systems, then
evaluates log-likelihoods of parameter points over and over (a sampler's batches, from a
handful of points to thousands, on images from 64 x 64 up), renders an image now and
then, and, when it samples with the network pre-screen, trains that network and runs it on
proposals.  Every case goes through those entry points (``Model``, ``GpuLikelihood``,
``Surrogate``).  Models, image sizes, rules, PSFs and batch sizes are those of
``workloads`` and of the benchmark, or lie between them.

``exact`` is the same forward model in 64 bits, written from the formulas with plain torch.
"""
import functools
import math

import numpy as np
import torch

import workloads as W
from paper_1505_07674_gb300.lensed import Model
from paper_1505_07674_gb300.posterior import GpuLikelihood
from paper_1505_07674_gb300.surrogate import Surrogate


def listed():
    return [
        # The benchmark: one HST-like image, 4,096 parameter points a call, with the launch
        # configuration that the autotuner picks for it.
        _like("hst_batch", "hst", 200, 200, 4096, "gl", 5, 21, "halo", "mixed_ff", 23),
        # The same image straight after Model(...): no configuration chosen, a smaller batch.
        _like("hst_batch_untuned", "hst", 200, 200, 512, "gl", 5, 21, "halo", "mixed_ff", -1),
        # A small cut-out, the benchmark's second workload (tuned configuration).
        _like("small_batch", "single", 64, 64, 1000, "gl", 5, 7, "gauss", "mixed_ff", 15),
        # One step of the sampler's random walks on a 400 x 400 image: unit-cube points from
        # the host in, log-likelihoods on the host out.
        _like("walk_step", "euclid", 400, 400, 500, "gl", 5, 15, "gauss", "mixed_ff", -1, path="walk"),
        # Many systems of different sizes, rules and PSFs in one call.
        _like("uneven_batch", "uneven", 0, 0, 64, "gl", 0, 0, "gauss", "mixed_ff", 23, systems=24),
        # Two lens galaxies, three lens lights, two sources and sky with the Gauss-Kronrod
        # rule g3k7 and an image-plane prior: 35 free parameters.
        _like("group_batch", "group", 160, 160, 256, "gk", 3, 15, "gauss", "mixed_ff", 23),
        # A handful of points through host buffers: launches and latency.
        _like("few_points_host", "single", 64, 64, 8, "gl", 5, 7, "gauss", "mixed_ff", -1, path="host"),
        # An odd-sized image with a PSF that is no sum of a few separable terms, in the
        # faster precision mode, near the posterior.
        _like("mixed_full_psf", "hst", 161, 143, 700, "gl", 4, 21, "full", "mixed", 11, spread=0.05),
        # Validation mode, everything in 64 bits.
        _like("validate_fp64", "single", 64, 64, 64, "gl", 5, 7, "gauss", "fp64", -1),
        # One model image and its integration-error map.
        _like("render_maps", "group", 160, 160, 1, "gk", 3, 15, "gauss", "mixed_ff", -1, path="render"),
        # The pre-screen network on one batch of proposals.
        {"name": "screen_forward", "path": "forward", "n_in": 18, "rows": 65536, "max_batch": 65536},
        # A stretch of the network's training loop.
        {"name": "screen_training", "path": "train", "n_in": 18, "rows": 8192, "steps": 12},
    ]


def _like(name, model, nx, ny, points, rule, order, psf, psf_kind, precision, config, path="batch",
          systems=1, spread=1.0):
    return {"name": name, "path": path, "model": model, "nx": nx, "ny": ny, "points": points,
            "rule": rule, "order": order, "psf": psf, "psf_kind": psf_kind, "precision": precision,
            "config": config, "systems": systems, "spread": spread}


MOST_RAYS = 1.5e9     # rays of a drawn case, 32-bit modes
MOST_RAYS_FP64 = 2e7  # 64-bit mode


def draw(rng):
    def log_uniform(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    path = rng.choice(["batch"] * 8 + ["walk", "walk", "host", "host", "render", "forward", "train"])
    if path == "forward":
        rows = log_uniform(200, 65536)
        return {"path": path, "n_in": rng.randint(5, 35), "rows": rows,
                "max_batch": rng.choice([8192, 65536])}
    if path == "train":
        return {"path": path, "n_in": rng.randint(5, 35), "rows": log_uniform(500, 8192),
                "steps": rng.randint(4, 12)}
    model = rng.choice(["single", "hst", "hst", "euclid", "group", "uneven"])
    precision = rng.choice(["mixed_ff"] * 6 + ["mixed", "fp32", "fp64"])
    if path in ("host", "walk", "render") and model == "uneven":
        model = "single"
    if path == "render":
        precision = "mixed_ff"
    if model == "uneven":
        case = _like(None, model, 0, 0, 0, "gl", 0, 0, "gauss", precision, 0, path,
                     systems=log_uniform(4, 48))
        rays = sum(s["nx"] * s["ny"] * s["rule"][1] ** 2 for s in W.c3_batch(case["systems"]))
        fewest, most = 4, 512
    else:
        lo, hi = {"single": (48, 160), "hst": (96, 280), "euclid": (160, 400), "group": (96, 200)}[model]
        nx, ny = log_uniform(lo, hi), log_uniform(lo, hi)
        rule, order = ("gk", rng.choice([3, 3, 3, 5])) if path == "render" else rng.choice(
            [("gl", 5)] * 5 + [("gl", 3), ("gl", 4), ("gl", 6), ("gl", 7), ("gk", 3), ("gk", 3), ("gk", 5),
                               ("sub", 4), ("sub", 2)])
        case = _like(None, model, nx, ny, 0, rule, order, 2 * rng.randint(3, 13) + 1,
                     rng.choice(["gauss", "halo", "halo", "full"]), precision, 0, path)
        rays = nx * ny * _nodes_per_row(rule, order) ** 2
        fewest, most = {"host": (1, 64), "walk": (128, 1000), "render": (1, 1)}.get(path, (64, 4096))
    most = min(most, int((MOST_RAYS_FP64 if precision == "fp64" else MOST_RAYS) / rays))
    case["points"] = log_uniform(min(fewest, max(1, most)), max(1, most))
    case["config"] = -1 if path in ("walk", "render", "host") else rng.choice(
        [-1, 15, 21, 23, 23] if precision == "mixed_ff" else [-1, 3, 11])
    case["spread"] = rng.choice([1.0, 1.0, 0.05])
    del case["name"]
    return case


# ---------------------------------------------------------------------------------------
# inputs

def _psf(kind, size, h):
    if kind == "gauss":
        return W.gaussian_psf(size, 0.1 if h < 0.1 else 0.18, h)
    if kind == "halo":
        return W.gaussian_psf(size, 0.1, h, halo_frac=0.1, halo_fwhm=0.5)
    # an instrument's PSF: an elongated core off the axes, two more lobes at other angles
    r = np.arange(size) - size // 2
    x, y = np.meshgrid(r, r)
    out = np.zeros((size, size))
    for amp, a, b, deg, x0, y0 in ((1.0, 1.6, 1.1, 25.0, 0.0, 0.0), (0.10, 6.0, 0.8, 40.0, 0.3, -0.2),
                                   (0.08, 5.0, 0.9, -52.0, -0.2, 0.4), (0.03, 7.0, 4.0, 10.0, 0.5, 0.5)):
        c, s = math.cos(math.radians(deg)), math.sin(math.radians(deg))
        u, v = (x - x0) * c + (y - y0) * s, (y - y0) * c - (x - x0) * s
        out += amp * np.exp(-0.5 * ((u / a) ** 2 + (v / b) ** 2))
    return out


def _specs(case):
    """The case's systems, as the dicts that Model takes."""
    model = case["model"]
    if model == "uneven":
        return W.c3_batch(case["systems"])
    spec = dict({"single": W.c1_small, "hst": W.c2_hst, "euclid": W.c4_euclid,
                 "group": lambda: W.j0808_like(image_prior=True)}[model]())
    spec["nx"], spec["ny"] = case["nx"], case["ny"]
    spec["rule"] = (case["rule"], case["order"])
    spec["psf"] = _psf(case["psf_kind"], case["psf"], spec["h"])
    if spec["mask"] is not None:
        spec["mask"] = W.annular_mask(case["nx"], case["ny"], spec["h"], 0.5, 3.0)
    return [spec]


def _unit_points(spec, P, spread, rng):
    """P points of the unit cube: the whole prior, or a box around the truth."""
    u = rng.random((P, spec["n_params"]))
    if spread < 1.0:
        lo, hi = np.asarray(spec["prior_lo"], float), np.asarray(spec["prior_hi"], float)
        t = (np.asarray(spec["truth"], float) - lo) / (hi - lo)
        u = np.clip(t + spread * (u - 0.5), 0.0, 1.0)
    return u


def _inputs(case, seed):
    """Systems, observations (the noiseless 64-bit image plus seeded noise) and unit-cube
    points, in host memory."""
    specs = _specs(case)
    obs, units = [], []
    for k, spec in enumerate(specs):
        rng = np.random.default_rng([seed, k])
        img = _images(spec, np.asarray(spec["truth"], float)[None])[0].cpu().numpy()
        obs.append(W.add_noise(spec, img, int(rng.integers(1 << 30))))
        units.append(_unit_points(spec, case["points"], case["spread"], rng))
    return specs, obs, units


def _to_params(spec, u):
    lo, hi = np.asarray(spec["prior_lo"], float), np.asarray(spec["prior_hi"], float)
    return lo + (hi - lo) * u


def _packed(specs, units):
    n = max(s["n_params"] for s in specs)
    out = np.zeros((len(specs), len(units[0]), n))
    for k, (s, u) in enumerate(zip(specs, units)):
        out[k, :, :s["n_params"]] = _to_params(s, u)
    return out


def _network(case, seed):
    """Weights (He-style, small nonzero biases), whitened inputs and standardised targets."""
    rng = np.random.default_rng(seed)
    d, H = case["n_in"], HIDDEN
    theta = np.concatenate([a.ravel() for a in (
        rng.standard_normal((H, d)) * math.sqrt(2.0 / d), rng.standard_normal(H) * 0.05,
        rng.standard_normal((H, H)) * math.sqrt(2.0 / H), rng.standard_normal(H) * 0.05,
        rng.standard_normal((H, H)) * math.sqrt(2.0 / H), rng.standard_normal(H) * 0.05,
        rng.standard_normal(H) * math.sqrt(1.0 / H), np.zeros(1))]).astype(np.float32)
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    X = torch.randn((case["rows"], d), device="cuda", generator=g)
    t = torch.log1p((X * X).sum(1))
    return theta, X, (t - t.mean()) / t.std()


HIDDEN = 256  # the width that every use of the network takes


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case = case
    path = case["path"]
    if path in ("forward", "train"):
        s.theta, s.X, s.t = _network(case, seed)
        s.net = Surrogate(case["n_in"], HIDDEN, case["max_batch"] if path == "forward" else 8192)
        s.net.set_params(s.theta)
        return s
    specs, obs, units = _inputs(case, seed)
    s.model = Model(specs, obs, precision=case["precision"])
    if case["config"] >= 0:
        s.model.set_config(case["config"])
    if path == "walk":
        s.like, s.u = GpuLikelihood(s.model, specs[0]), units[0]
    elif path == "render":
        s.points = torch.as_tensor(_to_params(specs[0], units[0])[0], device="cuda")
    elif path == "host":
        s.points = torch.as_tensor(_packed(specs, units)).pin_memory()
        s.out = torch.empty((len(specs), case["points"]), dtype=torch.float64).pin_memory()
    else:
        s.points = torch.as_tensor(_packed(specs, units), device="cuda")
    return s


def run(s):
    path = s.case["path"]
    if path == "batch":
        return s.model.loglike_batch(s.points)
    if path == "walk":
        return s.like(s.u)
    if path == "host":
        return s.model.loglike_batch_host(s.points, s.out)
    if path == "render":
        return {"image": s.model.render(0, s.points), "error": s.model.render_error(0, s.points)}
    if path == "forward":
        return s.net.forward(s.X)
    s.net.set_params(s.theta)
    for k in range(s.case["steps"]):
        loss = s.net.train_step(s.X, s.t, 1e-3)
    return {"loss": loss, "weights": s.net.get_params()}


# ---------------------------------------------------------------------------------------
# the work that no implementation can do without

_FLOPS = {"sie": 32, "shear": 10, "pointmass": 10, "sersic": 21, "devauc": 21, "gauss": 18, "sky": 1}


def _nodes_per_row(rule, order):
    return {"point": 1, "gk": 2 * order + 1}.get(rule, order)


def _needed(spec):
    """Weighted pixels, and the pixels that they see through the PSF."""
    ny, nx = spec["ny"], spec["nx"]
    if spec["mask"] is None:
        return nx * ny, nx * ny
    live = np.asarray(spec["mask"]) == 0
    h = spec["psf"].shape[0] // 2
    c = np.zeros((ny + 2 * h + 1, nx + 2 * h + 1))
    c[1:, 1:] = np.pad(live, h).cumsum(0).cumsum(1)
    w = 2 * h + 1
    seen = c[w:, w:] - c[:-w, w:] - c[w:, :-w] + c[:-w, :-w]
    return int(live.sum()), int((seen[:ny, :nx] > 0).sum()) if h else int(live.sum())


def work(case):
    path = case["path"]
    if path in ("forward", "train"):
        n, d, H = case["rows"], case["n_in"], HIDDEN
        mul = 2.0 * n * (d * H + 2 * H * H + H)
        params = 4 * (H * d + 2 * H * H + 4 * H + 1)
        if path == "forward":
            return {"bytes": 4 * n * (d + 1) + params, "flops": mul}
        # each step reads the batch and reads and writes the weights and Adam's two moments;
        # forward, and the two products of each layer's backward but the first's
        return {"bytes": case["steps"] * (4 * n * (d + 1) + 6 * params),
                "flops": case["steps"] * (3 * mul - 2.0 * n * d * H)}
    P, nbytes, flops = case["points"], 0.0, 0.0
    for spec in _specs(case):
        live, seen = _needed(spec)
        size = spec["psf"].shape[0]
        if path == "render":
            live = seen = spec["nx"] * spec["ny"]
        rays = seen * _nodes_per_row(*spec["rule"]) ** 2
        per_ray = 6 + sum(_FLOPS[c["type"]] for c in spec["components"]
                          if c["plane"] != "foreground" or any(k == "free" for k, _ in c["params"]))
        terms = {"gauss": 2 * size, "halo": 4 * size}.get(case["psf_kind"], size * size)
        flops += P * (rays * per_ray + live * (2 * terms + 4))
        nbytes += live * 8 + P * (8 * spec["n_params"] + 8)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------------------
# 64-bit values

def _rule(rule, order):
    """Nodes and weights on the unit pixel, and the embedded Gauss weights (or None)."""
    if rule == "point":
        return np.zeros(1), np.ones(1), None
    if rule == "sub":
        return (np.arange(order) + 0.5) / order - 0.5, np.full(order, 1.0 / order), None
    x, w = np.polynomial.legendre.leggauss(order)
    if rule == "gl":
        return 0.5 * x, 0.5 * w, None
    # Kronrod's extension: the roots of the polynomial E of degree N + 1 with
    # integral(P_N E P_k) = 0 for k <= N, and the weights that integrate P_0 .. P_2N
    leg = np.polynomial.legendre
    N = order
    xs, ws = leg.leggauss(2 * N + 8)
    V = leg.legvander(xs, N + 1)
    A = (V[:, :N + 1] * (ws * V[:, N])[:, None]).T @ V
    e = np.append(np.linalg.lstsq(A[:, :N + 1], -A[:, N + 1], rcond=None)[0], 1.0)
    nodes = np.sort(np.concatenate([x, leg.legroots(e).real]))
    rhs = np.zeros(2 * N + 1)
    rhs[0] = 2.0
    wk = np.linalg.solve(leg.legvander(nodes, 2 * N).T, rhs)
    wg = np.zeros(2 * N + 1)
    wg[1::2] = w
    return 0.5 * nodes, 0.5 * wk, 0.5 * wg


def _bn(n):
    """Half-light constant of the Sersic profile: P(2n, b) = 1/2."""
    lo, hi = torch.zeros_like(n), 2.0 * n
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        low = torch.special.gammainc(2.0 * n, mid) < 0.5
        lo, hi = torch.where(low, mid, lo), torch.where(low, hi, mid)
    return 0.5 * (lo + hi)


def _frame(x, y, x0, y0, pa):
    c, s = torch.cos(pa * (math.pi / 180)), torch.sin(pa * (math.pi / 180))
    dx, dy = x - x0, y - y0
    return dx * c + dy * s, dy * c - dx * s, c, s


def _deflection(kind, v, x, y):
    if kind == "sie":
        x0, y0, b, q, pa, core = v
        dx, dy, c, s = _frame(x, y, x0, y0, pa)
        e = torch.sqrt((1 - q) * (1 + q))
        psi = torch.sqrt(q * q * (core * core + dx * dx) + dy * dy)
        k = b * torch.sqrt(q) / e
        au, av = k * torch.atan(e * dx / (psi + core)), k * torch.atanh(e * dy / (psi + q * q * core))
        return au * c - av * s, au * s + av * c
    if kind == "shear":
        x0, y0, gamma, phi = v
        g1 = gamma * torch.cos(phi * (math.pi / 90))
        g2 = gamma * torch.sin(phi * (math.pi / 90))
        dx, dy = x - x0, y - y0
        return g1 * dx + g2 * dy, g2 * dx - g1 * dy
    x0, y0, theta = v
    dx, dy = x - x0, y - y0
    f = theta * theta / (dx * dx + dy * dy)
    return f * dx, f * dy


def _light(kind, v, x, y, h, zeropoint):
    if kind == "sky":
        return v[0] * h * h
    x0, y0, r, mag = v[:4]
    n = v[4] if kind == "sersic" else torch.full_like(r, 4.0)
    q, pa = v[-2], v[-1]
    dx, dy, _, _ = _frame(x, y, x0, y0, pa)
    flux = 10.0 ** (-0.4 * (mag - zeropoint))
    R2 = q * dx * dx + dy * dy / q
    if kind == "gauss":
        return flux * h * h / (2 * math.pi * r * r) * torch.exp(-0.5 * R2 / (r * r))
    b = _bn(n)
    I0 = flux * torch.exp(2 * n * torch.log(b) - torch.lgamma(2 * n)) / (2 * math.pi * n * r * r)
    return I0 * h * h * torch.exp(-b * (R2 / (r * r)) ** (0.5 / n))


def _images(spec, params, rules=None, convolved=True):
    """Model images [P][ny][nx] of the points, in 64 bits on the GPU."""
    ny, nx, h = spec["ny"], spec["nx"], spec["h"]
    t, w, _ = _rule(*spec["rule"]) if rules is None else (*rules, None)
    dev = dict(dtype=torch.float64, device="cuda")
    params = torch.as_tensor(params, **dev)
    px = ((torch.arange(nx, **dev) - 0.5 * (nx - 1)) * h)[None, None, :]
    py = ((torch.arange(ny, **dev) - 0.5 * (ny - 1)) * h)[None, :, None]
    out = torch.empty((len(params), ny, nx), **dev)
    step = max(1, (1 << 25) // (nx * ny))
    for p0 in range(0, len(params), step):
        part = params[p0:p0 + step]
        vals = [[part[:, int(v)].reshape(-1, 1, 1) if k == "free" else
                 torch.full((len(part), 1, 1), float(v), **dev) for k, v in c["params"]]
                for c in spec["components"]]
        lens = [(c["type"], v) for c, v in zip(spec["components"], vals) if c["plane"] == "lens"]
        for c, v in zip(spec["components"], vals):
            if c["plane"] == "source_image":  # given on the image plane: moved to theta - alpha(theta)
                ds = [_deflection(k, u, v[0], v[1]) for k, u in lens]
                v[0], v[1] = v[0] - sum(a for a, _ in ds), v[1] - sum(b for _, b in ds)
        acc = torch.zeros((len(part), ny, nx), **dev)
        for tb, wb in zip(t, w):
            for ta, wa in zip(t, w):
                if wa * wb == 0.0:
                    continue
                x, y = px + ta * h, py + tb * h
                sx, sy = x, y
                for k, v in lens:
                    a = _deflection(k, v, x, y)
                    sx, sy = sx - a[0], sy - a[1]
                for c, v in zip(spec["components"], vals):
                    if c["plane"] == "foreground":
                        acc += wa * wb * _light(c["type"], v, x, y, h, spec["zeropoint"])
                    elif c["plane"] != "lens":
                        acc += wa * wb * _light(c["type"], v, sx, sy, h, spec["zeropoint"])
        if convolved and spec["psf"] is not None:
            F = torch.as_tensor(np.asarray(spec["psf"], float), **dev)
            F = (F / F.sum()).flip(0, 1)
            p, q = F.shape[0] // 2, F.shape[1] // 2
            wide = torch.nn.functional.pad(acc[:, None], (q, q, p, p), mode="replicate")[:, 0]
            acc = torch.zeros_like(acc)
            for k in range(F.shape[0]):
                for m in range(F.shape[1]):
                    acc += F[k, m] * wide[:, k:k + ny, m:m + nx]
        out[p0:p0 + step] = acc
    return out


def _loglikes(spec, obs, params):
    d = np.asarray(obs["data"], float)
    var = np.asarray(obs["variance"], float) if "variance" in obs else (d + obs["offset"]) / obs["gain"]
    w = 1.0 / var
    if spec["mask"] is not None:
        w = np.where(np.asarray(spec["mask"]) != 0, 0.0, w)
    d, w = torch.as_tensor(d, device="cuda"), torch.as_tensor(w, device="cuda")
    out = []
    step = max(1, (1 << 25) // d.numel())
    for p0 in range(0, len(params), step):
        r = d - _images(spec, params[p0:p0 + step])
        out.append(-0.5 * (w * r * r).sum((1, 2)))
    return torch.cat(out)


def _unpack(theta, d, H):
    shapes = ((H, d), (H,), (H, H), (H,), (H, H), (H,), (H,), (1,))
    sizes = [int(np.prod(s)) for s in shapes]
    return [p.reshape(s) for p, s in zip(torch.split(theta, sizes), shapes)]


def _predict(theta, X, d, H):
    W1, b1, W2, b2, W3, b3, w4, b4 = _unpack(theta, d, H)
    silu = torch.nn.functional.silu
    return silu(silu(silu(X @ W1.T + b1) @ W2.T + b2) @ W3.T + b3) @ w4 + b4


def exact(case, seed):
    path = case["path"]
    if path in ("forward", "train"):
        theta, X, t = _network(case, seed)
        theta = torch.as_tensor(theta, device="cuda").double()
        X, t, predict = X.double(), t.double(), functools.partial(_predict, d=case["n_in"], H=HIDDEN)
        if path == "forward":
            return predict(theta, X)
        m = v = torch.zeros_like(theta)
        for k in range(1, case["steps"] + 1):
            theta = theta.detach().requires_grad_()
            loss = 0.5 * ((predict(theta, X) - t) ** 2).mean()
            g, = torch.autograd.grad(loss, theta)
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            theta = theta.detach() - 1e-3 * (m / (1 - 0.9 ** k)) / ((v / (1 - 0.999 ** k)).sqrt() + 1e-8)
        return {"loss": loss.detach().reshape(1), "weights": theta}
    specs, obs, units = _inputs(case, seed)
    if path == "render":
        spec, p = specs[0], _to_params(specs[0], units[0])
        t, wk, wg = _rule(*spec["rule"])
        image = _images(spec, p)[0]
        error = (_images(spec, p, (t, wk), False) - _images(spec, p, (t, wg), False)).abs()[0]
        return {"image": image, "error": error}
    out = torch.stack([_loglikes(s, o, _to_params(s, u)) for s, o, u in zip(specs, obs, units)])
    return out[0] if path == "walk" else out
