"""What a user of the framework has it compute, as cases that can be timed and checked.

Each case is one call (or one pair of calls) through the public Python binding: the projector
pair alone, as an autograd layer and inside the filtered backprojection, the Fourier
preconditioner, whole reconstructions (Alg. 4 and Alg. 5) and a batch of uneven slices, over
the sizes of the framework's configurations: images of 64^2 to 2048^2, 90 to 2048 views, even
and odd view counts, uniform and golden-ratio angles, FP32, FP64 and bfloat16 operands.
"""
import math

import numpy as np
import torch

from paper_1810_03275_gb300 import autograd, ctrecon

TAU = 1.0 / math.sqrt(8.0)


def listed():
    return [
        # a projector layer inside a small training loop: the smallest calls, launches count
        {"name": "layer_64", "kind": "layer", "n": 64, "views": 90, "bins": 95, "dtype": "f32", "angles": "uniform"},
        # one forward projection at the metal-artifact workload's size
        {"name": "forward_512", "kind": "forward", "n": 512, "views": 720, "bins": 729, "dtype": "f32",
         "angles": "uniform"},
        # one backprojection of a scan with an odd view count on a ragged image
        {"name": "adjoint_500_odd", "kind": "adjoint", "n": 500, "views": 725, "bins": 711, "dtype": "f32",
         "angles": "uniform"},
        # both projectors of the largest configuration, operands stored in bfloat16
        {"name": "pair_2048_bf16", "kind": "pair", "n": 2048, "views": 2048, "bins": 2897, "dtype": "bf16",
         "angles": "uniform"},
        # a golden-ratio (irregular) acquisition
        {"name": "pair_384_golden", "kind": "pair", "n": 384, "views": 600, "bins": 545, "dtype": "f32",
         "angles": "golden"},
        # the double-precision projectors
        {"name": "pair_256_f64", "kind": "pair", "n": 256, "views": 360, "bins": 363, "dtype": "f64",
         "angles": "uniform"},
        # the classical reconstruction, a preview of a large slice
        {"name": "fbp_1024", "kind": "fbp", "n": 1024, "views": 1440, "bins": 1449, "dtype": "f32",
         "angles": "uniform"},
        # the preconditioner alone, at a size that is not a power of two
        {"name": "precond_768", "kind": "precond", "n": 768, "views": 180, "bins": 1087, "dtype": "f32",
         "angles": "uniform"},
        # the plain double-precision reconstruction, scaling constants by power iteration
        {"name": "solve_64_f64", "kind": "solve", "n": 64, "views": 90, "bins": 95, "dtype": "f64",
         "angles": "uniform", "iters": 200, "metal": 0, "alpha": 0.01, "nonneg": False, "scaling": "power"},
        # the metal-artifact reconstruction: the headline workload
        {"name": "solve_512_metal", "kind": "solve", "n": 512, "views": 720, "bins": 729, "dtype": "f32",
         "angles": "uniform", "iters": 500, "metal": 3, "alpha": 0.3, "nonneg": False, "scaling": "power"},
        # a non-negative reconstruction of a scan with an odd view count, scaling constants kept
        {"name": "solve_432_nonneg", "kind": "solve", "n": 432, "views": 361, "bins": 611, "dtype": "f32",
         "angles": "uniform", "iters": 100, "metal": 0, "alpha": 0.1, "nonneg": True, "scaling": "kept"},
        # a batch of uneven slices solved together
        {"name": "batch_12", "kind": "batch", "count": 12, "seed_sizes": 3, "nmax": 1024, "iters": 15, "alpha": 0.3},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


#: image sizes 2^a 3^b, which the Fourier preconditioner takes
_SMOOTH = sorted(2 ** a * 3 ** b for a in range(3, 11) for b in range(4) if 64 <= 2 ** a * 3 ** b <= 1024)


def draw(rng):
    kind = rng.choice(["layer", "forward", "adjoint", "pair", "pair", "fbp", "precond", "solve", "solve", "batch"])
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(3, 10), "seed_sizes": rng.randrange(1 << 20), "nmax": 768,
                "iters": rng.randint(5, 15), "alpha": 0.3}
    case = {"kind": kind, "dtype": "f32", "angles": "uniform"}
    if kind == "solve":
        case["dtype"] = rng.choice(["f32", "f32", "f32", "f64"])
        top = 96 if case["dtype"] == "f64" else 512
        case["n"] = rng.choice([n for n in _SMOOTH if n <= top])
        case["views"] = min(720, max(45, int(case["n"] * rng.uniform(0.5, 1.5))))
        case["iters"] = _log_int(rng, 20, 200)
        case["metal"] = rng.randint(0, 4)
        case["alpha"] = round(10 ** rng.uniform(-2, -0.3), 4)
        case["nonneg"] = rng.random() < 0.3
        case["scaling"] = rng.choice(["power", "kept"])
    elif kind == "precond":
        case["n"] = rng.choice(_SMOOTH)
        case["views"] = 45
    else:
        case["dtype"] = rng.choice(["f32", "f32", "bf16", "f64"]) if kind == "pair" else "f32"
        if kind in ("pair", "forward", "adjoint") and rng.random() < 0.25:
            case["angles"] = "golden"
        top = 256 if case["dtype"] == "f64" else 1024 if case["angles"] == "golden" or kind == "layer" else 1536
        case["n"] = _log_int(rng, 64, top)
        case["views"] = min(2048, max(60, int(case["n"] * rng.uniform(0.5, 1.6))))
    case["bins"] = int(case["n"] * rng.uniform(1.38, 1.5)) + 1
    return case


# ---- inputs ---------------------------------------------------------------------------------


def _theta(case):
    v = np.arange(case["views"], dtype=np.float64)
    if case["angles"] == "golden":
        return np.mod(v * (math.pi * (math.sqrt(5.0) - 1.0) / 2.0), math.pi)
    return v * (math.pi / case["views"])


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _scan(n, theta, bins, seed, metal=0):
    """A phantom of eight ellipses and `metal` metal disks on an n x n grid: its image with a
    fine texture, its exact line integrals with 1 % noise, the noise level and the metal trace."""
    dev = _device()
    rs = np.random.Generator(np.random.PCG64(seed))
    R = 0.5 * n
    shapes = []
    for _ in range(8):
        r, t = 0.6 * R * math.sqrt(rs.uniform()), rs.uniform(0, 2 * math.pi)
        shapes.append((r * math.cos(t), r * math.sin(t), rs.uniform(0.05, 0.4) * R, rs.uniform(0.05, 0.4) * R,
                       rs.uniform(0, math.pi), rs.uniform(0, 1), False))
    for _ in range(metal):
        r, t = 0.35 * R * math.sqrt(rs.uniform()), rs.uniform(0, 2 * math.pi)
        rad = rs.uniform(4.0, 10.0)
        shapes.append((r * math.cos(t), r * math.sin(t), rad, rad, 0.0, 10.0, True))
    x = torch.arange(n, dtype=torch.float64, device=dev) - 0.5 * (n - 1)
    s = torch.arange(bins, dtype=torch.float64, device=dev) - 0.5 * (bins - 1)
    th = torch.as_tensor(theta, device=dev)[:, None]
    u = torch.zeros(n, n, dtype=torch.float64, device=dev)
    f = torch.zeros(len(theta), bins, dtype=torch.float64, device=dev)
    trace = torch.zeros(len(theta), bins, dtype=torch.uint8, device=dev)
    for cx, cy, a, b, phi, value, is_metal in shapes:
        dx, dy = x[:, None] - cx, x[None, :] - cy
        e1 = (math.cos(phi) * dx + math.sin(phi) * dy) / a
        e2 = (-math.sin(phi) * dx + math.cos(phi) * dy) / b
        u += value * (e1 * e1 + e2 * e2 <= 1)
        off = s[None, :] - (cx * torch.cos(th) + cy * torch.sin(th))
        half = (a * torch.cos(th - phi)) ** 2 + (b * torch.sin(th - phi)) ** 2
        f += value * 2 * a * b * torch.sqrt(torch.clamp(half - off * off, min=0)) / half
        if is_metal:
            trace |= (off.abs() < a + 1).to(torch.uint8)
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    level = 0.01 * float(f.max())
    f += level * torch.randn(f.shape, generator=g, dtype=torch.float64, device=dev)
    u += 0.02 * torch.randn(u.shape, generator=g, dtype=torch.float64, device=dev)
    return u, f, level, trace


_REAL = {"f32": torch.float32, "f64": torch.float64, "bf16": torch.float32}
_OPERAND = {"f32": torch.float32, "f64": torch.float64, "bf16": torch.bfloat16}


def _kept_scaling(n, views):
    """beta and c as a program keeps them for a geometry (upper estimates of ||R|| and of the
    preconditioned spectrum: the power iterations give 0.98 sqrt(n views) and 7 / n to 9 / n)."""
    return math.sqrt(n * views), 12.0 / n


def _batch_cases(case):
    rs = np.random.Generator(np.random.PCG64(case["seed_sizes"]))
    sizes = [n for n in (256, 384, 512, 768, 1024) if n <= case["nmax"]]
    out = []
    for _ in range(case["count"]):
        n, views = int(rs.choice(sizes)), int(rs.integers(180, 1441))
        out.append({"n": n, "views": views, "bins": math.ceil(math.sqrt(2) * n), "angles": "uniform"})
    return out


def _inputs(case, seed):
    if case["kind"] == "batch":
        scans = [_scan(c["n"], _theta(c), c["bins"], seed * 100 + i, 2) for i, c in enumerate(_batch_cases(case))]
        return {"f": [s[1].float() for s in scans], "mask": [s[3] for s in scans], "delta": [3 * s[2] for s in scans]}
    u, f, level, trace = _scan(case["n"], _theta(case), case["bins"], seed, case.get("metal", 0))
    real, operand = _REAL[case["dtype"]], _OPERAND[case["dtype"]]
    if case["kind"] in ("solve", "fbp"):
        return {"f": f.to(real), "mask": trace if case.get("metal") else None, "delta": 3 * level}
    return {"u": u.to(operand), "g": f.to(operand), "y": u.to(real)}


def prepare(case, seed):
    state = _inputs(case, seed)
    state["case"] = case
    if case["kind"] == "batch":
        cs = _batch_cases(case)
        state["batch"] = ctrecon.Batch([{"n": c["n"], "n_angles": c["views"], "n_bins": c["bins"]} for c in cs])
        state["betas"], state["cs"] = zip(*[_kept_scaling(c["n"], c["views"]) for c in cs])
        state["params"] = ctrecon.default_params()
        return state
    state["plan"] = ctrecon.Plan(case["n"], case["views"], case["bins"], angles=_theta(case), dtype=case["dtype"])
    if case["kind"] == "precond":
        state["params"] = ctrecon.default_params(c=_kept_scaling(case["n"], case["views"])[1])
    if case["kind"] == "solve":
        kw = {"nonneg": int(case["nonneg"])}
        if case["scaling"] == "kept":
            kw["beta"], kw["c"] = _kept_scaling(case["n"], case["views"])
        state["params"] = ctrecon.default_params(**kw)
    return state


# ---- the calls ------------------------------------------------------------------------------


def run(state):
    case, plan = state["case"], state.get("plan")
    kind = case["kind"]
    if kind == "forward":
        return plan.rh_forward(state["u"])
    if kind == "adjoint":
        return plan.rh_adjoint(state["g"])
    if kind == "pair":
        return {"g": plan.rh_forward(state["u"]), "u": plan.rh_adjoint(state["g"])}
    if kind == "layer":
        u = state["u"].detach().requires_grad_(True)
        g = autograd.radon(u, plan)
        g.backward(state["g"])
        return {"g": g.detach(), "grad": u.grad}
    if kind == "fbp":
        return plan.fbp(state["f"])
    if kind == "precond":
        return plan.precond_apply(state["y"], state["params"])
    if kind == "solve":
        u, diag = plan.tv_pd_solve(state["f"], state["mask"], case["alpha"], state["delta"], case["iters"],
                                   params=state["params"])
        return {"u": u, "objective": diag["objective"]}
    us, _ = state["batch"].solve(state["f"], state["mask"], [case["alpha"]] * case["count"], state["delta"],
                                 case["iters"], params=state["params"], betas=state["betas"], cs=state["cs"],
                                 want_diag=False)
    return us


def work(case):
    if case["kind"] == "batch":
        each = [dict(c, kind="solve", dtype="f32", iters=case["iters"], metal=2, scaling="kept")
                for c in _batch_cases(case)]
        total = [work(c) for c in each]
        return {k: sum(w[k] for w in total) for k in ("bytes", "flops")}
    n, views, bins = case["n"], case["views"], case["bins"]
    operand = {"f32": 4, "f64": 8, "bf16": 2}[case["dtype"]]
    real = 8 if case["dtype"] == "f64" else 4
    image, sino = n * n, views * bins
    projector = 4.0 * n * n * views               # two fused multiply-adds per (pixel, view)
    fft = 2 * 5.0 * image * math.log2(image)      # a complex transform there and back
    kind = case["kind"]
    if kind == "forward":
        return {"bytes": operand * image + real * sino, "flops": projector}
    if kind == "adjoint":
        return {"bytes": operand * sino + real * image, "flops": projector}
    if kind in ("pair", "layer"):
        return {"bytes": (operand + real) * (image + sino), "flops": 2 * projector}
    if kind == "fbp":
        return {"bytes": real * (sino + image), "flops": projector + 2 * 5.0 * views * 2 * bins * math.log2(2 * bins)}
    if kind == "precond":
        return {"bytes": 2 * real * image, "flops": fft / 2}
    pairs = case["iters"] + (100 if case["scaling"] == "power" else 0)
    return {"bytes": real * (sino + image) + (sino if case["metal"] else 0),
            "flops": pairs * (2 * projector + fft / 2)}


# ---- the same in 64 bits, from the definitions ----------------------------------------------


class _Radon64:
    """Linear-interpolation projector pair (h = ds = 1) in FP64, views in blocks."""

    def __init__(self, case):
        self.n, self.bins, self.dev = case["n"], case["bins"], _device()
        self.theta = _theta(case)
        self.step = max(1, (1 << 25) // (self.n * self.n))
        self.kept = {} if len(self.theta) * self.n * self.n <= 2_000_000_000 else None

    def _blocks(self):
        x = torch.arange(self.n, dtype=torch.float64, device=self.dev) - 0.5 * (self.n - 1)
        for at in range(0, len(self.theta), self.step):
            if self.kept is not None and at in self.kept:
                yield at, *self.kept[at]
                continue
            th = torch.as_tensor(self.theta[at:at + self.step], device=self.dev)[:, None, None]
            p = x[:, None] * torch.cos(th) + x[None, :] * torch.sin(th) + 0.5 * (self.bins - 1)
            k = torch.floor(p)
            w = torch.where(k < -1, 0.0, torch.where(k > self.bins - 1, 1.0, p - k))
            # bins shifted by one: slots 0 and bins + 1 stand for what is off the detector
            k = (k.clamp(-1, self.bins - 1) + 1).to(torch.int32)
            k += torch.arange(th.shape[0], dtype=torch.int32, device=self.dev)[:, None, None] * (self.bins + 2)
            if self.kept is not None:
                self.kept[at] = (k, w)
            yield at, k, w

    def forward(self, u):
        out = []
        for _, k, w in self._blocks():
            g = torch.zeros(k.shape[0] * (self.bins + 2), dtype=torch.float64, device=self.dev)
            k, hi = k.reshape(-1), (w * u).reshape(-1)
            g.index_add_(0, k, u.expand(w.shape).reshape(-1) - hi)
            g.index_add_(0, k + 1, hi)
            out.append(g.reshape(-1, self.bins + 2)[:, 1:-1])
        return torch.cat(out)

    def adjoint(self, g):
        u = torch.zeros(self.n, self.n, dtype=torch.float64, device=self.dev)
        pad = torch.nn.functional.pad(g, (1, 1))
        for at, k, w in self._blocks():
            row = pad[at:at + k.shape[0]].reshape(-1)
            lo = row[k]
            u += torch.lerp(lo, row[k + 1], w).sum(0)
        return u


def _grad64(u):
    p = torch.zeros(2, *u.shape, dtype=u.dtype, device=u.device)
    p[0, :-1], p[1, :, :-1] = u[1:] - u[:-1], u[:, 1:] - u[:, :-1]
    return p


def _div64(p):
    d = torch.zeros_like(p[0])
    d[:-1] += p[0, :-1]
    d[1:] -= p[0, :-1]
    d[:, :-1] += p[1, :, :-1]
    d[:, 1:] -= p[1, :, :-1]
    return d


def _frequencies64(n, dev):
    xi = 2 * math.pi * torch.fft.fftfreq(n, dtype=torch.float64, device=dev)
    norm = torch.sqrt(xi[:, None] ** 2 + xi[None, :] ** 2 + (math.pi / n) ** 2)
    s = 4 * torch.sin(math.pi * torch.arange(n, dtype=torch.float64, device=dev) / n) ** 2
    return norm, s[:, None] + s[None, :]


def _filter64(y, symbol):
    return torch.fft.ifft2(torch.fft.fft2(y) * symbol).real


def _power64(radon, steps=50, margin=1.05):
    """||R|| and c = margin * lambda_max of the preconditioned R^T R / ||R||^2, from the fixed start."""
    n, dev = radon.n, radon.dev
    plastic = 1.324717957244746
    i = torch.arange(n, dtype=torch.float64, device=dev)
    start = torch.frac(0.5 + i[:, None] / plastic + i[None, :] / plastic ** 2) - 0.5
    root = torch.sqrt(_frequencies64(n, dev)[0])
    x = start / start.norm()
    for _ in range(steps):
        y = radon.adjoint(radon.forward(x))
        beta = math.sqrt(float((x * y).sum()))
        x = y / y.norm()
    x = start / start.norm()
    for _ in range(steps):
        y = _filter64(radon.adjoint(radon.forward(_filter64(x, root))), root) / beta ** 2
        lam = float((x * y).sum())
        x = y / y.norm()
    return beta, margin * lam


def _solve64(radon, f, mask, alpha, delta, iters, nonneg, scaling):
    """Alg. 4 (and Alg. 5) of the thesis with sigma = 1 and tau = 1 / sqrt(8), from u = 0."""
    n = radon.n
    beta, c = scaling or _power64(radon)
    f = f.double()
    on = torch.zeros_like(f, dtype=torch.bool) if mask is None else mask.bool()
    w, a = (~on).double(), torch.where(on, 0.0, f) / beta
    lo = torch.where(on, 0.8 * f, f - delta) / beta
    hi = torch.where(on, math.inf, f + delta) / beta
    lam = alpha / beta ** 2
    norm, lap = _frequencies64(n, radon.dev)
    symbol = norm / ((norm if nonneg else 0.0) + c + TAU ** 2 * lap * norm)
    u = torch.zeros(n, n, dtype=torch.float64, device=radon.dev)
    bar, Ru = u.clone(), torch.zeros_like(f)
    v1, v2 = torch.zeros_like(f), torch.zeros(2, n, n, dtype=torch.float64, device=radon.dev)
    for _ in range(iters):
        y = -radon.adjoint(v1 + Ru) / beta + TAU * _div64(v2 + TAU * _grad64(u))
        if nonneg:
            y = y + bar - u
        u = u + _filter64(y, symbol)
        Ru = radon.forward(u) / beta
        z = v1 + 2 * Ru
        t = z - torch.minimum(torch.maximum((z + w * a) / (1 + w), lo), hi)
        v1 = t - Ru
        g = TAU * _grad64(u)
        z = v2 + 2 * g
        v2 = z / torch.clamp(TAU * torch.sqrt(z[0] ** 2 + z[1] ** 2) / lam, min=1.0) - g
        if nonneg:
            bar = bar + torch.clamp(2 * u - bar, min=0.0) - u
    g = _grad64(u)
    objective = 0.5 * (w * (beta * Ru - torch.where(on, 0.0, f)) ** 2).sum() + alpha * torch.sqrt(g[0] ** 2 + g[1] ** 2).sum()
    return u, float(objective)


def _ramp64(g):
    """The Ram-Lak filter of each view, a linear convolution over the bins."""
    bins = g.shape[1]
    m = torch.arange(bins, dtype=torch.float64, device=g.device)
    half = torch.where(m % 2 == 1, -1 / (math.pi * m.clamp(min=1)) ** 2, 0.0)
    half[0] = 0.25
    size = 2 * bins
    kernel = torch.zeros(size, dtype=torch.float64, device=g.device)
    kernel[:bins] = half
    kernel[size - bins + 1:] = half[1:].flip(0)
    return torch.fft.irfft(torch.fft.rfft(g, size) * torch.fft.rfft(kernel), size)[:, :bins]


def exact(case, seed):
    x = _inputs(case, seed)
    kind = case["kind"]
    if kind == "batch":
        out = []
        for i, c in enumerate(_batch_cases(case)):
            radon = _Radon64(c)
            out.append(_solve64(radon, x["f"][i], x["mask"][i], case["alpha"], x["delta"][i], case["iters"], False,
                                _kept_scaling(c["n"], c["views"]))[0])
        return out
    if kind == "precond":
        norm, lap = _frequencies64(case["n"], _device())
        c = _kept_scaling(case["n"], case["views"])[1]
        return _filter64(x["y"].double(), norm / (c + TAU ** 2 * lap * norm))
    radon = _Radon64(case)
    if kind == "forward":
        return radon.forward(x["u"].double())
    if kind == "adjoint":
        return radon.adjoint(x["g"].double())
    if kind == "pair":
        return {"g": radon.forward(x["u"].double()), "u": radon.adjoint(x["g"].double())}
    if kind == "layer":
        return {"g": radon.forward(x["u"].double()), "grad": radon.adjoint(x["g"].double())}
    if kind == "fbp":
        return math.pi / case["views"] * radon.adjoint(_ramp64(x["f"].double()))
    scaling = _kept_scaling(case["n"], case["views"]) if case["scaling"] == "kept" else None
    u, objective = _solve64(radon, x["f"], x["mask"], case["alpha"], x["delta"], case["iters"], case["nonneg"], scaling)
    return {"u": u, "objective": objective}
