"""The work that programs have this package do, as cases that can be timed and compared.

Every case is one call sequence of the public entry points: the stretched operator and the residual
(`operator`, `residual`), one application of the source-transfer preconditioner with the factors in hand
(`precondition`), a new geometry factored and applied once (`factor`), a new geometry factored and solved
(`solve`), and the initial-guess network's forward pass and loss gradient (`nn_forward`, `nn_gradient`).

Fields are complex128 with node (i, j) at i * ny + j.  Geometries are drawn from the seed: ellipses of eps
2 .. 12.1 in vacuum, wavy guides of eps 12.1 in 2.085, pillars of eps 12.1 on a substrate, and (where the
preconditioner itself is the output) a film on a substrate, at lambda / 24.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2509_20801_gb300 import Solver
from paper_2509_20801_gb300 import binding as stdd
from paper_2509_20801_gb300.learned import Network

PPW = 24
ADDITIVE, SYMMETRIC, RED_BLACK, FORWARD = 0, 1, 2, 3


def _problem(do, nx, ny, nsub, medium="ellipses", npml=20, overlap=8, ipml=20, precision="fp64", order=ADDITIVE,
             pivoting=0, band=0, nrhs=1):
    return dict(do=do, nx=nx, ny=ny, nsub=nsub, medium=medium, npml=npml, overlap=overlap, ipml=ipml,
                precision=precision, order=order, pivoting=pivoting, band=band, nrhs=nrhs)


def listed():
    return [
        # the smallest call: one operator product on the cylinder example's grid, a user's own iteration
        dict(_problem("operator", 200, 200, 2), name="operator-200x200"),
        # a residual check of a finished metalens field
        dict(_problem("residual", 4096, 1024, 16, "metalens", npml=30, overlap=12, ipml=30),
             name="residual-4096x1024"),
        # one preconditioner application on the smallest example: latency and launches
        dict(_problem("precondition", 200, 200, 2, "layers"), name="precondition-200x200"),
        # an odd grid with uneven strips
        dict(_problem("precondition", 874, 509, 9, "layers", npml=30, overlap=12, ipml=30),
             name="precondition-874x509"),
        # the sequential order that guided-wave networks are solved with: one strip after another
        dict(_problem("precondition", 2048, 512, 8, "layers", npml=32, overlap=16, ipml=32, order=SYMMETRIC),
             name="precondition-sequential-2048x512"),
        # the metalens configuration at full size, all strips at once
        dict(_problem("precondition", 4096, 1024, 16, "layers", npml=30, overlap=12, ipml=30),
             name="precondition-4096x1024"),
        # preprocessing of a new permittivity and the first application of its factors
        dict(_problem("factor", 1024, 512, 4, "layers", npml=30, overlap=12, ipml=30), name="factor-1024x512"),
        # the guided-wave network at its shrunk size: factored and solved in complex128
        dict(_problem("solve", 2048, 512, 8, "guides", npml=32, overlap=16, ipml=32, order=SYMMETRIC),
             name="solve-guides-2048x512"),
        # one geometry of the batched workload: complex64 factors pivoted within fronts, eight point sources
        dict(_problem("solve", 512, 512, 3, precision="c64", order=RED_BLACK, pivoting=1, nrhs=8),
             name="solve-c64-512x512x8"),
        # a metalens in complex128 through the interface bands, the way its own benchmark solves it
        dict(_problem("solve", 1024, 256, 4, "metalens", npml=30, overlap=12, ipml=30, band=1),
             name="solve-band-1024x256"),
        # the network's guess for one field of the evaluation size, and its gradient on a training batch
        dict(do="nn_forward", batch=1, height=512, width=1024, levels=6, base=32, widest=256,
             name="nn-forward-1024x512"),
        dict(do="nn_gradient", batch=8, height=512, width=512, levels=6, base=32, widest=256,
             name="nn-gradient-512x512x8"),
    ]


# Strip widths and heights of drawn preconditioners.  A separator's box is eliminated with its border held
# fixed, as a closed cavity, and one close to a resonance in air loses digits; these keep clear of that, so
# that a strip's field is determined to rounding by its operator.
CLEAR = {
    90: (101, 128, 200, 233, 256, 333, 384, 400, 509, 512, 640, 767),
    97: (101, 128, 200, 233, 333, 384, 509, 512, 640, 767),
    128: (101, 128, 200, 233, 256, 509, 512, 640),
    161: (101, 128, 200, 233, 256, 333, 384, 509, 512, 640, 767),
    200: (101, 128, 200, 233, 384, 509, 512, 640, 767),
    203: (101, 128, 200, 233, 384, 509, 512, 640, 767),
    256: (101, 128, 200, 333, 384, 509, 512, 640),
    301: (101, 128, 200, 233, 256, 333, 509, 640),
}


def _between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(("operator", "residual", "precondition", "precondition", "precondition", "factor", "solve",
                     "solve", "solve", "nn_forward", "nn_gradient"))
    if do in ("operator", "residual"):
        return _problem(do, _between(rng, 100, 4096), _between(rng, 100, 1024), 1)
    if do in ("nn_forward", "nn_gradient"):
        side = 32  # image sides are multiples of 2 ** (levels - 1)
        return dict(do=do, batch=1 if do == "nn_forward" else rng.choice((1, 2, 4, 8)),
                    height=side * _between(rng, 3, 16), width=side * _between(rng, 3, 16), levels=6, base=32,
                    widest=256)
    order = rng.choice((ADDITIVE, ADDITIVE, SYMMETRIC, RED_BLACK, FORWARD))
    if do != "solve":
        # strips of a width, the first perhaps one wider
        width = rng.choice(sorted(CLEAR))
        ny = rng.choice(CLEAR[width])
        nsub = rng.randint(2, 8)
        return _problem(do, width * nsub + rng.randint(0, 1), ny, nsub, "layers", 30, 12, 30, order=order)
    medium = rng.choice(("ellipses", "ellipses", "guides", "metalens"))
    npml, overlap, ipml = dict(ellipses=(20, 8, 20), guides=(32, 16, 32), metalens=(30, 12, 30))[medium]
    nx, ny = _between(rng, 200, 1024), _between(rng, 200, 512)
    nsub = rng.randint(1, max(1, nx // 100))
    # complex64 factors are met through a solve, whose FGMRES brings the field to complex128
    c64 = rng.random() < 0.5
    band = int(not c64 and order == ADDITIVE and rng.random() < 0.5)
    return _problem(do, nx, ny, nsub, medium, npml, overlap, ipml, "c64" if c64 else "fp64", order, int(c64), band,
                    rng.choice((1, 1, 2, 8)))


# ---------------------------------------------------------------- inputs

def _generator(seed, device):
    return torch.Generator(device=device).manual_seed(int(seed) & 0x7FFFFFFF)


def _permittivity(case, seed, device):
    """Node permittivity (nx, ny) float64: the mean of four samples around each node."""
    nx, ny, npml = case["nx"], case["ny"], case["npml"]
    r = np.random.default_rng(seed)
    x = (torch.arange(2 * nx, device=device, dtype=torch.float64) - 0.5) / (2 * PPW)   # wavelengths
    y = (torch.arange(2 * ny, device=device, dtype=torch.float64) - 0.5) / (2 * PPW)
    lx, ly = nx / PPW, ny / PPW
    if case["medium"] == "layers":
        # a film of 0.6 wavelengths on a substrate, each within its tolerance of the nominal permittivity
        floor = round(0.2 * ny) / PPW
        line = torch.ones(2 * ny, device=device, dtype=torch.float64)
        line[y <= floor + round(0.6 * PPW) / PPW] = 4.0 + 1e-4 * r.uniform(-1, 1)
        line[y <= floor] = 2.085 + 1e-4 * r.uniform(-1, 1)
        eps = line.expand(2 * nx, 2 * ny)
    elif case["medium"] == "guides":
        eps = torch.full((2 * nx, 2 * ny), 2.085, device=device, dtype=torch.float64)
        for q in range(3):
            middle, swing = ly * (0.25 + 0.25 * q), 0.04 * ly * r.uniform(-1, 1)
            start, length = lx * r.uniform(0.2, 0.6), lx * r.uniform(0.08, 0.15)
            t = ((x - start) / length).clamp(0, 1)
            yc = middle + 0.5 * swing * (1 - torch.cos(math.pi * t))
            eps[(y[None, :] - yc[:, None]).abs() <= 0.225] = 12.1
    elif case["medium"] == "metalens":
        eps = torch.ones((2 * nx, 2 * ny), device=device, dtype=torch.float64)
        floor = round(0.2 * ny) / PPW
        eps[:, y <= floor] = 2.085
        edge = (npml + 1) / PPW
        rows = (y > floor) & (y <= floor + round(0.6 * PPW) / PPW)
        count = int((lx - 2 * edge) / 0.5)
        half = torch.from_numpy(0.5 * r.uniform(0.1, 0.4, max(count, 1))).to(device)
        k = torch.floor((x - edge) / 0.5).long()
        inside = (k >= 0) & (k < count)
        k = k.clamp(0, max(count - 1, 0))
        inside &= (x - edge - 0.5 * (k + 0.5)).abs() <= half[k]
        eps[inside[:, None] & rows[None, :]] = 12.1
    else:
        eps = torch.ones((2 * nx, 2 * ny), device=device, dtype=torch.float64)
        edge = (npml + 0.5 * PPW) / PPW
        target, got, placed = r.uniform(0.15, 0.30) * max(0.0, lx - 2 * edge) * max(0.0, ly - 2 * edge), 0.0, []
        for _ in range(400):
            if got >= target:
                break
            a, b = r.uniform(0.2, 1.0, 2)
            big = max(a, b)
            if lx - 2 * (edge + big) <= 0 or ly - 2 * (edge + big) <= 0:
                continue
            cx, cy = r.uniform(edge + big, lx - edge - big), r.uniform(edge + big, ly - edge - big)
            angle, value = r.uniform(0, math.pi), r.uniform(2.0, 12.1)
            if any((cx - px) ** 2 + (cy - py) ** 2 < (big + pr) ** 2 for px, py, pr in placed):
                continue
            placed.append((cx, cy, big))
            got += math.pi * a * b
            i0, i1 = max(0, int((cx - big) * 2 * PPW)), min(2 * nx, int((cx + big) * 2 * PPW) + 3)
            j0, j1 = max(0, int((cy - big) * 2 * PPW)), min(2 * ny, int((cy + big) * 2 * PPW) + 3)
            u, v = x[i0:i1, None] - cx, y[None, j0:j1] - cy
            c, s = math.cos(angle), math.sin(angle)
            hit = ((u * c + v * s) / a) ** 2 + ((v * c - u * s) / b) ** 2 <= 1
            eps[i0:i1, j0:j1][hit] = value
    return eps.reshape(nx, 2, ny, 2).mean(dim=(1, 3)).contiguous()


def _sources(case, seed, device):
    """Right-hand sides (nrhs, nx, ny): point sources, a guide's mode-like column, or a line source."""
    nx, ny, npml = case["nx"], case["ny"], case["npml"]
    r = np.random.default_rng(seed + 1)
    b = torch.zeros((case["nrhs"], nx, ny), device=device, dtype=torch.complex128)
    for q in range(case["nrhs"]):
        if case["medium"] == "guides":
            j = torch.arange(ny, device=device, dtype=torch.float64)
            at = ny * (0.25 + 0.25 * ((q + seed) % 3))
            b[q, npml + 12] = -PPW * torch.exp(-((j - at) / (0.3 * PPW)) ** 2) * r.uniform(0.5, 2.0)
        elif case["medium"] in ("metalens", "layers"):
            b[q, :, npml + 10 + 3 * q % 24] = -PPW * r.uniform(0.5, 2.0)
        else:
            i = int(r.integers(npml + PPW // 2, nx - npml - PPW // 2))
            j = int(r.integers(npml + PPW // 2, ny - npml - PPW // 2))
            b[q, i, j] = -float(PPW * PPW)
    return b


def _field(case, seed, device):
    """A dense complex field, as Krylov vectors are."""
    g = _generator(seed + 2, device)
    return torch.view_as_complex(torch.randn((case["nx"], case["ny"], 2), generator=g, device=device,
                                             dtype=torch.float64))


def _solver(case, eps):
    d = 1.0 / PPW
    s = Solver(case["nx"], case["ny"], d, d, 1.0, eps, npml=(case["npml"],) * 4, nsub=case["nsub"],
               overlap=case["overlap"], interface_pml=case["ipml"],
               precision=stdd.STDD_PREC_C64 if case["precision"] == "c64" else stdd.STDD_PREC_FP64)
    stdd.stdd_set_option(s.ctx, stdd.STDD_OPT_ORDER, case["order"])
    stdd.stdd_set_option(s.ctx, stdd.STDD_OPT_PIVOTING, case["pivoting"])
    stdd.stdd_set_option(s.ctx, stdd.STDD_OPT_BAND, case["band"])
    return s


def _layers(case):
    """(cin, cout) of the network's convolutions in parameter order."""
    ch = [min(case["base"] << l, case["widest"]) for l in range(case["levels"])]
    out = []
    for l, c in enumerate(ch):
        out += [(3 if l == 0 else ch[l - 1], c), (c, c)]
    for l in range(case["levels"] - 2, -1, -1):
        out += [(ch[l + 1], ch[l]), (ch[l], ch[l])]
    return out + [(ch[0], 2)]


def _network_inputs(case, seed, device):
    """He-normal parameters with small biases, smooth images and targets."""
    r = np.random.default_rng(seed)
    parts = []
    for cin, cout in _layers(case):
        parts += [r.standard_normal(cout * cin * 9) * math.sqrt(2.0 / (9 * cin)), 0.01 * r.standard_normal(cout)]
    params = np.concatenate(parts).astype(np.float32)
    g = _generator(seed + 3, device)
    n, h, w = case["batch"], case["height"], case["width"]

    def images(channels):
        z = torch.randn((n, channels, h // 8, w // 8), generator=g, device=device)
        return torch.nn.functional.interpolate(z, size=(h, w), mode="bilinear").contiguous()

    return params, images(3), images(2)


def prepare(case, seed):
    device = torch.device("cuda", 0)
    if case["do"].startswith("nn_"):
        params, image, target = _network_inputs(case, seed, device)
        net = Network(case["levels"], case["base"], case["widest"], mode="tc")
        net.set_params(params)
        out = torch.empty((case["batch"], 2, case["height"], case["width"]), device=device)
        torch.cuda.synchronize()
        return dict(do=case["do"], net=net, image=image, target=target, out=out)
    eps = _permittivity(case, seed, device)
    v = _field(case, seed, device)
    state = dict(do=case["do"], eps=eps, v=v, z=torch.empty_like(v))
    if case["do"] == "residual":
        state["x"] = _field(case, seed + 10, device)
    if case["do"] == "solve":
        state["b"] = _sources(case, seed, device)
        state["x"] = torch.empty_like(state["b"])
    torch.cuda.synchronize()
    state["solver"] = s = _solver(case, eps)
    if case["do"] == "operator":
        # sets the operator up, as a program's first product does
        stdd.stdd_apply_operator(s.ctx, v, state["z"])
    elif case["do"] == "residual":
        stdd.stdd_residual(s.ctx, state["x"], v, state["z"])
    else:
        # the plan a program keeps: symbolic analysis, buffers and launch shapes
        s.factor()
    return state


def run(state):
    do = state["do"]
    if do == "nn_forward":
        state["net"].forward(state["image"], state["out"])
        return state["out"]
    if do == "nn_gradient":
        loss, grad = state["net"].gradient(state["image"], state["target"])
        return {"loss": loss, "grad": grad}
    s = state["solver"]
    if do == "operator":
        stdd.stdd_apply_operator(s.ctx, state["v"], state["z"])
        return state["z"]
    if do == "residual":
        rel = stdd.stdd_residual(s.ctx, state["x"], state["v"], state["z"])
        return {"r": state["z"], "rel": rel}
    if do == "precondition":
        stdd.stdd_apply_preconditioner(s.ctx, state["v"], state["z"])
        return state["z"]
    stdd.stdd_set_permittivity(s.ctx, state["eps"])
    s.factor()
    if do == "factor":
        stdd.stdd_apply_preconditioner(s.ctx, state["v"], state["z"])
        return state["z"]
    s.set_sources(state["b"])
    s.solve(state["x"], restart=50, maxit=2000, rtol=1e-12)
    return state["x"]


# ---------------------------------------------------------------- least work

def _parts(case):
    """(c0, c1, x0, x1, low PML, high PML) of every strip."""
    n, k, ext = case["nx"], case["nsub"], case["overlap"] + case["ipml"]
    cut = [0]
    for q in range(k):
        cut.append(cut[-1] + n // k + (1 if q < n % k else 0))
    return [(cut[q], cut[q + 1], cut[q] - ext if q else 0, cut[q + 1] + ext if q < k - 1 else n,
             case["ipml"] if q else case["npml"], case["ipml"] if q < k - 1 else case["npml"]) for q in range(k)]


@functools.lru_cache(maxsize=64)
def _elimination(width, height):
    """(complex entries, real flops) of the symmetric factors of a width x height box."""
    a = stdd.stdd_nd_analyze(width, height, 16)
    p, b = a["p"].astype(np.float64), a["b"].astype(np.float64)
    n = p + b
    cubes = lambda m: m * (m + 1) * (m + 2) / 6   # the triangles m (m + 1) / 2 of trailing blocks, summed
    return float((p * (p + 1) / 2 + p * b).sum()), float(8 * (cubes(n - 1) - cubes(b - 1)).sum())


def work(case):
    if case["do"].startswith("nn_"):
        h, w, lv = case["height"], case["width"], case["levels"]
        at = [l for l in range(lv) for _ in (0, 1)] + [l for l in range(lv - 2, -1, -1) for _ in (0, 1)] + [0]
        pixels = [case["batch"] * (h >> l) * (w >> l) for l in at]
        flops = sum(18.0 * cin * cout * px for (cin, cout), px in zip(_layers(case), pixels))
        params = sum(9 * cin * cout + cout for cin, cout in _layers(case))
        if case["do"] == "nn_forward":
            return {"bytes": 4.0 * (params + 5 * pixels[0]), "flops": flops}
        return {"bytes": 4.0 * (2 * params + 5 * pixels[0]), "flops": 3 * flops}
    n = case["nx"] * case["ny"]
    if case["do"] == "operator":
        return {"bytes": 40.0 * n, "flops": 40.0 * n}
    if case["do"] == "residual":
        return {"bytes": 56.0 * n, "flops": 52.0 * n}
    entries = flops = 0.0
    for _, _, x0, x1, _, _ in _parts(case):
        e, f = _elimination(x1 - x0, case["ny"])
        entries, flops = entries + e, flops + f
    size = 8.0 if case["precision"] == "c64" else 16.0
    times = 2.0 - 1.0 / case["nsub"] if case["order"] == SYMMETRIC else 1.0
    once = {"bytes": size * entries * times + 32.0 * n, "flops": 16.0 * entries * times}
    if case["do"] == "precondition":
        return once
    if case["do"] == "factor":
        return {"bytes": size * entries + 8.0 * n + once["bytes"], "flops": flops + once["flops"]}
    # a solve needs at least one iteration: its iteration count depends on the medium
    return {"bytes": size * entries + 8.0 * n + once["bytes"] + 32.0 * n * case["nrhs"],
            "flops": flops + once["flops"] * case["nrhs"]}


# ---------------------------------------------------------------- 64-bit values

def _profile(n, lo, hi):
    """Stretch at the nodes and half nodes of a line with PMLs of lo and hi cells."""
    d, k0, m, refl = 1.0 / PPW, 2 * math.pi, 3, 1e-8

    def sigma(pos):
        v = np.zeros_like(pos)
        for cells, depth in ((lo, (lo - 0.5) - pos), (hi, pos - (n - hi - 0.5))):
            if cells:
                v += (m + 1) * -math.log(refl) / (2 * k0 * cells * d) * (np.maximum(0.0, depth) / cells) ** m
        return v

    return 1 + 1j * sigma(np.arange(n, dtype=float)), 1 + 1j * sigma(np.arange(n + 1, dtype=float) - 0.5)


def _couplings(n, lo, hi, device):
    s, half = _profile(n, lo, hi)
    to = lambda a: torch.from_numpy(a * PPW ** 2).to(device)
    return to(1 / (s * half[:-1])), to(1 / (s * half[1:]))


def _coefficients(eps, px, py):
    """Couplings to i - 1, i + 1, j - 1, j + 1 and the diagonal of the stretched operator."""
    w, h = eps.shape
    cxm, cxp = _couplings(w, *px, eps.device)
    cym, cyp = _couplings(h, *py, eps.device)
    diag = (2 * math.pi) ** 2 * eps - (cxm + cxp)[:, None] - (cym + cyp)[None, :]
    return cxm, cxp, cym, cyp, diag


def _apply(co, x):
    cxm, cxp, cym, cyp, diag = co
    y = diag * x
    y[..., 1:, :] += cxm[1:, None] * x[..., :-1, :]
    y[..., :-1, :] += cxp[:-1, None] * x[..., 1:, :]
    y[..., :, 1:] += cym[1:] * x[..., :, :-1]
    y[..., :, :-1] += cyp[:-1] * x[..., :, 1:]
    return y


class _Direct:
    """Block elimination of the operator along its longer side, with one step of refinement."""

    def __init__(self, eps, px, py):
        self.co = _coefficients(eps, px, py)
        w, h = eps.shape
        self.swap = w > h   # blocks of the shorter side
        cxm, cxp, cym, cyp, diag = self.co
        if self.swap:
            cxm, cxp, cym, cyp, diag = cym, cyp, cxm, cxp, diag.T.contiguous()
        self.lo, self.hi = cym, cyp
        side, steps = diag.shape
        inner = torch.diag(cxm[1:], -1) + torch.diag(cxp[:-1], 1)
        self.inv = torch.empty((steps, side, side), dtype=torch.complex128, device=eps.device)
        for j in range(steps):
            block = inner + torch.diag(diag[:, j])
            if j:
                block = block - self.lo[j] * self.hi[j - 1] * self.inv[j - 1]
            self.inv[j] = torch.linalg.inv(block)

    def _once(self, t):
        t = t.transpose(-1, -2) if self.swap else t       # (rhs, side, steps)
        t = t.permute(2, 1, 0).clone(memory_format=torch.contiguous_format)   # (steps, side, rhs)
        for j in range(1, t.shape[0]):
            t[j] -= self.lo[j] * (self.inv[j - 1] @ t[j - 1])
        for j in range(t.shape[0] - 1, -1, -1):
            t[j] = self.inv[j] @ (t[j] - self.hi[j] * t[j + 1] if j + 1 < t.shape[0] else t[j])
        t = t.permute(2, 1, 0)
        return (t.transpose(-1, -2) if self.swap else t).contiguous()

    def __call__(self, t):
        x = self._once(t)
        return x + self._once(t - _apply(self.co, x))


def _cost(case):
    """Rough seconds of the 64-bit elimination."""
    if case["do"] == "solve":
        boxes = [(case["nx"], case["ny"])]
    else:
        boxes = [(x1 - x0, case["ny"]) for _, _, x0, x1, _, _ in _parts(case)]
    return sum(max(a, b) * (2e-3 + 3e-11 * min(a, b) ** 3) for a, b in boxes)


def exact(case, seed):
    device = torch.device("cuda", 0)
    if case["do"].startswith("nn_"):
        return _exact_network(case, seed, device)
    eps = _permittivity(case, seed, device)
    v = _field(case, seed, device)
    py = (case["npml"], case["npml"])
    whole = (case["npml"], case["npml"])
    if case["do"] == "operator":
        return _apply(_coefficients(eps, whole, py), v)
    if case["do"] == "residual":
        r = v - _apply(_coefficients(eps, whole, py), _field(case, seed + 10, device))
        return {"r": r, "rel": float(torch.linalg.vector_norm(r) / torch.linalg.vector_norm(v))}
    if _cost(case) > 18:
        return None
    if case["do"] == "solve":
        return _Direct(eps, whole, py)(_sources(case, seed, device))
    parts = _parts(case)
    solvers = [_Direct(eps[x0:x1].contiguous(), (lo, hi), py) for _, _, x0, x1, lo, hi in parts]
    co = _coefficients(eps, whole, py)
    z = torch.zeros_like(v)

    def add(group, residual):
        for k in group:
            c0, c1, x0, x1, _, _ = parts[k]
            t = torch.zeros((1, x1 - x0, case["ny"]), dtype=torch.complex128, device=device)
            t[0, c0 - x0:c1 - x0] = residual[c0:c1]
            z[x0:x1] += solvers[k](t)[0]

    n = len(parts)
    if case["order"] == ADDITIVE:
        groups = [range(n)]
    elif case["order"] == RED_BLACK:
        groups = [range(0, n, 2), range(1, n, 2)]
    else:
        groups = [[k] for k in range(n)]
        if case["order"] == SYMMETRIC:
            groups += [[k] for k in range(n - 2, -1, -1)]
    for q, group in enumerate(groups):
        add(group, v - _apply(co, z) if q else v)
    return z


def _exact_network(case, seed, device):
    conv, pool = torch.nn.functional.conv2d, torch.nn.functional.avg_pool2d
    params, image, target = _network_inputs(case, seed, device)
    grad = case["do"] == "nn_gradient"
    flat = torch.from_numpy(params.astype(np.float64)).to(device).requires_grad_(grad)

    def forward(x):
        at = 0
        weights = []
        for cin, cout in _layers(case):
            weights.append((flat[at:at + 9 * cin * cout].reshape(cout, cin, 3, 3),
                            flat[at + 9 * cin * cout:at + 9 * cin * cout + cout]))
            at += 9 * cin * cout + cout
        layer = iter(weights)
        step = lambda x: torch.relu(conv(x, *next(layer), padding=1))
        skips = []
        for l in range(case["levels"]):
            x = step(step(pool(x, 2) if l else x))
            skips.append(x)
        for l in range(case["levels"] - 2, -1, -1):
            x = x.repeat_interleave(2, dim=2).repeat_interleave(2, dim=3)
            x = step(step(x) + skips[l])
        return conv(x, *next(layer), padding=1)

    if not grad:
        with torch.no_grad():
            return forward(image.double())
    total, loss = target.numel(), 0.0
    for q in range(case["batch"]):   # one image at a time: the graph of a batch is large in 64 bits
        part = ((forward(image[q:q + 1].double()) - target[q:q + 1].double()) ** 2).sum() / total
        part.backward()
        loss += float(part.detach())
    return {"loss": loss, "grad": flat.grad}
