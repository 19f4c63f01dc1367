"""Work that a user of the solver has it do, through its public entry points, at the sizes it is used at.

A case is one call sequence of a user's program: a solve with its adjoint and gradient, a forward
solve, a differentiated focal intensity, a design step, a design iteration from host buffers, or a
batch of served requests.  Solves run a fixed number of iterations (tol = 0): a converged solve is
thousands of the same iterations, so a few blocks of them stand for it and the work is exact.

    listed()   the cases              prepare(case, seed)   what a program has in hand beforehand
    draw(rng)  one more of the range  run(state)            one pass
    work(case) its bytes and flops    exact(case, seed)     the same outputs in 64 bits by plain torch
"""
from __future__ import annotations

import math

import numpy as np
import torch

LAM = 1.064e-6                     # vacuum wavelength [m] of every configuration of the package
GENTLE = {"layer_round_trip": 1e-2, "layer_corner_max": True}   # the serving streams' layers


def _case(name, op, grid, ppl, pads, shape, iters, layers="default", source="plane", check=32, requests=1):
    return {"name": name, "op": op, "nx": grid[0], "ny": grid[1], "nz": grid[2], "ppl": ppl,
            "px": pads[0], "py": pads[1], "pz": pads[2], "shape": shape, "iters": iters, "layers": layers,
            "source": source, "check": check, "requests": requests}


def listed():
    return [
        # the smallest grid: the sphere workload and the first size of the serving streams, solved
        # for one gradient of the focal intensity (launches and their gaps count)
        _case("sphere_64", "solve", (64, 64, 64), 8, (8, 8, 8), "sphere", 32, "gentle"),
        # six requests of that size in flight at once, half of them with the adjoint
        _case("serve_64", "serve", (64, 64, 64), 8, (8, 8, 8), "mixed", 32, "gentle", requests=6),
        # one differentiated solve of a small design slab, warm-started from an earlier field
        _case("autograd_96x96x64", "autograd", (96, 96, 64), 8, (8, 8, 8), "slab", 16),
        # the coarse end of the lens resolution sweep (lambda / 6): axes with a factor 13
        _case("sweep_104x104x120", "forward", (104, 104, 120), 6, (6, 6, 36), "lens", 64, check=64),
        # a dipole in a sphere at the second size of the serving streams
        _case("dipole_128", "forward", (128, 128, 128), 8, (8, 8, 8), "sphere", 64, "gentle", "point"),
        # a caller's own source (a Gaussian beam's current sheet) at lambda / 10: odd axes
        _case("beam_175x175x198", "forward", (175, 175, 198), 10, (10, 10, 60), "lens", 32, source="user"),
        # one step of the design loop: map -> permittivity -> both solves -> dL/dh -> Adam
        _case("design_192x192x128", "design", (192, 192, 128), 8, (8, 8, 8), "lens", 16, "gentle"),
        # a design iteration from and to host memory on the 256 x 256 x 192 design volume
        _case("host_256x256x192", "host", (256, 256, 192), 8, (8, 8, 24), "slab", 16, check=16),
        # the Fresnel lens benchmark at lambda / 16: every axis odd
        _case("lens_275x275x315", "forward", (275, 275, 315), 16, (16, 16, 96), "lens", 32),
        # the largest size of the serving streams with its adjoint and gradient
        _case("solve_384x384x256", "solve", (384, 384, 256), 8, (8, 8, 8), "lens", 16, "gentle", check=16),
        # the paper-scale design volume (621 x 621 x 261 voxels at lambda / 6 and its layers)
        _case("paper_640x640x336", "solve", (640, 640, 336), 6, (6, 6, 36), "lens", 12, check=12),
    ]


def _smooth(n, odd=False):
    """The supported axis length (prime factors up to 13) nearest to n; odd: the nearest odd one."""
    def ok(m):
        for p in (2, 3, 5, 7, 11, 13):
            while m % p == 0:
                m //= p
        return m == 1
    return min((m for m in range(1, 1025) if ok(m) and (m % 2 or not odd)), key=lambda m: (abs(m - n), m))


def draw(rng):
    op = rng.choice(["solve", "solve", "forward", "forward", "forward", "autograd", "design", "host", "serve"])
    top = 384 * 384 * 256 if op in ("host", "serve") else 640 * 640 * 336
    vox = math.exp(rng.uniform(math.log(40 ** 3), math.log(top)))
    if op == "serve":
        vox = min(vox, 192 * 192 * 128)
    flat = math.exp(rng.uniform(math.log(0.5), math.log(2.0)))      # nz against nx
    skew = math.exp(rng.uniform(math.log(0.7), math.log(1.4)))      # ny against nx
    side = (vox / (flat * skew)) ** (1 / 3)
    grid = [max(24, min(1000, int(round(v)))) for v in (side, side * skew, side * flat)]
    if op == "design":
        grid[1] = grid[0]
    grid = [_smooth(v) for v in grid]
    if op != "design" and rng.random() < 0.3:                       # an odd axis more often than by chance
        k = rng.randrange(3)
        grid[k] = _smooth(grid[k], odd=True)
    ppl = rng.choice([6, 8, 10, 12, 16])
    pads = [min(ppl, n // 5) for n in grid]
    pads[2] = min(rng.choice([1, 3, 6]) * ppl, grid[2] // 4)
    n = grid[0] * grid[1] * grid[2]
    iters = max(4, min(rng.choice([16, 24, 32, 48]), int(12 * 640 * 640 * 336 / n)))
    source = rng.choice(["plane", "plane", "point", "user"]) if op == "forward" else "plane"
    shape = {"autograd": "slab", "host": "slab", "design": "lens", "serve": "mixed"}.get(op) or \
        rng.choice(["lens", "sphere", "slab"])
    c = _case("", op, grid, ppl, pads, shape, iters, rng.choice(["default", "gentle"]), source,
              rng.choice([8, 16, 32]), rng.choice([2, 3, 5, 8]) if op == "serve" else 1)
    del c["name"]
    return c


# ------------------------------------------------------------------------------------ inputs
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _rng(seed, k=0):
    return np.random.default_rng([int(seed) & 0x7FFFFFFF, k])


def _centred(n, dev, dtype=torch.float32):
    return torch.arange(n, device=dev, dtype=dtype) - (n - 1) / 2


def _height(c, dev, n_lens, scale):
    """Kinoform thickness map in voxels (ny, nx): one wrapped phase ramp per zone, NA 0.84."""
    x, y = _centred(c["nx"], dev, torch.float64), _centred(c["ny"], dev, torch.float64)
    r2 = x[None, :] ** 2 + y[:, None] ** 2
    radius = 0.5 * scale * (min(c["nx"], c["ny"]) - 2 * max(c["px"], c["py"]))
    f = radius / math.tan(math.asin(0.84))
    path = (torch.sqrt(r2 + f * f) - f) / c["ppl"]
    h = c["ppl"] / (n_lens - 1.0) * (1.0 - (path - torch.floor(path)))
    return torch.where(r2 <= radius ** 2, h, torch.zeros_like(h))


def _fill(c, h, n_lens, dev):
    """Permittivity of a height map above its base plane, filled by fractions along z."""
    k = torch.arange(c["nz"], device=dev, dtype=torch.float32) - (c["pz"] + 2)
    eps = torch.clamp(h.to(torch.float32)[None] - k[:, None, None], 0.0, 1.0)
    eps[: c["pz"] + 2] = 0.0
    return eps.mul_(n_lens ** 2 - 1.0).add_(1.0)


def _eps(c, seed, k=0):
    """Permittivity float32 (nz, ny, nx): a Fresnel lens, a sphere, or a noisy design slab."""
    dev, rng = _device(), _rng(seed, k)
    n_idx = float(rng.uniform(1.3, 1.6))
    shape = c["shape"] if c["shape"] != "mixed" else ("sphere", "lens")[k % 2]
    if shape == "sphere":
        radius = min(12.0, 0.3 * (min(c["nx"], c["ny"], c["nz"]) - 2 * max(c["px"], c["py"])))
        at = rng.uniform(-1.0, 1.0, 3)
        x, y, z = (_centred(c[a], dev) - float(o) for a, o in zip(("nx", "ny", "nz"), at))
        d = torch.sqrt(z[:, None, None] ** 2 + y[None, :, None] ** 2 + x[None, None, :] ** 2)
        return torch.clamp(radius - d + 0.5, 0.0, 1.0).mul_(n_idx ** 2 - 1.0).add_(1.0)
    h = _height(c, dev, n_idx, float(rng.uniform(0.6, 0.8)))
    eps = _fill(c, h, n_idx, dev)
    if shape == "slab":
        g = torch.Generator(device=dev)
        g.manual_seed(int(rng.integers(1 << 31)))
        z0 = c["pz"] + 2
        part = eps[z0: z0 + max(4, c["nz"] // 4), c["py"]: c["ny"] - c["py"], c["px"]: c["nx"] - c["px"]]
        part.add_(torch.rand(part.shape, generator=g, device=dev) * 0.2 - 0.1).clamp_(1.0, n_idx ** 2)
    return eps


def _beam(c, seed):
    """Current sheet of a Gaussian beam, (3, nz, ny, nx) complex64, its waist set by the seed."""
    dev, rng = _device(), _rng(seed, 7)
    pitch = LAM / c["ppl"]
    w = float(rng.uniform(0.2, 0.35)) * min(c["nx"], c["ny"])
    x, y = _centred(c["nx"], dev), _centred(c["ny"], dev)
    prof = torch.exp(-(x[None, :] ** 2 + y[:, None] ** 2) / (w * w))
    S = torch.zeros((3, c["nz"], c["ny"], c["nx"]), dtype=torch.complex64, device=dev)
    amp = -2j * (2 * math.pi / LAM) / pitch
    S[0, c["pz"]] = amp * prof
    S[1, c["pz"]] = 0.5j * amp * prof
    return S


def _earlier_field(c, seed):
    """A field a warm start begins from: the background's plane wave, a little off."""
    dev, rng = _device(), _rng(seed, 8)
    z = torch.arange(c["nz"], device=dev, dtype=torch.float64) - c["pz"]
    wave = torch.exp(1j * (2 * math.pi / c["ppl"]) * z.abs()) * float(rng.uniform(0.9, 1.1))
    E = torch.zeros((3, c["nz"], c["ny"], c["nx"]), dtype=torch.complex64, device=dev)
    E[0] = wave.to(torch.complex64)[:, None, None]
    return E


def _focus(c):
    """Objective voxel (x, y, z): on the source sheet, where the field of these iterations is strongest."""
    return (c["nx"] // 2, c["ny"] // 2, c["pz"])


def _dipole(c, seed):
    rng = _rng(seed, 9)
    pitch = LAM / c["ppl"]
    at = tuple(n // 2 + int(rng.integers(-2, 3)) for n in (c["nx"], c["ny"], c["nz"]))
    return at, tuple(complex(v) / pitch ** 3 for v in rng.standard_normal(3) + 1j * rng.standard_normal(3))


def _design_params(c):
    pitch_um = LAM / c["ppl"] * 1e6
    return dict(z_base=c["pz"] + 2, n_lens=1.54, aperture_um=0.7 * (c["nx"] - 2 * c["px"]) * pitch_um,
                h_max_um=LAM * 1e6 / 0.54, sigma_um=0.355, mirror=True)


def _design_map(c, seed):
    """Height map [um], (ny, nx): a Fresnel start with the deviations of a few earlier steps."""
    dev, rng = _device(), _rng(seed, 10)
    pitch_um = LAM / c["ppl"] * 1e6
    h = _height(c, dev, 1.54, 0.7) * pitch_um
    bump = torch.from_numpy(rng.uniform(-0.3, 0.3, (c["ny"], c["nx"]))).to(dev)
    return torch.where(h > 0, (h + bump).clamp(0.0, LAM * 1e6 / 0.54), h).to(torch.float32).contiguous()


# --------------------------------------------------------------------------------- one pass
def _plan(c):
    from paper_2506_15411_gb300 import CBSPlan
    pads = (c["px"], c["py"], c["pz"])
    return CBSPlan(c["nx"], c["ny"], c["nz"], LAM / c["ppl"], LAM, 1.0, pads, pads, tol=0.0, max_iter=c["iters"],
                   check_every=c["check"], **(GENTLE if c["layers"] == "gentle" else {}))


def prepare(case, seed):
    from paper_2506_15411_gb300 import PlaneWave, PointSource, UserSource
    c, s = case, {"case": case, "r0": _focus(case), "source": PlaneWave()}
    op = c["op"]
    if op == "serve":
        from paper_2506_15411_gb300.serve import GridSpec, Server
        pads = (c["px"], c["py"], c["pz"])
        s["grid"] = GridSpec(c["nx"], c["ny"], c["nz"], LAM / c["ppl"], LAM, 1.0, pads, pads,
                             **(GENTLE if c["layers"] == "gentle" else {}))
        s["server"] = Server(max_active=8, tol=0.0, max_iter=c["iters"], check_every=c["check"])
        s["eps"] = [_eps(c, seed, k) for k in range(c["requests"])]
        return s
    s["plan"] = _plan(c)
    if op == "design":
        from paper_2506_15411_gb300.design import Design
        s["design"] = Design(s["plan"], **_design_params(c))
        s["h"] = _design_map(c, seed)
        return s
    eps = _eps(c, seed)
    if op == "host":
        s["eps"] = eps.cpu().numpy()
        return s
    if op == "forward":                 # one permittivity, solved for a source
        s["plan"].set_permittivity(eps)
        if c["source"] == "point":
            at, pol = _dipole(c, seed)
            s["source"] = PointSource(at, pol)
        elif c["source"] == "user":
            s["source"] = UserSource(_beam(c, seed))
    if op == "autograd":
        eps.requires_grad_(True)
        s["E_init"] = _earlier_field(c, seed)
    s["eps"] = eps
    return s


def run(state):
    op, r0 = state["case"]["op"], state["r0"]
    if op == "serve":
        srv = state["server"]
        for k, eps in enumerate(state["eps"]):
            srv.submit(state["grid"], eps, state["source"], r0, adjoint=k % 2 == 1, want_field=True,
                       want_grad=k % 2 == 1, tag=k)
        done = sorted(srv.wait(len(state["eps"])), key=lambda r: r.tag)
        return [(r.E, r.grad) if r.grad is not None else (r.E,) for r in done]
    plan, source = state["plan"], state["source"]
    if op == "forward":
        E, _ = plan.forward(source)
        return {"E": E}
    if op == "solve":
        plan.set_permittivity(state["eps"])
        E, _ = plan.forward(source)
        E_adj, _ = plan.adjoint(r0, E)
        grad, _ = plan.gradient(E, E_adj, r0)
        return {"E": E, "E_adj": E_adj, "grad": grad}
    if op == "autograd":
        from paper_2506_15411_gb300.autograd import focal_intensity
        loss = focal_intensity(state["eps"], plan, source, r0, E_init=state["E_init"])
        grad, = torch.autograd.grad(loss, state["eps"])
        return {"grad": grad, "E": plan.last_field}
    if op == "host":
        grad, _, _, _ = plan.design_step_host(state["eps"], source, r0)
        return {"grad": grad}
    d = state["design"]                 # a design loop's step; the map is stepped in place
    h, grad_h = state["h"].clone(), torch.empty_like(state["h"])
    d.reset()
    d.step(h, source, r0, grad_h=grad_h)
    return {"E": d.E, "E_adj": d.E_adj, "grad_h": grad_h}


def work(case):
    """Per voxel and iteration a pass reads V and reads and writes E (56 bytes), and the spectrum
    crosses memory once each way between the transforms along x and those along y and z (48 bytes);
    six complex transforms per iteration count 5 N log2 N flops.  A gradient reads both fields."""
    c = case
    n = c["nx"] * c["ny"] * c["nz"]
    solves = {"forward": 1, "serve": c["requests"] + c["requests"] // 2}.get(c["op"], 2)
    grads = {"forward": 0, "serve": c["requests"] // 2}.get(c["op"], 1)
    its = solves * c["iters"]
    return {"bytes": 104.0 * n * its + 52.0 * n * grads, "flops": n * its * (30.0 * math.log2(n) + 150.0)}


# --------------------------------------------------------------------------------- in 64 bits
def _sigma_axis(n, pad, ppl, round_trip, dev):
    """Quadratic absorption profile of an axis: a normally incident wave keeps the amplitude
    round_trip after crossing the layer and back."""
    i = torch.arange(n, device=dev, dtype=torch.float64)
    if pad == 0:
        return torch.zeros_like(i)
    depth = torch.clamp(torch.maximum(pad - i, i - (n - 1 - pad)), min=0.0)
    return 3.0 * math.log(1.0 / round_trip) / (2 * math.pi / ppl * pad) * (depth / pad) ** 2


class _Exact:
    """The series in complex128 on the permittivity of a case, lengths in voxels."""

    def __init__(self, c, eps):
        dev = eps.device
        self.c, self.kv2 = c, (2 * math.pi / c["ppl"]) ** 2
        rt = 1e-2 if c["layers"] == "gentle" else 1e-4
        sx, sy, sz = (_sigma_axis(c[a], c[p], c["ppl"], rt, dev)
                      for a, p in (("nx", "px"), ("ny", "py"), ("nz", "pz")))
        if c["layers"] == "gentle":
            sig = torch.maximum(torch.maximum(sz[:, None, None], sy[None, :, None]), sx[None, None, :])
        else:
            sig = sz[:, None, None] + sy[None, :, None] + sx[None, None, :]
        re = self.kv2 * eps.double()
        im = self.kv2 * sig
        k0 = 0.5 * (re.min().item() + re.max().item())
        shift = torch.sqrt(((re - k0) ** 2 + im ** 2).max()).item()
        self.V = torch.complex(re - k0, im - shift)
        self.shift, self.kt2 = shift, complex(k0, shift)
        self.p, self.q = [], []
        for n, view in ((c["nx"], (1, 1, -1)), (c["ny"], (1, -1, 1)), (c["nz"], (-1, 1, 1))):
            p = 2 * math.pi * torch.fft.fftfreq(n, device=dev, dtype=torch.float64)
            q = p.clone()
            if n % 2 == 0:
                q[n // 2] = 0.0
            self.p.append(p.view(view))
            self.q.append(q.view(view))

    def solve(self, add_source, E=None):
        """iters iterations from E (zero if None); add_source(component, field) adds S in place."""
        c = self.c
        if E is None:
            E = torch.zeros((3,) + tuple(self.V.shape), dtype=torch.complex128, device=self.V.device)
        p2 = sum(v * v for v in self.p)
        q2 = sum(v * v for v in self.q)
        a, b = 1.0 / (p2 - self.kt2), 1.0 / (p2 - q2 - self.kt2)
        for _ in range(c["iters"]):
            X = []
            for k in range(3):
                x = self.V * E[k]
                add_source(k, x)
                X.append(torch.fft.fftn(x))
            dot = (self.q[0] * X[0] + self.q[1] * X[1] + self.q[2] * X[2]) * b
            for k in range(3):
                w = torch.fft.ifftn((X[k] + self.q[k] * dot) * a)
                X[k] = None
                E[k] -= (1j / self.shift) * self.V * (E[k] - w)
        return E

    def sheet(self):
        amp = -2j * (2 * math.pi / self.c["ppl"])

        def add(k, x):
            if k == 0:
                x[self.c["pz"]] += amp
        return add

    def adjoint(self, E, r0):
        x0, y0, z0 = r0
        amp = torch.conj(E[:, z0, y0, x0]) * (LAM / self.c["ppl"]) ** 2

        def add(k, x):
            x[z0, y0, x0] += amp[k]
        return self.solve(add)

    def gradient(self, E, E_adj):
        g = torch.zeros(tuple(self.V.shape), dtype=torch.float64, device=self.V.device)
        for k in range(3):
            g += (E_adj[k] * E[k]).real
        return g * (2 * (2 * math.pi / LAM) ** 2)


def _gauss(a, s):
    """Separable Gaussian of std s pixels, cut at ceil(4 s), normalised, zero outside."""
    r = int(math.ceil(4 * s))
    w = torch.exp(-torch.arange(-r, r + 1, device=a.device, dtype=torch.float64) ** 2 / (2 * s * s))
    w = w / w.sum()
    for dim in (0, 1):
        b = torch.zeros_like(a)
        n = a.shape[dim]
        for k in range(-r, r + 1):
            lo, hi = max(0, k), min(n, n + k)
            if lo < hi:
                b.narrow(dim, lo - k, hi - lo).add_(a.narrow(dim, lo, hi - lo), alpha=w[k + r].item())
        a = b
    return a


def _mirror(a):
    return 0.25 * (a + a.flip(0) + a.flip(1) + a.flip(0, 1))


def exact(case, seed):
    c, op, r0 = case, case["op"], _focus(case)
    if not torch.cuda.is_available() and c["nx"] * c["ny"] * c["nz"] * c["iters"] > 4e7:
        return None                     # minutes on host cores
    if op == "serve":
        out = []
        for k in range(c["requests"]):
            X = _Exact(c, _eps(c, seed, k))
            E = X.solve(X.sheet())
            out.append((E, X.gradient(E, X.adjoint(E, r0))) if k % 2 == 1 else (E,))
        return out
    if op == "design":
        prm, pitch_um = _design_params(c), LAM / c["ppl"] * 1e6
        de = prm["n_lens"] ** 2 - 1.0
        heff = _gauss(_mirror(_design_map(c, seed).double()), prm["sigma_um"] / pitch_um)
        k = torch.arange(c["nz"], device=heff.device, dtype=torch.float64) - prm["z_base"]
        fill = torch.clamp(heff[None] / pitch_um - k[:, None, None], 0.0, 1.0)
        fill[: prm["z_base"]] = 0.0
        X = _Exact(c, 1.0 + de * fill)
        E = X.solve(X.sheet())
        E_adj = X.adjoint(E, r0)
        z = prm["z_base"] + torch.floor(heff / pitch_um).long()
        slope = torch.gather(X.gradient(E, E_adj), 0, z.clamp(max=c["nz"] - 1)[None])[0] * (de / pitch_um)
        slope = torch.where(z < c["nz"], slope, torch.zeros_like(slope))
        return {"E": E, "E_adj": E_adj, "grad_h": _mirror(_gauss(slope, prm["sigma_um"] / pitch_um))}
    X = _Exact(c, _eps(c, seed))
    if op == "forward" and c["source"] == "point":
        at, pol = _dipole(c, seed)
        scale = (LAM / c["ppl"]) ** 2

        def add(k, x):
            x[at[2], at[1], at[0]] += pol[k] * scale
        return {"E": X.solve(add)}
    if op == "forward" and c["source"] == "user":
        S = _beam(c, seed)

        def add(k, x):
            x += S[k].to(torch.complex128) * (LAM / c["ppl"]) ** 2
        return {"E": X.solve(add)}
    E = X.solve(X.sheet(), _earlier_field(c, seed).to(torch.complex128) if op == "autograd" else None)
    if op == "forward":
        return {"E": E}
    E_adj = X.adjoint(E, r0)
    grad = X.gradient(E, E_adj)
    if op == "solve":
        return {"E": E, "E_adj": E_adj, "grad": grad}
    return {"grad": grad, "E": E} if op == "autograd" else {"grad": grad}
