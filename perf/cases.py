"""The work that users of this library have it do, through its public entry points:

* time integration of one problem on the device (``State.step``): classic RK4 on grids from a few
  thousand to millions of cells, FP64 and FP32 fields, uniform materials, grains, and stacks of
  unequal layers with per-cell material maps; adaptive Dormand-Prince and Fehlberg steps;
* one effective field with energies and torque, as a log line or a static analysis asks for it;
* gradients of an RK4 rollout with respect to the saturation magnetisation (inverse design);
* served batches: many small relax requests loaded into slots, advanced together and read back.

``listed`` holds the sizes of the repository's own workloads, tests and benchmark; ``draw`` gives
other sizes of the same kinds, odd and prime ones among them.  ``exact`` restates every result in
plain FP64 torch: Newell's tensor (point dipoles beyond 20 cells), an FFT convolution, the local
terms, and the Runge-Kutta methods.
"""
import math

import numpy as np
import torch

from paper_2302_08843_gb300.autodiff import rk4_observable
from paper_2302_08843_gb300.binding import Batch, State
from paper_2302_08843_gb300.serving import auto_capacity

MU0 = 4.0e-7 * math.pi
GAMMA = 2.21e5
NEAR = 20           # cells within which Newell's formula is used
RTOL = 1e-5
LAYERS_NM = (1.0, 0.6, 2.4, 0.8, 1.5, 0.6, 3.0, 1.1)


def listed():
    def c(name, kind, material, precision, nx, ny, nz, **more):
        return dict(name=name, kind=kind, material=material, precision=precision, nx=nx, ny=ny, nz=nz, **more)

    return [
        # a small box in plain FP64: launches and latency are all there is
        c("rk4 fp64 32x32x4", "rk4", "plain", "fp64", 32, 32, 4, steps=10),
        # the headline problem: a polycrystal that fills the device
        c("rk4 fp32 256x256x64 grains", "rk4", "grains", "fp32", 256, 256, 64, steps=5),
        # the same construction where FP64 is wanted
        c("rk4 fp64 128x128x32 grains", "rk4", "grains", "fp64", 128, 128, 32, steps=1),
        # extents that are no power of two
        c("rk4 fp32 192x192x48 grains", "rk4", "grains", "fp32", 192, 192, 48, steps=5),
        # a stack of unequal layers, every material constant per cell
        c("rk4 fp32 256x256x8 layers", "rk4", "layers", "fp32", 256, 256, 8, steps=5),
        # a thin film in a switched field, adaptive steps from a cautious first one
        c("dp45 fp32 512x128x1 film", "adaptive", "film", "fp32", 512, 128, 1, method="dp45", steps=4),
        c("dp45 fp64 512x128x1 film", "adaptive", "film", "fp64", 512, 128, 1, method="dp45", steps=4),
        # one field with energies and torque, DMI, ragged extents
        c("field fp32 100x65x27 dmi", "field", "dmi", "fp32", 100, 65, 27),
        # the gradient of a driven film's signal with respect to its density
        c("gradient fp32 128x128x1", "gradient", "density", "fp32", 128, 128, 1, steps=10, every=5),
        # full batch states of served relax requests, small, large and thick grids
        c("served fp32 64x64x1 x32", "served", "requests", "fp32", 64, 64, 1, slots=32, attempts=4),
        c("served fp32 256x256x1 x32", "served", "requests", "fp32", 256, 256, 1, slots=32, attempts=4),
        c("served fp32 100x100x8 x16", "served", "requests", "fp32", 100, 100, 8, slots=16, attempts=4),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """Another case of the ranges above: extents over their logarithm, any integer among them."""
    kind = rng.choice(["rk4", "rk4", "adaptive", "field", "gradient", "served"])
    case = dict(kind=kind, material="plain", precision=rng.choice(["fp32", "fp32", "fp64"]))
    most = 1 << 20 if case["precision"] == "fp32" else 1 << 17
    while True:
        nx, ny = _log_int(rng, 16, 512), _log_int(rng, 16, 512)
        nz = 1 if rng.random() < 0.3 else _log_int(rng, 2, 64)
        if kind in ("gradient", "adaptive") and rng.random() < 0.7:
            nz = 1
        if kind == "served":
            nx, ny, nz = min(nx, 300), min(ny, 300), min(nz, 8)
        cells = nx * ny * nz
        if (1 << 10) <= cells <= (most if kind in ("rk4", "field") else most >> 3):
            break
    if kind == "rk4":
        case.update(material=rng.choice(["plain", "grains", "layers"]), steps=rng.choice([2, 3, 5]))
        if case["material"] == "layers":
            nz = 2 + nz % 9
            nx, ny = min(nx, 256), min(ny, 256)
        if case["precision"] == "fp64":
            case["steps"] = 1
    elif kind == "adaptive":
        case.update(material="film", method=rng.choice(["dp45", "dp45", "rkf45"]), steps=4)
    elif kind == "field":
        case.update(material=rng.choice(["dmi", "grains", "film"]))
    elif kind == "gradient":
        case.update(material="density", steps=rng.choice([4, 6, 10]), every=rng.choice([2, 5]))
    else:
        case.update(material="requests", precision="fp32", slots=auto_capacity((nx, ny, nz)) - rng.choice([0, 0, 1, 3]),
                    attempts=4)
    case.update(nx=nx, ny=ny, nz=nz)
    return case


# ------------------------------------------------------------------ inputs --
def _unit(v, axis=0):
    return v / v.norm(dim=axis, keepdim=True)


def _problem(case, seed):
    """Inputs of a case, FP64 tensors on the GPU: vectors (3, nz, ny, nx), maps (nz, ny, nx)."""
    g = torch.Generator("cuda").manual_seed(int(seed))
    shape = (case["nz"], case["ny"], case["nx"])
    real = torch.float64 if case["precision"] == "fp64" else torch.float32

    def normal(*size):
        return torch.randn(*size, generator=g, device="cuda", dtype=torch.float64)

    def uniform(*size):
        return torch.rand(*size, generator=g, device="cuda", dtype=torch.float64)

    def pulse(t):       # 5 mT sinc of 20 GHz around 50 ps, along y
        x = 2.0 * math.pi * 20e9 * (t - 50e-12)
        return (0.0, 0.005 / MU0 * (1.0 if x == 0.0 else math.sin(x) / x), 0.0)

    kind = case["material"]
    p = dict(dx=(2e-9, 2e-9, 2e-9), Ms=8e5, A=1.3e-11, alpha=0.5, Ku=0.0, axis=(1.0, 0.0, 0.0), h=(0.0, 0.0, 0.0))
    if kind == "plain":
        p.update(dx=(2.5e-9, 2.5e-9, 3e-9), h=(0.010 / MU0, 0.0, 0.0), dt=1e-13)
    elif kind == "grains":      # 64 grains, each cell in that of the nearest seed, with random easy axes
        p.update(Ms=1e6, A=1.5e-11, alpha=0.1, Ku=4e5, dt=5e-14, table=_unit(normal(64, 3), 1))
        seeds = uniform(64, 3) * torch.tensor(shape[::-1], device="cuda", dtype=torch.float64)
        best = torch.full(shape, math.inf, device="cuda", dtype=torch.float64)
        ids = torch.zeros(shape, device="cuda", dtype=torch.uint8)
        at = [torch.arange(n, device="cuda", dtype=torch.float64) + 0.5 for n in shape]
        for k in range(64):
            d = ((at[0] - seeds[k, 2]) ** 2)[:, None, None] + ((at[1] - seeds[k, 1]) ** 2)[:, None] + (at[2] - seeds[k, 0]) ** 2
            ids = torch.where(d < best, k, ids).to(torch.uint8)
            best = torch.minimum(best, d)
        p["grain"] = ids
    elif kind == "layers":
        h = [LAYERS_NM[k % len(LAYERS_NM)] * 1e-9 for k in range(case["nz"])]
        per = [(1.1e6, 1.6e-11, 3e5) if v >= 1.5e-9 else (4e5, 0.4e-11, 0.0) if v <= 0.6e-9 else (8e5, 1.3e-11, 0.0) for v in h]
        maps = [torch.tensor([v[q] for v in per], device="cuda", dtype=torch.float64)[:, None, None].expand(shape).contiguous()
                for q in range(3)]
        p.update(dx=(2e-9, 2e-9, sum(h) / len(h)), layers=h, Ms=maps[0], A=maps[1], Ku=maps[2], alpha=0.1,
                 axis=(0.0, 0.0, 1.0), h=(0.020 / MU0, 0.0, 0.0), dt=2e-14)
    elif kind == "film":
        a = math.radians(170.0)
        p.update(dx=(3.90625e-9, 3.90625e-9, 3e-9), alpha=0.02, Ku=5e3, dt=2e-16,
                 h=(0.025 / MU0 * math.cos(a), 0.025 / MU0 * math.sin(a), 0.0))
        p["m0"] = _unit(1.0 / math.sqrt(3.0) + 0.01 * normal(3, *shape))
    elif kind == "dmi":
        p.update(Ms=5.8e5, A=1.5e-11, alpha=0.3, Ku=8e5, axis=(0.0, 0.0, 1.0), D=3e-3, h=(0.0, 0.0, 0.05 / MU0))
    elif kind == "density":     # Ms = sigmoid(w) Ms0, driven in a strip, the signal taken in a small window
        w = 0.1 * normal(*shape)
        weight = torch.zeros(shape, device="cuda", dtype=torch.float64)
        weight[:, :, :10] = 1.0
        probe = torch.zeros((3,) + shape, device="cuda", dtype=torch.float64)
        probe[1, :, shape[1] // 2 - 5: shape[1] // 2 + 5, -20:-10] = 1.0 / (100.0 * shape[0])
        m0 = torch.zeros((3,) + shape, device="cuda", dtype=torch.float64)
        m0[0] = 1.0
        p.update(dx=(5e-9, 5e-9, 5e-9), w=w, Ms=8e5 * torch.sigmoid(w), weight=weight, probe=probe.to(real), m0=m0,
                 h=pulse, alpha=0.05, dt=5e-14)
    else:                       # requests: each slot its own Ms, A and state, cautious first steps
        n = case["slots"]
        p.update(dx=(3e-9, 3e-9, 3e-9), Ms=6e5 + 6e5 * uniform(n), A=1e-11 + 1e-11 * uniform(n), alpha=1.0, dt=1e-16)
        p["m0"] = _unit(normal(n, 3, *shape), 1)
    if "m0" not in p:
        p["m0"] = _unit(normal(3, *shape))
    p["m0"] = p["m0"].to(real).contiguous()
    return p


def prepare(case, seed):
    p = _problem(case, seed)
    n = (case["nx"], case["ny"], case["nz"])
    if case["kind"] == "served":
        b = Batch(n, p["dx"], case["precision"], case["slots"], NEAR)
        # requests arrive in host memory
        return dict(case=case, batch=b, m0=p["m0"].cpu().numpy(), Ms=p["Ms"].tolist(), A=p["A"].tolist(), p=p)
    s = State(n, p["dx"], case["precision"])
    maps = isinstance(p["Ms"], torch.Tensor)
    more = {}
    if "grain" in p:
        more = dict(grain_id=p["grain"], axis_table=p["table"])
    if "layers" in p:
        more = dict(Ms_cell=p["Ms"], A_cell=p["A"], Ku1_cell=p["Ku"])
    s.set_material(Ms=0.0 if maps else p["Ms"], A=0.0 if "layers" in p else p["A"], alpha=p["alpha"],
                   Ku1=0.0 if "layers" in p else p["Ku"], ku_axis=p["axis"], **(more or (dict(Ms_cell=p["Ms"]) if maps else {})))
    weight = p.get("weight")
    if callable(p["h"]):
        s.set_zeeman(fn=p["h"], weight=weight)
    else:
        s.set_zeeman(h=p["h"], weight=weight)
    if "D" in p:
        s.set_dmi("interface", p["D"])
    if "layers" in p:
        s.set_layers(p["layers"])
    s.demag_setup(NEAR)
    s.set_m(p["m0"])
    if case["kind"] == "gradient":
        p["leaf"] = p["w"].to(p["m0"].dtype).clone().requires_grad_(True)
    torch.cuda.synchronize()
    return dict(case=case, s=s, p=p)


def run(state):
    case, p = state["case"], state["p"]
    kind = case["kind"]
    if kind == "rk4":           # a stretch of fixed steps from a given state
        s, t = state["s"], 0.0
        s.set_m(p["m0"])
        for _ in range(case["steps"]):
            t, _ = s.step(p["dt"], t, "rk4")
        return s.get_m()
    if kind == "adaptive":      # the first steps of an adaptive run, the step size fed back
        s, t, dt = state["s"], 0.0, p["dt"]
        s.set_m(p["m0"])
        for _ in range(case["steps"]):
            t, dt = s.step(dt, t, case["method"], RTOL)
        return s.get_m(), t, dt
    if kind == "field":
        return state["s"].heff(p["m0"], t=0.0, energies=True, torque=True)
    if kind == "gradient":      # signal of a rollout and its gradient with respect to the design
        leaf = p["leaf"]
        leaf.grad = None
        signal = rk4_observable(8e5 * torch.sigmoid(leaf), state["s"], p["m0"], p["probe"], p["dt"], case["steps"],
                                case["every"], dict(A=p["A"], alpha=p["alpha"], ku_axis=p["axis"]))
        signal.mean().backward()
        return signal.detach().to(leaf.dtype), leaf.grad     # in the precision the fields have
    b = state["batch"]          # a server's cycle: load the slots, advance, collect
    for k in range(case["slots"]):
        b.set_slot(k, state["Ms"][k], state["A"][k], p["alpha"], state["m0"][k], p["dt"])
    b.begin(case["attempts"], RTOL, 1e-3, 20000)
    status, steps, torque = b.end()
    m = [b.get_m(k) for k in range(case["slots"])]
    for k in range(case["slots"]):
        b.clear_slot(k)
    # the torque of FP32 fields, in the precision it has
    return status, steps, torque.astype(m[0].dtype), np.stack(m)


# -------------------------------------------------------------------- work --
def _evaluations(case):
    """Field evaluations of one pass."""
    kind = case["kind"]
    if kind == "rk4":
        return 4 * case["steps"]
    if kind == "adaptive":
        return 1 + 6 * case["steps"] if case["method"] == "dp45" else 6 * case["steps"]
    if kind == "gradient":      # forward, and per step of the reverse sweep the stages and their transposes
        return (4 + 8) * case["steps"]
    if kind == "served":
        return case["slots"] * (1 + 6 * case["attempts"])
    return 1


def work(case):
    n = [case["nx"], case["ny"], case["nz"]]
    size = 8 if case["precision"] == "fp64" else 4
    cells = n[0] * n[1] * n[2]
    pad = [1 if v == 1 else 2 * v for v in n]
    lg = [math.log2(v) if v > 1 else 0.0 for v in pad]
    kx = pad[0] // 2 + 1
    # transforms that skip the padding, half of them along x for real rows, and 30 operations per wave number
    flops = 6 * n[1] * n[2] * 2.5 * pad[0] * lg[0] + 6 * n[2] * kx * 5 * pad[1] * lg[1]
    flops += kx * pad[1] * (30 * pad[2] + 30 * pad[2] * lg[2]) + 150 * cells
    spectrum = 6 * size * kx * (pad[1] // 2 + 1) * (pad[2] // 2 + 1)
    if case["material"] == "layers":
        flops += kx * pad[1] * 36 * n[2] * n[2] - kx * pad[1] * (30 * pad[2] + 30 * pad[2] * lg[2])
        spectrum = 6 * size * kx * (pad[1] // 2 + 1) * (n[2] * (n[2] + 1) // 2)
    e = _evaluations(case)
    # per evaluation: the state in, the tensor's spectrum once, the result out (a batch shares the spectrum)
    share = case.get("slots", 1)
    return {"bytes": float(e * (6 * cells * size + spectrum / share)), "flops": float(e * flops)}


# ------------------------------------------------------------------- exact --
def _f(x, y, z):
    x, y, z = x.abs(), y.abs(), z.abs()
    r = torch.sqrt(x * x + y * y + z * z)

    def ash(a, b, c):
        d = torch.sqrt(b * b + c * c)
        return torch.where(d > 0, torch.asinh(a / d.clamp_min(1e-300)), torch.zeros_like(d))

    v = (2 * x * x - y * y - z * z) * r / 6
    v = v + 0.5 * y * (z * z - x * x) * ash(y, x, z) + 0.5 * z * (y * y - x * x) * ash(z, x, y)
    return v - x * y * z * torch.atan2(y * z, x * r)


def _g(x, y, z):
    s = torch.sign(x) * torch.sign(y)
    x, y, z = x.abs(), y.abs(), z.abs()
    r = torch.sqrt(x * x + y * y + z * z)

    def ash(a, b, c):
        d = torch.sqrt(b * b + c * c)
        return torch.where(d > 0, torch.asinh(a / d.clamp_min(1e-300)), torch.zeros_like(d))

    v = x * y * z * ash(z, x, y) + y / 6 * (3 * z * z - y * y) * ash(x, y, z) + x / 6 * (3 * z * z - x * x) * ash(y, x, z)
    v = v - z ** 3 / 6 * torch.atan2(x * y, z * r) - z * y * y / 2 * torch.atan2(x * z, y * r)
    return s * (v - z * x * x / 2 * torch.atan2(y * z, x * r) - x * y * r / 3)


_COMPONENTS = ((_f, (0, 1, 2)), (_g, (0, 1, 2)), (_g, (0, 2, 1)), (_f, (1, 0, 2)), (_g, (1, 2, 0)), (_f, (2, 1, 0)))
_AXES = ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))


def _pairs(nx, ny, dx, dy, z0, hi, hj, gap):
    """Tensor (6, K, Py, Px) between boxes of heights hi (target) and hj whose lower faces are z0
    apart, `gap` layers apart, at every lateral offset, negative ones wrapped."""
    px, py, dev = (1 if nx == 1 else 2 * nx), (1 if ny == 1 else 2 * ny), z0.device
    i = torch.fft.fftfreq(px, 1.0 / px, device=dev, dtype=torch.float64)
    j = torch.fft.fftfreq(py, 1.0 / py, device=dev, dtype=torch.float64)
    x, y = (i * dx)[None, None, :], (j * dy)[None, :, None]
    z = (z0 + 0.5 * (hi - hj))[:, None, None]       # between the centres
    r = torch.sqrt(x * x + y * y + z * z)
    far = torch.maximum(torch.maximum(i.abs()[None, None, :], j.abs()[None, :, None]), gap.abs()[:, None, None]) > NEAR
    safe = torch.where(far, r, torch.ones_like(r))
    d = (x, y, z)
    vol = (dx * dy * hj / (4 * math.pi))[:, None, None]
    out = torch.stack([torch.where(far, vol * ((1.0 if a == b else 0.0) / safe ** 3 - 3 * d[a] * d[b] / safe ** 5), 0.0)
                       for a, b in _AXES])
    # the lateral second difference of the four corner terms where the boxes are near
    ni, nj = i[i.abs() <= NEAR], j[j.abs() <= NEAR]
    ks = torch.nonzero(gap.abs() <= NEAR)[:, 0]
    at = torch.arange(-1, 2, device=dev, dtype=torch.float64)
    gx = ((ni[:, None] + at) * dx)[None, None, :, None, :]
    gy = ((nj[:, None] + at) * dy)[None, :, None, :, None]
    wgt = torch.tensor([-1.0, 2.0, -1.0], device=dev, dtype=torch.float64)
    near = torch.zeros(6, len(ks), len(nj), len(ni), device=dev, dtype=torch.float64)
    for sign, zz in ((1, z0), (-1, z0 + hi), (-1, z0 - hj), (1, z0 + hi - hj)):
        gz = zz[ks][:, None, None, None, None]
        for c, (fn, order) in enumerate(_COMPONENTS):
            v = fn(*[(gx, gy, gz)[q] for q in order])
            near[c] += sign * torch.einsum("kjiba,b,a->kji", v, wgt, wgt)
    near /= (4 * math.pi * dx * dy * hi[ks])[None, :, None, None]
    jx, ix = torch.nonzero(j.abs() <= NEAR)[:, 0], torch.nonzero(i.abs() <= NEAR)[:, 0]
    block = out[:, ks][:, :, jx][:, :, :, ix]
    keep = far[ks][:, jx][:, :, ix]
    full = out.clone()
    full[:, ks[:, None, None], jx[None, :, None], ix[None, None, :]] = torch.where(keep, block, near)
    # the wrapped offset n itself is no offset between two cells
    if nx > 1:
        full[..., nx] = 0
    if ny > 1:
        full[:, :, ny] = 0
    return full


class _Exact:
    """The field and the right-hand side in plain FP64 for states (..., 3, nz, ny, nx)."""

    def __init__(self, case, p):
        self.n = n = (case["nz"], case["ny"], case["nx"])
        self.p, nm = p, 1e-9
        self.pad = [1 if v == 1 else 2 * v for v in n]
        self.dx = [v / nm for v in p["dx"]]
        dev = p["m0"].device

        def t(v):
            return torch.tensor(v, device=dev, dtype=torch.float64)

        if "layers" in p:
            self.h = t(p["layers"]) / nm
            low = torch.cumsum(self.h, 0) - self.h
            a, b = [v.reshape(-1) for v in torch.meshgrid(torch.arange(n[0], device=dev), torch.arange(n[0], device=dev), indexing="ij")]
            ten = _pairs(n[2], n[1], self.dx[0], self.dx[1], low[a] - low[b], self.h[a], self.h[b], (a - b).double())
            self.K = torch.fft.rfft2(ten).reshape(6, n[0], n[0], self.pad[1], -1)
        else:
            self.h = None
            k = torch.fft.fftfreq(self.pad[0], 1.0 / self.pad[0], device=dev, dtype=torch.float64)
            hz = torch.full_like(k, self.dx[2])
            ten = _pairs(n[2], n[1], self.dx[0], self.dx[1], k * self.dx[2], hz, hz, k)
            if n[0] > 1:
                ten[:, n[0]] = 0
            self.K = torch.fft.rfftn(ten, dim=(1, 2, 3))

    def demag(self, M):
        index = ((0, 1, 2), (1, 3, 4), (2, 4, 5))
        z, y, x = self.n
        if self.h is not None:
            F = torch.fft.rfft2(M, s=self.pad[1:])
            H = torch.stack([sum(torch.einsum("ijyx,...jyx->...iyx", self.K[index[a][b]], F[..., b, :, :, :]) for b in range(3))
                             for a in range(3)], dim=-4)
            return -torch.fft.irfft2(H, s=self.pad[1:])[..., :y, :x]
        F = torch.fft.rfftn(M, s=self.pad, dim=(-3, -2, -1))
        H = torch.stack([sum(self.K[index[a][b]] * F[..., b, :, :, :] for b in range(3)) for a in range(3)], dim=-4)
        return -torch.fft.irfftn(H, s=self.pad, dim=(-3, -2, -1))[..., :z, :y, :x]

    @staticmethod
    def _cells(v):
        """A per-request value or a per-cell map, against states (..., 3, nz, ny, nx)."""
        if not isinstance(v, torch.Tensor):
            return v
        return v[:, None, None, None, None] if v.dim() == 1 else v

    def terms(self, m, t, Ms=None):
        p, nm = self.p, 1e-9
        Ms = self._cells(p["Ms"] if Ms is None else Ms)
        A, Ku = self._cells(p["A"]), p["Ku"]
        demag = self.demag(Ms * m)
        ex, dmi = torch.zeros_like(m), torch.zeros_like(m)
        e = ((0.0, 1.0, 0.0), (-1.0, 0.0, 0.0), (0.0, 0.0, 0.0))
        for axis in range(3):           # x, y, z
            dim, n = -1 - axis, self.n[2 - axis]
            if n == 1:
                continue
            lo, hi = m.narrow(dim, 0, n - 1), m.narrow(dim, 1, n - 1)
            link, d2 = A, (self.dx[axis] * nm) ** 2
            per_cell = isinstance(A, torch.Tensor) and A.dim() == 3
            if per_cell:
                a, b = A.narrow(dim, 0, n - 1), A.narrow(dim, 1, n - 1)
                if axis == 2 and self.h is not None:
                    h = self.h * nm
                    ha, hb = h[:-1, None, None], h[1:, None, None]
                    link = (ha + hb) * a * b / (ha * b + hb * a)
                else:
                    link = 2 * a * b / (a + b)
            flow = link * (hi - lo)
            pad = [0, 0] * axis
            up, down = torch.nn.functional.pad(flow, pad + [0, 1]), torch.nn.functional.pad(flow, pad + [1, 0])
            if axis == 2 and self.h is not None:
                h = self.h * nm
                mid = 0.5 * (h[:-1] + h[1:])
                zero = mid.new_zeros(1)
                ex = ex + up * torch.cat([1 / (h[:-1] * mid), zero])[:, None, None]
                ex = ex - down * torch.cat([zero, 1 / (h[1:] * mid)])[:, None, None]
            else:
                ex = ex + (up - down) / d2
            if "D" in p:
                pull = torch.nn.functional.pad(hi, pad + [0, 1]) - torch.nn.functional.pad(lo, pad + [1, 0])
                v = torch.tensor(e[axis], device=m.device, dtype=m.dtype)[:, None, None, None].expand_as(m)
                dmi = dmi + p["D"] * torch.linalg.cross(v, pull, dim=-4) / (2 * self.dx[axis] * nm)
        ex, dmi = 2 / (MU0 * Ms) * ex, 2 / (MU0 * Ms) * dmi
        if "grain" in p:
            axis = p["table"][p["grain"].long()].permute(3, 0, 1, 2)
        else:
            axis = torch.tensor(p["axis"], device=m.device, dtype=m.dtype)[:, None, None, None]
        ani = 2 * Ku / (MU0 * Ms) * (m * axis).sum(-4, keepdim=True) * axis
        h = p["h"](t) if callable(p["h"]) else p["h"]
        zee = torch.tensor(h, device=m.device, dtype=m.dtype)[:, None, None, None] * p.get("weight", 1.0)
        return demag, ex, ani, zee + torch.zeros_like(m), dmi

    def rhs(self, m, t, Ms=None, field=False):
        h = sum(self.terms(m, t, Ms))
        c = torch.linalg.cross(m, h, dim=-4)
        a = self.p["alpha"]
        k = -GAMMA / (1 + a * a) * (c + a * torch.linalg.cross(m, c, dim=-4))
        return (k, c) if field else k

    def rk4(self, m, t, dt, Ms=None):
        k1 = self.rhs(m, t, Ms)
        k2 = self.rhs(m + 0.5 * dt * k1, t + 0.5 * dt, Ms)
        k3 = self.rhs(m + 0.5 * dt * k2, t + 0.5 * dt, Ms)
        k4 = self.rhs(m + dt * k3, t + dt, Ms)
        return _unit(m + dt / 6 * (k1 + 2 * k2 + 2 * k3 + k4), -4)

    def adaptive(self, m, t, dt, method):
        """One accepted step: the new state, the next step size and the torque at the last stage.
        The cases start with steps so small that each one is accepted and grows by the largest factor."""
        rows, high, low = _DP45 if method == "dp45" else _RKF45
        k, y, c = [], m, None
        for row in rows:
            y = m + dt * sum(a * v for a, v in zip(row, k)) if row else m
            v, c = self.rhs(y, t + dt * sum(row), field=True)
            k.append(v)
        new = m + dt * sum(a * v for a, v in zip(high, k))
        err = dt * sum((a - b) * v for a, b, v in zip(high, low, k))
        err = float((err.abs() / (RTOL + RTOL * torch.maximum(m.abs(), new.abs()))).max())
        factor = 5.0 if err == 0 else min(5.0, max(0.2, 0.9 * err ** -0.2))
        Ms = self._cells(self.p["Ms"])
        torque = (c.norm(dim=-4, keepdim=True) / Ms).amax((-4, -3, -2, -1))
        assert err <= 1
        return _unit(new, -4), dt * factor, torque


_DP45 = ([[], [1 / 5], [3 / 40, 9 / 40], [44 / 45, -56 / 15, 32 / 9],
          [19372 / 6561, -25360 / 2187, 64448 / 6561, -212 / 729],
          [9017 / 3168, -355 / 33, 46732 / 5247, 49 / 176, -5103 / 18656],
          [35 / 384, 0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84]],
         [35 / 384, 0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84, 0],
         [5179 / 57600, 0, 7571 / 16695, 393 / 640, -92097 / 339200, 187 / 2100, 1 / 40])
_RKF45 = ([[], [1 / 4], [3 / 32, 9 / 32], [1932 / 2197, -7200 / 2197, 7296 / 2197],
           [439 / 216, -8, 3680 / 513, -845 / 4104], [-8 / 27, 2, -3544 / 2565, 1859 / 4104, -11 / 40]],
          [25 / 216, 0, 1408 / 2565, 2197 / 4104, -1 / 5, 0],
          [16 / 135, 0, 6656 / 12825, 28561 / 56430, -9 / 50, 2 / 55])


def exact(case, seed):
    p = _problem(case, seed)
    x = _Exact(case, p)
    m, t, kind = p["m0"].double(), 0.0, case["kind"]
    if kind == "rk4":
        for _ in range(case["steps"]):
            m, t = x.rk4(m, t, p["dt"]), t + p["dt"]
        return m
    if kind == "adaptive":
        dt = p["dt"]
        for _ in range(case["steps"]):
            m, new, _ = x.adaptive(m, t, dt, case["method"])
            t, dt = t + dt, new
        return m, t, dt
    if kind == "field":
        terms = x.terms(m, 0.0)
        h = sum(terms)
        f = -0.5 * MU0 * p["dx"][0] * p["dx"][1] * p["dx"][2] * p["Ms"]
        energies = [float(f * (2 if k == 3 else 1) * (m * v).sum()) for k, v in enumerate(terms)]
        return h, energies, float(torch.linalg.cross(m, h, dim=-4).norm(dim=-4).max() / p["Ms"])
    if kind == "gradient":
        w = p["w"].to(p["m0"].dtype).double().requires_grad_(True)
        Ms, signal = 8e5 * torch.sigmoid(w), []
        for _ in range(case["steps"]):
            m, t = x.rk4(m, t, p["dt"], Ms), t + p["dt"]
            signal.append((p["probe"].double() * m).sum())
        signal = torch.stack(signal)
        signal.mean().backward()
        return signal.detach(), w.grad
    dt, torque = p["dt"], None
    out, last = [], []
    for k in range(case["slots"]):      # slot by slot: a batch's states fit the card, its spectra need not
        q = dict(p, Ms=float(p["Ms"][k]), A=float(p["A"][k]))
        x.p, mk, dt = q, m[k], p["dt"]
        for _ in range(case["attempts"]):
            mk, dt, torque = x.adaptive(mk, 0.0, dt, "dp45")
        out.append(mk)
        last.append(torque.reshape(()))
    return None, None, torch.stack(last), torch.stack(out)
