"""Timed cases of the probed-gradient library, through its public entry points.

Each case is one call that a program makes on a batch of shots: modelling, a
gradient (probed, full storage, replayed from graphs, through autograd), an
image, range-finding probes.  Sizes are those of the repository's workloads
and of its serving mix, with ragged neighbours; the time axes of the 3-D cases
are cut so that a pass takes a fraction of a second.

    listed()              the cases
    draw(rng)             one more case of the same ranges
    prepare(case, seed)   model, wavelet, records, problem (and captured graph) on the GPU
    run(state)            one pass, its outputs
    work(case)            bytes and operations the path cannot do without
    exact(case, seed)     the outputs in 64 bits, by plain torch and numpy

The equations of ``exact`` are those of include/tprobe.h: leapfrog in time,
centred order-4 or order-8 Laplacian, zero values outside the grid, u[0] =
u[1] = 0, the adjoint the exact transpose, dJ/dm of the least-squares misfit.
"""
import math

import numpy as np
import torch

from paper_2104_00794_gb300 import api
from paper_2104_00794_gb300.autograd import modeling

# Courant numbers v dt / h at which the scheme stops being stable, per (ndim, order)
CFL = {(2, 4): 0.6124, (2, 8): 0.5546, (3, 4): 0.5000, (3, 8): 0.4529}
W2 = {4: (-5 / 2, 4 / 3, -1 / 12), 8: (-205 / 72, 8 / 5, -1 / 5, 8 / 315, -1 / 560)}
W1 = {4: (2 / 3, -1 / 12), 8: (4 / 5, -1 / 5, 4 / 105, -1 / 280)}


def _case(name, kind, nx, nz, nt, *, ny=1, shots=1, order=8, h=10.0, dt=1e-3, f0=8.0, r=0, probe="rademacher", T=128,
          acc="f32", sponge=0):
    c = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "nt": nt, "shots": shots, "order": order, "h": h, "dt": dt,
         "f0": f0, "r": r, "probe": probe, "T": T, "acc": acc, "sponge": sponge}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one shot on a small grid, as a line search evaluates its misfit
        _case("forward_2d_small", "forward", 101, 101, 500, order=4, f0=10.0),
        # the smallest gradient: the same shot with four probes
        _case("gradient_2d_small", "probed", 101, 101, 500, order=4, f0=10.0, r=4),
        # an inversion's iteration in 2-D: all its shots in one batch, sixteen Gaussian probes
        _case("gradient_2d_shots", "probed", 601, 201, 3000, shots=16, h=12.5, r=16, probe="gaussian"),
        # differentiable modelling: the forward pass and the backward pass of a larger 2-D batch
        _case("autograd_2d", "autograd", 801, 301, 2500, shots=8, r=16, probe="gaussian"),
        # migration: one shot of a large 2-D section, the probed fields' gradient image
        _case("image_2d_large", "image", 1001, 401, 1000, r=16, T=64),
        # the conventional gradient in 2-D, which keeps the whole history, on a ragged section
        _case("full_2d", "full", 397, 401, 1000, shots=4),
        # a gradient with an absorbing layer around the section (field-like boundaries)
        _case("sponge_2d", "probed", 601, 201, 1500, shots=4, h=12.5, r=8, T=32, sponge=20),
        # modelling in 3-D on a ragged grid at order 4: two shots' records
        _case("forward_3d_ragged", "forward", 131, 107, 400, ny=119, shots=2, order=4, dt=8e-4, f0=10.0),
        # a served 3-D request: one captured gradient, replayed, with a single accumulator set
        _case("graphed_3d_small", "graphed", 128, 128, 1000, ny=128, dt=8e-4, f0=10.0, r=16, T=64, acc="f32_fold"),
        # the flagship 3-D gradient (shorter time axis), a receiver at every surface node
        _case("gradient_3d", "probed", 256, 256, 500, ny=256, dt=8e-4, f0=10.0, r=32, T=32),
        # the conventional gradient in 3-D
        _case("full_3d", "full", 192, 144, 400, ny=160, dt=8e-4, f0=10.0),
        # range-finding probes from a batch of observed records, once per model update
        _case("qr_2d", "qr", 801, 301, 2500, shots=8, r=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forward", "probed", "probed", "autograd", "image", "full", "graphed", "qr"])
    three = kind != "qr" and rng.random() < 0.4
    order = rng.choice([4, 8, 8])
    r = 0 if kind in ("forward", "full") else rng.choice([4, 8, 16, 16, 32]) if not three else rng.choice([8, 16, 32])
    T = rng.choice([32, 64, 128])
    probe = rng.choice(["rademacher", "gaussian"])
    acc = rng.choice(["f32", "f32", "f32_fold"]) if kind in ("probed", "graphed") else "f32"
    sponge = rng.choice([0, 0, 0, rng.randint(8, 24)]) if kind in ("forward", "probed", "full") else 0
    if three:
        nx, ny, nz = (_log(rng, 48, 256) for _ in range(3))
        n, shots = nx * ny * nz, rng.choice([1, 1, 1, 2])
        most = 3e9 if kind == "full" else 6e9 if kind != "forward" else 8e9  # history in memory; time of a pass
        nt = min(_log(rng, 100, 1000), max(60, int(most / (n * shots))))
        return _case(None, kind, nx, nz, nt, ny=ny, shots=shots, order=order, dt=8e-4, f0=10.0, r=r, probe=probe, T=T,
                     acc=acc, sponge=sponge)
    nx, nz, shots = _log(rng, 64, 1001), _log(rng, 64, 401), _log(rng, 1, 16)
    most = 1.2e9 if kind == "full" else 2.5e9
    nt = min(_log(rng, 200, 3000), max(150, int(most / (nx * nz * shots))))
    if kind == "qr":
        nt = max(nt, 300)
    return _case(None, kind, nx, nz, nt, shots=shots, order=order, h=rng.choice([10.0, 12.5]), r=r, probe=probe, T=T,
                 acc=acc, sponge=sponge)


# ------------------------------------------------------------------ inputs
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _shape(c):
    return (c["nz"], c["ny"], c["nx"]) if c["ny"] > 1 else (c["nz"], c["nx"])


def _smooth(x, sigma):
    """Separable Gaussian filter over every axis, by reflection at the faces."""
    m = int(3 * sigma)
    k = torch.exp(-0.5 * (torch.arange(-m, m + 1, device=x.device, dtype=x.dtype) / sigma) ** 2)
    k = k / k.sum()
    for ax in range(x.dim()):
        y = x.movedim(ax, -1)
        flat = y.reshape(-1, 1, y.shape[-1])
        w = min(m, y.shape[-1] - 1)
        out = torch.nn.functional.conv1d(torch.nn.functional.pad(flat, (w, w), mode="reflect"), k[m - w:m + w + 1][None, None])
        x = out.reshape(y.shape).movedim(-1, ax)
    return x


def _ricker(tau, f0):
    a = (math.pi * f0 * tau) ** 2
    return (1.0 - 2.0 * a) * torch.exp(-a)


def _inputs(c, seed):
    """Velocity, wavelet, records, geometry and the velocity bound, from the seed alone."""
    dev = _device()
    g = torch.Generator(device="cpu").manual_seed(seed)
    shape, order = _shape(c), c["order"]
    bound = 0.9 * CFL[len(shape), order] * c["h"] / c["dt"]
    coarse = tuple(min(n, -(-n // 4) + 2) for n in shape)  # perturbations a few cells wide
    field = _smooth(torch.randn(coarse, generator=g, dtype=torch.float32).to(dev), 1.5)
    field = torch.nn.functional.interpolate(field[None, None], size=shape, mode="trilinear" if len(shape) == 3 else "bilinear")[0, 0]
    field = field / field.abs().max()
    z = torch.linspace(0, 1, shape[0], device=dev).reshape(-1, *[1] * (len(shape) - 1))
    if len(shape) == 3:
        z = torch.floor(z * 7.999) / 7.0  # eight layers
    top = min(4000.0, 0.95 * bound)
    vel = ((1500.0 + (top - 1500.0) * z) * (1.0 + 0.05 * field)).clamp(max=bound).contiguous()
    nx, ny, nt, shots = c["nx"], c["ny"], c["nt"], c["shots"]
    # sources two cells deep along the middle line (jittered), a receiver at every surface node
    xs = torch.linspace(0, nx - 1, shots + 2)[1:-1].round().to(torch.int64)
    xs = (xs + torch.randint(-3, 4, (shots,), generator=g)).clamp(0, nx - 1)
    src = ((2 * ny + ny // 2) * nx + xs)[:, None]
    rec = torch.arange(nx * ny, dtype=torch.int64)[None].expand(shots, -1).contiguous()
    t = torch.arange(nt, device=dev, dtype=torch.float32) * c["dt"]
    f = c["f0"] * (0.95 + 0.1 * torch.rand(1, generator=g).item())
    wavelet = _ricker(t - 1.0 / f, f)[None, :, None].expand(shots, -1, 1).contiguous()
    # records: a few arrivals with hyperbolic moveout from each source
    cols = torch.arange(nx * ny, device=dev)
    rx, ry = (cols % nx).float(), (cols // nx).float()
    d = torch.zeros((shots, nt, nx * ny), device=dev)
    amp = 0.02 if len(shape) == 3 else 0.5
    for s in range(shots):
        off = torch.hypot(rx - float(xs[s]), ry - float(ny // 2)) * c["h"]
        for e in range(3):
            t0, v, a = (torch.rand(3, generator=g) * torch.tensor([0.8, 1500.0, 1.0]) + torch.tensor([0.05, 1600.0, 0.2])).tolist()
            t0 *= nt * c["dt"]
            tau = t[:, None] - (torch.sqrt(t0 * t0 + (off / v) ** 2) + 1.0 / f)[None]
            d[s] += (amp * a / (1.0 + e)) * _ricker(tau, f)
    noise = torch.Generator(device=dev).manual_seed(seed)
    d += 0.01 * amp * torch.randn(d.shape, generator=noise, device=dev)  # the sensors' own noise
    eta = 3.0 * bound * math.log(1e3) / (2.0 * c["sponge"] * c["h"]) if c["sponge"] else 0.0
    return {"vel": vel, "wavelet": wavelet, "d": d, "src": src, "rec": rec, "vmax": bound, "eta": eta,
            "probe_seed": 2104 + seed}


def prepare(case, seed):
    i = _inputs(case, seed)
    p = api.Problem(3 if case["ny"] > 1 else 2, case["nx"], case["ny"], case["nz"], case["h"], case["dt"], case["nt"],
                    case["order"], i["src"], i["rec"], vmax=i["vmax"], sponge=case["sponge"], sponge_eta=i["eta"])
    s = {"case": case, "problem": p, "vel": i["vel"], "wavelet": i["wavelet"], "d": i["d"], "seed": i["probe_seed"]}
    if case["r"]:
        s["probe"] = api.ProbeSpec(kind=case["probe"], r=case["r"], T=case["T"], seed=i["probe_seed"], acc=case["acc"])
    if case["kind"] == "graphed":
        s["graph"] = api.GraphedGradient(p, s["probe"])
    if case["kind"] == "image":
        s["state"] = p.new_state(s["probe"])
    return s


def run(state):
    p, kind, vel, wavelet, d = state["problem"], state["case"]["kind"], state["vel"], state["wavelet"], state["d"]
    if kind == "forward":
        return p.forward(vel, wavelet)
    if kind == "probed":
        return p.gradient_probed(vel, wavelet, d, state["probe"])
    if kind == "full":
        return p.gradient_full(vel, wavelet, d)
    if kind == "graphed":
        return state["graph"](vel, wavelet, d)
    if kind == "qr":
        return p.qr_probes(d, state["case"]["r"], seed=state["seed"], kind=state["case"]["probe"])
    if kind == "image":  # the records drive the adjoint field, as in migration
        p.probed_forward(vel, wavelet, state["probe"], state["state"])
        return p.probed_image(vel, d, state["probe"], state["state"], cond="gradient")
    v = vel.detach().requires_grad_(True)
    syn = modeling(v, p, wavelet, state["probe"])
    (0.5 * (syn - d).square().sum()).backward()
    return syn.detach(), v.grad


def work(case):
    c = case
    n, nt, shots = c["nx"] * c["ny"] * c["nz"], c["nt"], c["shots"]
    nrec, nd = c["nx"] * c["ny"], 3 if c["ny"] > 1 else 2
    rows = float(shots * nt * nrec)
    if c["kind"] == "qr":  # two products with the records and the Gram-Schmidt passes
        return {"bytes": 4 * (rows + shots * nt * c["r"]), "flops": 4 * rows * c["r"] + 4 * shots * nt * c["r"] ** 2}
    # a stencil step: per distance 2 nd - 1 sums and one product, four operations to advance
    step = float(n) * nt * shots * (c["order"] // 2 * (2 * nd + 1) + 4)
    if c["kind"] == "forward":
        return {"bytes": 4 * (n + shots * nt + rows), "flops": step}
    if c["kind"] == "full":  # the history is written once and read once
        return {"bytes": 4 * (2 * n + shots * nt + rows + 2.0 * n * nt * shots), "flops": 3 * step}
    out = rows if c["kind"] == "autograd" else 0
    return {"bytes": 4 * (2 * n + shots * nt + rows + out), "flops": 2 * step + 4.0 * n * nt * shots * c["r"]}


# ------------------------------------------------------------------ 64 bits
def _mix(s, n):
    """n-th output of SplitMix64 from state s (arrays of uint64)."""
    z = s + n * np.uint64(0x9E3779B97F4A7C15)
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def _probes(c, seed):
    """The shots' random probes [shots, nt, r]: key chain seed, shot, column; draws indexed by time."""
    with np.errstate(over="ignore"):
        shot = _mix(np.full(c["shots"], seed, np.uint64), np.arange(1, c["shots"] + 1, dtype=np.uint64))
        col = _mix(shot[:, None], np.arange(1, c["r"] + 1, dtype=np.uint64)[None])[:, None, :]
        t = np.arange(c["nt"], dtype=np.uint64)[None, :, None]
        if c["probe"] == "rademacher":
            z = np.where(_mix(col, t + np.uint64(1)) >> np.uint64(63), -1.0, 1.0)
        else:  # sum of twelve uniforms, floored to steps of 2^-20, at the odd multiples of 2^-21
            s = np.zeros((c["shots"], c["nt"], c["r"]), np.int64)
            for k in range(12):
                s += (_mix(col, np.uint64(12) * t + np.uint64(k + 1)) >> np.uint64(32)).astype(np.int64)
            z = (2 * ((s - (6 << 32)) // 4096) + 1) * 2.0 ** -21
    return torch.from_numpy(z).to(_device())


class _Scheme:
    """The discrete system in 64 bits on fields [shots, (nz, ny, nx) or (nz, nx)]."""

    def __init__(self, c, i):
        self.c, self.shape, self.S = c, _shape(c), c["shots"]
        self.R, self.nd = c["order"] // 2, len(_shape(c))
        self.h, self.dt = float(np.float32(c["h"])), float(np.float32(c["dt"]))
        self.v2 = i["vel"].double() ** 2
        self.k = self.dt ** 2 * self.v2
        self.src, self.rec = i["src"].to(_device()), i["rec"].to(_device())
        self.a = self._damping(i["eta"]) if c["sponge"] else None

    def _damping(self, eta):
        w, d = self.c["sponge"], None
        for ax, n in enumerate(self.shape):
            x = torch.arange(n, device=_device(), dtype=torch.float64).reshape([-1 if j == ax else 1 for j in range(self.nd)])
            e = n - 1 - x if ax == 0 else torch.minimum(x, n - 1 - x)  # the top face is free
            d = e if d is None else torch.minimum(d, e)
        return 0.5 * float(np.float32(eta)) * self.dt * torch.where(d < w, (w - d) / w, torch.zeros_like(d)) ** 2

    def lap(self, u):
        """Laplacian, zero outside the grid."""
        w = W2[self.c["order"]]
        out = u * (self.nd * w[0])
        for ax in range(1, self.nd + 1):
            n = u.shape[ax]
            for k in range(1, self.R + 1):
                if k < n:
                    out.narrow(ax, 0, n - k).add_(u.narrow(ax, k, n - k), alpha=w[k])
                    out.narrow(ax, k, n - k).add_(u.narrow(ax, 0, n - k), alpha=w[k])
        return out.div_(self.h ** 2)

    def grad(self, u, ax):
        """Centred first difference along an axis, zero outside the grid."""
        out, n = torch.zeros_like(u), u.shape[ax]
        for k, w in enumerate(W1[self.c["order"]], 1):
            if k < n:
                out.narrow(ax, 0, n - k).add_(u.narrow(ax, k, n - k), alpha=w)
                out.narrow(ax, k, n - k).add_(u.narrow(ax, 0, n - k), alpha=-w)
        return out.div_(self.h)

    def at(self, u, idx):
        return u.reshape(u.shape[0], -1).gather(1, idx)

    def put(self, u, idx, val):
        u.reshape(u.shape[0], -1).scatter_add_(1, idx, val)

    def step(self, u, old, idx, val):
        """The level after u (old before it), with val entering at idx."""
        f = self.lap(u)
        self.put(f, idx, val)
        f.mul_(self.k)
        if self.a is None:
            return f.add_(u, alpha=2.0).sub_(old)
        return f.add_(u, alpha=2.0).sub_((1.0 - self.a) * old).div_(1.0 + self.a)

    def zero(self):
        return torch.zeros((self.S, *self.shape), dtype=torch.float64, device=_device())

    def forward(self, q, each=None):
        """Records [shots, nt, nrec]; each(t, u[t]) on the way."""
        nt, old, u = self.c["nt"], self.zero(), self.zero()
        d = torch.zeros((self.S, nt, self.rec.shape[1]), dtype=torch.float64, device=_device())
        for t in range(1, nt - 1):
            old, u = u, self.step(u, old, self.src, q[:, t])
            d[:, t + 1] = self.at(u, self.rec)
            if each:
                each(t + 1, u)
        return d

    def adjoint(self, s, each):
        old, lam = self.zero(), self.zero()
        for j in range(self.c["nt"] - 1, 1, -1):
            old, lam = lam, self.step(lam, old, self.rec, s[:, j])
            each(j, lam)

    def projector(self, Q, shift, lo, hi):
        """(each, fields): fields[s, i] = sum of Q[s, t + shift, i] times the level t, lo <= t <= hi."""
        P = torch.zeros((self.S, Q.shape[2], math.prod(self.shape)), dtype=torch.float64, device=_device())
        held = []

        def flush():
            if held:
                q = torch.stack([Q[:, t + shift] for t, _ in held], 2)  # [shots, r, levels]
                for s in range(self.S):
                    P[s].addmm_(q[s], torch.stack([u[s].reshape(-1) for _, u in held]))
                held.clear()

        def each(t, u):
            if lo <= t <= hi:
                held.append((t, u))
                if len(held) == 24:
                    flush()

        return each, flush, P


def exact(case, seed):
    if case["ny"] * case["nx"] * case["nz"] * case["nt"] * case["shots"] > 9e9:
        return None
    i = _inputs(case, seed)
    if case["kind"] == "qr":
        Z, D = _probes(case, i["probe_seed"]), i["d"].double()
        Q, R = torch.linalg.qr(D @ (D.transpose(1, 2) @ Z))
        return Q * torch.sign(torch.diagonal(R, dim1=1, dim2=2))[:, None, :]
    m, q, nt, kind = _Scheme(case, i), i["wavelet"].double(), case["nt"], case["kind"]
    if kind == "forward":
        return m.forward(q)
    dobs = i["d"].double()
    if kind == "full":
        hist = {1: m.zero()}
        d = m.forward(q, lambda t, u: hist.__setitem__(t, u))
        g = torch.zeros(m.shape, dtype=torch.float64, device=_device())

        def term(j, lam):
            f = m.lap(hist.pop(j - 1))
            m.put(f, m.src, q[:, j - 1])
            g.sub_((lam * f).sum(0).mul_(m.v2))

        hist.pop(nt - 1, None)
        res = d - dobs
        m.adjoint(res, term)
        return g, torch.stack([0.5 * res.square().sum(), g.norm()])
    Q = _probes(case, i["probe_seed"])
    each, flush, P = m.projector(Q, 1, 2, nt - 2)
    d = m.forward(q, each)
    flush()
    res = dobs if kind == "image" else d - dobs
    each, flush, V = m.projector(Q, 0, 2, nt - 1)
    m.adjoint(res, each)
    flush()
    g = torch.zeros(m.shape, dtype=torch.float64, device=_device())
    qbar = torch.einsum("sti,stk->ski", Q[:, 2:nt], q[:, 1:nt - 1])  # [shots, nsrc, r]
    for k in range(case["r"]):
        p, v = (x[:, k].reshape(m.S, *m.shape) for x in (P, V))
        if kind == "image":
            for ax in range(1, m.nd + 1):
                g.add_((m.grad(p, ax) * m.grad(v, ax)).sum(0))
        else:
            f = m.lap(p)
            m.put(f, m.src, qbar[:, :, k])
            g.sub_((f * v).sum(0).mul_(m.v2))
    g.div_(case["r"])
    if kind == "image":
        return g
    if kind == "autograd":
        return d, g * (-2.0 / i["vel"].double() ** 3)
    return g, torch.stack([0.5 * res.square().sum(), g.norm()])
