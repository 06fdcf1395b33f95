"""Workloads of the lattice Boltzmann library for timing, each a whole use of its public calls.

A case is a dict of plain values with a "kind":

  step    lbm_init, lbm_step(steps), lbm_get_state: a simulation run, any operator, storage,
          network and boundary; with forced=True the spectral forcing's draws are queued and
          (spectrum=True) the energy spectrum is taken at the end, as a turbulence run does
          every 100 steps;
  batch   many uneven instances stepped by lbm_batch_step;
  unroll  one training step through autograd.NCOUnroll: forward with recording, a velocity
          loss, backward to the gradient of the network's parameters;
  ke      one training step of the kinetic-energy curve through
          autograd.NCOKineticEnergyUnroll and dissipation_mse (reduced Taylor-Green domain).

Every pass starts from its inputs (lbm_init, or the unroll's f0), so it can be repeated.
exact(case, seed) restates the method in 64 bits with plain torch on the same inputs.
"""

import math

import numpy as np
import torch

import paper_2412_08229_gb300 as P
from paper_2412_08229_gb300.autograd import NCOKineticEnergyUnroll, NCOUnroll, dissipation_mse

DEV = "cuda"
RE = 1600.0
NET_FLOPS = 2 * (6 * 540 + 48 * 400) + 6 * 20 * 24 + 2 * 4 * 20  # per cell, with the group average's exact folds
DEEP_FLOPS = NET_FLOPS + 2 * 48 * 400                            # a third hidden layer
OP_FLOPS = {"bgk": 250, "reg": 400, "kbc": 500, "nco": 400}       # collision without the network, per cell
SIZES = {False: (27, 20, 20, 4), True: (27, 20, 20, 20, 4)}
STORAGE_BYTES = {"f32": 4, "f16": 2}


def _step(name, n, op, storage, net="f32", steps=10, boundary="periodic", field="hit", deep=False, forced=False,
          spectrum=False):
    nx, ny, nz = (n, n, n) if isinstance(n, int) else n
    c = dict(kind="step", nx=nx, ny=ny, nz=nz, op=op, storage=storage, net=net, steps=steps, boundary=boundary,
             field=field, deep=deep, forced=forced, spectrum=spectrum)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest grid anyone steps: the 16^3 parity and unit-test runs, launch-bound
        _step("bgk_f32_16", 16, "bgk", "f32", steps=100, field="tgv"),
        # the baseline operators at production size: FP16 f - w storage doubles what fits and is half the traffic
        _step("bgk_f16_256", 256, "bgk", "f16", field="tgv"),
        # an entropic run on a box that is no power of two along any axis
        _step("kbc_f32_197x131x149", (197, 131, 149), "kbc", "f32"),
        # the headline: the learned operator in its mixed form on the 256^3 Re 1600 Taylor-Green vortex
        _step("nco_mixed_256", 256, "nco", "f16", "bf16", steps=4, field="tgv"),
        # FP32 populations with the BF16 network (the long-horizon form) on a ragged box
        _step("nco_f32_bf16net_101x75x53", (101, 75, 53), "nco", "f32", "bf16"),
        # the FP32-class tensor-core form, used where BF16 rates are not exact enough
        _step("nco_f32_x3net_128", 128, "nco", "f32", "bf16x3", steps=5, field="tgv"),
        # the three-hidden-layer network on a symmetric octant (evaluating a trained deep operator)
        _step("nco_deep_mixed_octant_96", 96, "nco", "f16", "bf16", steps=5, boundary="mirror", field="octant", deep=True),
        # forced isotropic turbulence between two stored spectra (100 steps), baseline and learned
        _step("hit64_bgk_f32", 64, "bgk", "f32", steps=100, forced=True, spectrum=True),
        _step("hit64_nco_mixed", 64, "nco", "f16", "bf16", steps=100, forced=True, spectrum=True),
        # many uneven instances at once: a parameter sweep, every second one forced
        dict(name="batch_16_uneven", kind="batch", sizes="96,32,64,48,32,64,48,96,32,48,64,32,48,32,64,48", steps=10),
        # one training step of the differentiation form: 32^3 octant, 200 steps, checkpoint every 20
        dict(name="train_octant_32", kind="unroll", n=32, boundary="mirror", steps=200, k=20, deep=False),
        # one training step on the kinetic-energy curve: reduced Taylor-Green 16^3, t in [0, 3], deep network
        dict(name="train_ke_reduced_16", kind="ke", n=16, every=26, samples=21, deep=True),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _ragged(rng, cells):
    """Three edge lengths whose product is about `cells`, within a factor of two of a cube."""
    side = cells ** (1.0 / 3.0)
    nx, ny = (max(5, round(side * _log(rng, 0.7, 1.4))) for _ in range(2))
    return nx, ny, max(5, round(cells / (nx * ny)))


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["forced"] * 2 + ["batch", "unroll", "ke"])
    if kind == "step":
        op = rng.choice(["bgk", "kbc", "reg", "nco", "nco", "nco"])
        storage = rng.choice(["f32", "f16"])
        net = rng.choice(["bf16", "bf16", "bf16x3", "f32"]) if op == "nco" else "f32"
        deep = op == "nco" and rng.random() < 0.25
        steps = rng.randint(4, 20)
        # at most the cell updates (or, for the slower networks, the time) of the 256^3 learned run
        most = {"bf16": 4 * 256 ** 3, "bf16x3": 4 * 144 ** 3, "f32": 4 * 112 ** 3}[net] if op == "nco" else 10 * 256 ** 3
        cells = _log(rng, 12 ** 3, min(256 ** 3, most / steps / (2 if deep else 1)))
        boundary = rng.choice(["periodic", "periodic", "periodic", "mirror", "tgv_reduced"])
        if boundary == "tgv_reduced":
            n = max(6, min(96, round(cells ** (1.0 / 3.0))))
            return _step(None, n, op, storage, net, steps, boundary, "reduced", deep)
        if boundary == "mirror":
            return _step(None, max(6, round(cells ** (1.0 / 3.0))), op, storage, net, steps, boundary, "octant", deep)
        return _step(None, _ragged(rng, cells), op, storage, net, steps, boundary, "hit", deep)
    if kind == "forced":
        op = rng.choice(["bgk", "kbc", "nco", "nco"])
        n = rng.choice([24, 32, 48, 64, 96, 128])
        return _step(None, n, op, rng.choice(["f32", "f16"]), "bf16" if op == "nco" else "f32",
                     rng.randint(10, 100 if n <= 64 else 20), forced=True, spectrum=rng.random() < 0.7)
    if kind == "batch":
        sizes = [round(_log(rng, 16, 96)) for _ in range(rng.randint(4, 24))]
        return dict(kind="batch", sizes=",".join(map(str, sizes)), steps=rng.randint(4, 20))
    if kind == "unroll":
        deep = rng.random() < 0.3
        return dict(kind="unroll", n=rng.randint(10, 26 if deep else 32), boundary=rng.choice(["mirror", "periodic"]),
                    steps=rng.randint(20, 200), k=rng.randint(5, 30), deep=deep)
    n = rng.choice([10, 12, 16, 20])
    return dict(kind="ke", n=n, every=rng.randint(6, 26 if n <= 16 else 16), samples=rng.randint(6, 21),
                deep=rng.random() < 0.7)


# --- inputs ------------------------------------------------------------------

def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + salt) & 0x7FFFFFFF)
    return g


def _wavenumbers(shape):
    ks = [torch.fft.fftfreq(m, d=1.0 / m, device=DEV) for m in shape]
    return torch.meshgrid(*ks, indexing="ij")  # kz, ky, kx


def _isotropic(shape, seed, rms):
    """Random-phase solenoidal velocity with E(k) ~ k^4 exp(-2 (k/4)^2) and the given rms per axis."""
    kz, ky, kx = _wavenumbers(shape)
    noise = torch.randn((3,) + tuple(shape), generator=_gen(seed, 1), device=DEV)
    uh = torch.fft.fftn(noise, dim=(1, 2, 3))
    k2 = kx * kx + ky * ky + kz * kz
    k2s = torch.where(k2 == 0, torch.ones_like(k2), k2)
    dot = (kx * uh[0] + ky * uh[1] + kz * uh[2]) / k2s
    uh = torch.stack([uh[0] - kx * dot, uh[1] - ky * dot, uh[2] - kz * dot])
    uh = uh * (k2 * torch.exp(-k2 / 16.0)) / k2s.sqrt() * (k2 > 0)
    u = torch.fft.ifftn(uh, dim=(1, 2, 3)).real
    return (u * (rms / u.square().mean().sqrt())).float().contiguous()


def _taylor_green(shape, u0, period, shift):
    """u0 (sin x cos y cos z, -cos x sin y cos z, 0); `period` nodes per 2 pi along each axis."""
    z, y, x = torch.meshgrid(*[(torch.arange(m, device=DEV, dtype=torch.float64) + shift) * (2 * math.pi / p)
                               for m, p in zip(shape, period)], indexing="ij")
    return u0 * torch.stack([x.sin() * y.cos() * z.cos(), -x.cos() * y.sin() * z.cos(), torch.zeros_like(x)])


def _fields(kind, shape, seed):
    """rho, u (float32) and the velocity and length scale of one run's initial flow."""
    u0 = 0.04 + 0.01 * float(torch.rand(1, generator=_gen(seed, 2), device=DEV))
    length = shape[2]
    if kind == "hit":
        u0 = 0.8 * u0
        u = _isotropic(shape, seed, u0)
    elif kind == "tgv":  # with the small disturbance that breaks its symmetries
        u = (_taylor_green(shape, u0, shape, 0.0) + _isotropic(shape, seed, 0.02 * u0)).float()
    elif kind == "octant":
        length = 2 * shape[2]
        full = [2 * m for m in shape]
        u = _taylor_green(shape, u0, full, 0.5)
        u = (u + 0.2 * _taylor_green(shape, u0, [m // 2 for m in full], 0.5)).float()
    else:
        length = 4 * shape[2]
        u = _taylor_green(shape, u0, [4 * m for m in shape], 0.5).float()
    rho = torch.ones(shape, device=DEV)
    if kind in ("hit", "tgv"):
        rho += 0.002 * torch.randn(shape, generator=_gen(seed, 3), device=DEV).clamp_(-3, 3)
    return rho, u.contiguous(), u0, length


def _theta(seed, deep):
    """Kaiming-uniform parameters as nn.Linear draws them, flattened layer by layer (W, then b)."""
    g = torch.Generator()
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    parts = []
    for a, b in zip(SIZES[deep][:-1], SIZES[deep][1:]):
        parts += [(2 * torch.rand(b * a, generator=g) - 1) / math.sqrt(a), (2 * torch.rand(b, generator=g) - 1) / math.sqrt(a)]
    return torch.cat(parts).to(DEV)


def _power(u, nu):
    """The viscous dissipation nu <|grad u|^2> of a field: the power a forced run puts in."""
    g2 = sum(float(((torch.roll(u[a], -1, d) - torch.roll(u[a], 1, d)).double() / 2).square().mean())
             for a in range(3) for d in range(3))
    return nu * g2


def _draws(seed, steps):
    rng = np.random.default_rng([int(seed), 7])
    return rng.uniform(0, math.pi, (steps, 16)), rng.uniform(0, 2 * math.pi, (steps, 16))


def _shape(case):
    return (case["nz"], case["ny"], case["nx"])


def _step_inputs(case, seed):
    rho, u, u0, length = _fields(case["field"], _shape(case), seed)
    nu = 0.0015 if case["forced"] else u0 * length / (2 * math.pi * RE)
    return rho, u, nu


def _batch_inputs(case, seed):
    """Per instance: n, rho, u, nu, power (None: a Taylor-Green instance), draws."""
    rng = np.random.default_rng([int(seed), 11])
    out = []
    for i, n in enumerate(int(v) for v in case["sizes"].split(",")):
        rho, u, u0, length = _fields("hit" if i % 2 else "tgv", (n, n, n), seed * 64 + i)
        nu = u0 * length / (2 * math.pi * math.exp(rng.uniform(math.log(400.0), math.log(4000.0))))
        out.append((n, rho, u, nu, _power(u, nu) if i % 2 else None, _draws(seed * 64 + i, case["steps"])))
    return out


def _train_inputs(case, seed):
    n = case["n"]
    field = "reduced" if case["kind"] == "ke" else {"mirror": "octant", "periodic": "hit"}[case["boundary"]]
    rho, u, u0, length = _fields(field, (n, n, n), seed)
    re = RE if case["kind"] == "ke" else 3000.0
    f0 = _equilibrium(rho.double(), u.double(), *_lattice()).float()
    return f0, u, u0, length, u0 * length / (2 * math.pi * re)


def prepare(case, seed):
    s = dict(case=case)
    if case["kind"] == "step":
        rho, u, nu = _step_inputs(case, seed)
        forcing = dict(power=_power(u, nu)) if case["forced"] else None
        ctx = P.lbm_create(case["nx"], case["ny"], case["nz"], nu, op=case["op"], storage=case["storage"],
                           net=case["net"], boundary=case["boundary"], forcing=forcing)
        if case["op"] == "nco":
            P.nco_set_weights(ctx, _theta(seed, case["deep"]))
        s.update(ctx=ctx, rho=rho, u=u, f=torch.empty((27,) + _shape(case), device=DEV))
        if case["forced"]:
            s["draws"] = _draws(seed, case["steps"])
        if case["spectrum"]:
            s["E"] = torch.empty(max(_shape(case)) // 2 + 1, dtype=torch.float64, device=DEV)
    elif case["kind"] == "batch":
        inst = _batch_inputs(case, seed)
        batch = P.lbm_batch_create([dict(nx=n, ny=n, nz=n, nu=nu, storage="f16",
                                         forcing=None if power is None else dict(power=power))
                                    for n, _, _, nu, power, _ in inst])
        P.lbm_batch_set_weights(batch, _theta(seed, False))
        s.update(batch=batch, inst=inst, f=[torch.empty((27, n, n, n), device=DEV) for n, *_ in inst])
    else:
        f0, u, u0, length, nu = _train_inputs(case, seed)
        boundary = "tgv_reduced" if case["kind"] == "ke" else case["boundary"]
        n = case["n"]
        s.update(ctx=P.lbm_create(n, n, n, nu, op="nco", boundary=boundary), f0=f0, u0=u0,
                 theta=_theta(seed, case["deep"]), target=0.9 * u)
        if case["kind"] == "ke":
            tc = length / (2 * math.pi * u0)  # steps per unit of t = L / U0
            s.update(dt=case["every"] / tc, eps=torch.full((case["samples"] - 1,), 0.01, dtype=torch.float64, device=DEV))
    torch.cuda.synchronize()
    return s


def run(s):
    case = s["case"]
    if case["kind"] == "step":
        ctx = s["ctx"]
        P.lbm_init(ctx, s["rho"], s["u"])
        if case["forced"]:
            P.lbm_force_draws(ctx, *s["draws"])
        P.lbm_step(ctx, case["steps"])
        P.lbm_get_state(ctx, s["f"])
        out = {"f": s["f"]}
        if case["spectrum"]:
            P.lbm_energy_spectrum(ctx, s["E"])
            out["E"] = s["E"].float()  # kept in the populations' own precision
        return out
    if case["kind"] == "batch":
        batch = s["batch"]
        for i, (n, rho, u, nu, power, draws) in enumerate(s["inst"]):
            P.lbm_init(batch[i], rho, u)
            if power is not None:
                P.lbm_force_draws(batch[i], *draws)
        P.lbm_batch_step(batch, case["steps"])
        for i, f in enumerate(s["f"]):
            P.lbm_get_state(batch[i], f)
        return s["f"]
    theta = s["theta"].detach().requires_grad_(True)
    if case["kind"] == "unroll":
        rho, u = NCOUnroll.apply(theta, s["ctx"], s["f0"], case["steps"], case["k"])
        _velocity_loss(u, s["target"]).backward()
        return {"rho": rho.detach(), "u": u.detach(), "grad": theta.grad}
    obs = [case["every"] * j for j in range(case["samples"] + 1)]
    ke = NCOKineticEnergyUnroll.apply(theta, s["ctx"], s["f0"], obs, case["every"])
    dissipation_mse(ke / s["u0"] ** 2, s["dt"], s["eps"]).backward()
    return {"ke": ke.detach().float(), "grad": theta.grad}


def _velocity_loss(u, target):
    d = u - target
    return (d * d).sum() / (target * target).sum()


def work(case):
    """Populations of every step read and written once, inputs and results once; the
    collision's and the network's operations. A gradient is one more forward (recomputed
    between checkpoints) and a backward of twice the forward's operations per step, whose
    cotangents are read and written once."""
    if case["kind"] == "step":
        cells = case["nx"] * case["ny"] * case["nz"]
        sb = STORAGE_BYTES[case["storage"]]
        net = (DEEP_FLOPS if case["deep"] else NET_FLOPS) if case["op"] == "nco" else 0
        b = cells * (case["steps"] * 54 * sb + 16 + 27 * sb + 27 * sb + 108)
        fl = cells * case["steps"] * (OP_FLOPS[case["op"]] + net + (400 if case["forced"] else 0))
        if case["spectrum"]:
            b += cells * (27 * sb + 3 * 6 * 8)
            fl += cells * 3 * 5 * math.log2(cells)
        return {"bytes": b, "flops": fl}
    if case["kind"] == "batch":
        ns = [int(v) for v in case["sizes"].split(",")]
        cells = sum(n ** 3 for n in ns)
        return {"bytes": cells * (case["steps"] * 108 + 16 + 54 + 54 + 108),
                "flops": cells * case["steps"] * (OP_FLOPS["nco"] + NET_FLOPS)}
    steps = case["steps"] if case["kind"] == "unroll" else case["every"] * case["samples"]
    cells = case["n"] ** 3
    net = DEEP_FLOPS if case["deep"] else NET_FLOPS
    return {"bytes": cells * (steps * (216 + 216 + 324) + 2 * 108 + 32), "flops": cells * steps * 4 * (net + OP_FLOPS["nco"])}


# --- the method in 64 bits, plain torch ---------------------------------------

NAMES = ["", "x", "y", "z", "xx", "xy", "xz", "yy", "yz", "zz", "xxy", "xxz", "xyy", "xyz", "xzz", "yyz", "yzz", "xxyy",
         "xxyz", "xxzz", "xyyz", "xyzz", "yyzz", "xxyyz", "xxyzz", "xyyzz", "xxyyzz"]


def _velocities():
    return np.array([(cx, cy, cz) for cz in (-1, 0, 1) for cy in (-1, 0, 1) for cx in (-1, 0, 1)], dtype=np.int64)


def _lattice():
    c = _velocities()
    w1 = {-1: 1 / 6, 0: 2 / 3, 1: 1 / 6}
    w = np.array([w1[a] * w1[b] * w1[d] for a, b, d in c])
    return torch.tensor(c, dtype=torch.float64, device=DEV), torch.tensor(w, dtype=torch.float64, device=DEV)


def _hermite():
    """M (printed row order) and the order of each row."""
    xi = math.sqrt(3.0) * _velocities()
    he = [np.ones_like(xi), xi, xi * xi - 1]
    rows = [np.prod([he[name.count("xyz"[a])][:, a] for a in range(3)], axis=0) for name in NAMES]
    return np.array(rows), np.array([len(name) for name in NAMES])


def _group():
    """Velocity permutations pi of the 48 cube symmetries: c[pi[i]] = R c[i]."""
    c = _velocities()
    index = {tuple(v): i for i, v in enumerate(c)}
    out = []
    for p in ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)):
        for s in range(8):
            sign = np.array([1 - 2 * (s & 1), 1 - (s & 2), 1 - (s & 4) // 2])
            out.append([index[tuple(sign * v[list(p)])] for v in c])
    return np.array(out)


def _equilibrium(rho, u, c, w):
    cu = torch.einsum("ia,a...->i...", c, u)
    usq = (u * u).sum(0)
    shape = (27,) + (1,) * rho.dim()
    return w.reshape(shape) * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * usq)


class _Exact:
    """One run in 64 bits: collide and stream on f (27, cells)."""

    def __init__(self, shape, nu, op, boundary, deep=False):
        self.shape, self.op, self.boundary, self.deep = shape, op, boundary, deep
        self.tau = 3.0 * nu + 0.5
        self.c, self.w = _lattice()
        M, order = _hermite()
        self.M = torch.tensor(M, dtype=torch.float64, device=DEV)
        self.Mi = torch.tensor(np.linalg.inv(M), dtype=torch.float64, device=DEV)
        self.order = order
        inv = np.linalg.inv(M)
        self.Pg = torch.tensor(np.array([np.rint(M @ np.eye(27)[pi] @ inv) for pi in _group()]), dtype=torch.float64, device=DEV)
        self.index = _reduced_index(shape[0]) if boundary == "tgv_reduced" else None

    def macro(self, f):
        rho = f.sum(0)
        return rho, (self.c.T @ f) / rho

    def layers(self, theta):
        out, off, sizes = [], 0, SIZES[self.deep]
        for a, b in zip(sizes[:-1], sizes[1:]):
            out.append((theta[off:off + a * b].reshape(b, a), theta[off + a * b:off + a * b + b]))
            off += a * b + b
        return out

    def rates(self, m, theta):
        (W1, b1), *mid, (W3, b3) = self.layers(theta)
        first = (W1 @ self.Pg).reshape(-1, 27)
        h = torch.relu(first @ m + b1.repeat(48)[:, None]).reshape(48, 20, -1)
        for W, b in mid:
            h = torch.relu(W @ h + b[:, None])
        t = W3 @ h.mean(0) + b3[:, None]
        return 1.0 / (0.5 / (1.0 + torch.exp(t)) + 0.5)

    def collide(self, f, theta=None, force=None):
        rho, u = self.macro(f)
        feq = _equilibrium(rho, u, self.c, self.w)
        if self.op == "bgk":
            out = f - (f - feq) / self.tau
        elif self.op == "kbc":
            dm = self.M @ (f - feq)
            second = torch.tensor((self.order == 2).astype(float), device=DEV)[:, None]
            ds = self.Mi @ (dm * second)
            dh = self.Mi @ (dm * torch.tensor((self.order >= 3).astype(float), device=DEV)[:, None])
            sh, hh = (ds * dh / feq).sum(0), (dh * dh / feq).sum(0)
            beta = 1.0 / (2.0 * self.tau)
            safe = hh >= 1e-30
            gamma = torch.where(safe, 1 / beta - (2 - 1 / beta) * sh / torch.where(safe, hh, torch.ones_like(hh)),
                                torch.full_like(hh, 2.0))
            out = f - beta * (2 * ds + gamma * dh)
        else:
            m = self.M @ f
            dm = m - self.M @ feq
            r = self.rates(m, theta) if self.op == "nco" else torch.ones((4, f.shape[1]), dtype=f.dtype, device=DEV)
            one = torch.ones_like(r[:1])
            table = torch.cat([one, one, one / self.tau, r])  # by order 0..6
            out = f - self.Mi @ (table[torch.tensor(self.order, device=DEV)] * dm)
        if force is not None:
            out = out + _equilibrium(rho, u + force / rho, self.c, self.w) - feq
        return out

    def stream(self, f):
        nz, ny, nx = self.shape
        c = _velocities()
        if self.boundary == "tgv_reduced":
            return f.reshape(-1)[self.index].reshape(27, -1)
        f = f.reshape(27, nz, ny, nx)
        if self.boundary == "periodic":
            return torch.stack([torch.roll(f[i], tuple(int(v) for v in c[i][::-1]), (0, 1, 2)) for i in range(27)]).reshape(27, -1)
        for a in range(3):  # mirror planes half a spacing outside the nodes: axis by axis
            d = 2 - a
            place = {tuple(v): i for i, v in enumerate(c)}
            new = [None] * 27
            for i, v in enumerate(c):
                flip = v.copy()
                flip[a] = -flip[a]
                j, n = place[tuple(flip)], self.shape[d]
                if v[a] == 0:
                    new[i] = f[i]
                elif v[a] > 0:
                    new[i] = torch.cat([f[j].narrow(d, 0, 1), f[i].narrow(d, 0, n - 1)], d)
                else:
                    new[i] = torch.cat([f[i].narrow(d, 1, n - 1), f[j].narrow(d, n - 1, 1)], d)
            f = torch.stack(new)
        return f.reshape(27, -1)

    def step(self, f, theta=None, force=None, chunk=1 << 17):
        if f.requires_grad or f.shape[1] <= chunk:
            return self.stream(self.collide(f, theta, force))
        out = torch.empty_like(f)
        for a in range(0, f.shape[1], chunk):
            out[:, a:a + chunk] = self.collide(f[:, a:a + chunk], theta, None if force is None else force[:, a:a + chunk])
        return self.stream(out)


def _reduced_index(n):
    """Pull index (27 * cells) of the reduced Taylor-Green domain [0, pi/2]^3: a source outside
    it is mapped back, with its direction, by the flow symmetry x -> A x + (pi/2) k of its block."""
    c = _velocities()
    place = {tuple(v): i for i, v in enumerate(c)}
    pts = np.random.default_rng(3).uniform(0, 2 * math.pi, (32, 3))

    def flow(x):
        return np.stack([np.sin(x[:, 0]) * np.cos(x[:, 1]) * np.cos(x[:, 2]),
                         -np.cos(x[:, 0]) * np.sin(x[:, 1]) * np.cos(x[:, 2]), 0 * x[:, 0]], 1)

    sym = []
    for p in ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)):
        for s in range(8):
            A = np.zeros((3, 3), dtype=np.int64)
            for a in range(3):
                A[a, p[a]] = 1 - 2 * ((s >> a) & 1)
            for k in np.ndindex(4, 4, 4):
                if np.allclose(flow(pts @ A.T + np.array(k) * math.pi / 2), flow(pts) @ A.T, atol=1e-9):
                    sym.append((A, np.array(k)))
    z, y, x = np.meshgrid(*[np.arange(n)] * 3, indexing="ij")
    node = np.stack([x, y, z], -1).reshape(-1, 3)
    out = np.empty((27, n ** 3), dtype=np.int64)
    for i, v in enumerate(c):
        src = node - v
        block = np.floor_divide(src, n)
        out[i] = -1
        for b in np.unique(block, axis=0):
            at = np.all(block == b, axis=1)
            s, d = src[at], i
            if np.any(b):
                for A, k in sym:  # the one that maps the block's centre into the domain
                    if np.all((A @ (2 * b + 1) + 2 * k) % 8 == 1):
                        s = (((2 * s + 1) @ A.T + 2 * n * k) % (8 * n) - 1) // 2
                        d = place[tuple(A @ v)]
                        break
            out[i, at] = d * n ** 3 + (s[:, 2] * n + s[:, 1]) * n + s[:, 0]
    return torch.tensor(out.reshape(-1), device=DEV)


class _Forcing:
    """The spectral force on the half-space modes 1 <= |k| <= 2, in 64 bits."""

    def __init__(self, shape, power, draws, kf=1.5, c=0.5, ka=1.0, kb=2.0):
        modes = [(kx, ky, kz) for kz in range(-2, 3) for ky in range(-2, 3) for kx in range(-2, 3)
                 if 1 <= kx * kx + ky * ky + kz * kz <= 4
                 and (kz > 0 or (kz == 0 and ky > 0) or (kz == 0 and ky == 0 and kx > 0))]
        modes.sort(key=lambda k: (k[0] ** 2 + k[1] ** 2 + k[2] ** 2, k[2], k[1], k[0]))
        self.draws = draws
        k = np.array(modes, dtype=np.float64)
        kk, kh = np.sqrt((k * k).sum(1)), np.sqrt(k[:, 0] ** 2 + k[:, 1] ** 2)
        safe = np.where(kh > 0, kh, 1.0)
        self.e1 = np.where(kh[:, None] > 0, np.stack([k[:, 1], -k[:, 0], 0 * kh], 1) / safe[:, None], [1.0, 0.0, 0.0])
        self.e2 = np.where(kh[:, None] > 0, np.stack([k[:, 0] * k[:, 2], k[:, 1] * k[:, 2], -kh * kh], 1) / (safe * kk)[:, None],
                           [0.0, 1.0, 0.0])
        integral = 0.5 * math.sqrt(math.pi * c) * (math.erf((kb - kf) / math.sqrt(c)) - math.erf((ka - kf) / math.sqrt(c)))
        self.amp = np.sqrt(power / integral * np.exp(-((kk - kf) ** 2) / c) / (2 * math.pi * kk * kk))
        z, y, x = torch.meshgrid(*[torch.arange(m, dtype=torch.float64, device=DEV) / m for m in shape], indexing="ij")
        t = torch.tensor(k, device=DEV)
        arg = 2 * math.pi * (t[:, 0, None] * x.reshape(-1) + t[:, 1, None] * y.reshape(-1) + t[:, 2, None] * z.reshape(-1))
        self.cos, self.sin = arg.cos(), arg.sin()

    def project(self, u):
        n = u.shape[1]
        return ((u @ self.cos.T - 1j * (u @ self.sin.T)) / n).T.cpu().numpy()  # (16, 3)

    def field(self, t, uh):
        phi, psi = self.draws[0][t], self.draws[1][t]
        x1, x2 = (uh * self.e1).sum(1), (uh * self.e2).sum(1)
        ga, gb, sp, cp = np.sin(2 * phi), np.cos(2 * phi), np.sin(psi), np.cos(psi)
        num = ga * x1.real + gb * (sp * x2.imag + cp * x2.real)
        den = -ga * x1.imag + gb * (sp * x2.real - cp * x2.imag)
        th = np.arctan2(num, den)
        F = (self.amp * ga * np.exp(1j * th))[:, None] * self.e1 + (self.amp * gb * np.exp(1j * (th + psi)))[:, None] * self.e2
        F = torch.tensor(F, device=DEV)
        return 2 * (F.real.T @ self.cos - F.imag.T @ self.sin)


def _spectrum(u, shape, nbins):
    uh = torch.fft.fftn(u.reshape((3,) + tuple(shape)), dim=(1, 2, 3)) / math.prod(shape)
    e = 0.5 * uh.abs().square().sum(0).reshape(-1)
    kz, ky, kx = _wavenumbers(shape)
    shell = (kx.double() ** 2 + ky.double() ** 2 + kz.double() ** 2).sqrt().round().long().reshape(-1)
    E = torch.zeros(int(shell.max()) + 1, dtype=torch.float64, device=DEV).index_add_(0, shell, e)
    return E[:nbins]


def _exact_run(shape, rho, u, nu, op, boundary, steps, theta=None, deep=False, power=None, draws=None):
    sim = _Exact(shape, nu, op, boundary, deep)
    f = _equilibrium(rho.double().reshape(-1), u.double().reshape(3, -1), sim.c, sim.w)
    forcing = None if power is None else _Forcing(shape, power, draws)
    uh = forcing.project(u.double().reshape(3, -1)) if forcing else None
    th = None if theta is None else theta.double()
    for t in range(steps):
        force = None
        if forcing:
            force = forcing.field(t, uh)
            uh = forcing.project(sim.macro(f)[1])
        f = sim.step(f, th, force)
    return sim, f


def _exact_updates(case):
    """Cell updates of exact(), a learned one counted ten times (its 90k operations per cell)."""
    return case["nx"] * case["ny"] * case["nz"] * case["steps"] * (10 if case["op"] == "nco" else 1)


def exact(case, seed):
    if case["kind"] == "step":
        if _exact_updates(case) > 11 * 256 ** 3 * 4:
            return None
        rho, u, nu = _step_inputs(case, seed)
        power = _power(u, nu) if case["forced"] else None
        with torch.no_grad():
            sim, f = _exact_run(_shape(case), rho, u, nu, case["op"], case["boundary"], case["steps"],
                                _theta(seed, case["deep"]) if case["op"] == "nco" else None, case["deep"], power,
                                _draws(seed, case["steps"]) if case["forced"] else None)
            out = {"f": f.reshape((27,) + _shape(case))}
            if case["spectrum"]:
                out["E"] = _spectrum(sim.macro(f)[1], _shape(case), max(_shape(case)) // 2 + 1)
        return out
    if case["kind"] == "batch":
        theta, out = _theta(seed, False), []
        with torch.no_grad():
            for n, rho, u, nu, power, draws in _batch_inputs(case, seed):
                f = _exact_run((n, n, n), rho, u, nu, "nco", "periodic", case["steps"], theta, False, power, draws)[1]
                out.append(f.reshape(27, n, n, n))
        return out
    from torch.utils.checkpoint import checkpoint
    f0, u, u0, length, nu = _train_inputs(case, seed)
    n = case["n"]
    sim = _Exact((n, n, n), nu, "nco", "tgv_reduced" if case["kind"] == "ke" else case["boundary"], case["deep"])
    theta = _theta(seed, case["deep"]).double().requires_grad_(True)
    f = f0.double().reshape(27, -1).requires_grad_(True)

    def segment(g, th, count):
        for _ in range(count):
            g = checkpoint(sim.step, g, th, use_reentrant=False)
        return g

    if case["kind"] == "unroll":
        left = case["steps"]
        while left:
            k = min(left, case["k"])
            f = checkpoint(segment, f, theta, k, use_reentrant=False)
            left -= k
        rho, v = sim.macro(f)
        _velocity_loss(v, 0.9 * u.double().reshape(3, -1)).backward()
        return {"rho": rho.detach().reshape(n, n, n), "u": v.detach().reshape(3, n, n, n), "grad": theta.grad}
    ke = []
    for j in range(case["samples"] + 1):
        if j:
            f = checkpoint(segment, f, theta, case["every"], use_reentrant=False)
        ke.append(0.5 * (sim.macro(f)[1] ** 2).sum(0).mean())
    ke = torch.stack(ke)
    d = -((ke[2:] - ke[:-2]) / u0 ** 2) / (2 * case["every"] * 2 * math.pi * u0 / length) - 0.01
    (d * d).mean().backward()
    return {"ke": ke.detach(), "grad": theta.grad}
