"""The work whose speed is measured: one pass of each kind of program that uses this package.

A case is a dict of plain values.  Its "kind" says which program it stands for:

  step       a run of Algorithm 4 on the device (`Simulation`): some steps, then the
             positions in particle order in the caller's device arrays, where asked
             with the FP64 diagnostics of the new state
  host       the same run driven from pinned host memory: positions sent, one step,
             positions read back
  batch      an ensemble of independent runs advanced together (`Batch`)
  adjoint    forward and reverse sweep through `SipfDensity` (torch autograd)
  plane      the two-dimensional system (`Simulation2D`)
  operators  a caller's own particle-mesh solve with the stateless operators

Inputs come from the seed alone.  `exact` is the same mathematics in 64-bit torch.
"""
import math

import numpy as np
import torch

from paper_2512_03452_gb300 import (DEPOSIT_ATOMIC, DEPOSIT_DETERMINISTIC, SPLIT_HALF, SPLIT_PLAIN, Batch, Simulation,
                                    Simulation2D, _abi, make_params)
from paper_2512_03452_gb300.adjoint import Adjoint, SipfDensity

TWO_PI = 2.0 * math.pi

# Physical parameters of the runs.  "ring" and "blowup" are the workloads' own supercritical
# data, whose density collapses within some tens of steps and then stays so; the others have
# their shapes, boxes and time steps with a mass below the critical one, so their density
# spreads and stays spread however many passes are made.
SYSTEMS = {
    "blob": dict(shape="gaussian", sigma=0.1, L=1.0, mass=2.0, mu=1.0, eps=1.0, k=1.0, dt=1e-3),
    "drop": dict(shape="gaussian", sigma=0.1, L=1.0, mass=2.0, mu=1.0, eps=1.0, k=1.0, dt=1e-4),
    "blowup": dict(shape="gaussian", sigma=0.05, L=2.0, mass=200.0, mu=1.0, eps=1.0, k=0.5, dt=1e-4),
    "ring": dict(shape="torus", sigma=0.03, L=1.0, mass=300.0, mu=0.5, eps=1.0, k=1.0, dt=5e-5),
    "thin_ring": dict(shape="torus", sigma=0.03, L=1.0, mass=5.0, mu=0.5, eps=1.0, k=1.0, dt=5e-5),
    "ball": dict(shape="ball", sigma=0.125, L=8.0, mass=40.0, mu=1.0, eps=1e-4, k=0.1, dt=1e-5),
}


def listed():
    return [
        # the smallest run in earnest: double precision on a small grid, where launches and latency count
        dict(name="step64_P1e4_H16", kind="step", system="blob", P=10_000, H=16, precision=64, steps=20),
        # one run of the convergence study at its default size
        dict(name="step32_P16384_H32", kind="step", system="ball", P=16_384, H=32, precision=32, steps=20),
        # the blow-up study: a million particles, diagnostics watched along the way
        dict(name="step32_P1e6_H64", kind="step", system="blowup", P=1_000_000, H=64, precision=32, steps=5,
             diagnostics=True),
        # the benchmark's run: the largest number of particles
        dict(name="step32_P1e7_H128", kind="step", system="ring", P=10_000_000, H=128, precision=32, steps=4),
        # the finest grid of the convergence study: the field solve counts
        dict(name="step32_P2e20_H256", kind="step", system="ball", P=1 << 20, H=256, precision=32, steps=4),
        # the double-precision form at an ordinary, ragged size
        dict(name="step64_P1e6_H64", kind="step", system="drop", P=999_983, H=64, precision=64, steps=2),
        # bit-reproducible sums and the plain Euler-Maruyama move
        dict(name="fixed32_P2e6_H128", kind="step", system="thin_ring", P=2_000_003, H=128, precision=32, steps=4,
             deterministic=True, plain=True),
        # coupled to a program whose positions live in host memory
        dict(name="host32_P4e6_H128", kind="host", system="drop", P=4_000_003, H=128, precision=32),
        # a parameter study: many small runs of uneven size, read back at the end
        dict(name="batch32_24runs", kind="batch", runs=24, P_min=10_000, P_max=100_000, steps=192, precision=32),
        # gradients of an observable of the final density
        dict(name="adjoint32_P2e5_H64", kind="adjoint", system="drop", P=200_003, H=64, precision=32, steps=40),
        # the two-dimensional critical-mass experiment
        dict(name="plane32_P2e20_H256", kind="plane", P=1 << 20, H=256, precision=32, steps=50),
        # the operators by themselves, on unsorted particles
        dict(name="operators32_P1e6_H128", kind="operators", P=1_000_003, H=128, precision=32, comps=3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "host", "batch", "adjoint", "plane", "operators"])
    if kind == "step":
        precision = rng.choice([32, 32, 32, 64])
        H = rng.choice([16, 32, 64, 128, 256] if precision == 32 else [16, 32, 64])
        most = (10_000_000 if H < 256 else 4_000_000) if precision == 32 else 1_000_000
        P = _log_int(rng, 3_000, most)
        return dict(kind=kind, system=rng.choice(["blob", "drop", "thin_ring", "ball"]), P=P, H=H, precision=precision,
                    steps=2 if precision == 64 and P > 200_000 else 4 if P > 500_000 else rng.choice([4, 10, 20]),
                    deterministic=rng.random() < 0.25, plain=rng.random() < 0.25, diagnostics=rng.random() < 0.25)
    if kind == "host":
        return dict(kind=kind, system="drop", P=_log_int(rng, 100_000, 8_000_000), H=rng.choice([32, 64, 128]),
                    precision=32)
    if kind == "batch":
        P_min = _log_int(rng, 3_000, 12_000)
        return dict(kind=kind, runs=rng.randint(8, 24), P_min=P_min, P_max=P_min * rng.randint(2, 6), steps=192,
                    precision=32)
    if kind == "adjoint":
        return dict(kind=kind, system="drop", P=_log_int(rng, 20_000, 400_000), H=rng.choice([32, 64]), precision=32,
                    steps=rng.choice([20, 30, 40]))
    if kind == "plane":
        return dict(kind=kind, P=_log_int(rng, 30_000, 2_000_000), H=rng.choice([64, 128, 256]), precision=32, steps=50)
    return dict(kind=kind, P=_log_int(rng, 30_000, 4_000_000), H=rng.choice([32, 64, 128, 256]),
                precision=rng.choice([32, 32, 64]), comps=rng.choice([1, 3]))


# ------------------------------------------------------------------ inputs
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _sample(shape, P, L, sigma, precision, g):
    """P i.i.d. positions of one initial shape, (P, 3) float64 on the device, exact in the run's precision."""
    def normal(*s):
        return torch.randn(*s, device="cuda", dtype=torch.float64, generator=g)

    def uniform(*s):
        return torch.rand(*s, device="cuda", dtype=torch.float64, generator=g)

    if shape == "gaussian":
        X = normal(P, 3) * (sigma * L)
    elif shape == "torus":   # a ring of radius L/4 and 5% uniform background
        phi = uniform(P) * TWO_PI
        r = 0.25 * L + sigma * L * normal(P)
        X = torch.stack([r * phi.cos(), r * phi.sin(), sigma * L * normal(P)], dim=1)
        back = uniform(P) < 0.05
        X[back] = (uniform(int(back.sum()), 3) - 0.5) * L
    elif shape == "ball":    # uniform ball of radius sigma L
        v = normal(P, 3)
        X = v / v.norm(dim=1, keepdim=True) * (sigma * L * uniform(P, 1) ** (1.0 / 3.0))
    else:
        raise ValueError(shape)
    X = X - L * torch.floor(X / L + 0.5)
    return X.float().double() if precision == 32 else X


def _system(case, seed):
    s = dict(SYSTEMS[case["system"]])
    s.update(P=case["P"], H=case["H"], precision=case["precision"], seed=int(seed), chi=1.0,
             plain=bool(case.get("plain")), deterministic=bool(case.get("deterministic")))
    return s


def _params(s):
    return make_params(s["P"], s["H"], L=s["L"], mass=s["mass"], chi=s["chi"], mu=s["mu"], eps=s["eps"], k=s["k"],
                       dt=s["dt"], seed=s["seed"], precision=s["precision"],
                       splitting=SPLIT_PLAIN if s["plain"] else SPLIT_HALF,
                       deposit_mode=DEPOSIT_DETERMINISTIC if s["deterministic"] else DEPOSIT_ATOMIC)


def _ensemble(case, seed):
    """Runs of a parameter study: log-uniform P, H in {32, 64} (of the case), chi, mass and noise of their own."""
    sizes, rng = np.random.default_rng(case["runs"] + case["P_min"]), np.random.default_rng(int(seed))
    runs = []
    for i in range(case["runs"]):
        s = dict(SYSTEMS["drop"], precision=case["precision"], plain=False, deterministic=False, seed=int(seed) + i)
        s["P"] = int(math.exp(sizes.uniform(math.log(case["P_min"]), math.log(case["P_max"]))))
        s["H"] = 64 if i % 2 else 32
        s["chi"] = float(np.float32(rng.uniform(0.5, 2.0)))
        s["mass"] = float(rng.uniform(0.5, 2.0))
        runs.append(s)
    return runs


def _ensemble_positions(runs, seed):
    g = _generator(seed)
    return [_sample(s["shape"], s["P"], s["L"], s["sigma"], s["precision"], g) for s in runs]


def _plane(case, seed):
    """Unit disk of mass near the critical 8 pi in a box of side 10."""
    g = _generator(seed)
    r = torch.rand(case["P"], device="cuda", dtype=torch.float64, generator=g).sqrt()
    phi = TWO_PI * torch.rand(case["P"], device="cuda", dtype=torch.float64, generator=g)
    X = torch.stack([r * phi.cos(), r * phi.sin()], dim=1)
    s = dict(P=case["P"], H=case["H"], L=10.0, mass=24.6, chi=1.0, mu=1.0, eps=0.0, k=0.0, dt=5e-4, seed=int(seed),
             precision=case["precision"])
    return s, X.float().double() if case["precision"] == 32 else X


def _real(precision):
    return torch.float64 if precision == 64 else torch.float32


def _host(X):
    return np.ascontiguousarray(X.cpu().numpy())


def prepare(case, seed):
    kind, T = case["kind"], _real(case["precision"])
    if kind == "batch":
        runs = _ensemble(case, seed)
        return dict(case=case, batch=Batch([_params(s) for s in runs], [_host(X) for X in _ensemble_positions(runs, seed)]))
    if kind == "plane":
        s, X = _plane(case, seed)
        p = make_params(s["P"], s["H"], L=s["L"], mass=s["mass"], chi=s["chi"], mu=s["mu"], eps=s["eps"], k=s["k"],
                        dt=s["dt"], seed=s["seed"], precision=s["precision"])
        return dict(case=case, sim=Simulation2D(p, _host(X)))
    if kind == "operators":
        X, green = _operator_inputs(case, seed)
        P, H = case["P"], case["H"]
        return dict(case=case, x=X.t().to(T).contiguous(), green=green.to(T),
                    grid=torch.empty(H, H, H, dtype=T, device="cuda"),
                    spec=torch.empty(H, H, H // 2 + 1, dtype=torch.complex128 if T == torch.float64 else torch.complex64,
                                     device="cuda"),
                    field=torch.empty(case["comps"], H, H, H, dtype=T, device="cuda"),
                    values=torch.empty(case["comps"], P, dtype=T, device="cuda"))
    s = _system(case, seed)
    X = _sample(s["shape"], s["P"], s["L"], s["sigma"], s["precision"], _generator(seed))
    if kind == "adjoint":
        return dict(case=case, engine=Adjoint(_params(s), _host(X), nsteps=case["steps"]), X0=X.to(T),
                    weight=_observable(s), chi=torch.tensor(s["chi"], dtype=T), mu=torch.tensor(s["mu"], dtype=T))
    if kind == "host":
        src = X.t().to(T).contiguous().cpu().pin_memory()
        return dict(case=case, sim=Simulation(_params(s), _host(X)), src=src, dst=torch.empty_like(src).pin_memory())
    stream = torch.cuda.Stream()
    return dict(case=case, stream=stream, sim=Simulation(_params(s), _host(X), stream=stream.cuda_stream),
                x=torch.empty(3, s["P"], dtype=T, device="cuda"))


def _operator_inputs(case, seed):
    """Positions of a Gaussian cloud in particle order and the screened Green's function of the unit box."""
    X = _sample("gaussian", case["P"], 1.0, 0.12, case["precision"], _generator(seed))
    H = case["H"]
    q = torch.fft.fftfreq(H, 1.0 / H, device="cuda", dtype=torch.float64) * TWO_PI
    qz = torch.arange(H // 2 + 1, device="cuda", dtype=torch.float64) * TWO_PI
    return X, 1.0 / (1.0 + q[:, None, None] ** 2 + q[None, :, None] ** 2 + qz[None, None, :] ** 2)


def _observable(s):
    """Smooth weight of the observable sum_j w_j rho_j h^3 on the grid nodes."""
    H, L = s["H"], s["L"]
    j = torch.arange(H, device="cuda", dtype=torch.float64)
    x2 = (torch.where(j < H / 2, j, j - H) * (L / H) / (0.15 * L)) ** 2
    return (L / H) ** 3 * torch.exp(-0.5 * (x2[:, None, None] + x2[None, :, None] + x2[None, None, :]))


# ------------------------------------------------------------------ one pass
def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "step":
        sim, x = st["sim"], st["x"]
        st["stream"].wait_stream(torch.cuda.current_stream())   # whoever reads x is done with it
        sim.step(case["steps"])
        sim.positions_dev(x[0].data_ptr(), x[1].data_ptr(), x[2].data_ptr())
        torch.cuda.current_stream().wait_stream(st["stream"])
        if not case.get("diagnostics"):
            return {"positions": x}
        R = np.float64 if case["precision"] == 64 else np.float32
        return {"positions": x, **{k: R(v) for k, v in sim.diagnostics().items() if k != "step"}}
    if kind == "host":
        sim, src, dst = st["sim"], st["src"], st["dst"]
        _abi.sipf_upload_soa(sim.ctx, src[0].data_ptr(), src[1].data_ptr(), src[2].data_ptr())
        sim.step(1)
        _abi.sipf_download_soa(sim.ctx, dst[0].data_ptr(), dst[1].data_ptr(), dst[2].data_ptr())
        sim.sync()
        return {"positions": dst}
    if kind == "batch":
        batch = st["batch"]
        batch.step(case["steps"])
        R = np.float64 if case["precision"] == 64 else np.float32
        return [batch.positions(r).astype(R) for r in range(len(batch))]
    if kind == "adjoint":
        X0 = st["X0"].detach().requires_grad_(True)
        chi, mu = st["chi"].clone().requires_grad_(True), st["mu"].clone().requires_grad_(True)
        rho = SipfDensity.apply(X0, chi, mu, st["engine"])
        (rho * st["weight"]).sum().backward()
        return {"rho": rho.detach().to(X0.dtype), "X0": X0.grad, "chi": chi.grad, "mu": mu.grad}
    if kind == "plane":
        sim = st["sim"]
        sim.step(case["steps"])
        X = sim.positions()
        return {"positions": X if case["precision"] == 64 else X.astype(np.float32)}
    P, H, prec = case["P"], case["H"], case["precision"]
    x, grid, field, values = st["x"], st["grid"], st["field"], st["values"]
    s = torch.cuda.current_stream().cuda_stream
    _abi.sipf_deposit_dev(prec, x[0].data_ptr(), x[1].data_ptr(), x[2].data_ptr(), P, H, 1.0, 10.0 / P, 4, grid.data_ptr(), s)
    _abi.sipf_forward_ft_dev(prec, H, 1.0, grid.data_ptr(), st["spec"].data_ptr(), s)
    for c in range(case["comps"]):
        spec = st["spec"] * st["green"] ** (c + 1)
        _abi.sipf_inverse_ft_dev(prec, H, spec.data_ptr(), field[c].data_ptr(), s)
    _abi.sipf_gather_dev(prec, x[0].data_ptr(), x[1].data_ptr(), x[2].data_ptr(), P, H, 1.0, field.data_ptr(), case["comps"], 2,
                         values.data_ptr(), s)
    return {"grid": grid, "spectrum": st["spec"], "field": field, "values": values}


def work(case):
    """Bytes and operations of one pass: positions and spectrum read and written once per step, transforms as
    5 N log2 N (half for real data), 10 operations a stencil node and particle, about 60 for the noise."""
    kind, esz = case["kind"], case["precision"] // 8

    def grid_flops(H, transforms):
        return transforms * 2.5 * H ** 3 * 3 * math.log2(H)

    def step_work(P, H):
        spectrum = H * H * (H // 2 + 1) * 2
        return esz * (6 * P + 2 * spectrum), P * (40 * 10 + 60) + grid_flops(H, 4)

    if kind == "plane":
        P, H = case["P"], case["H"]
        return {"bytes": case["steps"] * esz * (4 * P + H * (H + 2)) + 16 * P,
                "flops": case["steps"] * (P * (16 * 10 + 40) + 3 * 2.5 * H * H * 2 * math.log2(H))}
    if kind == "operators":
        P, H, C = case["P"], case["H"], case["comps"]
        N = H ** 3
        return {"bytes": esz * (2 * 3 * P + C * P + (2 + C) * N + (2 + 2 * C) * N), "flops": P * (320 + 16 * C) + grid_flops(H, 1 + C)}
    if kind == "batch":
        P = (case["P_max"] - case["P_min"]) / math.log(case["P_max"] / case["P_min"])   # mean of the log-uniform sizes
        b, f = 0.0, 0.0
        for H in (32, 64):
            w = step_work(P, H)
            b, f = b + case["runs"] / 2 * w[0], f + case["runs"] / 2 * w[1]
        return {"bytes": case["steps"] * b + case["runs"] * P * 24, "flops": case["steps"] * f}
    b, f = step_work(case["P"], case["H"])
    if kind == "adjoint":   # a forward and a reverse step of about twice its work
        return {"bytes": 3 * case["steps"] * b + 48 * case["P"], "flops": 3 * case["steps"] * f}
    if kind == "host":
        return {"bytes": b + 6 * esz * case["P"], "flops": f}
    return {"bytes": case["steps"] * b + 3 * esz * case["P"], "flops": case["steps"] * f}


# ------------------------------------------------------------------ the same in 64 bits
def _philox(seed, n, P, block):
    """Philox4x32-10 of counters (p, 0, n, block), key = seed: four words in [0, 2^32) as int64 tensors."""
    m32 = 0xFFFFFFFF
    c = [torch.arange(P, device="cuda"), *(torch.full((P,), v, device="cuda", dtype=torch.int64) for v in (0, n, block))]
    k0, k1 = seed & m32, (seed >> 32) & m32

    def mulhilo(a, m):   # 32 x 32 -> (high, low), in 16-bit pieces so that nothing passes 2^63
        lo, hi = a * (m & 0xFFFF), a * (m >> 16)
        s = lo + ((hi & 0xFFFF) << 16)
        return (hi >> 16) + (s >> 32), s & m32

    for _ in range(10):
        h0, l0 = mulhilo(c[0], 0xD2511F53)
        h1, l1 = mulhilo(c[2], 0xCD9E8D57)
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return c


def _normals(seed, n, P, count):
    words = _philox(seed, n, P, 0) + (_philox(seed, n, P, 1) if count > 4 else [])
    z = []
    for j in range(count // 2):
        u, v = ((w.double() + 0.5) * 2.0 ** -32 for w in words[2 * j:2 * j + 2])
        r = torch.sqrt(-2.0 * torch.log(u))
        z += [r * torch.cos(TWO_PI * v), r * torch.sin(TWO_PI * v)]
    return z


def _stencil(X, H, L, order):
    """(flat node indices, weights) of every node of the 2- or 4-point stencils of positions X (P, d)."""
    d = X.shape[1]
    u = X * (H / L)
    cell = torch.floor(u.detach())
    lam = u - cell
    cell = cell.long()
    lin = [[1.0 - lam[:, a], lam[:, a]] for a in range(d)]
    bump = [lam[:, a] * (1.0 - lam[:, a]) for a in range(d)]

    def index(off):
        i = torch.zeros_like(cell[:, 0])
        for a in range(d):
            i = i * H + (cell[:, a] + off[a]) % H
        return i

    def product(off, skip=None):
        w = torch.ones_like(lam[:, 0])
        for a in range(d):
            if a != skip:
                w = w * lin[a][off[a]]
        return w

    for m in range(2 ** d):
        off = [(m >> a) & 1 for a in range(d)]
        w = product(off)
        yield index(off), w if order == 2 else w * (1.0 + 0.5 * sum(bump))
        if order == 4:
            for a in range(d):   # the node beyond off on axis a: index -1 for 0, 2 for 1
                far = list(off)
                far[a] = -1 if off[a] == 0 else 2
                cubic = -((2.0 - lam[:, a]) if off[a] == 0 else (1.0 + lam[:, a])) * bump[a] / 6.0
                yield index(far), cubic * product(off, skip=a)


def _deposit(X, w, H, L, order=4):
    phi = torch.zeros(H ** X.shape[1], dtype=torch.float64, device="cuda")
    for i, f in _stencil(X, H, L, order):
        phi = phi.index_add(0, i, f * w)
    return phi.reshape((H,) * X.shape[1])


def _gather(fields, X, H, L, order=2):
    out = [0.0] * len(fields)
    for i, f in _stencil(X, H, L, order):
        out = [o + f * g.reshape(-1)[i] for o, g in zip(out, fields)]
    return out


def _modes(H, d):
    """Integer modes of the half spectrum per axis (q in [-H/2, H/2)) and |q|^2."""
    full = torch.fft.fftfreq(H, 1.0 / H, device="cuda", dtype=torch.float64).round()
    half = torch.arange(H // 2 + 1, device="cuda", dtype=torch.float64)
    half[-1] = -H // 2
    axes = [full] * (d - 1) + [half]
    q = [axes[a].reshape([-1 if b == a else 1 for b in range(d)]) for a in range(d)]
    return q, sum(v ** 2 for v in q)


def _filter_scale(H, L):
    return math.ceil(8.0 * H ** (8.0 / 13.0) * L ** (5.0 / 13.0) - 1e-9)


class _Exact:
    """Algorithm 4 (or its plane form) for one run in 64 bits."""

    def __init__(self, s, d):
        self.s, self.d = s, d
        self.q, self.q2 = _modes(s["H"], d)
        self.phi_hat = torch.exp(-2.0 * math.pi ** 2 / _filter_scale(s["H"], s["L"]) ** 2 * self.q2)

    def forward(self, grid):
        return torch.fft.rfftn(grid) / self.s["L"] ** self.d

    def inverse(self, spec):
        return torch.fft.irfftn(spec, s=(self.s["H"],) * self.d, norm="forward")

    def step(self, X, alpha, n, chi=None, mu=None):
        s, H, L, tau = self.s, self.s["H"], self.s["L"], self.s["dt"]
        chi, mu = s["chi"] if chi is None else chi, s["mu"] if mu is None else mu
        beta = self.forward(_deposit(X, s["mass"] / s["P"], H, L))
        lam = (TWO_PI / L) ** 2 * self.q2 + s["k"] ** 2
        if s["eps"] == 0.0:
            new = torch.where(lam > 0, beta / lam.clamp(min=1e-300), torch.zeros_like(beta))
            drive = new
        else:
            new = alpha / (1.0 + tau / s["eps"] * lam) + beta / (lam + s["eps"] / tau)
            drive = alpha
        grads = [self.inverse(torch.where(q == -H // 2, torch.zeros_like(drive), 1j * (TWO_PI / L) * q * self.phi_hat * drive))
                 for q in self.q]
        z = torch.stack(_normals(s["seed"], n, s["P"], 2 * self.d), dim=1)
        amp = (mu * tau) ** 0.5 if not s.get("plain") else (2.0 * mu * tau) ** 0.5
        Y = X if s.get("plain") else X + amp * z[:, :self.d]
        noise = z[:, :self.d] if s.get("plain") else z[:, self.d:]
        Z = Y + chi * tau * torch.stack(_gather(grads, Y, H, L), dim=1) + amp * noise
        return Z - L * torch.floor(Z.detach() / L + 0.5), new

    def alpha0(self):
        H = self.s["H"]
        return torch.zeros((H,) * (self.d - 1) + (H // 2 + 1,), dtype=torch.complex128, device="cuda")

    def run(self, X, steps):
        alpha = self.alpha0()
        for n in range(1, steps + 1):
            X, alpha = self.step(X, alpha, n)
        return X, alpha

    def diagnostics(self, X, alpha):
        s = self.s
        phi = _deposit(X, s["mass"] / s["P"], s["H"], s["L"])
        energy = alpha.abs() ** 2 * torch.where((self.q[-1] == 0) | (self.q[-1] == -s["H"] // 2), 1.0, 2.0)
        return {"mass": float(phi.sum()), "alpha0": float(alpha.reshape(-1)[0].real),
                "peak": float(self.inverse(self.phi_hat * self.forward(phi)).max()),
                "hf_frac": float(energy[self.q2 >= 16].sum() / energy.sum()), "m2": float((X ** 2).sum(1).mean()),
                "ring_radius": float((X[:, 0] ** 2 + X[:, 1] ** 2).sqrt().mean())}


def exact(case, seed):
    kind = case["kind"]
    if kind == "operators":
        X, green = _operator_inputs(case, seed)
        H = case["H"]
        grid = _deposit(X, 10.0 / case["P"], H, 1.0)
        spec = torch.fft.rfftn(grid)
        field = torch.stack([torch.fft.irfftn(spec * green ** (c + 1), s=(H,) * 3, norm="forward") for c in range(case["comps"])])
        return {"grid": grid, "spectrum": spec, "field": field, "values": torch.stack(_gather(field, X, H, 1.0))}
    if kind == "batch":   # the first two runs, one of each grid size
        runs = _ensemble(case, seed)
        X = _ensemble_positions(runs, seed)
        return [_Exact(s, 3).run(X[i], case["steps"])[0] if i < 2 else None for i, s in enumerate(runs)]
    if kind == "plane":
        s, X = _plane(case, seed)
        return {"positions": _Exact(s, 2).run(X, case["steps"])[0]}
    s = _system(case, seed)
    X = _sample(s["shape"], s["P"], s["L"], s["sigma"], s["precision"], _generator(seed))
    E = _Exact(s, 3)
    if kind == "adjoint":
        from torch.utils.checkpoint import checkpoint
        X0 = X.clone().requires_grad_(True)
        chi, mu = (torch.tensor(s[k], dtype=torch.float64, device="cuda", requires_grad=True) for k in ("chi", "mu"))
        Xn, alpha = X0, E.alpha0()
        for n in range(1, case["steps"] + 1):
            Xn, alpha = checkpoint(E.step, Xn, alpha, n, chi, mu, use_reentrant=False)
        rho = _deposit(Xn, s["mass"] / s["P"], s["H"], s["L"]) / (s["L"] / s["H"]) ** 3
        (rho * _observable(s)).sum().backward()
        return {"rho": rho.detach(), "X0": X0.grad, "chi": chi.grad, "mu": mu.grad}
    X, alpha = E.run(X, 1 if kind == "host" else case["steps"])
    out = {"positions": X.t().contiguous()}
    if case.get("diagnostics"):
        out.update(E.diagnostics(X, alpha))
    return out
