"""What the performance of this framework is measured on.

Every case is work that a user of the library has it do through
``paper_1603_08221_gb300.binding`` (or ``autograd``, ``diagnostics``): time
steps of one channel from the smallest to the largest, in every storage type
and with the options in use, monitored and steady-state runs, parametric
sweeps, moment fields, and gradients by the adjoint.  The sizes are those of
``workloads.PRESETS``, of the paper's 20 x 700 lattice, of the parametric
study, and odd ones beside them.

``exact`` restates the method in 64 bits with plain torch operations (the
lattice Boltzmann step of Sec. 3 of arXiv:1603.08221 on full populations, its
gradients by torch's own reverse mode), independently of the library.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.utils.checkpoint

from paper_1603_08221_gb300 import autograd, binding, diagnostics, workloads

HE, NE, AR = workloads.HE, workloads.NE, workloads.AR


# ------------------------------------------------------------------- cases
def listed():
    return [
        # README use: a He-Ar 320 x 16 channel with the default parameters
        # (a diagnostic record every step), watched every few steps the way
        # CL(t) histories are taken.  The smallest calls.
        dict(name="monitor_320x16", kind="monitor", m_a=HE, m_b=AR, N=16, N_x=320, theta=2.0,
             Kn_out=0.1, C_l=0.5, steps=100, every=10),
        # One run of the paper's Table 1 on its own lattice, advanced to a
        # steady residual in check blocks (default diag_every).
        dict(name="steady_700x20", kind="steady", m_a=HE, m_b=AR, N=20, N_x=700, theta=2.0,
             Kn_out=0.3, C_l=0.5, steps=400, every=200, diag_every=1),
        # The sensitivity workload's channel stepped in FP32: a lone channel
        # of middle size.
        dict(name="step_1280x64", kind="step", m_a=HE, m_b=AR, N=64, N_x=1280, theta=2.0,
             Kn_out=0.2, C_l=0.5, steps=100, diag_every=100),
        # A ragged channel (37 rows, 1001 columns) under the bounce-back /
        # specular wall and the other readings of Eq. R and lambda_sigma.
        dict(name="bsr_1001x37", kind="step", m_a=HE, m_b=AR, N=37, N_x=1001, theta=1.5,
             Kn_out=0.25, C_l=0.4, steps=60, diag_every=20, wall=1, r_form=1,
             lambda_pressure=1),
        # The throughput workload: FP32 storage, larger than the caches.
        dict(name="step_32768x512", kind="step", m_a=NE, m_b=AR, N=512, N_x=32768, theta=3.0,
             Kn_out=0.05, C_l=0.3, steps=4, diag_every=100),
        # The reduced-precision workload: BF16 storage, stochastic rounding.
        dict(name="bf16_16384x256", kind="step", m_a=NE, m_b=AR, N=256, N_x=16384, theta=2.5,
             Kn_out=0.5, C_l=0.5, steps=8, diag_every=100, storage=1),
        # FP16 storage rounded to nearest on a ragged channel of middle size.
        dict(name="fp16_5001x130", kind="step", m_a=NE, m_b=AR, N=130, N_x=5001, theta=2.0,
             Kn_out=0.2, C_l=0.5, steps=20, diag_every=20, storage=2, rounding=1),
        # The paper's whole Table 1: 52 channels of 700 x 20 as one sweep.
        dict(name="table1_sweep", kind="table1", N=20, L_over_H=35, steps=200, every=100),
        # A parametric study over mixed gases and sizes (N = 16 ... 128,
        # L/H = 10 ... 50).
        dict(name="mixed_sweep", kind="sweep", n=24, N_max=128, steps=100, every=50),
        # Forward run and gradient of CL on the sensitivity workload, every
        # step kept.
        dict(name="adjoint_1280x64", kind="adjoint", m_a=HE, m_b=AR, N=64, N_x=1280, theta=2.0,
             Kn_out=0.2, C_l=0.5, steps=60, keep=60),
        # The torch.autograd path as an optimisation loop calls it: a small
        # channel, its default checkpointing, the outlet flux.
        dict(name="autograd_320x16", kind="autograd", m_a=HE, m_b=AR, N=16, N_x=320, theta=2.0,
             Kn_out=0.1, C_l=0.5, steps=150, keep=70),
        # Fields on the device and the outlet volume flow after a few steps,
        # as a visualisation or a coupling to another code reads them.
        dict(name="fields_16384x256", kind="fields", m_a=NE, m_b=AR, N=256, N_x=16384,
             theta=2.5, Kn_out=0.5, C_l=0.5, steps=2, diag_every=100),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["monitor", "steady", "step", "step", "step16", "step16", "table1", "sweep",
                       "adjoint", "autograd", "fields"])
    gas = rng.choice([HE, NE])
    c = dict(m_a=gas, m_b=AR, theta=round(rng.uniform(1.2, 2.5), 3),
             Kn_out=round(_log(rng, 0.1, 1.0), 4), C_l=rng.choice([0.3, 0.5, 0.7]))

    def channel(n_lo, n_hi, most):
        n = int(_log(rng, n_lo, n_hi))
        nx = int(n * rng.uniform(15.0, 64.0)) + rng.randrange(3)
        return n, max(64, min(nx, most // n))

    if kind == "monitor":
        n, nx = channel(10, 48, 60_000)
        every = rng.choice([5, 10, 25])
        return dict(c, kind=kind, N=n, N_x=nx, steps=4 * every, every=every)
    if kind == "steady":
        n, nx = channel(10, 96, 300_000)
        return dict(c, kind=kind, N=n, N_x=nx, steps=200, every=100,
                    diag_every=rng.choice([1, 100]))
    if kind in ("step", "step16"):
        n, nx = channel(12, 512, 8_000_000) if kind == "step" else channel(32, 512, 12_000_000)
        steps = 2 * max(2, min(40, int(1.2e7 / (n * nx))))
        c = dict(c, kind="step", N=n, N_x=nx, steps=steps, diag_every=rng.choice([1, 20, 100]))
        if kind == "step16":
            return dict(c, storage=rng.choice([1, 2]), rounding=rng.choice([0, 0, 1]))
        if rng.random() < 0.3:
            c.update(wall=1, r_form=rng.randrange(3), lambda_pressure=rng.randrange(2))
        elif rng.random() < 0.2:
            c.update(x_periodic=1)
        return c
    if kind == "table1":
        return dict(kind=kind, N=rng.randrange(16, 33), L_over_H=rng.randrange(25, 46),
                    steps=100, every=50)
    if kind == "sweep":
        return dict(kind=kind, n=rng.randrange(8, 33), N_max=rng.choice([32, 64]), steps=100,
                    every=50, pick=rng.randrange(1000))
    if kind == "adjoint":
        n, nx = channel(16, 64, 80_000)
        steps = rng.randrange(30, 60)
        return dict(c, kind=kind, N=n, N_x=nx, steps=steps, keep=rng.choice([steps, 20]))
    if kind == "autograd":
        n, nx = channel(10, 24, 12_000)
        return dict(c, kind=kind, N=n, N_x=nx, steps=rng.randrange(60, 150), keep=70)
    n, nx = channel(32, 300, 4_000_000)
    return dict(c, kind="fields", N=n, N_x=nx, steps=2, diag_every=100)


_STREAMS: list = []


def _stream():
    if not _STREAMS:
        _STREAMS.append(torch.cuda.Stream())
    return _STREAMS[0]


_PARAMS = ("m_a", "m_b", "theta", "Kn_out", "C_l", "C_l_out", "N", "N_x", "storage", "rounding",
           "wall", "r_form", "lambda_pressure", "x_periodic", "diag_every")


def _params(case):
    return {k: case[k] for k in _PARAMS if k in case}


def _sweep_params(case, seed):
    """The channels of a sweep case: sizes and gases from the case alone (the
    study's own lists), pressure ratios, Knudsen numbers and end compositions
    around the study's from the seed."""
    rng = np.random.default_rng(seed)
    out = []
    if case["kind"] == "table1":
        for _, p in workloads.paper_table1(case["N"], float(case["L_over_H"])):
            p = dict(p)
            p["theta"] *= 1.0 + 0.02 * rng.random()
            p["Kn_out"] *= 1.0 + 0.1 * rng.random()
            out.append(p)
        return out
    sizes = np.random.default_rng(case.get("pick", 0))
    rows = [n for n in (16, 32, 64, 128) if n <= case["N_max"]]
    for k in range(case["n"]):
        out.append(dict(m_a=HE if k % 2 == 0 else NE, m_b=AR, C_l=(0.1, 0.3, 0.5, 0.7, 0.9)[k % 5],
                        N=int(sizes.choice(rows)), L_over_H=float(sizes.choice([10.0, 20.0, 50.0])),
                        theta=float(rng.uniform(1.5, 3.0)), Kn_out=float(10.0 ** rng.uniform(-1, 0))))
    return out


def _alpha(case, seed):
    """A wall accommodation field 1 - U(0, 0.05), bottom wall then top."""
    return workloads.random_accommodation(case["N_x"], seed=seed, spread=0.05)


def _constants(p):
    """Masses, mole fractions and rest weights shared by the inputs and the
    64-bit restatement (masses in units of the lighter one)."""
    m_min = min(p["m_a"], p["m_b"])
    mh = (p["m_a"] / m_min, p["m_b"] / m_min)
    light = 0 if p["m_a"] <= p["m_b"] else 1
    c_in = p["C_l"]
    c_out = p.get("C_l_out", -1.0)
    c_out = c_in if c_out < 0 else c_out
    w = [[(9 - 5 / m) / 9] + [1 / m / 9] * 4 + [1 / m / 36] * 4 for m in mh]
    return mh, light, c_in, c_out, w


def _rest_density(p, nx, device):
    """Species densities [2][N_x] of the linear initial profile."""
    mh, light, c_in, c_out, _ = _constants(p)
    t = torch.arange(nx, dtype=torch.float64, device=device) / (nx - 1)
    if p.get("x_periodic"):
        t = torch.ones_like(t)
    n = p["theta"] + (1.0 - p["theta"]) * t if not p.get("x_periodic") else torch.ones_like(t)
    cl = c_in + (c_out - c_in) * t
    c = [cl, 1 - cl] if light == 0 else [1 - cl, cl]
    return torch.stack([n * c[s] * mh[s] for s in range(2)])


def _developed_state(case, seed):
    """Populations [2][9][N][N_x] (FP32, host) of a flow under way: the linear
    density profile bent and rippled by a few per cent, a parabolic velocity
    with slip, and non-equilibrium parts of 1e-4, all from the seed."""
    dev = "cuda"
    g = torch.Generator(device=dev).manual_seed(seed)
    N, nx = case["N"], case["N_x"]
    mh, _, _, _, w = _constants(case)

    def rand(*shape):
        return torch.rand(*shape, generator=g, device=dev, dtype=torch.float32)

    a = rand(8)
    x = torch.arange(nx, device=dev, dtype=torch.float32) / nx
    y = (torch.arange(N, device=dev, dtype=torch.float32) + 0.5) / N
    rho0 = _rest_density(case, nx, dev).float()
    wave = 2 * math.pi
    ux = (0.01 + 0.005 * a[0]) * (4 * y * (1 - y) + 0.3)[:, None] * (1 + 0.1 * torch.sin(wave * (x + a[1])))
    uy = 1e-4 * torch.sin(wave * (y[:, None] + a[2])) * torch.cos(wave * (x + a[3]))
    usq = ux * ux + uy * uy
    cx, cy = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)
    lam = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
    f = np.empty((2, 9, N, nx), dtype=np.float32)
    for s in range(2):
        rho = rho0[s] * (1 + 0.03 * torch.sin(wave * (x / 2 + a[4 + s])) +
                         2e-3 * torch.sin(wave * (y[:, None] + 3 * x + a[6 + s])))
        for i in range(9):
            cu = cx[i] * ux + cy[i] * uy
            feq = rho * (w[s][i] + lam[i] * (3 * cu + 4.5 * cu * cu - 1.5 * usq))
            f[s, i] = (feq * (1 + 1e-4 * (rand(N, nx) - 0.5))).cpu().numpy()
    return f


# --------------------------------------------------------------- prepare, run
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("table1", "sweep"):
        sweep = binding.LbmSweep(_sweep_params(case, seed))
        sweep.init()
        return dict(case=case, sweep=sweep)
    alpha = _alpha(case, seed)
    if kind == "adjoint":
        return dict(case=case, adj=binding.LbmAdjoint(_params(case), case["steps"], case["keep"],
                                                      alpha=alpha))
    if kind == "autograd":
        t = dict(theta=torch.tensor(case["theta"], dtype=torch.float64, requires_grad=True),
                 kn=torch.tensor(case["Kn_out"], dtype=torch.float64, requires_grad=True),
                 alpha=torch.tensor(alpha.reshape(2, -1), requires_grad=True))
        return dict(case=case, **t)
    # the channel steps on the program's torch stream, so that the state can
    # be read through zero-copy views: one channel at a time, its calls in order
    stream = _stream()
    sim = binding.LbmMix(stream=stream, **_params(case))
    sim.set_accommodation_field(alpha)
    sim.set_post_state(_developed_state(case, seed))
    state = dict(case=case, sim=sim, stream=stream)
    if kind == "fields":
        state["out"] = torch.empty((6, case["N"], case["N_x"]), dtype=torch.float64, device="cuda")
    return state


def _populations(sim, owner=None):
    """The stored state, viewed in place.  The view keeps the library object
    that owns the memory alive (torch holds on to the array it views)."""
    array = sim.device_views()["populations"]
    array.owner = owner or sim
    v = torch.as_tensor(array, device="cuda")
    return v.view(torch.bfloat16) if sim.params.storage == binding.LBM_BF16 else v


# Diagnostics and moments of a channel are reported in FP64 but computed from
# an FP32 (or 16-bit) state in FP32 arithmetic: they come back as FP32 values.
def _f32(v):
    return np.asarray(v, dtype=np.float32)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("table1", "sweep"):
        sweep = state["sweep"]
        _, residual, _ = sweep.run_to_steady(1e-14, case["steps"], case["every"])
        return dict(residual=_f32(residual),
                    populations=[_populations(sweep.instance(k), sweep) for k in range(sweep.n)])
    if kind == "adjoint":
        cl, flux = state["adj"].forward()
        return dict(CL=cl, flux=flux, **state["adj"].gradient(binding.LBM_ADJ_CL))
    if kind == "autograd":
        j = autograd.channel_objective(state["theta"], state["kn"], state["alpha"], _params(case),
                                       case["steps"], case["keep"], binding.LBM_ADJ_FLUX)
        grads = torch.autograd.grad(j, (state["theta"], state["kn"], state["alpha"]))
        return dict(flux=j.detach(), theta=grads[0], Kn_out=grads[1], alpha=grads[2])
    sim = state["sim"]
    with torch.cuda.stream(state["stream"]):
        if kind == "monitor":
            _, cl, ct, qv = diagnostics.separation_history(sim, case["steps"], case["every"])
            return dict(CL=_f32(cl), Cl_tilde=_f32(ct), Q_v=_f32(qv), populations=_populations(sim))
        if kind == "steady":
            _, _, residual = sim.run_to_steady(1e-14, case["steps"], case["every"])
            s = sim.separation()
            return dict(residual=_f32([residual]), Cl_profile=_f32(s["Cl_profile"]),
                        mdot=_f32([s["mdot_a"], s["mdot_b"]]), populations=_populations(sim))
        if kind == "fields":
            sim.step(case["steps"])
            binding.lbm_mix_moments_device(sim.h, state["out"].data_ptr())
            q = sim.volume_flow()
            return dict(moments=state["out"].float(), Q_v=_f32([q]))
        sim.step(case["steps"])
        sums = torch.as_tensor(sim.device_views()["colsum"], device="cuda")
        return dict(colsum=sums.float(), populations=_populations(sim))


# ---------------------------------------------------------------------- work
#: floating-point operations of one node's step (both species: moments, six
#: evaluations of psi, equilibria and collision), of the FP64 forward step and
#: of its reverse
NODE_FLOPS, ADJ_FLOPS = 450, 1500


def work(case):
    """State (or field) in and out once, and the arithmetic of every step."""
    kind = case["kind"]
    if kind in ("table1", "sweep"):
        nodes = sum(p["N"] * workloads.n_x(p) for p in _sweep_params(case, 0))
    else:
        nodes = case["N"] * case["N_x"]
    elem = 2 if case.get("storage") else 4
    if kind in ("adjoint", "autograd"):
        # the accommodation field in, its gradient out
        return {"bytes": 8.0 * 4 * case["N_x"], "flops": float(ADJ_FLOPS) * nodes * case["steps"]}
    nbytes = 2.0 * 18 * elem * nodes
    if kind == "fields":
        nbytes += 6 * 8 * nodes
    return {"bytes": nbytes, "flops": float(NODE_FLOPS) * nodes * case["steps"]}


# --------------------------------------------------------- the method in 64 bits
CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
M = torch.tensor([
    [1, 1, 1, 1, 1, 1, 1, 1, 1], [-4, -1, -1, -1, -1, 2, 2, 2, 2], [4, -2, -2, -2, -2, 1, 1, 1, 1],
    [0, 1, 0, -1, 0, 1, -1, -1, 1], [0, -2, 0, 2, 0, 1, -1, -1, 1], [0, 0, 1, 0, -1, 1, 1, -1, -1],
    [0, 0, -2, 0, 2, 1, 1, -1, -1], [0, 1, -1, 1, -1, 0, 0, 0, 0], [0, 0, 0, 0, 0, 1, -1, 1, -1],
], dtype=torch.float64)


def _e1(a):
    """E_1(a), a > 0: the convergent series up to 2, the continued fraction
    (evaluated from its 40th term) beyond."""
    lo = a.clamp(max=2.0)
    term, total = torch.ones_like(lo), torch.zeros_like(lo)
    for k in range(1, 32):
        term = term * (-lo / k)
        total = total - term / k
    small = -0.57721566490153286061 - torch.log(lo) + total
    hi = a.clamp(min=2.0)
    t = hi + 81.0
    for k in range(40, 0, -1):
        t = hi + (2 * k - 1) - k * k / t
    return torch.where(a <= 2.0, small, torch.exp(-hi) / t)


class _Psi(torch.autograd.Function):
    """psi(a) = 1 + (a - 1) e^-a - a^2 E_1(a) and psi'(a) = 2 e^-a - 2 a E_1(a)."""

    @staticmethod
    def forward(ctx, a):
        e, x = _e1(a), torch.exp(-a)
        d = 2 * x - 2 * a * e
        ctx.save_for_backward(d, e)
        return 1 + (a - 1) * x - a * a * e, d

    @staticmethod
    def backward(ctx, g, gd):
        d, e = ctx.saved_tensors
        return g * d - 2 * gd * e


class _Model:
    """One channel: step(f, alpha) on full populations [2][9][N][N_x]."""

    def __init__(self, p, nx, theta=None, kn=None, device="cuda"):
        self.p, self.N, self.nx = p, p["N"], nx
        self.mh, self.light, self.c_in, c_out, w = _constants(p)
        self.w = torch.tensor(w, dtype=torch.float64, device=device)[:, :, None, None]
        self.M = M.to(device)
        self.norm = (self.M * self.M).sum(1)
        self.periodic = p.get("x_periodic", 0)
        self.theta = p["theta"] if theta is None else theta
        kn = p["Kn_out"] if kn is None else kn
        ci = (self.c_in, 1 - self.c_in) if self.light == 0 else (1 - self.c_in, self.c_in)
        co = (c_out, 1 - c_out) if self.light == 0 else (1 - c_out, c_out)
        self.s = [1 / m for m in self.mh]
        self.rho_in = [self.theta * ci[k] * self.mh[k] for k in range(2)]
        self.rho_out = [co[k] * self.mh[k] for k in range(2)]
        mx_out = co[0] * self.mh[0] + co[1] * self.mh[1]
        # lambda = (mu/p) sqrt(pi k_B T / (2 m)) with k_B T = 1/3, p = n/3
        self.mu = kn * self.N / 3 / math.sqrt(math.pi / (6 * mx_out))
        self.y = torch.arange(self.N, dtype=torch.float64, device=device)[:, None] + 0.5
        half = (self.N + 1) // 2
        self.bottom = (torch.arange(self.N, device=device) < half)[:, None]

    def initial(self):
        """Rest equilibrium of the linear profiles, differentiable in theta."""
        dev = self.w.device
        t = torch.arange(self.nx, dtype=torch.float64, device=dev) / (self.nx - 1)
        c_out = self.rho_out[self.light] / self.mh[self.light]
        cl = self.c_in + (c_out - self.c_in) * t
        n = self.theta + (1 - self.theta) * t
        c = [cl, 1 - cl] if self.light == 0 else [1 - cl, cl]
        rho = torch.stack([n * c[k] * self.mh[k] for k in range(2)])
        return self.w * rho[:, None, None, :].expand(2, 9, self.N, self.nx)

    def mean_free_path(self, n, m):
        return 3 * self.mu * math.sqrt(math.pi / 6) / (n * torch.sqrt(m))

    def confined(self, lam):
        """lambda_e / lambda at every row."""
        return 0.5 * (_Psi.apply(self.y / lam)[0] + _Psi.apply((self.N - self.y) / lam)[0])

    def slip(self, f, wall, alpha):
        """r of Eq. R (bounce-back fraction under the BSR wall), per species."""
        row = 0 if wall == 0 else self.N - 1
        rho = f[:, :, row].sum(1)
        mx = (rho[0] + rho[1]) / (self.s[0] * rho[0] + self.s[1] * rho[1])
        form = self.p.get("r_form", 0)
        x0 = self.p.get("c_m0", 1.016) * (2 - alpha[wall]) / alpha[wall] * torch.sqrt(math.pi * mx / 6)
        if form == 2:
            x0 = x0 * torch.sqrt(mx)
        out = []
        for k in range(2):
            X = x0 if form == 0 else x0 / math.sqrt(self.mh[k])
            out.append(1 / (1 + X) if self.p.get("wall") else 2 - 2 / (1 + X))
        return torch.stack(out)

    def pull(self, f, alpha):
        """Pre-collision populations of every column (the updated ones are
        used): streaming, the walls and the extrapolated ghost columns."""
        if not self.periodic:
            rho = f.sum((1, 2))
            cols = []
            for tgt, x1, x2 in ((self.rho_in, 1, 2), (self.rho_out, self.nx - 2, self.nx - 3)):
                k = torch.stack([self.N * tgt[s] / (2 * rho[s, x1] - rho[s, x2]) for s in range(2)])
                cols.append(k[:, None, None] * (2 * f[..., x1] - f[..., x2]))
            f = torch.cat([cols[0][..., None], f[..., 1:-1], cols[1][..., None]], -1)
        r = [self.slip(f, 0, alpha), self.slip(f, 1, alpha)]

        def shift(v, i):
            return torch.roll(v, CX[i], -1)

        g = [f[:, 0]]
        low, high = f[:, :, 0], f[:, :, -1]
        for i in range(1, 9):
            v = shift(f[:, i], i)
            if CY[i] == 0:
                g.append(v)
                continue
            up = CY[i] > 0
            edge, out, rr = (low, (4, 7, 8), r[0]) if up else (high, (2, 5, 6), r[1])
            opp = (0, 3, 4, 1, 2, 7, 8, 5, 6)[i]
            if self.p.get("wall"):
                mirror = (0, 1, 4, 3, 2, 8, 7, 6, 5)[i]
                b = edge[:, opp] if CX[i] == 0 else rr * edge[:, opp] + (1 - rr) * shift(edge[:, mirror], i)
            else:
                total = edge[:, out[0]] + edge[:, out[1]] + edge[:, out[2]]
                b = (1 - rr) * edge[:, opp] + rr * total * (2 / 3 if CX[i] == 0 else 1 / 6)
            b = b[:, None]
            g.append(torch.cat([b, v[:, :-1]], 1) if up else torch.cat([v[:, 1:], b], 1))
        return torch.stack(g, 1)

    def tau_q(self, g, wall, alpha):
        row = 0 if wall == 0 else self.N - 1
        rho = g[:, :, row].sum(1)
        n = self.s[0] * rho[0] + self.s[1] * rho[1]
        mx = (rho[0] + rho[1]) / n
        lam = self.mean_free_path(n, mx)
        c = torch.sqrt(6 / (math.pi * mx))
        psi, dpsi = _Psi.apply(self.N / lam)
        ts = 0.5 * lam * psi * c
        dts = 0.5 * c * (2 - dpsi)
        al = alpha[wall]
        a1 = (2 - al) / al * (1 - 0.1817 * al)
        a2 = 1 / math.pi + 0.5 * a1 * a1
        v = math.sqrt(math.pi / 6)
        return 0.5 + (3 + 24 * v * v * ts * ts * a2) / (16 * ts) + dts * (12 + 30 * ts * v * a1) / (16 * ts * ts)

    def rates(self, rho, n, mx):
        """1/tau_s and 1/tau_d of every node."""
        lam = self.mean_free_path(n, mx)
        om_s = 1 / (0.5 + lam * self.confined(lam) * torch.sqrt(6 / (math.pi * mx)))
        br = 0
        for k in range(2):
            xs = self.s[k] * rho[k] / n
            ls = self.mean_free_path(n if self.p.get("lambda_pressure") else self.s[k] * rho[k],
                                     torch.full_like(n, self.mh[k]))
            br = br + 1 / torch.sqrt(xs * ls * self.confined(ls))
        c_td = 1.5 * math.sqrt(3 * (self.mh[0] + self.mh[1]) * self.mh[0] * self.mh[1])
        return om_s, 1 / (0.5 + c_td / (mx * br * br))

    def step(self, f, alpha):
        g = self.pull(f, alpha)
        m = torch.einsum("ki,sijx->skjx", self.M, g)
        rho, jx, jy = m[:, 0], m[:, 3], m[:, 5]
        rt = rho[0] + rho[1]
        n = self.s[0] * rho[0] + self.s[1] * rho[1]
        ux, uy = (jx[0] + jx[1]) / rt, (jy[0] + jy[1]) / rt
        om_s, om_d = self.rates(rho, n, rt / n)
        om_q = torch.where(self.bottom, 1 / self.tau_q(g, 0, alpha), 1 / self.tau_q(g, 1, alpha))
        zero = torch.zeros_like(n)
        om = torch.stack([zero, zero + 1 / self.p.get("tau_e", 1.1), zero + 1 / self.p.get("tau_eps", 1.2),
                          om_d, om_q, om_d, om_q, om_s, om_s])
        u2 = ux * ux + uy * uy
        meq = torch.stack([rho[k] * torch.stack([zero + 1, 3 * u2 - 4 + 2 * self.s[k],
                                                 4 - 3 * self.s[k] - 3 * u2, ux, -ux, uy, -uy,
                                                 ux * ux - uy * uy, ux * uy]) for k in range(2)])
        d = om * (m - meq) / self.norm[:, None, None]
        new = g - torch.einsum("ki,skjx->sijx", self.M, d)
        self.momentum = jx - 0.5 * om_d * (jx - rho * ux)
        if self.periodic:
            return new
        return torch.cat([f[..., :1], new[..., 1:-1], f[..., -1:]], -1)

    def light_fraction(self, f):
        n = [self.s[k] * f[k].sum((0, 1)) for k in range(2)]
        return n[self.light] / (n[0] + n[1])


def _strips(f, ref, w):
    """Full populations -> deviations from the reference in the strip layout."""
    d = f - w * ref[:, None, None, :]
    n, nx = d.shape[2], d.shape[3]
    d = torch.nn.functional.pad(d, (0, -nx % 32))
    return d.reshape(2, 9, n, -1, 32).permute(3, 2, 1, 4, 0).reshape(-1)


def _reference(p, nx):
    """The stored deviations' reference densities and weights (FP32 values)."""
    ref = _rest_density(p, nx, "cuda").float().double()
    w = []
    for m in _constants(p)[0]:
        s = float(np.float32(1 / m))
        w.append([float(np.float32(v)) for v in ((9 - 5 * s) / 9,) + (s / 9,) * 4 + (s / 36,) * 4])
    return ref, torch.tensor(w, dtype=torch.float64, device="cuda")[:, :, None, None]


def _diagnostics(model, f):
    """CL, C~_l, C_l(x) and the mass flows of the state f of the last step."""
    nx = model.nx
    inside = slice(None) if model.periodic else slice(1, nx - 1)
    cl = model.light_fraction(f)
    mdot = model.momentum.sum(1)[:, inside].mean(1)
    prof = cl.clone()
    c_out = model.rho_out[model.light] / model.mh[model.light]
    if not model.periodic:
        prof[0], prof[-1] = model.c_in, c_out
    CL = (model.c_in - cl[inside].min()) / model.c_in
    return CL, (prof - model.c_in).sum() / (nx * model.c_in), prof, mdot


def _fields(model, f_prev, alpha):
    """Moment fields [6][N][N_x] of the state streamed from f_prev."""
    g = model.pull(f_prev, alpha)
    rho = g.sum(1)
    jx = torch.einsum("i,sijx->sjx", model.M[3], g)
    jy = torch.einsum("i,sijx->sjx", model.M[5], g)
    rt = rho[0] + rho[1]
    n = model.s[0] * rho[0] + model.s[1] * rho[1]
    _, om_d = model.rates(rho, n, rt / n)
    out = [rho[0], rho[1]]
    for k in range(2):
        for j in (jx, jy):
            u = (j[0] + j[1]) / rt
            out.append(((1 - om_d / 2) * j[k] + om_d / 2 * rho[k] * u) / rho[k])
    out = torch.stack(out)
    if not model.periodic:
        for tgt, x0, x1, x2 in ((model.rho_in, 0, 1, 2),
                                (model.rho_out, model.nx - 1, model.nx - 2, model.nx - 3)):
            v = 2 * out[..., x1] - out[..., x2]
            for k in range(2):
                v[k] = v[k] * (model.N * tgt[k] / v[k].sum())
            out[..., x0] = v
    return out


def _volume_flow(model, fields):
    x = 0 if model.periodic else model.nx - 2
    ra, rb, ua, ub = (fields[k, :, x] for k in (0, 1, 2, 4))
    return ((ra * ua + rb * ub) / (ra + rb)).sum()


def _column_sums(model, f):
    sums = torch.cat([f.sum((1, 2)), model.momentum.sum(1)])
    if not model.periodic:
        sums[:, 0] = sums[:, -1] = 0
    return sums


def _residual(old, new, k):
    return float(((new - old).norm() / (k * new.norm())).item())


def exact(case, seed):
    kind = case["kind"]
    if kind in ("adjoint", "autograd"):
        return _exact_gradient(case, seed)
    with torch.no_grad():
        if kind in ("table1", "sweep"):
            return _exact_sweep(case, seed)
        f = torch.from_numpy(_developed_state(case, seed)).cuda().double()
        ghosts = f[..., [0, -1]].clone()
        model = _Model(_params(case), case["N_x"])
        alpha = torch.as_tensor(_alpha(case, seed), device="cuda").reshape(2, -1)
        watch = case.get("every", case["steps"])
        rows, sums, res, prev = [], None, math.inf, f
        for t in range(1, case["steps"] + 1):
            prev, f = f, model.step(f, alpha)
            if kind in ("monitor", "steady") and t % watch == 0:
                d = _diagnostics(model, f)
                if kind == "monitor":
                    rows.append((d[0], d[1], _volume_flow(model, _fields(model, prev, alpha))))
                now = _column_sums(model, f)
                if sums is not None:
                    res = _residual(sums, now, watch)
                sums = now
        if kind == "fields":
            fields = _fields(model, prev, alpha)
            return dict(moments=fields, Q_v=_volume_flow(model, fields).reshape(1))
        # an even number of steps ends in the buffer of the upload, whose
        # boundary columns it leaves as they were
        assert case["steps"] % 2 == 0
        if not model.periodic:
            f[..., [0, -1]] = ghosts
        pops = _strips(f, *_reference(_params(case), case["N_x"]))
        if kind == "monitor":
            cl, ct, qv = (torch.stack([r[k] for r in rows]) for k in range(3))
            return dict(CL=cl, Cl_tilde=ct, Q_v=qv, populations=pops)
        if kind == "steady":
            return dict(residual=np.array([res]), Cl_profile=d[2], mdot=d[3], populations=pops)
        return dict(colsum=_column_sums(model, f), populations=pops)


def _exact_sweep(case, seed):
    """The first channels of a sweep (all of them would take too long)."""
    params = _sweep_params(case, seed)
    pops = []
    for p in params:
        nx = workloads.n_x(p)
        if len(pops) >= 6 or p["N"] * nx > 300_000:
            pops.append(None)
            continue
        model = _Model(p, nx)
        ref, w = _reference(p, nx)
        f = w * ref[:, None, None, :].expand(2, 9, p["N"], nx)  # at rest
        alpha = torch.ones(2, nx, dtype=torch.float64, device="cuda")
        for _ in range(case["steps"]):
            f = model.step(f, alpha)
        pops.append(_strips(f, ref, w))
    return dict(residual=None, populations=pops)


def _exact_gradient(case, seed):
    """Objective and gradients by torch's reverse mode through every step."""
    dev = "cuda"
    theta = torch.tensor(case["theta"], dtype=torch.float64, device=dev, requires_grad=True)
    kn = torch.tensor(case["Kn_out"], dtype=torch.float64, device=dev, requires_grad=True)
    alpha = torch.tensor(_alpha(case, seed).reshape(2, -1), device=dev, requires_grad=True)
    model = _Model(_params(case), case["N_x"], theta, kn)
    f = model.initial()

    def step(f, alpha, theta, kn):
        return _Model(_params(case), case["N_x"], theta, kn).step(f, alpha)

    for _ in range(case["steps"]):
        f = torch.utils.checkpoint.checkpoint(step, f, alpha, theta, kn, use_reentrant=False)
    cl = (model.c_in - model.light_fraction(f)[1:-1].min()) / model.c_in
    l = model.light
    flux = torch.einsum("i,ij->", model.M[3], f[l, :, :, -2])
    j = flux if case["kind"] == "autograd" else cl
    g = torch.autograd.grad(j, (theta, kn, alpha))
    out = dict(theta=g[0], Kn_out=g[1], alpha=g[2])
    if case["kind"] == "autograd":
        return dict(flux=flux.detach(), **out)
    return dict(CL=float(cl), flux=float(flux), theta=float(g[0]), Kn_out=float(g[1]),
                alpha=g[2])
