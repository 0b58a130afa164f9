"""Performance cases of the solver, through the calls a program makes.

Every case is one pass of a running program: load a state (a checkpoint, or
the previous parameter point's state), propagate a block of split steps,
evaluate the observables and read the state back; or the same for a batch of
condensates; or one training step of the learned start.  The states are
smooth vortex states in the middle of a run, drawn from the seed alone.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1906_06327_gb300 import inputs
from paper_1906_06327_gb300.rotgp import Batch, Solver, WarmStart

OBS = ("norm", "mu", "energy", "mu_c", "energy_c", "rms_x", "rms_y", "rms_z", "rms_r",
       "max_density", "mu4", "energy4")


def _steps(name, n, h, *, precision="fp32", mode="imag", steps, g, omega, dt, nu=1.0, lam=1.0):
    n, h = list(n) + [0] * (3 - len(n)), list(h) + [0.0] * (3 - len(h))
    c = dict(kind="steps", dim=3 if n[2] else 2, nx=n[0], ny=n[1], nz=n[2], hx=h[0], hy=h[1],
             hz=h[2], precision=precision, mode=mode, steps=steps, g=g, omega=omega, dt=dt, nu=nu,
             lam=lam)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: a short block between two looks at the observables
        # on the 128^2 grid (convergence checks, interactive runs)
        _steps("2d_128_fp32_short", (128, 128), (0.1, 0.1), steps=20, g=100.0, omega=0.5, dt=1e-3),
        # the same grid in double precision: the precision of the paper's own
        # programs, and what a user validates a single-precision run against
        _steps("2d_128_fp64", (128, 128), (0.1, 0.1), precision="fp64", steps=100, g=100.0,
               omega=0.5, dt=1e-3),
        # Table 1's larger 2D grid (441^2 points): millions of these steps per lattice
        _steps("2d_440_fp32", (440, 440), (0.05, 0.05), steps=200, g=500.0, omega=0.92, dt=2.5e-4),
        # an odd, uneven 2D grid (a stretched trap), where rows are not 16-byte multiples
        _steps("2d_301x215_fp32", (301, 215), (0.06, 0.07), steps=100, g=300.0, omega=0.8, dt=4e-4,
               nu=1.3),
        # real-time ramp of the rotation frequency on the 512^2 grid
        _steps("2d_512_fp32_ramp", (512, 512), (0.05, 0.05), mode="ramp", steps=50, g=1000.0,
               omega=0.9, dt=1e-4, nu=1.05),
        # a finely resolved 2D state larger than L2 whose line carries decay slowly
        _steps("2d_4096_fp32", (4096, 4096), (0.01, 0.01), steps=10, g=1000.0, omega=0.9,
               dt=2.5e-4, nu=1.05),
        # the 3D benchmark: imaginary time, and its real-time part
        _steps("3d_256x256x128_fp32", (256, 256, 128), (0.08, 0.08, 0.1), steps=50, g=3000.0,
               omega=0.85, dt=2e-4, lam=0.5),
        _steps("3d_256x256x128_fp32_real", (256, 256, 128), (0.08, 0.08, 0.1), mode="real",
               steps=25, g=3000.0, omega=0.85, dt=1e-4, lam=0.5),
        # the 3D state larger than L2
        _steps("3d_512x512x128_fp32", (512, 512, 128), (0.08, 0.08, 0.1), steps=10, g=3000.0,
               omega=0.85, dt=2e-4, lam=0.5),
        # Table 1's 3D disk (257 x 257 x 33 points) in double precision
        _steps("3d_256x256x32_fp64", (256, 256, 32), (0.05, 0.05, 0.025), precision="fp64",
               steps=5, g=100.0, omega=0.8, dt=2.5e-4, lam=100.0),
        # the batched parameter sweep: 64 condensates of 128^2 .. 512^2
        dict(name="batch_64_fp32", kind="batch", count=64, spec_seed=0, steps=50),
        # one training step of the learned start on a batch of its 128^2 grid
        dict(name="ws_train_128", kind="ws_train", grid=128, batch=16, half_width=12.0),
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    k = rng.choice(("2d", "2d", "2d", "ramp", "fp64", "long", "3d", "3d", "3dreal", "3dfp64",
                    "batch", "ws"))
    kappa = math.exp(rng.uniform(math.log(0.008), math.log(0.04)))
    g, omega = rng.uniform(50.0, 1500.0), rng.uniform(0.3, 0.95)
    nu = rng.uniform(1.0, 1.2)
    if k == "batch":
        return dict(kind="batch", count=_log(rng, 4, 64), spec_seed=rng.randrange(1, 1 << 20),
                    steps=rng.randrange(10, 51))
    if k == "ws":
        return dict(kind="ws_train", grid=16 * rng.randrange(3, 9), batch=rng.randrange(2, 17),
                    half_width=round(rng.uniform(8.0, 14.0), 3))
    if k in ("2d", "ramp", "fp64", "long"):
        lo, hi = {"2d": (48, 1200), "ramp": (96, 640), "fp64": (48, 300), "long": (1500, 4096)}[k]
        nx = _log(rng, lo, hi)
        ny = max(lo // 2, min(hi, int(nx * rng.uniform(0.6, 1.0))))
        half = rng.uniform(6.0, 13.0) if k != "long" else rng.uniform(12.0, 20.0)
        hx = 2.0 * half / nx
        hy = hx * rng.uniform(0.9, 1.2)
        if k == "long":
            kappa = rng.uniform(0.1, 0.6)
        steps = {"2d": 100, "ramp": 40, "fp64": 40, "long": 6}[k]
        return _steps(None, (nx, ny), (hx, hy), precision="fp64" if k == "fp64" else "fp32",
                      mode="ramp" if k == "ramp" else rng.choice(("imag", "imag", "real")),
                      steps=rng.randrange(steps // 2, steps + 1), g=g, omega=omega,
                      dt=min(2e-3, 4.0 * hx * hx * kappa), nu=nu)
    most = 1.2e6 if k == "3dfp64" else 2.0e7
    while True:
        nx, ny, nz = (_log(rng, 32, 128 if k == "3dfp64" else 448), _log(rng, 32, 320),
                      _log(rng, 24, 200))
        if nx * ny * nz <= most:
            break
    hx = 2.0 * rng.uniform(5.0, 10.0) / nx
    hy, hz = hx * rng.uniform(0.9, 1.2), hx * rng.uniform(0.9, 1.4)
    return _steps(None, (nx, ny, nz), (hx, hy, hz), precision="fp64" if k == "3dfp64" else "fp32",
                  mode="real" if k == "3dreal" else "imag",
                  steps=4 if k == "3dfp64" else rng.randrange(8, 25), g=g, omega=omega,
                  dt=min(2e-3, 4.0 * hx * hx * kappa), nu=nu, lam=rng.uniform(0.5, 3.0))


# ------------------------------------------------------------------ inputs
def _vortex_state(n, h, nu, seed, dtype):
    """A smooth vortex state on all (N+1)^d points (edges zero), from the
    seed: a Thomas-Fermi-like profile with vortices at drawn places and long
    density waves, unit norm up to the normalisation on load."""
    rng = np.random.default_rng(seed)
    dev = "cuda"
    f64 = dict(dtype=torch.float64, device=dev)
    ax = [(torch.arange(v + 1, **f64) - 0.5 * v) * d for v, d in zip(n, h)]
    x, y = ax[0][None, :], ax[1][:, None]
    half = [0.5 * v * d for v, d in zip(n, h)]
    rx = 0.62 * half[0] * rng.uniform(0.9, 1.05)
    ry = min(rx / nu, 0.65 * half[1])
    count = int(rng.integers(5, 13))
    psi = torch.ones((n[1] + 1, n[0] + 1), dtype=torch.complex128, device=dev)
    for _ in range(count):
        r, a = math.sqrt(rng.uniform(0, 1)) * 0.75, rng.uniform(0, 2 * math.pi)
        zeta = torch.complex((x - r * rx * math.cos(a)).expand(psi.shape),
                             (y - r * ry * math.sin(a)).expand(psi.shape))
        psi *= zeta / torch.sqrt(zeta.abs() ** 2 + (0.08 * rx) ** 2)
    for _ in range(4):
        kx, ky = rng.uniform(-6, 6, 2) / rx
        psi *= 1.0 + 0.05 * torch.cos(kx * x + ky * y + rng.uniform(0, 2 * math.pi))
    u = (x / rx) ** 2 + (y / ry) ** 2
    soft = torch.nn.functional.softplus
    if len(n) == 2:
        psi *= torch.sqrt(0.1 * soft((1.0 - u) / 0.1))
    else:
        rz = 0.6 * half[2]
        out = torch.empty((n[2] + 1, n[1] + 1, n[0] + 1), dtype=dtype, device=dev)
        for k in range(n[2] + 1):
            tilt = complex(math.cos(0.3 * float(ax[2][k]) / rz), math.sin(0.3 * float(ax[2][k]) / rz))
            out[k] = (psi * tilt * torch.sqrt(0.1 * soft((1.0 - u - (ax[2][k] / rz) ** 2) / 0.1))
                      ).to(dtype)
        psi = out
        psi[0] = psi[-1] = 0
    psi = psi.to(dtype)
    psi[..., 0, :] = psi[..., -1, :] = 0
    psi[..., :, 0] = psi[..., :, -1] = 0
    vol = math.prod(h)
    norm = vol * sum(float(p.abs().double().square().sum()) for p in psi.reshape(-1, n[1] + 1, n[0] + 1))
    psi *= 1.0 / math.sqrt(norm)
    return psi.contiguous()


def _grid(case):
    d = case["dim"]
    return ([case["nx"], case["ny"], case["nz"]][:d], [case["hx"], case["hy"], case["hz"]][:d])


def _cdtype(case):
    return torch.complex128 if case.get("precision") == "fp64" else torch.complex64


def _ramp(case):
    """Omega of each step: a linear ramp down by a ninth over 20000 such steps."""
    return case["omega"] * (1.0 - np.arange(case["steps"]) / 180000.0)


def _specs(case):
    return inputs.batch_specs(case["count"], case["spec_seed"])


def _sizes(specs):
    """Instances by grid size, in a fixed order."""
    groups = {}
    for i, sp in enumerate(specs):
        groups.setdefault(sp["n"][0], []).append(i)
    return dict(sorted(groups.items()))


def _ws_inputs(case, seed):
    rng = np.random.default_rng(seed)
    prm = inputs.warmstart_params(case["batch"], int(rng.integers(1 << 30)))
    grid = case["grid"]
    layers = ((6, 32), (32, 32), (32, 64), (64, 64), (64, 128), (128, 128), (128, 128),
              (128, 128), (128, 64), (64, 32), (32, 32), (32, 2))
    parts = []
    for ci, co in layers:
        parts.append((rng.standard_normal(9 * ci * co) * math.sqrt(2.0 / (9 * ci))))
        parts.append(0.01 * rng.standard_normal(co))
    h = 2.0 * case["half_width"] / grid
    psi = torch.stack([_vortex_state((grid, grid), (h, h), float(prm[i, 2]),
                                     int(rng.integers(1 << 30)), torch.complex128)
                       for i in range(case["batch"])])
    return prm, np.concatenate(parts).astype(np.float32), psi


def prepare(case, seed):
    stream = torch.cuda.current_stream().cuda_stream
    if case["kind"] == "steps":
        n, h = _grid(case)
        s = Solver(n, h, gamma=1.0, nu=case["nu"], lam=case["lam"], g=case["g"],
                   omega=case["omega"], dt=case["dt"], precision=case["precision"], stream=stream)
        psi = _vortex_state(n, h, case["nu"], seed, _cdtype(case))
        return dict(case=case, solver=s, psi=psi, out=torch.empty_like(psi), ramp=_ramp(case))
    if case["kind"] == "batch":
        specs = _specs(case)
        b = Batch(specs, stream=stream)
        psi, out, where = {}, {}, [None] * len(specs)
        for size, members in _sizes(specs).items():
            psi[size] = torch.stack([_vortex_state(specs[i]["n"], specs[i]["h"], specs[i]["nu"],
                                                   seed * 1000 + i, torch.complex64)
                                     for i in members])
            out[size] = torch.empty_like(psi[size])
            for k, i in enumerate(members):
                where[i] = (size, k)
        return dict(case=case, batch=b, psi=psi, out=out, where=where)
    prm, params, psi = _ws_inputs(case, seed)
    ws = WarmStart(case["grid"], case["batch"], stream=stream)
    ws.set_params(params)
    return dict(case=case, ws=ws, prm=prm, psi=psi)


# ------------------------------------------------------------------ the pass
def _obs(o):
    return {k: o[k] for k in OBS}


def run(state):
    case = state["case"]
    if case["kind"] == "steps":
        s = state["solver"]
        s.set_psi(state["psi"], normalise=case["mode"] == "imag")
        if case["mode"] == "imag":
            s.step_imag(case["steps"])
        elif case["mode"] == "real":
            s.step_real(case["steps"])
        else:
            s.step_schedule(state["ramp"])
        o = s.observables()
        s.get_psi(state["out"])
        return {"psi": state["out"], "obs": _obs(o), "vortices": o["vortices"]}
    if case["kind"] == "batch":
        b = state["batch"]
        for inst, (size, k) in zip(b.instances, state["where"]):
            inst.set_psi(state["psi"][size][k], normalise=True)
        b.step_imag(case["steps"], mode="persistent")
        obs = b.observables()
        for inst, (size, k) in zip(b.instances, state["where"]):
            inst.get_psi(state["out"][size][k])
        return {"psi": {str(k): v for k, v in state["out"].items()},
                "obs": np.array([[o[k] for k in OBS] for o in obs], dtype=np.float32),
                "vortices": np.array([o["vortices"] for o in obs])}
    ws = state["ws"]
    loss = ws.train_step(state["prm"], case["half_width"], state["psi"], 1e-3)
    return {"loss": loss, "params": ws.get_params()}


# ------------------------------------------------------------------ work
def _step_work(sites, dim, itemsize):
    """One split step: the state read and written once; per site and sweep two
    complex multiply-adds forward and one back, and the pointwise factor."""
    return 2.0 * itemsize * sites, sites * (24.0 * dim + 20.0)


def work(case):
    if case["kind"] == "ws_train":
        g2, macs = case["grid"] ** 2, 0.0
        for ci, co, div in ((6, 32, 1), (32, 32, 1), (32, 64, 2), (64, 64, 2), (64, 128, 4),
                            (128, 128, 4), (128, 128, 8), (128, 128, 8), (128, 64, 4),
                            (64, 32, 2), (32, 32, 1), (32, 2, 1)):
            macs += 9.0 * ci * co * g2 / div ** 2
        # forward, data gradient and weight gradient; weights and Adam state, targets
        return {"bytes": 684642 * 4.0 * 7 + 16.0 * (case["grid"] + 1) ** 2 * case["batch"],
                "flops": 6.0 * macs * case["batch"]}
    if case["kind"] == "batch":
        bytes_, flops = 0.0, 0.0
        for sp in _specs(case):
            sites = sp["n"][0] * sp["n"][1]
            b, f = _step_work(sites, 2, 8)
            bytes_ += case["steps"] * b + 3 * 8.0 * sites
            flops += case["steps"] * f
        return {"bytes": bytes_, "flops": flops}
    n, _ = _grid(case)
    size = 16 if case["precision"] == "fp64" else 8
    b, f = _step_work(math.prod(n), len(n), size)
    # load, observables and read back beside the steps
    return {"bytes": case["steps"] * b + 3.0 * size * math.prod(n), "flops": case["steps"] * f}


# ------------------------------------------------------------------ 64-bit values
class _Line:
    """Crank-Nicolson sweep along one axis of psi (B, [nz,] ny, nx) interior
    points: (1 - K) x = (1 + K) psi with K = kap second difference + tau
    first difference, by the Thomas algorithm in complex double."""

    def __init__(self, axis, m, kap, tau):
        self.axis, self.kap, self.tau = axis, kap, tau
        am, a0, ap = -kap + tau, 1.0 + 2.0 * kap + 0.0 * tau, -kap - tau
        self.am = am
        self.c, self.m = [], []
        c = torch.zeros_like(a0)
        for _ in range(m):
            inv = 1.0 / (a0 - am * c)
            cn = ap * inv
            self.m.append(inv)
            self.c.append(cn)
            if len(self.c) > 1 and bool((cn == c).all()):
                break
            c = cn

    def __call__(self, psi):
        p = psi.movedim(self.axis, 0).contiguous()
        m = p.shape[0]
        b = (1.0 - 2.0 * self.kap) * p
        b[:-1] += (self.kap + self.tau) * p[1:]
        b[1:] += (self.kap - self.tau) * p[:-1]
        last = len(self.m) - 1
        d = torch.zeros_like(p[0])
        for i in range(m):
            d = torch.mul(torch.addcmul(b[i], self.am.expand_as(d), d, value=-1),
                          self.m[min(i, last)], out=b[i])
        for i in range(m - 2, -1, -1):
            b[i].addcmul_(self.c[min(i, last)].expand_as(d), b[i + 1], value=-1)
        return b.movedim(0, self.axis)


class _Exact:
    """Split steps and observables of B condensates of one grid size in
    complex double (spacings and physics may differ)."""

    def __init__(self, n, specs, dev):
        self.n, self.dim, self.dev = n, len(n), dev
        col = lambda v: torch.tensor(v, dtype=torch.float64, device=dev).reshape(  # noqa: E731
            [-1] + [1] * self.dim)
        self.h = [col([sp["h"][a] for sp in specs]) for a in range(self.dim)]
        self.trap = [col([sp.get(k, 1.0) for sp in specs]) for k in ("gamma", "nu", "lam")]
        self.g, self.omega, self.dt = (col([sp[k] for sp in specs]) for k in ("g", "omega", "dt"))
        self.x = []
        for a in range(self.dim):
            i = torch.arange(1, n[a], dtype=torch.float64, device=dev) - 0.5 * n[a]
            self.x.append(i.reshape([-1] + [1] * a) * self.h[a])
        self.V = sum(0.5 * w * w * x * x for w, x in zip(self.trap, self.x))
        self.vol = math.prod(self.h)

    def lines(self, imag, omega):
        out = []
        for a in range(self.dim):
            axis = self.dim - a  # of psi (B, [z,] y, x)
            dtau = self.dt.to(torch.complex128) * (1.0 if imag else 1j)
            kap = (dtau / (4.0 * self.h[a] ** 2)).squeeze(axis)
            sign = {0: -1.0, 1: 1.0, 2: 0.0}[a]
            other = self.x[{0: 1, 1: 0, 2: 0}[a]]
            tau = (sign * (dtau / 1j) * omega / (4.0 * self.h[a]) * other).squeeze(axis)
            out.append(_Line(axis, self.n[a] - 1, kap, tau))
        return out

    def norm(self, psi):
        return (psi.abs() ** 2).sum(dim=tuple(range(1, psi.dim())), keepdim=True) * self.vol

    def step(self, psi, lines, imag):
        en = self.V + self.g * psi.abs() ** 2
        psi = psi * (torch.exp(-self.dt * en) if imag else torch.exp(-1j * self.dt * en))
        for ln in lines:
            psi = ln(psi)
        return psi / torch.sqrt(self.norm(psi)) if imag else psi

    def observables(self, psi):
        d = list(range(1, psi.dim()))
        total = lambda v: v.sum(dim=d)  # noqa: E731
        pad = torch.nn.functional.pad(psi, [2, 2] * self.dim)
        lap, lap4, der, der4 = 0.0, 0.0, [], []
        for a in range(self.dim):
            axis = self.dim - a

            def at(o):
                v = pad
                for q in d:
                    v = v.narrow(q, 2 + (o if q == axis else 0), psi.shape[q])
                return v

            p1, m1, p2, m2 = at(1), at(-1), at(2), at(-2)
            h = self.h[a]
            lap = lap + (p1 - 2.0 * psi + m1) / (h * h)
            lap4 = lap4 + (-p2 + 16.0 * p1 - 30.0 * psi + 16.0 * m1 - m2) / (12.0 * h * h)
            der.append((p1 - m1) / (2.0 * h))
            der4.append((-p2 + 8.0 * p1 - 8.0 * m1 + m2) / (12.0 * h))
            del p1, m1, p2, m2
        x, y = self.x[0], self.x[1]
        rot, rot4 = y * der[0] - x * der[1], y * der4[0] - x * der4[1]
        del der, der4, pad
        re, im, rho = psi.real, psi.imag, psi.abs() ** 2
        s2, sr, si = total(rho), total(re * re), total(im * im)
        om, g = self.omega, self.g
        swap = sr < 1e-3 * s2
        lin_r = total(re * (-0.5 * lap.real + self.V * re + om * rot.imag))
        lin_i = total(im * (-0.5 * lap.imag + self.V * im - om * rot.real))
        lin = torch.where(swap, lin_i, lin_r)
        nl = torch.where(swap, total(g * rho * im * im), total(g * rho * re * re))
        den = torch.where(swap, si, sr)
        lin_c = total((psi.conj() * (-0.5 * lap + self.V * psi - 1j * om * rot)).real)
        lin_4 = total((psi.conj() * (-0.5 * lap4 + self.V * psi - 1j * om * rot4)).real)
        nl_c = total(g * rho * rho)
        r2 = [total(v * v * rho) / s2 for v in self.x]
        z2 = r2[2] if self.dim == 3 else torch.zeros_like(s2)
        return dict(norm=s2 * self.vol.reshape(-1), mu=(lin + nl) / den,
                    energy=(lin + 0.5 * nl) / den, mu_c=(lin_c + nl_c) / s2,
                    energy_c=(lin_c + 0.5 * nl_c) / s2, rms_x=r2[0].sqrt(), rms_y=r2[1].sqrt(),
                    rms_z=z2.sqrt(), rms_r=(r2[0] + r2[1] + z2).sqrt(), max_density=rho.amax(dim=d),
                    mu4=(lin_4 + nl_c) / s2, energy4=(lin_4 + 0.5 * nl_c) / s2)

    def full(self, psi):
        return torch.nn.functional.pad(psi, [1, 1] * self.dim)


def _interior(psi, dim):
    return psi[(Ellipsis,) + (slice(1, -1),) * dim].to(torch.complex128)


def _exact_ws(case, seed):
    prm, params, psi = _ws_inputs(case, seed)
    dev, G, L = psi.device, case["grid"], case["half_width"]
    col = lambda k: torch.tensor(prm[:, k], device=dev).reshape(-1, 1, 1)  # noqa: E731
    om, g, nu = col(0), col(1), col(2)
    c = -L + torch.arange(G, dtype=torch.float64, device=dev) * (2.0 * L / G)
    x, y = c[None, None, :].expand(1, G, G), c[None, :, None].expand(1, G, G)
    gx2, gy2 = (1.0 - om * om).clamp(min=1e-3), (nu * nu - om * om).clamp(min=1e-3)
    mu = torch.sqrt(g * torch.sqrt(gx2 * gy2) / math.pi)
    tf = (mu - 0.5 * (gx2 * x * x + gy2 * y * y)).clamp(min=0.0) / g
    planes = [2.0 * L * tf.sqrt(), x / L, y / L, om, g / 1000.0, (nu - 1.0) / 0.1]
    v = torch.stack([p.expand(case["batch"], G, G) for p in planes], dim=1)
    target = 2.0 * L * torch.view_as_real(psi[:, :G, :G]).permute(0, 3, 1, 2)
    flat = torch.tensor(params, dtype=torch.float64, device=dev, requires_grad=True)
    layers, off = [], 0
    for ci, co in ((6, 32), (32, 32), (32, 64), (64, 64), (64, 128), (128, 128), (128, 128),
                   (128, 128), (128, 64), (64, 32), (32, 32), (32, 2)):
        w = flat[off:off + 9 * ci * co].reshape(3, 3, ci, co).permute(3, 2, 0, 1)
        layers.append((w, flat[off + 9 * ci * co:off + 9 * ci * co + co]))
        off += 9 * ci * co + co
    F = torch.nn.functional

    def conv(t, i, relu=True):
        # a 3 x 3 correlation as nine shifted products
        w, b = layers[i]
        p = F.pad(t, [1, 1, 1, 1])
        hh, ww = t.shape[2:]
        out = b.reshape(1, -1, 1, 1)
        for ky in range(3):
            for kx in range(3):
                out = out + torch.einsum("bchw,oc->bohw", p[:, :, ky:ky + hh, kx:kx + ww],
                                         w[:, :, ky, kx])
        return F.relu(out) if relu else out

    up = lambda t: t.repeat_interleave(2, 2).repeat_interleave(2, 3)  # noqa: E731
    e1 = conv(conv(v, 0), 1)
    e3 = conv(conv(F.avg_pool2d(e1, 2), 2), 3)
    e5 = conv(conv(F.avg_pool2d(e3, 2), 4), 5)
    b7 = conv(conv(F.avg_pool2d(e5, 2), 6), 7)
    d8 = conv(up(b7) + e5, 8)
    d9 = conv(up(d8) + e3, 9)
    out = conv(conv(up(d9) + e1, 10), 11, relu=False)
    loss = ((out - target) ** 2).mean()
    grad, = torch.autograd.grad(loss, flat)
    new = flat.detach() - 1e-3 * grad / (grad.abs() + 1e-8)
    return {"loss": float(loss), "params": new}


def exact(case, seed):
    if case["kind"] == "ws_train":
        return _exact_ws(case, seed)
    if case["kind"] == "batch":
        specs = _specs(case)
        psis, obs = {}, [None] * len(specs)
        for size, members in _sizes(specs).items():
            p = torch.stack([_interior(_vortex_state(specs[i]["n"], specs[i]["h"], specs[i]["nu"],
                                                     seed * 1000 + i, torch.complex64), 2)
                             for i in members])
            ex = _Exact(specs[members[0]]["n"], [specs[i] for i in members], p.device)
            p = p / torch.sqrt(ex.norm(p))
            lines = ex.lines(True, ex.omega)
            for _ in range(case["steps"]):
                p = ex.step(p, lines, True)
            o = ex.observables(p)
            for k, i in enumerate(members):
                obs[i] = [float(o[q][k]) for q in OBS]
            psis[str(size)] = ex.full(p)
        return {"psi": psis, "obs": np.array(obs), "vortices": None}
    n, h = _grid(case)
    p = _interior(_vortex_state(n, h, case["nu"], seed, _cdtype(case)), len(n))[None]
    ex = _Exact(n, [dict(h=h, nu=case["nu"], lam=case["lam"], g=case["g"], omega=case["omega"],
                         dt=case["dt"])], p.device)
    imag = case["mode"] == "imag"
    if imag:
        p = p / torch.sqrt(ex.norm(p))
    lines = ex.lines(imag, ex.omega)
    for k in range(case["steps"]):
        if case["mode"] == "ramp":
            ex.omega = torch.full_like(ex.omega, float(_ramp(case)[k]))
            lines = ex.lines(imag, ex.omega)
        p = ex.step(p, lines, imag)
    o = ex.observables(p)
    return {"psi": ex.full(p)[0], "obs": {k: float(v[0]) for k, v in o.items()},
            "vortices": None}
