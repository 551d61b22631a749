"""Performance cases: what a program that uses this library has it do.

Every case is one pass through the public binding (``fcn.Solver``,
``fcn.SolverXY``): the fields are set from device tensors, the pulses advance
by fixed or adaptive Strang steps, and the resulting fields are read back into
device tensors.  ``listed`` gives the fixed cases, ``draw`` more of the same
ranges, ``exact`` the same result in plain 64-bit torch arithmetic.
"""
import math

import numpy as np
import torch

from paper_1507_05988_gb300 import fcn, workloads as W

C_LIGHT, EPS0, M_E = 299792458.0, 8.8541878128e-12, 9.1093837015e-31      # CODATA 2018
Q_E, H_BAR = 1.602176634e-19, 1.054571817e-34


# ---- cases ----
def _radial(name, nr, nt, pulses, prec, dz, n, w0, tp, power, n4=0.0, core=0.0, record=False):
    """pulses pulses on an nr x nt radial grid, n fixed steps of dz; core:
    peak intensity of a narrow filament core on top of the input beam (0:
    none); record: the run also reads energy and profiles, as a run that logs
    its distance does."""
    return dict(name=name, kind="run", nr=nr, nt=nt, pulses=pulses, prec=prec, dz=dz, n=n, w0=w0, tp=tp,
                power=power, n4=n4, core=core, record=record)


def _adaptive(name, nr, nt, pulses, dz, k, w0, tp, power, n4):
    """Step doubling at rtol 1e-4 from dz over dz (2^k - 1): at least k
    attempts, as the step law at most doubles a step."""
    return dict(name=name, kind="adaptive", nr=nr, nt=nt, pulses=pulses, prec="f32", dz=dz, k=k, w0=w0, tp=tp,
                power=power, n4=n4, core=0.0)


def _uneven(name, pulses, n, seed, nr_lo, nr_hi, nt_lo, nt_hi):
    """pulses pulses with grids, powers and widths of their own in one context."""
    return dict(name=name, kind="uneven", pulses=pulses, prec="f32", dz=2e-3, n=n, seed=seed, nr_lo=nr_lo,
                nr_hi=nr_hi, nt_lo=nt_lo, nt_hi=nt_hi)


def _cart(name, nx, ny, nt, prec, dz, n, w0, tp, power):
    """One pulse on an nx x ny x nt Cartesian transverse grid, n steps of dz."""
    return dict(name=name, kind="cart", nx=nx, ny=ny, nt=nt, prec=prec, dz=dz, n=n, w0=w0, tp=tp, power=power)


def listed():
    return [
        # the smallest call: a program that steps a small grid and looks at it after every step
        _radial("step_128x256_f32", 128, 256, 1, "f32", 1e-2, 1, 1e-3, 100e-15, 3.0),
        # the plain double-precision run on the small grid (validation, parameter scans)
        _radial("run_128x256_f64", 128, 256, 1, "f64", 1e-2, 64, 1e-3, 100e-15, 3.0),
        # the long application run on its ragged grid, filamented, logging between its blocks of steps
        _radial("run_1350x1024_f32", 1350, 1024, 1, "f32", 1e-3, 40, 18e-3, 300e-15, 53.3, core=2e17, record=True),
        # one pulse of the filamentation workload: the ordinary single-pulse run
        _radial("run_1024x4096_f32", 1024, 4096, 1, "f32", 2e-3, 24, 2e-3, 50e-15, 5.0, n4=W.N4),
        # eight such pulses advancing together: the throughput form
        _radial("run_1024x4096x8_f32", 1024, 4096, 8, "f32", 2e-3, 16, 2e-3, 50e-15, 5.0, n4=W.N4),
        # the same pulse in double precision: the reference run every mixed-precision result is held to
        _radial("run_1024x4096_f64", 1024, 4096, 1, "f64", 2e-3, 3, 2e-3, 50e-15, 5.0, n4=W.N4),
        # the long-distance grid, the largest single pulse
        _radial("run_2048x8192_f32", 2048, 8192, 1, "f32", 2e-3, 8, 5e-3, 100e-15, 10.0, n4=W.N4),
        # a parameter scan: many small pulses of uneven grids in one context
        _uneven("scan_16_uneven_f32", 16, 16, 7, 64, 256, 512, 1024),
        # adaptive propagation of one pulse
        _adaptive("adaptive_1024x4096_f32", 1024, 4096, 1, 2.5e-4, 4, 2e-3, 50e-15, 5.0, W.N4),
        # adaptive propagation of a batch with one common step
        _adaptive("adaptive_1024x4096x8_f32", 1024, 4096, 8, 2.5e-4, 4, 2e-3, 50e-15, 5.0, W.N4),
        # a beam without cylindrical symmetry: the Cartesian grid
        _cart("cart_255x255x256_f32", 255, 255, 256, "f32", 1e-2, 10, 1e-3, 100e-15, 3.0),
        # a small ragged Cartesian grid in double precision
        _cart("cart_97x65x128_f64", 97, 65, 128, "f64", 1e-2, 4, 1e-3, 100e-15, 3.0),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    w0 = math.exp(rng.uniform(math.log(5e-4), math.log(5e-3)))
    tp = rng.uniform(30e-15, 200e-15)
    power = rng.uniform(1.0, 10.0)
    dz = 2e-3 * min(1.0, (w0 / 2e-3) ** 2)
    kind = rng.choice(["run", "run", "run64", "adaptive", "cart", "cart64", "uneven"])
    if kind == "uneven":
        lo = log_int(48, 128)
        return {k: v for k, v in _uneven("", rng.randint(9, 24), rng.randint(4, 24), rng.randint(0, 1 << 20), lo,
                                         lo * rng.randint(2, 4), 512, rng.choice([1024, 2048])).items() if k != "name"}
    if kind.startswith("cart"):
        nx, ny, nt = log_int(33, 255), log_int(33, 255), rng.choice([64, 128, 256, 512])
        prec = "f64" if kind == "cart64" else "f32"
        while nx * ny * nt > (4e6 if prec == "f64" else 16e6):
            nt //= 2
        n = max(1, min(rng.randint(2, 40), int((6e6 if prec == "f64" else 160e6) / (nx * ny * nt))))
        c = _cart("", nx, ny, nt, prec, dz, n, w0, tp, power)
    elif kind == "adaptive":
        nr, nt = log_int(128, 2048), rng.choice([512, 1024, 2048, 4096, 8192])
        while nr * nt > 4 << 20:
            nt //= 2
        n4 = rng.choice([0.0, W.N4])               # with it the steps that meet rtol are much shorter
        c = _adaptive("", nr, nt, max(1, min(rng.randint(1, 8), (32 << 20) // (nr * nt))),
                      dz / 2 if n4 == 0.0 else min(dz / 2, 2.5e-4), rng.randint(2, 4), w0, tp, power, n4)
    else:
        nr, nt = log_int(64, 2048), rng.choice([256, 512, 1024, 2048, 4096, 8192])
        if kind == "run64":
            while nr * nt > 4 << 20:
                nt //= 2
            n = max(1, min(rng.randint(1, 64), int(12e6 / (nr * nt))))
            c = _radial("", nr, nt, 1, "f64", dz, n, w0, tp, power, rng.choice([0.0, W.N4]))
        else:
            pulses = rng.choice([1, 1, rng.randint(2, 8)])
            while nr * nt * pulses > 33 << 20:
                pulses = max(1, pulses // 2)
            n = max(1, min(rng.randint(1, 64), int(500e6 / (nr * nt * pulses))))
            c = _radial("", nr, nt, pulses, "f32", dz, n, w0, tp, power, rng.choice([0.0, W.N4]))
    return {k: v for k, v in c.items() if k != "name"}


# ---- inputs ----
def _workloads(case):
    """The workload description of every pulse of the case."""
    if case["kind"] == "cart":
        return [W.WorkloadXY("case", case["nx"], case["ny"], case["nt"], case["w0"], case["tp"], case["power"])]
    if case["kind"] == "uneven":
        rng = np.random.Generator(np.random.PCG64(case["seed"]))
        nts = [nt for nt in (512, 1024, 2048, 4096, 8192) if case["nt_lo"] <= nt <= case["nt_hi"]]
        return [W.Workload("case", int(rng.integers(case["nr_lo"], case["nr_hi"] + 1)), int(rng.choice(nts)),
                           float(rng.uniform(0.5e-3, 5e-3)), float(rng.uniform(30e-15, 200e-15)),
                           float(rng.uniform(1.0, 10.0))) for _ in range(case["pulses"])]
    wl = W.Workload("case", case["nr"], case["nt"], case["w0"], case["tp"], case["power"],
                    n2j=(W.N2, case["n4"], 0.0, 0.0))
    return [wl] * case["pulses"]


def _axis(n, width):
    return -0.5 * width + torch.arange(n, dtype=torch.float64, device="cuda") * (width / (n - 1))


def _fields(case, seed):
    """One input field per pulse, in the working precision: the Gaussian pulse
    with 1 % amplitude noise (and the filament core, where the case has one)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    out = []
    for wl in _workloads(case):
        tau = -0.5 * wl.t_window + torch.arange(wl.nt, dtype=torch.float64, device="cuda") * (wl.t_window / wl.nt)
        tt = (tau / wl.tp) ** 2
        if case["kind"] == "cart":
            x, y = _axis(wl.nx, wl.x_width), _axis(wl.ny, wl.y_width)
            r2 = (x[:, None] ** 2 + y[None, :] ** 2)[..., None]
        else:
            r2 = ((torch.arange(wl.nr, dtype=torch.float64, device="cuda") * (wl.r_max / (wl.nr - 1))) ** 2)[:, None]
        a = math.sqrt(wl.i0) * torch.exp(-r2 / wl.w0 ** 2 - tt)
        if case.get("core"):
            a = a + math.sqrt(case["core"]) * torch.exp(-r2 / (wl.w0 / 50) ** 2 - (tau / (wl.tp / 5)) ** 2)
        a = a * (0.99 + 0.02 * torch.rand(a.shape, generator=gen, device="cuda", dtype=torch.float64))
        out.append(a.to(torch.complex128 if case["prec"] == "f64" else torch.complex64).contiguous())
    return out


def prepare(case, seed):
    prec = fcn.FCN_FP64 if case["prec"] == "f64" else fcn.FCN_FP32_MIXED
    wls = _workloads(case)
    if case["kind"] == "cart":
        solver = fcn.SolverXY(wls[0].grid(), wls[0].physics(), precision=prec)
    else:
        solver = fcn.Solver([wl.physics() for wl in wls] if len(wls) > 1 else wls[0].physics(), precision=prec)
    fields = _fields(case, seed)
    return dict(case=case, solver=solver, fields=fields, out=[torch.empty_like(f) for f in fields])


def run(state):
    case, s = state["case"], state["solver"]
    if case["kind"] == "cart":
        s.set_field_device(state["fields"][0])
        s.step(case["dz"], case["n"])
        s.get_field_device(state["out"][0])
        return state["out"]
    for i, f in enumerate(state["fields"]):
        s.set_field_device(f, i)
    if case["kind"] == "adaptive":
        s.propagate(case["dz"] * (2 ** case["k"] - 1), case["dz"], rtol=1e-4)
    else:
        s.step(case["dz"], case["n"])
    for i, f in enumerate(state["out"]):
        s.get_field_device(f, i)
    if case.get("record"):
        energy = s.diag()["energy"]
        power, fluence = s.profiles()
        return state["out"] + [np.float32(energy), power.astype(np.float32), fluence.astype(np.float32)]
    return state["out"]


def work(case):
    """Of one pass.  A step's stages run along different axes over the whole
    field (the transforms and the nonlinear part along tau, one linear solve
    per transverse axis), so each reads and writes the field once; the
    arithmetic is two transforms (5 N log2 N), about 34 operations per point
    and linear solve and 60 for two nonlinear half steps.  An adaptive run
    takes at least k attempts of three steps."""
    size = 16 if case["prec"] == "f64" else 8
    axes = 2 if case["kind"] == "cart" else 1
    steps = 3 * case["k"] if case["kind"] == "adaptive" else case["n"]
    nbytes = flops = 0.0
    for wl in _workloads(case):
        nbytes += 2.0 * size * (1 + axes) * wl.points * steps
        flops += (10.0 * math.log2(wl.nt) + 34.0 * axes + 60.0) * wl.points * steps
    return {"bytes": nbytes, "flops": flops}


# ---- the same in 64 bits ----
def _recurrence(alpha, v, reverse=False):
    """v_j <- v_j + alpha_j v_{j-1} (j+1 when reverse) along axis -2, in place."""
    n = v.shape[-2]
    order = range(n - 2, -1, -1) if reverse else range(1, n)
    for j in order:
        p = v[..., j + 1 if reverse else j - 1, :]
        torch.addcmul(v[..., j, :], alpha[j], p, out=v[..., j, :])


class _Factor:
    """Crank-Nicolson factor of one axis: M_abc x' = M_def x along axis -2 for
    every frequency (last axis): sub-diagonal -i lo, super-diagonal -i hi,
    diagonal 1 + i (c0 - delta); rows with keep = 0 are walls (x' = 0)."""

    def __init__(self, lo, hi, c0, keep, delta):
        n, q = len(lo), delta.numel()
        lo, hi, c0, keep = (torch.tensor(v, dtype=torch.float64, device="cuda")[:, None] for v in (lo, hi, c0, keep))
        self.cd = c0 - delta[None, :]
        b = torch.complex(torch.ones(n, q, dtype=torch.float64, device="cuda"), self.cd) * keep + (1 - keep)
        inv = torch.empty_like(b)
        inv[0] = 1.0 / b[0]
        for j in range(1, n):                     # piv_j = b_j + lo_j hi_{j-1} / piv_{j-1}
            inv[j] = 1.0 / (b[j] + (lo[j] * hi[j - 1]) * inv[j - 1])
        self.inv, self.lo, self.hi, self.keep = inv, lo, hi, keep
        self.alpha, self.gamma = 1j * lo * inv, 1j * hi * inv

    def apply(self, x):
        w = -self.cd * x
        w[..., 1:, :] += self.lo[1:] * x[..., :-1, :]
        w[..., :-1, :] += self.hi[:-1] * x[..., 1:, :]
        y = (x + 1j * w) * self.keep * self.inv
        _recurrence(self.alpha, y)
        _recurrence(self.gamma, y, reverse=True)
        return y


class _Exact:
    """The Strang step of one grid in complex128 torch arithmetic."""

    def __init__(self, wl, cart):
        self.wl, self.cart, self.factors = wl, cart, {}
        self.k0 = 2 * math.pi * wl.n0 / wl.lambda0
        w = 2 * math.pi * C_LIGHT / wl.lambda0
        self.rho_c = EPS0 * M_E * w * w / Q_E ** 2
        self.beta = wl.K * H_BAR * w * wl.sigma_k * wl.rho_nt
        self.dtau = wl.t_window / wl.nt
        q = torch.arange(wl.nt, dtype=torch.float64, device="cuda")
        self.omega2 = (torch.where(q < wl.nt // 2, q, q - wl.nt) * (2 * math.pi / wl.t_window)) ** 2

    def half(self, a, h):
        wl = self.wl
        i = a.real ** 2 + a.imag ** 2
        x = wl.sigma_k * self.dtau * i ** wl.K
        xm = wl.sigma_k * self.dtau * (0.5 * (i[..., :-1] + i[..., 1:])) ** wl.K
        xa, xb = x[..., :-1], x[..., 1:]
        t1 = 1 - 0.5 * xa
        t2 = 1 - 0.5 * xm * t1
        t3 = 1 - xm * t2
        c = (xa + 2 * xm * (t1 + t2) + xb * t3) / 6
        u = torch.zeros_like(i)
        u[..., 1:] = -torch.expm1(torch.cumsum(torch.log1p(-c), -1))
        dn = sum(n2 * i ** (j + 1) for j, n2 in enumerate(wl.n2j) if n2)
        phi = h * (self.k0 / wl.n0 * dn - self.k0 / (2 * wl.n0 ** 2 * self.rho_c) * wl.rho_nt * u)
        return a * torch.polar(torch.exp(-0.5 * h * self.beta * i ** (wl.K - 1)), phi)

    def linear_factors(self, dz):
        if dz not in self.factors:
            wl, delta = self.wl, self.omega2 * (W.K2 * dz / 4)
            if self.cart:
                out = []
                for n, width, d in ((wl.nx, wl.x_width, 0 * delta), (wl.ny, wl.y_width, delta)):
                    s = dz / (4 * self.k0 * (width / (n - 1)) ** 2)
                    inner = [0.0] + [1.0] * (n - 2) + [0.0]
                    out.append(_Factor([s * v for v in inner], [s * v for v in inner], [2 * s * v for v in inner],
                                       inner, d))
            else:
                n, s = wl.nr, dz / (4 * self.k0 * (wl.r_max / (wl.nr - 1)) ** 2)
                lo = [0.0] + [s * (1 - 0.5 / j) for j in range(1, n - 1)] + [0.0]
                hi = [4 * s] + [s * (1 + 0.5 / j) for j in range(1, n - 1)] + [0.0]
                out = [_Factor(lo, hi, [4 * s] + [2 * s] * (n - 2) + [0.0], [1.0] * (n - 1) + [0.0], delta)]
            if len(self.factors) > 2:
                self.factors.clear()
            self.factors[dz] = out
        return self.factors[dz]

    def step(self, a, dz):
        a = torch.fft.fft(self.half(a, 0.5 * dz))
        f = self.linear_factors(dz)
        if self.cart:                              # x lines, then y lines
            a = f[0].apply(a.transpose(0, 1).contiguous()).transpose(0, 1).contiguous()
            a = f[1].apply(a)
        else:
            a = f[0].apply(a)
        return self.half(torch.fft.ifft(a), 0.5 * dz)

    def adaptive(self, a, dz0, z_end, rtol=1e-4):
        z, dz = 0.0, dz0
        while z < z_end:
            last = z + dz >= z_end
            h = z_end - z if last else dz
            one = self.step(a, h)
            two = self.step(self.step(a, 0.5 * h), 0.5 * h)
            err = max(float((t - o).norm() / t.norm()) for t, o in zip(two, one))
            fac = min(2.0, max(0.2, 0.9 * (rtol / err) ** (1 / 3)))
            if err <= rtol:
                a, z = two, (z_end if last else z + h)
            dz = h * fac
        return a


def exact(case, seed):
    wls, fields = _workloads(case), _fields(case, seed)
    fields = [f.to(torch.complex128) for f in fields]
    if case["kind"] in ("cart", "uneven"):
        out = []
        for wl, a in zip(wls, fields):
            ex = _Exact(wl, case["kind"] == "cart")
            for _ in range(case["n"]):
                a = ex.step(a, case["dz"])
            out.append(a)
        return out
    wl = wls[0]
    a, ex = torch.stack(fields), _Exact(wl, False)
    if case["kind"] == "adaptive":
        a = ex.adaptive(a, case["dz"], case["dz"] * (2 ** case["k"] - 1))
    else:
        for _ in range(case["n"]):
            a = ex.step(a, case["dz"])
    out = list(a)
    if case.get("record"):
        i = a[0].real ** 2 + a[0].imag ** 2
        dr = wl.r_max / (wl.nr - 1)
        weight = torch.arange(wl.nr, dtype=torch.float64, device="cuda")
        weight[0] = 0.125
        power = 2 * math.pi * dr * dr * (weight[:, None] * i).sum(0)
        out += [power.sum() * ex.dtau, power, i.sum(1) * ex.dtau]
    return out
