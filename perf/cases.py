"""Measured cases of the free-surface solver: what its users run, through the
public Python binding (`paper_2310_19840_gb300.sbi`).

A pass is one forecast segment: the state of every member in, a few time steps
(or one diagnostic), the new state (or the surface velocity) out.  Fields of a
single-precision context are handed on as float32, the precision they were
computed in and the one an analysis program keeps; double-precision contexts
return float64.
"""
import math

import torch

from paper_2310_19840_gb300 import sbi

G = 9.81
KP = 0.28 / (0.05 * math.sqrt(2.0))      # peak wavenumber of the seas [rad/m]
LAM = 2.0 * math.pi / KP
POINTS_PER_WAVE = 25.6                   # 256 points on ten wavelengths

_BASE = {"kind": "step", "grids": "", "scene": "sea", "steps": 1, "order": 7, "alpha": 0.5,
         "precision": "fp32", "integrator": "rk4", "diagnostic": "esbi", "filter": False}


def _case(name, **kw):
    return dict(_BASE, name=name, **kw)


def listed():
    return [
        # one solitary wave in a 1-D channel, between two outputs: the smallest
        # run, all launches
        _case("solitary_256", grids="256x1*1", scene="solitary", steps=8),
        # a numerical wave flume: submerged bar, wavemaker, absorbing layer
        _case("flume_1024", grids="1024x1*1", scene="flume", steps=4),
        # waves over a finely resolved submerged bar with sponge layers
        _case("bar_4096", grids="4096x1*1", scene="bar", steps=4),
        # one directional sea in deep water, the usual single forecast
        _case("sea_512", grids="512x512*1", steps=4),
        # the surface velocity of one wide sea over a barred bottom (forces on
        # a structure, a nested model's boundary)
        _case("velocity_1024x512", kind="velocity", grids="1024x512*1", scene="barred"),
        # a small ensemble of two resolutions
        _case("ensemble_12", grids="256x256*8+512x512*4", steps=2, filter=True),
        # the benchmark's ensemble of crossing seas
        _case("ensemble_96", grids="256x256*64+512x512*32", steps=1, filter=True),
        # an ensemble read from pinned host memory, the forecast left on the
        # device for the program that consumes it
        _case("ensemble_48_from_host", kind="stream", grids="256x256*32+512x512*16", steps=1, filter=True),
        # one sea of 64 x 32 wavelengths over bars, the largest grid
        _case("large_4096x2048", grids="4096x2048*1", scene="barred", steps=1, filter=True),
        # the double-precision reference run of a few members
        _case("ensemble_6_fp64", grids="256x256*4+512x512*2", steps=1, precision="fp64", filter=True),
        # the integrating-factor scheme on an ensemble
        _case("ensemble_24_lawson", grids="256x256*16+512x512*8", steps=1, integrator="lawson", filter=True),
        # the perturbation expansion users compare against, wide flat members
        _case("ensemble_8_hos", grids="512x128*8", steps=1, order=5, diagnostic="hos", filter=True),
    ]


def draw(rng):
    c = dict(_BASE, order=rng.choice([3, 4, 5, 6, 7, 7, 7, 7]))
    kind = rng.choice(["1d", "one", "one", "ensemble", "ensemble", "ensemble", "velocity", "stream"])
    if kind == "1d":
        c["scene"] = rng.choice(["solitary", "bar", "flume"])
        nx = 2 ** (rng.randint(6, 10) if c["scene"] == "solitary" else rng.randint(9, 12))
        c.update(grids="%dx1*1" % nx, steps=rng.randint(1, 9))
        return c
    # a wide sea or a narrow one, from 2^10 to 2^22 points in all
    c["scene"] = rng.choice(["sea", "sea", "barred"])
    total = 2.0 ** rng.uniform(10.0, 22.0)

    def grid(points):
        shape = rng.uniform(-1.5, 1.5)
        nx = min(12, max(5, round(0.5 * math.log2(points) + shape)))
        ny = min(11, max(4, round(math.log2(points) - nx)))
        return 2 ** nx, 2 ** ny

    if kind in ("one", "velocity"):
        nx, ny = grid(total)
        c.update(grids="%dx%d*1" % (nx, ny), kind="step" if kind == "one" else "velocity")
    else:
        parts = []
        for _ in range(rng.randint(1, 3)):
            n = rng.choice([1, 2, 3, 5, 7, 12, 17, 31])
            nx, ny = grid(max(1024.0, total / n))
            parts.append("%dx%d*%d" % (nx, ny, n))
        c.update(grids="+".join(parts), kind="stream" if kind == "stream" else "step")
    if rng.random() < 0.2 and _points(c) <= 2 ** 19:
        c["precision"] = "fp64"
    if c["kind"] == "velocity":
        return c
    c["filter"] = rng.random() < 0.6
    c["integrator"] = rng.choice(["rk4", "rk4", "rk4", "lawson"])
    if rng.random() < 0.15 and c["scene"] == "sea":
        c.update(diagnostic="hos", order=min(c["order"], 5))
    if rng.random() < 0.2:
        # a wider or a narrower band of kept modes, on a gentler sea
        c.update(alpha=rng.choice([1.0 / 3.0, 0.75]), order=min(c["order"], 5))
    c["steps"] = max(1, min(4, int(rng.uniform(1.0, 5.0)), 2 ** 22 // _points(c)))
    return c


# ---------------------------------------------------------------------------
# grids and inputs
# ---------------------------------------------------------------------------
def _grids(case):
    """(nx, ny, members) per part of the ensemble, in member order."""
    out = []
    for part in case["grids"].split("+"):
        size, n = part.split("*")
        nx, ny = size.split("x")
        out.append((int(nx), int(ny), int(n)))
    return out


def _points(case):
    return sum(nx * ny * n for nx, ny, n in _grids(case))


def _rng(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _freq(n, L, dev="cuda"):
    return torch.fft.fftfreq(n, d=L / n, dtype=torch.float64, device=dev) * (2.0 * math.pi)


def _dispersion(omega, h):
    k = omega * omega / G
    for _ in range(100):
        f = G * k * math.tanh(k * h) - omega * omega
        k -= f / (G * math.tanh(k * h) + G * k * h / math.cosh(k * h) ** 2)
    return k


def _sea(n, ny, nx, Lx, Ly, h, hs, alpha, gen):
    """n random seas, two JONSWAP systems at +-20 degrees each, in the band of
    kept modes: eta, phi~ (n, ny, nx)."""
    a = min(alpha, 0.5)
    KY, KX = torch.meshgrid(_freq(ny, Ly), _freq(nx, Lx), indexing="ij")
    K = torch.hypot(KX, KY)
    ok = K > 0
    k = torch.where(ok, K, torch.ones_like(K))
    w = torch.sqrt(G * k * torch.tanh(k * h))
    wp = math.sqrt(G * KP * math.tanh(KP * h))
    sig = torch.where(w <= wp, 0.07, 0.09)
    peak = torch.exp(-((w - wp) ** 2) / (2.0 * sig ** 2 * wp ** 2))
    S = w ** -5.0 * torch.exp(-1.25 * (wp / w) ** 4) * 3.3 ** peak
    kh2 = (2.0 * k * h).clamp(max=600.0)
    S = torch.where(ok, S * 0.5 * w / k * (1.0 + kh2 / torch.sinh(kh2)) / k, torch.zeros_like(K))
    mx = torch.arange(nx, device="cuda")
    my = torch.arange(ny, device="cuda")
    band = (torch.minimum(my, ny - my) < a * ny / 2 - 1e-9)[:, None] & (torch.minimum(mx, nx - mx) < a * nx / 2 - 1e-9)[None, :]
    theta = torch.atan2(KY, KX)
    C = torch.zeros((n, ny, nx), dtype=torch.complex128, device="cuda")
    for th0 in (math.radians(20.0), -math.radians(20.0)):
        d = torch.remainder(theta - th0 + math.pi, 2.0 * math.pi) - math.pi
        D = torch.where(d.abs() < 0.5 * math.pi, torch.cos(d) ** 2, torch.zeros_like(d))
        a2 = S * D * band
        m0 = float(0.5 * a2.sum())
        amp = torch.sqrt(a2 * ((hs / 4.0) ** 2 / m0 if m0 > 0 else 0.0))
        ph = torch.rand((n, ny, nx), generator=gen, dtype=torch.float64, device="cuda") * (2.0 * math.pi)
        C += torch.polar(amp.expand(n, -1, -1).contiguous(), ph)
    eta = torch.fft.ifft2(C).real * (nx * ny)
    phi = torch.fft.ifft2(C * (ok * (-1j * G) / w)).real * (nx * ny)
    return eta.contiguous(), phi.contiguous()


def _bar_depth(x, h0, toe):
    h = torch.full_like(x, h0)
    up, top, down = (x >= toe) & (x < toe + 6), (x >= toe + 6) & (x < toe + 8), (x >= toe + 8) & (x < toe + 11)
    h = torch.where(up, h0 - (x - toe) / 20.0, h)
    h = torch.where(top, torch.full_like(x, 0.1), h)
    return torch.where(down, 0.1 + (x - toe - 8.0) / 10.0, h)


def _scene(case, seed):
    """Everything that describes the problem: per part of the ensemble its box,
    depth, bottom and initial state; and the options shared by all members."""
    gen = _rng(seed)
    u = torch.rand(4, generator=gen, dtype=torch.float64, device="cuda").tolist()
    s = {"parts": [], "sponge": None, "nu": 0.0, "wave": None, "k_ref": 1.0,
         "dt": 0.0, "beta": (8.0, 30.0) if case["filter"] else (0.0, 0.0)}
    if case["scene"] in ("sea", "barred"):
        barred = case["scene"] == "barred"
        h = (1.5 if barred else 5.0) / KP
        hs = 0.05 if abs(case["alpha"] - 0.5) < 0.01 else 0.02
        for nx, ny, n in _grids(case):
            Lx, Ly = nx / POINTS_PER_WAVE * LAM, ny / POINTS_PER_WAVE * LAM
            eta, phi = _sea(n, ny, nx, Lx, Ly, h, hs, case["alpha"], gen)
            delta = None
            if barred:   # ten bars of half a wavelength across the middle of the box
                lb = min(0.5 * LAM, Lx / 20.0)
                x = torch.arange(nx, dtype=torch.float64, device="cuda") * (Lx / nx) - (0.5 * Lx - 5.0 * lb)
                ramp = torch.minimum(x, 10.0 * lb - x).clamp(0.0, 0.5 * lb) / (0.5 * lb)
                d = 0.3 * h * torch.sin(2.0 * math.pi * x / lb) * 0.5 * (1.0 - torch.cos(math.pi * ramp))
                delta = d.expand(n, ny, nx).contiguous()
            s["parts"].append({"nx": nx, "ny": ny, "n": n, "Lx": Lx, "Ly": Ly, "h0": h, "eta": eta, "phi": phi,
                               "delta": delta})
        s["dt"] = 2.0 * math.pi / math.sqrt(G * KP * math.tanh(KP * h)) / 32.0
        s["k_ref"] = KP
        return s
    nx, _, _ = _grids(case)[0]
    p = {"nx": nx, "ny": 1, "n": 1, "Ly": 1.0, "delta": None}
    if case["scene"] == "solitary":
        L, h, a, x0 = 100.0, 1.0, 0.2 + 0.1 * u[0], 25.0 + 50.0 * u[1]
        x = torch.arange(nx, dtype=torch.float64, device="cuda") * (L / nx)
        d = torch.remainder(x - x0 + 0.5 * L, L) - 0.5 * L
        eta = a / torch.cosh(math.sqrt(3.0 * a / (4.0 * h * h * (h + a))) * d) ** 2
        U = torch.fft.fft(math.sqrt(G * (h + a)) * eta / (h + eta))
        k = _freq(nx, L)
        k[0] = 1.0
        U = U / (1j * k)
        U[0] = 0.0
        U[nx // 2] = 0.0
        phi = torch.fft.ifft(U).real
        s["dt"] = 0.01 * min(1.0, 256.0 / nx)
    else:
        flume = case["scene"] == "flume"
        L, h, T = (64.0 if flume else 80.0), 0.4, 2.02
        a, w = 0.008 + 0.004 * u[0], 2.0 * math.pi / T
        x = torch.arange(nx, dtype=torch.float64, device="cuda") * (L / nx)
        k = _dispersion(w, h)
        env = a * torch.exp(-((x - 18.0 - 4.0 * u[1]) ** 2) / 32.0)
        eta, phi = env * torch.cos(k * x), (G / w) * env * torch.sin(k * x)
        p["delta"] = (h - _bar_depth(x, h, 10.0 if flume else 30.0)).reshape(1, 1, nx)
        if flume:
            d = torch.remainder(x - 7.0 / 8.0 * L + 0.5 * L, L) - 0.5 * L
            s["sponge"] = torch.exp(-(k * d / (4.0 * math.pi)) ** 2).reshape(1, nx)
            s["wave"] = {"amp": a, "omega": w, "phase": 2.0 * math.pi * u[2], "k": k, "t0": 3.0 * u[3]}
        else:
            edge = torch.maximum(10.0 - x, x - 70.0).clamp(min=0.0) / 10.0
            s["sponge"] = (torch.sin(0.5 * math.pi * edge) ** 2).reshape(1, nx)
        s["nu"] = w
        s["dt"] = 0.005 if nx >= 2048 else 0.01
    # the band a state of this solver has (modes below a quarter of the grid)
    kept = torch.arange(nx // 2 + 1, device="cuda") < nx // 4
    eta, phi = [torch.fft.irfft(torch.fft.rfft(v) * kept, n=nx) for v in (eta, phi)]
    p.update(Lx=L, h0=h, eta=eta.reshape(1, 1, nx).contiguous(), phi=phi.reshape(1, 1, nx).contiguous())
    s["parts"].append(p)
    return s


def _flat(parts, key):
    return torch.cat([p[key].reshape(-1) for p in parts]).contiguous()


def prepare(case, seed):
    s = _scene(case, seed)
    parts = s["parts"]
    grids, depths = [], []
    for p in parts:
        grids += [(p["nx"], p["ny"], p["Lx"], p["Ly"])] * p["n"]
        depths += [None] * p["n"] if p["delta"] is None else [d.cpu().numpy() for d in (p["h0"] - p["delta"])]
    ctx = sbi.Context(
        grids, G, depths, h0=parts[0]["h0"], order=case["order"], alias_frac=case["alpha"],
        precision=sbi.SBI_FP64 if case["precision"] == "fp64" else sbi.SBI_FP32,
        filt_beta1=s["beta"][0], filt_beta2=s["beta"][1], k_ref=s["k_ref"],
        sponge_w=None if s["sponge"] is None else s["sponge"].cpu().numpy(), sponge_nu=s["nu"],
        integrator=sbi.SBI_LAWSON_RK4 if case["integrator"] == "lawson" else sbi.SBI_RK4,
        diagnostic=sbi.SBI_DIAG_HOS if case["diagnostic"] == "hos" else sbi.SBI_DIAG_ESBI)
    if s["wave"]:
        w = s["wave"]
        ctx.set_wavemaker([w["amp"]], [w["omega"]], [w["phase"]], 0.0)
    eta, phi = _flat(parts, "eta"), _flat(parts, "phi")
    state = {"ctx": ctx, "case": case, "dt": s["dt"], "t0": s["wave"]["t0"] if s["wave"] else None,
             "out": (torch.empty_like(eta), torch.empty_like(phi))}
    if case["kind"] == "stream":
        eta, phi = eta.cpu().pin_memory(), phi.cpu().pin_memory()
    state["in"] = (eta, phi)
    return state


def _keep(case, t):
    return t.float() if case["precision"] == "fp32" else t


def run(state):
    ctx, case = state["ctx"], state["case"]
    (eta, phi), (eta_out, phi_out) = state["in"], state["out"]
    if case["kind"] == "velocity":
        ctx.set_state_all(eta, phi)
        ctx.vertical_velocity(0, out=eta_out)
        return {"V": _keep(case, eta_out)}
    if case["kind"] == "stream":
        ctx.step_streamed(eta, phi, state["dt"], case["steps"], eta_out, phi_out)
    else:
        ctx.set_state_all(eta, phi)
        if state["t0"] is not None:
            ctx.set_time(state["t0"])
        ctx.step(state["dt"], case["steps"])
        ctx.get_state_all(eta_out, phi_out)
    return {"eta": _keep(case, eta_out), "phi": _keep(case, phi_out)}


def work(case):
    """State in and out once (and the bottom); two-dimensional real transforms
    of the scheme at 2.5 N log2 N operations each."""
    size = 8.0
    bottom = case["scene"] in ("barred", "bar", "flume")
    M, fields, nbytes, flops = case["order"], 4 if case["kind"] != "velocity" else 3, 0.0, 0.0
    stages = 1 if case["kind"] == "velocity" else 4 * case["steps"]
    for nx, ny, n in _grids(case):
        N, dims = float(nx * ny), 2 if ny > 1 else 1
        if case["diagnostic"] == "hos":
            tr = M * (M - 1) + 2 * M + 2
        else:
            # physical V_l and grad phi~, the products eta^j V_l and eta^l grad phi~
            tr = (M - 1) + dims + M * (M - 1) // 2 + dims * (M - 1) + 1
            if bottom:   # grad varphi_l and the products delta^j grad varphi_l
                tr += dims * ((M - 1) + M * (M - 1) // 2)
        if case["kind"] != "velocity":
            tr += dims + 1
        nbytes += n * N * (fields * size + (size if bottom else 0.0))
        flops += n * stages * tr * 2.5 * N * math.log2(N)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
# the same results in 64 bits, with plain torch transforms
# ---------------------------------------------------------------------------
class _Exact:
    """One part of the ensemble: the scheme of arXiv 2310.19840 in float64."""

    def __init__(self, case, s, p):
        self.case, self.s, self.p = case, s, p
        nx, ny = p["nx"], p["ny"]
        self.two_d = ny > 1
        ky = _freq(ny, p["Ly"]) if self.two_d else torch.zeros(1, dtype=torch.float64, device="cuda")
        kx = _freq(nx, p["Lx"])[: nx // 2 + 1].abs()
        self.KY, self.KX = torch.meshgrid(ky, kx, indexing="ij")
        self.K = torch.hypot(self.KX, self.KY)
        self.inv = torch.where(self.K > 0, 1.0 / self.K.clamp(min=1e-300), torch.zeros_like(self.K))
        h = p["h0"]
        self.th = torch.tanh(self.K * h)
        e = torch.exp(-self.K * h)
        self.sech = 2.0 * e / (1.0 + e * e)
        a = case["alpha"]
        mx = torch.arange(nx // 2 + 1, device="cuda")
        my = torch.arange(ny, device="cuda")
        kept = (mx < a * nx / 2 - 1e-12) & (mx < nx // 2)
        my = torch.minimum(my, ny - my)
        kept_y = (my < a * ny / 2 - 1e-12) & (my < ny // 2) if self.two_d else my >= 0
        self.mask = (kept_y[:, None] & kept[None, :]).double()
        self.lam = self.mask
        b1, b2 = s["beta"]
        if b1 > 0:
            self.lam = self.mask * torch.exp(-(self.K / (b1 * s["k_ref"])) ** b2)

    def f(self, v):
        return torch.fft.rfft2(v)

    def g(self, v):
        return torch.fft.irfft2(v, s=(self.p["ny"], self.p["nx"]))

    def kp(self, n):
        return self.K ** n if n >= 0 else self.inv ** (-n)

    def grad(self, v):
        return [self.g(1j * self.KX * v)] + ([self.g(1j * self.KY * v)] if self.two_d else [])

    def div(self, a):
        v = 1j * self.KX * self.f(a[0])
        return v + 1j * self.KY * self.f(a[1]) if self.two_d else v

    def velocity(self, eta, phi):
        """Spectrum of V and the gradient of phi~."""
        M = self.case["order"]
        ph = self.f(phi) * self.mask
        gphi = self.grad(ph)
        if self.case["diagnostic"] == "hos":
            return self.hos(eta, ph, gphi), gphi
        delta, T = self.p["delta"], [torch.ones_like(self.th), self.th]
        Vh = {1: self.K * self.th * ph}
        V = {1: self.g(Vh[1])}
        gb = {1: self.grad(self.sech * ph)} if delta is not None else {}
        ep = [torch.ones_like(eta)]
        dp = [torch.ones_like(eta)]
        for _ in range(M):
            ep.append(ep[-1] * eta)
            if delta is not None:
                dp.append(dp[-1] * delta)
        for l in range(2, M + 1):
            A = torch.zeros_like(ph)
            B = torch.zeros_like(ph)
            for j in range(1, l):
                F = self.f(ep[j] * V[l - j])
                A = A - self.kp(j) / math.factorial(j) * T[j % 2] * F
                if j % 2:
                    B = B - self.kp(j - 1) / math.factorial(j) * self.sech * F
                if delta is not None:
                    D = self.div([dp[j] * q for q in gb[l - j]])
                    if j % 2:
                        A = A + self.kp(j - 1) / math.factorial(j) * self.sech * D
                    B = B + (-1.0) ** j * self.kp(j - 2) / math.factorial(j) * T[j % 2] * D
            Q = self.div([ep[l - 1] * q for q in gphi]) / math.factorial(l - 1)
            A = A - T[l % 2] * self.kp(l - 2) * Q
            if l % 2:
                B = B - self.sech * self.kp(l - 3) * Q
            Vh[l] = A * self.mask
            V[l] = self.g(Vh[l])
            if delta is not None:
                gb[l] = self.grad(B * self.mask)
        return sum(Vh.values()), gphi

    def hos(self, eta, ph, gphi):
        M, T = self.case["order"], [torch.ones_like(self.th), self.th]
        dz = lambda v, n: self.g(self.K ** n * T[n % 2] * v)
        P = {1: ph}
        for m in range(2, M + 1):
            v = -sum(eta ** n / math.factorial(n) * dz(P[m - n], n) for n in range(1, m))
            P[m] = self.f(v) * self.mask
        W = sum(eta ** n / math.factorial(n) * dz(sum(P[m] for m in range(1, M - n + 1)), n + 1) for n in range(M))
        W = self.g(self.f(W) * self.mask)
        ge = self.grad(self.f(eta) * self.mask)
        V = W * (1.0 + sum(q * q for q in ge)) - sum(q * r for q, r in zip(ge, gphi))
        return self.f(V) * self.mask

    def rhs(self, eta, phi, t):
        """Spectra of eta_t and phi~_t."""
        Vh, gphi = self.velocity(eta, phi)
        V, ge = self.g(Vh), self.grad(self.f(eta) * self.mask)
        dot = sum(q * r for q, r in zip(ge, gphi))
        N = -G * eta + 0.5 * ((V + dot) ** 2 / (1.0 + sum(q * q for q in ge)) - sum(q * q for q in gphi))
        if self.s["wave"]:
            N = N - self.pressure(t)
        F = self.f(N)
        if self.s["sponge"] is not None:
            F = F + self.s["nu"] * self.inv ** 2 * self.div([self.s["sponge"] * q for q in gphi])
        return Vh, F * self.mask

    def pressure(self, t):
        w, L, h, nx = self.s["wave"], self.p["Lx"], self.p["h0"], self.p["nx"]
        x = torch.arange(nx, dtype=torch.float64, device="cuda") * (L / nx)
        d = torch.remainder(x + 0.5 * L, L) - 0.5 * L
        k = w["k"]
        f = G * w["amp"] * math.sqrt(math.e / (2.0 * math.pi)) * (1.0 + 2.0 * k * h / math.sinh(2.0 * k * h))
        return f * torch.exp(-0.5 * (k * d) ** 2) * math.sin(w["omega"] * t + w["phase"])

    def rk4(self, eta, phi, t, dt):
        def rate(e, q, tt):
            a, b = self.rhs(e, q, tt)
            return self.g(a), self.g(b)
        k1 = rate(eta, phi, t)
        k2 = rate(eta + 0.5 * dt * k1[0], phi + 0.5 * dt * k1[1], t + 0.5 * dt)
        k3 = rate(eta + 0.5 * dt * k2[0], phi + 0.5 * dt * k2[1], t + 0.5 * dt)
        k4 = rate(eta + dt * k3[0], phi + dt * k3[1], t + dt)
        return [y + dt / 6.0 * (a + 2.0 * b + 2.0 * c + d)
                for y, a, b, c, d in zip((eta, phi), k1, k2, k3, k4)]

    def lawson(self, eta, phi, t, dt):
        w = torch.sqrt(G * self.K * self.th)
        wi = torch.where(w > 0, 1.0 / w.clamp(min=1e-300), torch.zeros_like(w))

        def E(tau, u):
            c, sn = torch.cos(w * tau), torch.sin(w * tau)
            sg = torch.where(w > 0, G * wi * sn, torch.full_like(w, G * tau))
            return c * u[0] + self.K * self.th * wi * sn * u[1], c * u[1] - sg * u[0]

        def N(u, tt):
            e, q = self.g(u[0]), self.g(u[1])
            a, b = self.rhs(e, q, tt)
            lin = self.K * self.th * u[1] * self.mask
            return a - lin, b + G * u[0] * self.mask

        ax = lambda u, c, v: (u[0] + c * v[0], u[1] + c * v[1])
        u = (self.f(eta) * self.mask, self.f(phi) * self.mask)
        k1 = N(u, t)
        uh, k1h = E(0.5 * dt, u), E(0.5 * dt, k1)
        k2 = N(ax(uh, 0.5 * dt, k1h), t + 0.5 * dt)
        k3 = N(ax(uh, 0.5 * dt, k2), t + 0.5 * dt)
        u1 = E(dt, u)
        k4 = N(ax(u1, dt, E(0.5 * dt, k3)), t + dt)
        for c, k in ((dt / 6.0, E(dt, k1)), (dt / 3.0, E(0.5 * dt, k2)), (dt / 3.0, E(0.5 * dt, k3)), (dt / 6.0, k4)):
            u1 = ax(u1, c, k)
        return [self.g(u1[0]), self.g(u1[1])]

    def run(self):
        band = lambda v, m: self.g(self.f(v) * m)
        eta, phi = band(self.p["eta"], self.mask), band(self.p["phi"], self.mask)
        if self.case["kind"] == "velocity":
            return self.g(self.velocity(eta, phi)[0]), None
        t, dt = self.s["wave"]["t0"] if self.s["wave"] else 0.0, self.s["dt"]
        step = self.lawson if self.case["integrator"] == "lawson" else self.rk4
        for _ in range(self.case["steps"]):
            eta, phi = [band(v, self.lam) for v in step(eta, phi, t, dt)]
            t += dt
        return eta, phi


def exact(case, seed):
    s = _scene(case, seed)
    done = []
    for p in s["parts"]:
        rows = []
        some = max(1, 2 ** 22 // (p["nx"] * p["ny"]))      # members at a time
        for m in range(0, p["n"], some):
            q = dict(p, **{key: p[key][m:m + some] for key in ("eta", "phi", "delta") if p[key] is not None})
            rows.append(_Exact(case, s, q).run())
        done.append([torch.cat([r[i].reshape(-1) for r in rows]) if rows[0][i] is not None else None for i in (0, 1)])
    if case["kind"] == "velocity":
        return {"V": done[0][0]}
    return {"eta": torch.cat([d[0] for d in done]), "phi": torch.cat([d[1] for d in done])}
