"""The work that this library is measured on, through its public Python entry points.

Every case is a plain dict.  ``kind`` says which calls a pass makes:

  propagate    set_fields, propagate, get_fields of one simulation (device buffers)
  batch        set_fields of every instance, one Batch.run, get_fields of every instance
  adjoint      adjoint_forward and adjoint_backward: the gradient of one objective
  diagnostics  set_fields and the power trace and spectrum of the fields
  thermal      set_fields, the heat load of the fields and the thermal map it gives

``fields`` names the set of coupled fields: ``shg`` (SH, F, no dispersion), ``mix``
(pump, signal, idler with walk-off, group-velocity mismatch and dispersion, driven at
signal and idler), ``opg`` (the same, driven at the pump, signal and idler from noise),
``lossy`` (``mix`` with third-order dispersion and loss).
"""
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

import paper_2609_08384_gb300 as br
from paper_2609_08384_gb300 import workloads as wl

C0, EPS0 = 299792458.0, 8.8541878128e-12
UM, FS, MM = 1e-6, 1e-15, 1e-3
D_EFF = 14e-12
KAPPA_TH, DKDT, REP_RATE = 4.0, 150.0, 1e6

# lengths that a grid axis may have (small and large ones beside those of the listed cases)
LENGTHS = (8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512, 768, 1024)
MOST_POINT_STEPS = 3 * 256 * 256 * 512 * 20  # fields x points x steps of the largest case


def _case(name, kind, nx, ny, nt, fields, nz, dx, dt, **more):
    c = {"name": name, "kind": kind, "nx": nx, "ny": ny, "nt": nt, "fields": fields, "nz": nz, "dx": dx, "dt": dt,
         "dz": 10 * UM, "dk": 0.0, "profile": False, "fanout": False, "count": 1}
    c.update(more)
    return c


def listed():
    return [
        # the smallest problem of the workloads (32x32x64 SHG over 1 mm): 400 dependent launches of microseconds each
        _case("shg_32x32x64", "propagate", 32, 32, 64, "shg", 100, 12.5 * UM, 50 * FS),
        # a mid-size member of the parameter sweeps, run by itself with a per-step mismatch profile
        _case("shg_96x96x192_profile", "propagate", 96, 96, 192, "shg", 50, 12.5 * UM, 50 * FS, profile=True),
        # three fields with every linear term on a ragged grid of 3 2^k lengths
        _case("lossy_48x192x384", "propagate", 48, 192, 384, "lossy", 30, 6.25 * UM, 25 * FS, dk=30.0),
        # the sum-frequency workload: 128x128x256, three fields, mismatched
        _case("sfg_128x128x256", "propagate", 128, 128, 256, "mix", 40, 3.75 * UM, 15.625 * FS, dk=20.0),
        # the benchmark's workload: parametric generation from noise, 256x256x512, phase matched
        _case("opg_256x256x512", "propagate", 256, 256, 512, "opg", 20, 3.125 * UM, 31.25 * FS),
        # the same in a fan-out grating: a mismatch map across x
        _case("opg_256x256x512_fanout", "propagate", 256, 256, 512, "opg", 12, 3.125 * UM, 31.25 * FS, fanout=True),
        # continuous-wave focused SHG: a large transverse grid without a time axis
        _case("cw_1024x1024", "propagate", 1024, 1024, 1, "shg", 60, 0.5 * UM, 1 * FS, dk=-223.0, dz=14.5 * UM),
        # a parameter sweep over small grids, one graph launch
        _case("batch_32x32x64", "batch", 32, 32, 64, "shg", 60, 12.5 * UM, 50 * FS, count=32),
        # a sweep over the two larger grids of the sweeps (every other instance has half the points per axis)
        _case("batch_128x128x256", "batch", 128, 128, 256, "shg", 24, 12.5 * UM, 50 * FS, count=8),
        # one gradient of the pulse-shaping and poling design loop (checkpointed forward, reverse sweep)
        _case("adjoint_128x128x256", "adjoint", 128, 128, 256, "shg", 36, 12.5 * UM, 50 * FS, dz=50 * UM, dk=200.0),
        # power trace and spectrum of a large state
        _case("diagnostics_256x256x512", "diagnostics", 256, 256, 512, "opg", 1, 3.125 * UM, 31.25 * FS),
        # one thermal iteration: heat load of the fields, heat equation, mismatch map
        _case("thermal_512x512x64", "thermal", 512, 512, 64, "lossy", 1, 3.125 * UM, 62.5 * FS),
    ]


def draw(rng):
    """One more case of the same ranges: every kind, lengths spread over their logarithm."""

    def length(low, high):
        return rng.choice([n for n in LENGTHS if low <= n <= high])

    kind = rng.choice(["propagate"] * 6 + ["batch", "batch", "adjoint", "diagnostics", "thermal"])
    fields = rng.choice(["shg", "mix", "opg", "lossy"]) if kind in ("propagate", "diagnostics", "thermal") else "shg"
    fields = "lossy" if kind == "thermal" else fields  # the heat load is the absorbed power
    nf = 2 if fields == "shg" else 3
    flat = kind == "propagate" and rng.random() < 0.15
    while True:
        nx, ny, nt = length(16, 512), length(8, 512), length(8, 768)
        if flat:
            nx, ny, nt = length(128, 1024), length(128, 1024), 1
        if kind in ("batch", "adjoint"):
            nx, ny, nt = length(32, 128), length(32, 128), length(32, 256)
        if kind in ("diagnostics", "thermal"):
            nx, ny = length(64, 512), length(64, 512)
        if 8192 <= nx * ny * nt and nf * nx * ny * nt <= 3 * 256 * 256 * 512:
            break
    count = rng.randint(3, 30) if kind == "batch" else 1
    low, high = (1, 1) if kind in ("diagnostics", "thermal") else (16, 40) if kind == "adjoint" else (8, 100)
    most = MOST_POINT_STEPS // (nf * nx * ny * nt * (4 if kind == "adjoint" else 1))
    if kind == "batch":
        count = max(1, min(count, most // low, (1 << 25) // (nx * ny * nt)))
        most //= count
    nz = max(1, min(most, int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))))
    # windows of 0.4 to 0.8 mm and 3.2 to 16 ps, as in the workloads
    return {"kind": kind, "nx": nx, "ny": ny, "nt": nt, "fields": fields, "nz": nz,
            "dx": rng.uniform(400, 800) * UM / max(nx, ny), "dt": rng.uniform(3200, 16000) * FS / max(nt, 8),
            "dz": rng.choice([5, 10]) * UM if kind != "adjoint" else rng.uniform(1.0, 2.0) * MM / nz, "dk": rng.choice([0.0, rng.uniform(-200.0, 200.0)]),
            "profile": kind == "propagate" and rng.random() < 0.3, "fanout": kind == "propagate" and rng.random() < 0.2,
            "count": count}


# ------------------------------------------------------------------ the problem, as plain numbers
def _fields_of(case):
    """(lambda, n, delta, k2, k3, rho, alpha) of every field."""
    if case["fields"] == "shg":
        return [(532e-9, 2.234, 0.0, 0.0, 0.0, 0.0, 0.0), (1064e-9, 2.156, 0.0, 0.0, 0.0, 0.0, 0.0)]
    gvm, gvd = 100 * FS / MM, FS * FS / MM
    lossy = case["fields"] == "lossy"
    k3, alpha = (40 * FS**3 / MM, 20.0) if lossy else (0.0, 0.0)
    rho = (2e-3, 0.0, 1e-3) if case["fields"] != "mix" else (0.0, 0.0, 2e-3)
    return [(1064e-9, 2.15, gvm, 200 * gvd, k3, rho[0], alpha),
            (1450e-9, 2.14, 0.0, 100 * gvd, 0.5 * k3, rho[1], 0.5 * alpha),
            (3997e-9, 2.08, -gvm, 50 * gvd, 0.25 * k3, rho[2], 2 * alpha)]


def _members(case, seed):
    """The instances of a batch: (nx, ny, nt, nz, dk) each."""
    r = np.random.default_rng(seed)
    got = []
    for i in range(case["count"]):
        h = 2 if case["count"] < 16 and i % 2 and min(case["nx"], case["ny"], case["nt"]) >= 64 else 1
        # step counts from half the longest up; the longest is always there, so passes of other inputs cost alike
        nz = case["nz"] if i < 2 else max(1, case["nz"] - (i * case["nz"]) // (2 * case["count"]))
        got.append((case["nx"] // h, case["ny"] // h, case["nt"] // h, nz, float(r.uniform(-200.0, 200.0))))
    return got


def _axis(n, d):
    return (torch.arange(n, dtype=torch.float64, device="cuda") - n // 2) * d


def _pulse(nx, ny, nt, dx, dt, lam, n, w0, tau0, intensity, delay, length):
    """Focused Gaussian beam (waist at length / 2) times a Gaussian pulse, complex64 [nt, ny, nx]."""
    a0 = math.sqrt(2.0 * intensity / (C0 * EPS0 * n))
    q = 1.0 - 1j * (0.5 * length / (math.pi * n / lam * w0 * w0))
    ex = torch.exp(-_axis(nx, dx) ** 2 / (w0 * w0 * q))
    ey = torch.exp(-_axis(ny, dx) ** 2 / (w0 * w0 * q)) * (a0 / q)
    et = torch.exp(-(((_axis(nt, dt) - delay) / tau0) ** 2)) if nt > 1 else torch.ones(1, dtype=torch.float64, device="cuda")
    return (et[:, None, None].to(torch.complex64) * (ey[:, None] * ex[None, :]).to(torch.complex64)[None]).contiguous()


def _noise(shape, rms, g):
    return torch.view_as_complex(torch.randn(*shape, 2, generator=g, device="cuda", dtype=torch.float32) * (rms / math.sqrt(2.0)))


def _inputs(case, seed, member=None):
    """The initial envelopes, from the seed alone: peak intensity, waist, duration and delay vary with it."""
    r = np.random.default_rng(seed if member is None else [seed, member])
    nx, ny, nt = (case["nx"], case["ny"], case["nt"]) if member is None else _members(case, seed)[member][:3]
    dx, dt = case["dx"], case["dt"]
    wx, wt = dx * min(nx, ny), dt * max(nt, 8)
    length = case["nz"] * case["dz"]
    w0, tau0 = wx * r.uniform(0.11, 0.14), wt * r.uniform(0.06, 0.09)
    power, late = 1e13 * r.uniform(0.7, 1.3), wt * r.uniform(-0.02, 0.02)
    f = _fields_of(case)
    g = torch.Generator(device="cuda")
    g.manual_seed(int(r.integers(1 << 60)))
    pulse = lambda k, w, t, p, d: _pulse(nx, ny, nt, dx, dt, f[k][0], f[k][1], w, t, p, d, length)  # noqa: E731
    if case["fields"] == "shg":
        a = pulse(1, w0, tau0, power, late)
        return [torch.zeros_like(a), a]
    if case["fields"] == "opg":
        rms = 1e-6 * math.sqrt(2.0 * power / (C0 * EPS0 * f[0][1]))
        return [pulse(0, w0, tau0, power, late), _noise((nt, ny, nx), rms, g), _noise((nt, ny, nx), rms, g)]
    s = pulse(1, w0, tau0, power, late)
    i = pulse(2, 1.3 * w0, 1.4 * tau0, 0.8 * power, -late)
    return [torch.zeros_like(s), s, i]


def _profile(case, seed):
    """Mismatch of every step, 1/m."""
    if not case["profile"] and case["kind"] != "adjoint":
        return np.full(case["nz"], case["dk"])
    return case["dk"] + np.random.default_rng([seed, 7]).normal(0.0, 100.0, case["nz"])


def _fanout(case):
    """Mismatch map [ny, nx] of a fan-out grating: linear across x, 1/m."""
    x = (np.arange(case["nx"]) - case["nx"] // 2) / case["nx"]
    return np.ascontiguousarray(np.broadcast_to(400.0 * x, (case["ny"], case["nx"])))


def _phase(case, seed):
    return np.random.default_rng([seed, 8]).normal(0.0, 0.1, case["nt"])


def _weights(case, inputs):
    f = _fields_of(case)
    return [f[0][1] / (f[1][1] * float(inputs[1].abs().double().square().sum())), 0.0]


# ------------------------------------------------------------------ the calls
def prepare(case, seed):
    f = [wl.FieldParams(*v) for v in _fields_of(case)]
    if case["kind"] == "batch":
        members = _members(case, seed)
        b = br.Batch()
        inputs = []
        for i, (nx, ny, nt, nz, dk) in enumerate(members):
            b.add(wl.Grid(nx, ny, nt, case["dx"], case["dx"], case["dt"]), f, D_EFF, dk, nz, case["dz"])
            inputs.append(_inputs(case, seed, i))
            b.set_fields(i, inputs[-1])
        b.run()  # the sweep is laid out and captured once
        b.sync()
        return {"case": case, "batch": b, "inputs": inputs}
    g = wl.Grid(case["nx"], case["ny"], case["nt"], case["dx"], case["dx"], case["dt"])
    s = br.Solver(g, f, D_EFF, case["dk"])
    inputs = _inputs(case, seed)
    st = {"case": case, "solver": s, "inputs": inputs}
    if case["kind"] == "propagate":
        st["out"] = [torch.empty_like(a) for a in inputs]
        if case["profile"]:
            s.set_dk_profile(_profile(case, seed))
        if case["fanout"]:
            s.set_dk_map(_fanout(case))
    if case["kind"] == "adjoint":
        st["dk"], st["phi"], st["weights"] = _profile(case, seed), _phase(case, seed), _weights(case, inputs)
    if case["kind"] == "thermal":
        s.set_fields(inputs)
        s.heat_accumulate(REP_RATE)  # the model's tables and planes are there from the first iteration on
    return st


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        b = state["batch"]
        for i, a in enumerate(state["inputs"]):
            b.set_fields(i, a)
        b.run()
        return [b.get_fields(i, on_device=True) for i in range(len(state["inputs"]))]
    s = state["solver"]
    if case["kind"] == "propagate":
        s.set_fields(state["inputs"])
        s.propagate(case["nz"], case["dz"])
        return s.get_fields(out=state["out"], on_device=True)
    if case["kind"] == "adjoint":
        j = s.adjoint_forward(state["inputs"], state["dk"], case["nz"], case["dz"], state["weights"], phi=state["phi"])
        gphi, gdk = s.adjoint_backward()
        # single precision, as the fields they come from and as an optimiser of float32 parameters takes them
        return {"j": np.float32(j), "phi": gphi.astype(np.float32), "dk": gdk.astype(np.float32)}
    if case["kind"] == "diagnostics":
        s.set_fields(state["inputs"])
        power, spectrum = s.diagnostics()
        return {"power": power.astype(np.float32), "spectrum": spectrum.astype(np.float32)}
    s.set_fields(state["inputs"])
    s.heat_set(None)
    s.heat_accumulate(REP_RATE)
    return s.thermal_map(KAPPA_TH, DKDT)


# ------------------------------------------------------------------ what a pass cannot do without
def _step_flops(nx, ny, nt, nf):
    """Two transforms of every axis, the propagator, two RK4 half steps."""
    n = nx * ny * nt
    return n * (nf * (10 * math.log2(n) + 6) + 2 * (222 if nf == 3 else 148))


def work(case):
    nx, ny, nt, nf = case["nx"], case["ny"], case["nt"], len(_fields_of(case))
    n = nx * ny * nt
    if case["kind"] == "batch":
        m = _members(case, 0)
        return {"bytes": sum(2 * 16 * a * b * c for a, b, c, _, _ in m),
                "flops": sum(z * _step_flops(a, b, c, 2) for a, b, c, z, _ in m)}
    if case["kind"] == "propagate":
        return {"bytes": 2 * 8 * nf * n, "flops": case["nz"] * _step_flops(nx, ny, nt, nf)}
    if case["kind"] == "adjoint":
        # forward, and the reverse step (the linear step and the vector-Jacobian products, about twice the RK4 work)
        return {"bytes": 8 * nf * n, "flops": 2 * case["nz"] * (_step_flops(nx, ny, nt, nf) + 148 * n)}
    if case["kind"] == "diagnostics":
        return {"bytes": 8 * nf * n, "flops": nf * n * (5 * math.log2(max(nt, 2)) + 8)}
    return {"bytes": 8 * nf * n + 16 * nx * ny, "flops": 4 * nf * n + 10 * nx * ny * math.log2(nx * ny)}


# ------------------------------------------------------------------ the same in 64 bits
def _freq(n, d):
    return 2.0 * math.pi * torch.fft.fftfreq(n, d, dtype=torch.float64, device="cuda")


def _propagators(case, nx, ny, nt):
    """exp(dz L) of every field, as the factors along x, y and tau."""
    kx, ky, om = _freq(nx, case["dx"]), _freq(ny, case["dx"]), _freq(nt, case["dt"])
    if nt == 1:
        om = torch.zeros_like(om)
    dz, got = case["dz"], []
    for lam, n, delta, k2, k3, rho, alpha in _fields_of(case):
        k = 2.0 * math.pi * n / lam
        px = torch.exp(-1j * dz * (kx * kx / (2 * k) + math.tan(rho) * kx))
        py = torch.exp(-1j * dz * ky * ky / (2 * k))
        pt = torch.exp(dz * (-0.5 * alpha - 1j * delta * om + 0.5j * k2 * om**2 - 1j * k3 / 6.0 * om**3))
        got.append((px[None, None, :], py[None, :, None], pt[:, None, None]))
    return got


def _kappas(case):
    f = _fields_of(case)
    k = [2.0 * math.pi * D_EFF / (v[1] * v[0]) for v in f]
    if len(f) == 2:
        k[0] *= 0.5
    return k


def _slope(a, k, e):
    """The coupling terms at a phase e = exp(i Phi)."""
    if len(a) == 2:
        return [1j * k[0] * e.conj() * a[1] * a[1], 1j * k[1] * e * a[0] * a[1].conj()]
    u = e * a[0]
    return [1j * k[0] * e.conj() * a[1] * a[2], 1j * k[1] * u * a[2].conj(), 1j * k[2] * u * a[1].conj()]


def _half(a, k, phi, slope, h):
    """One RK4 step of length h from phase phi, which grows at `slope`."""
    e = [torch.exp(1j * (phi + slope * (0.5 * h * s))) for s in range(3)]
    k1 = _slope(a, k, e[0])
    k2 = _slope([x + 0.5 * h * d for x, d in zip(a, k1)], k, e[1])
    k3 = _slope([x + 0.5 * h * d for x, d in zip(a, k2)], k, e[1])
    k4 = _slope([x + h * d for x, d in zip(a, k3)], k, e[2])
    return [x + (h / 6.0) * (p + 2 * q + 2 * r + s) for x, p, q, r, s in zip(a, k1, k2, k3, k4)]


def _step(a, props, k, phi, dk, dz):
    """One split step; phi: the phase at its start, dk its slope (numbers or [ny, nx])."""
    a = _half(a, k, phi, dk, 0.5 * dz)
    a = [torch.fft.ifftn(torch.fft.fftn(x) * p[0] * p[1] * p[2]) for x, p in zip(a, props)]
    return _half(a, k, phi + 0.5 * dz * dk, dk, 0.5 * dz)


def _propagate(case, inputs, nz, dks, dk_map=None):
    a = [x.to(torch.complex128) for x in inputs]
    nt, ny, nx = a[0].shape
    props, k = _propagators(case, nx, ny, nt), _kappas(case)
    m = torch.zeros((), dtype=torch.float64, device="cuda") if dk_map is None else torch.from_numpy(dk_map).cuda()
    phi = torch.zeros_like(m)
    for j in range(nz):
        slope = m + float(dks[j])
        a = _step(a, props, k, phi, slope, case["dz"])
        phi = phi + slope * case["dz"]
    return a


def _gradient(case, seed):
    a = [x.to(torch.complex128) for x in _inputs(case, seed)]
    w = _weights(case, _inputs(case, seed))
    phi = torch.from_numpy(_phase(case, seed)).cuda().requires_grad_()
    dk = torch.from_numpy(_profile(case, seed)).cuda().requires_grad_()
    props, k, dz = _propagators(case, case["nx"], case["ny"], case["nt"]), _kappas(case), case["dz"]
    turn = torch.exp(1j * torch.fft.ifftshift(phi))[:, None, None]
    a[1] = torch.fft.ifft(torch.fft.fft(a[1], dim=0) * turn, dim=0)
    at = torch.zeros((), dtype=torch.float64, device="cuda")
    for j in range(case["nz"]):
        a = checkpoint(lambda x, y, p, d: tuple(_step([x, y], props, k, p, d, dz)), a[0], a[1], at, dk[j], use_reentrant=False)
        at = at + dk[j] * dz
    value = sum(c * (x.real.square() + x.imag.square()).sum() for c, x in zip(w, a))
    value.backward()
    return {"j": value.detach(), "phi": phi.grad, "dk": dk.grad}


def _temperature(case, inputs):
    """The heat equation of the heat load, by the sine transforms that diagonalise its stencil."""
    nx, ny, dx = case["nx"], case["ny"], case["dx"]
    q = torch.zeros(ny, nx, dtype=torch.float64, device="cuda")
    pulsed = REP_RATE * case["dt"] if case["nt"] > 1 else 1.0
    for a, v in zip(inputs, _fields_of(case)):
        q += v[6] * 0.5 * C0 * EPS0 * v[1] * pulsed * a.to(torch.complex128).abs().square().sum(0)

    def sines(n):
        p = torch.arange(1, n + 1, dtype=torch.float64, device="cuda")
        s = torch.sin(math.pi * p[:, None] * (torch.arange(n, dtype=torch.float64, device="cuda") + 0.5)[None] / n)
        s = s / s.square().sum(1, keepdim=True).sqrt()
        return s, 4.0 * torch.sin(math.pi * p / (2 * n)) ** 2 / dx**2

    sx, mx = sines(nx)
    sy, my = sines(ny)
    t = (sy @ q @ sx.T) / (KAPPA_TH * (my[:, None] + mx[None]))
    return sy.T @ t @ sx


def exact(case, seed):
    """What run() returns, in 64 bits with plain torch."""
    if case["kind"] == "batch":
        return [_propagate(case, _inputs(case, seed, i), nz, np.full(nz, dk)) for i, (_, _, _, nz, dk) in enumerate(_members(case, seed))]
    if case["kind"] == "adjoint":
        return _gradient(case, seed)
    inputs = _inputs(case, seed)
    if case["kind"] == "propagate":
        return _propagate(case, inputs, case["nz"], _profile(case, seed), _fanout(case) if case["fanout"] else None)
    if case["kind"] == "diagnostics":
        power, spectrum = [], []
        for a, v in zip(inputs, _fields_of(case)):
            c = 0.5 * C0 * EPS0 * v[1] * case["dx"] ** 2
            a = a.to(torch.complex128)
            power.append(c * a.abs().square().sum((1, 2)))
            spectrum.append(c * case["dt"] / case["nt"] * torch.fft.fft(a, dim=0).abs().square().sum((1, 2)))
        return {"power": torch.stack(power), "spectrum": torch.stack(spectrum)}
    return _temperature(case, inputs)
