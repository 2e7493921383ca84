"""The measured cases: what users of this package have it do, through its public entry points.

A condensate (`GP`) is advanced from a field the program holds on the GPU and
its psi and observables are read; many uneven condensates (`Batch`) are
relaxed from their Gaussians together; an axially symmetric one (`AxialGP`)
is relaxed; the warm-start network (`warmstart.Net`) gives a loss and its
gradient.  Grids, spacings, steps and traps are those of the package's own
workloads (`inputs.py`), of its documents and tests, or drawn around them.
"""
import ctypes
import math

import numpy as np
import torch

from paper_1601_04641_gb300 import _native as N
from paper_1601_04641_gb300 import inputs
from paper_1601_04641_gb300.solver import GP, AxialGP, Batch
from paper_1601_04641_gb300.warmstart import Net

OBS = ("norm", "mu", "energy", "rms_x", "rms_y", "rms_z")


def _grid(name, n, d, dt_factor, omega, g, precision, field, mode, steps, splitting=1, track=0):
    """A single condensate: grid n, equal spacings d (0: sized to the condensate), dt = dt_factor min(d)^2."""
    return {"name": name, "kind": "grid", "nx": n[0], "ny": n[1], "nz": n[2], "d": d, "dt_factor": dt_factor,
            "gamma": omega[0], "nu": omega[1], "lam": omega[2], "g": g, "precision": precision, "field": field,
            "mode": mode, "steps": steps, "splitting": splitting, "track": track}


def listed():
    trap = (0.5, 1.0, 1.5)
    return [
        # the smallest call: one real-time step and its observables, as an interactive program or a control loop does
        _grid("real_tiny_c64", (48, 40, 32), 0.2, 0.02, trap, 10.0, "f32", "complex", "real", 1),
        # a small ground-state search on the plain method's settings (the 64x48x40 workload)
        _grid("imag_small_f64r", (64, 48, 40), 0.2, 0.1, (1.0, 1.4, 2.0), 10.0, "f64", "real", "imag", 100),
        # the FP64 real-time quench on the grid the paper's programs are set up for
        _grid("real_medium_f64", (240, 200, 160), 0.1, 0.02, trap, 40.0, "f64", "complex", "real", 10),
        # production dynamics: the complex64 quench on the large grid, observables every 10 steps
        _grid("real_large_c64", (480, 400, 320), 0.05, 0.02, trap, 40.0, "f32", "complex", "real", 10),
        # the large grid's ground state on a real field, observables every 10 steps
        _grid("imag_large_f32r", (480, 400, 320), 0.05, 0.1, trap, 20.0, "f32", "real", "imag", 10),
        # odd node counts (a node at the trap centre): rows and line pairs off every alignment
        _grid("imag_odd_c64", (241, 201, 161), 0.1, 0.1, trap, 20.0, "f32", "complex", "imag", 10),
        # second-order splitting with a record on the device every 5 steps, on the real-time programs' default grid
        _grid("real_strang_c64", (200, 160, 120), 0.1, 0.02, trap, 40.0, "f32", "complex", "real", 20, 2, 5),
        # the coarse level of a dt schedule (ten times the fine step): wide windows
        _grid("imag_coarse_f32r", (320, 240, 200), 0.075, 1.0, trap, 20.0, "f32", "real", "imag", 10),
        # the batched form: 64 uneven condensates
        {"name": "batch64_c64", "kind": "batch", "count": 64, "shapes": 0, "g_max": 200.0, "field": "complex",
         "dt_scale": 1.0, "steps": 100},
        # ground states for the warm start's training set: real fields through the coarse and the fine level
        {"name": "batch64_schedule_f32r", "kind": "batch", "count": 64, "shapes": 1, "g_max": 500.0, "field": "real",
         "dt_scale": 10.0, "steps": 100},
        # an axially symmetric ground state, checked every 10 steps
        {"name": "axial_f64r", "kind": "axial", "nx": 120, "nz": 241, "d": 0.05, "dt": 1e-3, "gamma": 1.0, "lam": 2.0,
         "g": 50.0, "precision": "f64", "field": "real", "mode": "imag", "steps": 100},
        # one training batch of the warm start: loss and gradient (forward and backward)
        {"name": "nn_grad", "kind": "nn", "count": 8, "points": 32768},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("grid", "grid", "grid", "grid", "grid", "batch", "axial", "nn"))
    if kind == "batch":
        return {"kind": "batch", "count": _log_int(rng, 4, 64), "shapes": rng.randrange(1 << 20),
                "g_max": rng.choice((200.0, 500.0)), "field": rng.choice(("complex", "real")),
                "dt_scale": rng.choice((1.0, 3.0, 10.0)), "steps": rng.randrange(20, 101)}
    if kind == "axial":
        field = rng.choice(("real", "complex"))
        return {"kind": "axial", "nx": _log_int(rng, 48, 320), "nz": _log_int(rng, 64, 512), "d": rng.uniform(0.04, 0.1),
                "dt": math.exp(rng.uniform(math.log(2e-4), math.log(2e-3))), "gamma": rng.uniform(0.5, 3.0),
                "lam": rng.uniform(0.5, 3.0), "g": math.exp(rng.uniform(0.0, math.log(200.0))),
                "precision": rng.choice(("f64", "f32")), "field": field,
                "mode": rng.choice(("imag", "real")) if field == "complex" else "imag", "steps": rng.randrange(20, 101)}
    if kind == "nn":
        return {"kind": "nn", "count": rng.randrange(2, 13), "points": 128 * _log_int(rng, 8, 256)}
    precision, field, mode, most = rng.choice((("f32", "complex", "real", 61440000), ("f32", "complex", "imag", 61440000),
                                               ("f32", "real", "imag", 61440000), ("f64", "real", "imag", 7680000),
                                               ("f64", "complex", "real", 7680000), ("f16", "real", "imag", 61440000)))
    sites = math.exp(rng.uniform(math.log(3e4), math.log(most)))
    while True:
        a, b = rng.uniform(0.6, 1.6), rng.uniform(0.6, 1.6)
        side = (sites / (a * b)) ** (1.0 / 3.0)
        n = [int(side * a), int(side * b), int(side)]
        rng.shuffle(n)
        if precision == "f16":  # half-precision storage is for whole 16-byte rows
            n[2] = max(56, n[2] // 8 * 8)
        if min(n) >= 20 and n[0] * n[1] * n[2] <= most:
            break
    factor = math.exp(rng.uniform(math.log(0.05), math.log(1.0))) if mode == "imag" else math.exp(
        rng.uniform(math.log(0.01), math.log(0.1)))
    if precision == "f16":
        factor = rng.uniform(0.5, 1.0)  # its steps are a schedule's coarse ones
    split = mode == "real" and rng.random() < 0.3
    c = _grid("", n, 0.0, factor, [rng.uniform(0.5, 3.0) for _ in range(3)],
              math.exp(rng.uniform(0.0, math.log(200.0))), precision, field, mode, rng.randrange(1, 11), 2 if split else 1,
              rng.choice((0, 0, 5)))
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs
def _problem(c):
    n, w = (c["nx"], c["ny"], c["nz"]), (c["gamma"], c["nu"], c["lam"])
    if c["d"] > 0.0:
        return inputs.Problem(n, (c["d"],) * 3, c["dt_factor"] * c["d"] ** 2, w, c["g"])
    return inputs.sized_box(n, w, c["g"], c["dt_factor"])


def _coords(n, d):
    return (torch.arange(n, dtype=torch.float64, device="cuda") - 0.5 * (n - 1)) * d


def _field(shape, d, omega, complex_, seed):
    """A condensate that has been stirred: two displaced, squeezed Gaussians of the trap's widths, with a small momentum
    each where the field is complex; zero on the boundary, norm 1.  float64 or complex128 on the GPU."""
    rng = np.random.default_rng(seed)
    out = None
    for amp in (1.0, rng.uniform(0.2, 0.6)):
        f = []
        for n, h, w in zip(shape, d, omega):
            x, a = _coords(n, h), 1.0 / math.sqrt(w)
            width, x0, k = a * rng.uniform(0.9, 1.6), a * rng.uniform(-0.5, 0.5), rng.uniform(-1.0, 1.0) / a
            v = torch.exp(-0.5 * ((x - x0) / width) ** 2)
            v[0] = v[-1] = 0.0
            f.append(v * torch.exp(1j * k * x) if complex_ else v)
        part = amp * f[0][:, None, None] * f[1][None, :, None] * f[2][None, None, :]
        out = part if out is None else out.add_(part)
    return out / math.sqrt(float((out.abs() ** 2).sum()) * d[0] * d[1] * d[2])


_TORCH = {("f64", "complex"): torch.complex128, ("f32", "complex"): torch.complex64, ("f64", "real"): torch.float64,
          ("f32", "real"): torch.float32, ("f16", "real"): torch.float16}


def _start(c, seed):
    p = _problem(c)
    psi = _field(p.shape, p.d, p.omega, c["field"] == "complex", seed)
    return p, psi.to(_TORCH[(c["precision"], c["field"])])


def _axial_field(c, seed):
    """A squeezed, displaced (and, where complex, moving) Gaussian of norm 1, on the host as the entry point takes it."""
    rng = np.random.default_rng(seed)
    x = (np.arange(c["nx"]) - 0.5) * c["d"]
    z = (np.arange(c["nz"]) - 0.5 * (c["nz"] - 1)) * c["d"]
    psi = (np.exp(-0.5 * c["gamma"] * rng.uniform(0.6, 1.2) * x ** 2)[:, None] *
           np.exp(-0.5 * c["lam"] * rng.uniform(0.6, 1.2) * (z - rng.uniform(-0.3, 0.3)) ** 2)[None, :])
    if c["field"] == "complex":
        psi = psi * np.exp(1j * rng.uniform(-1.0, 1.0) * z)[None, :]
    psi[0] = psi[-1] = 0.0
    psi[:, 0] = psi[:, -1] = 0.0
    w = 2.0 * math.pi * x[1:-1] * c["d"] ** 2
    psi = psi / math.sqrt(float((w[:, None] * np.abs(psi[1:-1]) ** 2).sum()))
    return np.ascontiguousarray(psi.astype({("f64", "complex"): np.complex128, ("f32", "complex"): np.complex64,
                                            ("f64", "real"): np.float64, ("f32", "real"): np.float32}[
                                                (c["precision"], c["field"])]))


def _batch_problems(c, seed):
    """The grids are the case's, the traps and nonlinearities the seed's."""
    rng = np.random.default_rng(seed)
    ps = []
    for q in inputs.batch_problems(c["count"], c["shapes"], c["g_max"]):
        omega = tuple(float(x) for x in rng.uniform(0.5, 3.0, size=3))
        ps.append(inputs.sized_box(q.shape, omega, float(math.exp(rng.uniform(0.0, math.log(c["g_max"]))))))
    return ps


_NN = {"h": 64, "in": 16, "used": 9}


def _nn_inputs(c, seed):
    """Targets (amplitudes of displaced Gaussians), sample points and Glorot weights."""
    rng = np.random.default_rng(seed)
    ps, data = [], []
    for q in inputs.batch_problems(c["count"], 7, 500.0):
        omega = tuple(float(x) for x in rng.uniform(0.5, 3.0, size=3))
        p = inputs.sized_box(q.shape, omega, float(math.exp(rng.uniform(0.0, math.log(500.0)))))
        ps.append(p)
        data.append(_field(p.shape, p.d, p.omega, False, int(rng.integers(1 << 30))).to(torch.float32).reshape(-1))
    offsets = np.concatenate([[0], np.cumsum([t.numel() for t in data])[:-1]]).astype(np.int64)
    inst = rng.integers(0, c["count"], size=c["points"]).astype(np.int32)
    sites = np.array([p.sites for p in ps], dtype=np.int64)[inst]
    site = np.minimum((rng.random(c["points"]) * sites).astype(np.int64), sites - 1)
    h, i = _NN["h"], _NN["in"]
    theta = []
    for fan_in, fan_out in ((i, h), (h, h), (h, h), (h, 1)):
        a = math.sqrt(6.0 / (fan_in + fan_out))
        w = rng.uniform(-a, a, size=(fan_in, fan_out))
        if fan_in == i:
            w[_NN["used"]:] = 0.0
        theta += [w.reshape(-1), rng.uniform(-0.1, 0.1, size=fan_out)]
    theta = np.concatenate(theta).astype(np.float32)
    return ps, data, offsets, [float(t.max()) for t in data], inst, site, theta


def prepare(c, seed):
    if c["kind"] == "grid":
        p, psi = _start(c, seed)
        gp = GP(p.shape, p.d, p.dt, p.omega, p.g, c["precision"], c["field"])
        if c["splitting"] == 2:
            gp.set_splitting(2)
        return {"c": c, "gp": gp, "psi": psi}
    if c["kind"] == "batch":
        ps = _batch_problems(c, seed)
        b = Batch(ps, "f32", c["field"])
        dtype = torch.complex64 if c["field"] == "complex" else torch.float32
        return {"c": c, "b": b, "ps": ps, "out": torch.empty(sum(p.sites for p in ps), dtype=dtype, device="cuda")}
    if c["kind"] == "axial":
        a = AxialGP(c["nx"], c["nz"], c["d"], c["d"], c["dt"], c["gamma"], c["lam"], c["g"], c["precision"], c["field"])
        return {"c": c, "a": a, "psi": _axial_field(c, seed)}
    ps, data, offsets, psi_max, inst, site, theta = _nn_inputs(c, seed)
    net = Net(0)
    net.params = theta
    net.set_data(ps, torch.cat(data), offsets, psi_max)
    return {"c": c, "net": net, "inst": inst, "site": site}


def run(s):
    c = s["c"]
    if c["kind"] == "grid":
        gp = s["gp"]
        gp.set_psi(s["psi"])
        if c["track"]:
            gp.set_tracking(c["track"])
        (gp.step_imag if c["mode"] == "imag" else gp.step_real)(c["steps"])
        obs = gp.observables()
        out = {"psi": gp.get_psi(as_numpy=False), "obs": np.array([obs[k] for k in OBS])}
        if c["track"]:
            out["track"] = np.array([[o[k] for k in OBS] for o in gp.tracking(1024)]).reshape(-1, len(OBS))
        return out
    if c["kind"] == "batch":
        b = s["b"]
        b.init_gaussian()
        if c["dt_scale"] == 1.0:
            b.step_imag(c["steps"])
        else:  # two levels that stop at their step counts
            b.run_imag_schedule([(c["dt_scale"], 1e-30), (1.0, 1e-30)], 10, c["steps"])
        obs = b.observables()
        off = 0
        for i, p in enumerate(s["ps"]):  # on the device, as the training targets are read
            t = s["out"][off:off + p.sites]
            N.check(b.lib.gp_batch_get_psi(b.h, i, ctypes.c_void_p(t.data_ptr()), 1), b.h, batch=True)
            off += p.sites
        return {"psi": s["out"], "obs": np.array([[o[k] for k in OBS] for o in obs])}
    if c["kind"] == "axial":
        a = s["a"]
        a.set_psi(s["psi"])
        if c["mode"] == "imag":
            a.run_imag_until(1e-30, 10, c["steps"])
        else:
            a.step_real(c["steps"])
        obs = a.observables()
        return {"psi": a.get_psi(), "obs": np.array([obs[k] for k in OBS])}
    loss, grad = s["net"].loss_grad(s["inst"], s["site"])
    return {"loss": loss, "grad": grad}


# ---------------------------------------------------------------- work
_BYTES = {"f64": 8, "f32": 4, "f16": 2}


def work(c):
    """A step reads the field once and writes it once (the next step needs all of it); per site and step about 20 (real)
    or 45 (complex) operations of the three line solves and 10 of the kick, and 15 of each set of observables."""
    if c["kind"] == "grid":
        sites, cplx = c["nx"] * c["ny"] * c["nz"], c["field"] == "complex"
        return {"bytes": 2.0 * sites * _BYTES[c["precision"]] * (2 if cplx else 1) * c["steps"],
                "flops": sites * ((80.0 if cplx else 35.0) * c["steps"] + 15.0)}
    if c["kind"] == "batch":
        sites, cplx = sum(p.sites for p in inputs.batch_problems(c["count"], c["shapes"], c["g_max"])), c["field"] == "complex"
        steps = c["steps"] * (1 if c["dt_scale"] == 1.0 else 2)
        return {"bytes": 2.0 * sites * (8 if cplx else 4) * steps, "flops": sites * ((80.0 if cplx else 35.0) * steps + 15.0)}
    if c["kind"] == "axial":
        sites, cplx = c["nx"] * c["nz"], c["field"] == "complex"
        return {"bytes": 2.0 * sites * _BYTES[c["precision"]] * (2 if cplx else 1) * c["steps"],
                "flops": sites * (70.0 if cplx else 30.0) * c["steps"]}
    macs = 16 * 64 + 2 * 64 * 64 + 64
    return {"bytes": c["points"] * 16.0 + 4.0 * 2 * 9408, "flops": 6.0 * macs * c["points"]}


# ---------------------------------------------------------------- the same in 64 bits
def _cn(n, c):
    """The dense CN operator of a line of n nodes (zero on the two end nodes)."""
    m = n - 2
    t = 2.0 * np.eye(m) - np.eye(m, k=1) - np.eye(m, k=-1)
    out = np.zeros((n, n), dtype=np.complex128 if isinstance(c, complex) else np.float64)
    out[1:-1, 1:-1] = np.linalg.solve(np.eye(m) + c * t, np.eye(m) - c * t)
    return torch.from_numpy(out).cuda()


def _sweeps(psi, ops):
    nx, ny, nz = psi.shape
    psi = (ops[0] @ psi.reshape(nx, -1)).reshape(nx, ny, nz)
    psi = torch.matmul(ops[1], psi)
    return torch.matmul(psi, ops[2].T)


def _exact_grid(n, d, dt, omega, g, psi, imag, steps, splitting=1, track=0):
    c = [dt / (4.0 * h * h) for h in d]
    ops = [_cn(m, x if imag else 1j * x).to(psi.dtype) for m, x in zip(n, c)]
    xs = [_coords(m, h) for m, h in zip(n, d)]
    dv = d[0] * d[1] * d[2]
    vx = [0.5 * w * w * x * x for w, x in zip(omega, xs)]
    v = vx[0][:, None, None] + vx[1][None, :, None] + vx[2][None, None, :]

    def rho(f):
        return f.real ** 2 + f.imag ** 2 if f.is_complex() else f * f

    def kick(f, h):
        a = v + g * rho(f)
        return f * (torch.exp(-h * a) if imag else torch.polar(torch.ones_like(a), -h * a))

    def observe(f):
        r = rho(f)
        nrm = dv * float(r.sum())
        kin = 0.5 * dv * sum(float(rho(f.diff(dim=q)).sum()) / (d[q] * d[q]) for q in range(3))
        pot, inter = dv * float((v * r).sum()), dv * float((r * r).sum())
        rms = [math.sqrt(dv * float((r.sum(dim=tuple(a for a in range(3) if a != q)) * xs[q] ** 2).sum()) / nrm)
               for q in range(3)]
        return [nrm, (kin + pot + g * inter) / nrm, (kin + pot + 0.5 * g * inter) / nrm] + rms

    records = []
    for s in range(1, steps + 1):
        psi = _sweeps(kick(psi, 0.5 * dt if splitting == 2 else dt), ops)
        if splitting == 2:
            psi = kick(psi, 0.5 * dt)
        if imag:
            psi = psi / math.sqrt(dv * float(rho(psi).sum()))
        if track and s % track == 0:
            records.append(observe(psi))
    return psi, observe(psi), records


def _exact_axial(c, seed):
    nx, nz, d, dt, imag = c["nx"], c["nz"], c["d"], c["dt"], c["mode"] == "imag"
    psi = torch.from_numpy(_axial_field(c, seed).astype(np.complex128 if c["field"] == "complex" else np.float64)).cuda()
    k = dt / (4.0 * d * d)
    k = k if imag else 1j * k
    r = (np.arange(1, nx - 1) - 0.5) * d
    lo, hi = (r - 0.5 * d) / r, (r + 0.5 * d) / r
    t = np.diag(lo + hi) - np.diag(hi[:-1], 1) - np.diag(lo[1:], -1)
    m = np.zeros((nx, nx), dtype=np.float64 if imag else np.complex128)
    m[1:-1, 1:-1] = np.linalg.solve(np.eye(nx - 2) + k * t, np.eye(nx - 2) - k * t)
    radial, axial = torch.from_numpy(m).cuda(), _cn(nz, k)
    if c["field"] == "complex":
        radial, axial = radial.to(torch.complex128), axial.to(torch.complex128)
    rho_, z = torch.from_numpy(r).cuda()[:, None], _coords(nz, d)[None, :]
    rr = torch.from_numpy((np.arange(nx) - 0.5) * d).cuda()[:, None]
    v = 0.5 * (c["gamma"] ** 2 * rr ** 2 + c["lam"] ** 2 * z ** 2)
    w = 2.0 * math.pi * rho_ * d * d

    def dens(f):
        return f.real ** 2 + f.imag ** 2 if f.is_complex() else f * f

    for _ in range(c["steps"]):
        a = dt * (v + c["g"] * dens(psi))
        psi = radial @ (psi * (torch.exp(-a) if imag else torch.polar(torch.ones_like(a), -a)))
        psi = torch.matmul(psi, axial.T)
        if imag:
            psi = psi / math.sqrt(float((w * dens(psi)[1:-1]).sum()))
    q = dens(psi)[1:-1]
    nrm, x2 = float((w * q).sum()), float((w * rho_ ** 2 * q).sum())
    kin = 0.5 * float((2.0 * math.pi * (rho_ + 0.5 * d) * dens(psi.diff(dim=0))[1:]).sum() +
                      (2.0 * math.pi * rho_ * dens(psi.diff(dim=1))[1:-1]).sum())
    pot, inter = float((w * v[1:-1] * q).sum()), float((w * q * q).sum())
    rms = math.sqrt(0.5 * x2 / nrm)
    return {"psi": psi, "obs": np.array([nrm, (kin + pot + c["g"] * inter) / nrm, (kin + pot + 0.5 * c["g"] * inter) / nrm,
                                         rms, rms, math.sqrt(float((w * z ** 2 * q).sum()) / nrm)])}


def _exact_nn(c, seed):
    ps, data, _, psi_max, inst, site, theta = _nn_inputs(c, seed)
    inst, site = torch.from_numpy(inst.astype(np.int64)).cuda(), torch.from_numpy(site).cuda()

    def per(vals):
        return torch.tensor(np.array(vals, dtype=np.float64), device="cuda")[inst]

    n = torch.tensor([p.shape for p in ps], device="cuda")[inst]
    k, j = site % n[:, 2], site // n[:, 2] % n[:, 1]
    idx = torch.stack([site // (n[:, 2] * n[:, 1]), j, k], 1)
    x = (idx - 0.5 * (n - 1)) * per([p.d for p in ps])
    w = per([p.omega for p in ps])
    mu = per([0.5 * (15.0 * abs(p.g) * p.omega[0] * p.omega[1] * p.omega[2] / (4.0 * math.pi)) ** 0.4 for p in ps])
    u = x * x * w
    sq = (x * w).pow(2).sum(1) / (2.0 * mu)
    f = torch.zeros(len(site), _NN["in"], dtype=torch.float64, device="cuda")
    f[:, :3] = 0.125 * u.clamp(max=16.0) - 1.0
    f[:, 3] = 0.5 * sq.clamp(max=4.0) - 1.0
    f[:, 4] = 0.125 * u.sum(1).clamp(max=16.0) - 1.0
    f[:, 5] = per([(math.log(max(abs(p.g), 1e-12)) - 3.1) / 3.1 for p in ps])
    f[:, 6:9] = (w - 1.75) / 1.25
    target = torch.zeros(len(site), dtype=torch.float64, device="cuda")
    for q, t in enumerate(data):
        target[inst == q] = t[site[inst == q]].double() / psi_max[q]
    par, at, h = [], 0, _NN["h"]
    for shape in ((_NN["in"], h), (h,), (h, h), (h,), (h, h), (h,), (h, 1), (1,)):
        size = int(np.prod(shape))
        par.append(torch.from_numpy(theta[at:at + size].astype(np.float64).reshape(shape)).cuda().requires_grad_())
        at += size
    a = f
    for q in range(0, 6, 2):
        a = torch.tanh(a @ par[q] + par[q + 1])
    y = torch.nn.functional.softplus((a @ par[6] + par[7])[:, 0])
    loss = ((y - target) ** 2).mean()
    loss.backward()
    return {"loss": float(loss), "grad": torch.cat([p.grad.reshape(-1) for p in par])}


def exact(c, seed):
    if c["kind"] == "grid":
        p, psi = _start(c, seed)
        psi = psi.to(torch.complex128 if c["field"] == "complex" else torch.float64)
        psi, obs, records = _exact_grid(p.shape, p.d, p.dt, p.omega, p.g, psi, c["mode"] == "imag", c["steps"],
                                        c["splitting"], c["track"])
        out = {"psi": psi, "obs": np.array(obs)}
        if c["track"]:
            out["track"] = np.array(records).reshape(-1, len(OBS))
        return out
    if c["kind"] == "batch":
        out, obs = [], []
        for p in _batch_problems(c, seed):
            psi = 1.0
            for q, (n, d, w) in enumerate(zip(p.shape, p.d, p.omega)):
                x = _coords(n, d)
                v = (w / math.pi) ** 0.25 * torch.exp(-0.5 * w * x * x)
                v[0] = v[-1] = 0.0
                psi = psi * v.reshape([-1 if a == q else 1 for a in range(3)])
            psi = psi / math.sqrt(float((psi * psi).sum()) * p.d[0] * p.d[1] * p.d[2])
            for scale in ((1.0,) if c["dt_scale"] == 1.0 else (c["dt_scale"], 1.0)):
                psi, o, _ = _exact_grid(p.shape, p.d, p.dt * scale, p.omega, p.g, psi, True, c["steps"])
            out.append(psi.reshape(-1))
            obs.append(o)
        psi = torch.cat(out)  # a complex field stays real from a real start in imaginary time
        return {"psi": torch.complex(psi, torch.zeros_like(psi)) if c["field"] == "complex" else psi, "obs": np.array(obs)}
    return _exact_axial(c, seed) if c["kind"] == "axial" else _exact_nn(c, seed)
