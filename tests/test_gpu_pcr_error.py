"""The error of FP64 steps against sweeps in extended precision (numpy
longdouble on the host): by cyclic reduction it is no larger than by the
two-pass solve, in the largest and in the mean, beyond what one of 107 520
rounded values may add to the largest (a quarter).  The error is taken
without its part along the field itself: that is the renormalisation
factor's, one rounding of one number a step, the same rounding for both."""
import numpy as np
import pytest

from paper_1601_04641_gb300 import build

pytestmark = pytest.mark.gpu

SHAPE, H, OMEGA, G, STEPS = (48, 56, 40), 0.2, (1.0, 1.4, 2.0), 100.0, 6
LD = np.longdouble


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _line(p, c):
    """CN solve of (1 + c T) phi = (1 - c T) p along axis 0, zero end nodes."""
    q, n = p[1:-1], p.shape[0] - 2
    lo, hi = np.concatenate([0 * q[:1], q[:-1]]), np.concatenate([q[1:], 0 * q[:1]])
    r, cp, d = q + c * (lo - 2 * q + hi), [], []
    for t in range(n):
        den = 1 + 2 * c + (c * cp[-1] if t else 0)
        d.append((r[t] + (c * d[-1] if t else 0)) / den)
        cp.append(-c / den)
    out = np.zeros_like(p)
    out[n] = d[n - 1]
    for t in range(n - 2, -1, -1):
        out[t + 1] = d[t] - cp[t] * out[t + 2]
    return out


def _reference(psi, dt, imag):
    psi, dt, h = psi.astype(LD if not np.iscomplexobj(psi) else np.clongdouble), LD(dt), LD(H)
    x = [(np.arange(n).astype(LD) - LD(0.5) * (n - 1)) * h for n in SHAPE]
    v = [LD(0.5) * LD(w) ** 2 * a * a for w, a in zip(OMEGA, x)]
    v = v[0][:, None, None] + v[1][None, :, None] + v[2][None, None, :]
    c = dt / (4 * h * h) * (LD(1) if imag else np.clongdouble(1j))
    for _ in range(STEPS):
        a = dt * (v + LD(G) * (psi.real ** 2 + psi.imag ** 2))
        psi = psi * (np.exp(-a) if imag else np.cos(a) - 1j * np.sin(a))
        for ax in range(3):
            psi = np.moveaxis(_line(np.moveaxis(psi, ax, 0), c), 0, ax)
        if imag:
            psi = psi / np.sqrt((psi.real ** 2 + psi.imag ** 2).sum() * h ** 3)
    return psi


@pytest.mark.parametrize("form,factor", [("real", 0.05), ("real", 0.8), ("complex", 0.1), ("realtime", 0.02), ("realtime", 0.1)])
def test_error_is_no_larger_than_the_two_pass_solves(form, factor):
    from paper_1601_04641_gb300.solver import GP
    f = []
    for n, w in zip(SHAPE, OMEGA):
        x = (np.arange(n) - 0.5 * (n - 1)) * H
        v = np.exp(-0.4 * w * (x - 0.2) ** 2) * (1.0 if form == "real" else np.exp(0.5j * x))
        v[0] = v[-1] = 0.0
        f.append(v)
    psi = f[0][:, None, None] * f[1][None, :, None] * f[2][None, None, :]
    psi = np.ascontiguousarray(psi / np.sqrt((np.abs(psi) ** 2).sum() * H ** 3))
    dt, imag = factor * H * H, form != "realtime"
    exact, errors = _reference(psi, dt, imag), []
    for two_pass in (False, True):
        gp = GP(SHAPE, (H, H, H), dt, OMEGA, G, "f64", "real" if form == "real" else "complex")
        if two_pass:
            gp.set_window(0)
        gp.set_psi(psi)
        (gp.step_imag if imag else gp.step_real)(STEPS)
        e = gp.get_psi().astype(exact.dtype) - exact
        e = np.abs(e - exact * ((exact.conj() * e).sum() / (exact.conj() * exact).sum()))
        errors.append((float(e.max()), float(np.sqrt((e * e).mean()))))
        gp.close()
    assert errors[0][1] <= errors[1][1] and errors[0][0] <= 1.25 * errors[1][0]
