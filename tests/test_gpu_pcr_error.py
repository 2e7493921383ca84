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


def _fma(a, b, c):
    return (a.astype(LD) * b + c).astype(np.float64)


def _modelled_real_time(psi, dt):
    """The two-pass real-time step as its kernel rounds it: a sweep has two roundings a node at the size of the field in the
    right-hand side and u = r + i k d, two in u / den and ONE in the back substitution, phi = d - (cp phi'), whose product
    is rounded at its own small size."""
    re, im = psi.real.copy(), psi.imag.copy()
    x = [(np.arange(n) - 0.5 * (n - 1)) * H for n in SHAPE]
    px = [dt * 0.5 * w * w * a * a for w, a in zip(OMEGA, x)]
    pot, k = px[0][:, None, None] + (px[1][:, None] + px[2][None, :])[None], dt / (4.0 * H * H)
    kk = np.float64(k)

    def horner(x2, cs):
        v = np.full_like(x2, cs[0])
        for c in cs[1:]:
            v = _fma(x2, v, np.float64(c))
        return v

    for _ in range(STEPS):
        th = _fma(np.full_like(re, dt * G), _fma(re, re, im * im), pot)
        x2 = th * th
        sn = th * horner(x2, (1.0 / 362880.0, -1.0 / 5040.0, 1.0 / 120.0, -1.0 / 6.0, 1.0))
        cs = horner(x2, (-1.0 / 3628800.0, 1.0 / 40320.0, -1.0 / 720.0, 1.0 / 24.0, -0.5, 1.0))
        re, im = _fma(cs, re, sn * im), _fma(cs, im, -sn * re)
        for ax in range(3):
            a, b = np.moveaxis(re, ax, 0), np.moveaxis(im, ax, 0)
            n = a.shape[0] - 2
            z = np.zeros_like(a[0])
            cp, d = [], []
            for t in range(n):
                e = 2j * k + (1j * k * cp[-1] if t else 0.0)
                cp.append(-1j * k / (1.0 + e))
                ip = -e / (1.0 + e)
                lo, hi = (a[t] if t else z, b[t] if t else z), (a[t + 2] if t < n - 1 else z, b[t + 2] if t < n - 1 else z)
                dre = _fma(np.full_like(z, -2.0), a[t + 1], lo[0] + hi[0])
                dim = _fma(np.full_like(z, -2.0), b[t + 1], lo[1] + hi[1])
                r = _fma(np.full_like(z, -kk), dim, a[t + 1]), _fma(np.full_like(z, kk), dre, b[t + 1])
                p = d[-1] if t else (z, z)
                u, v = _fma(np.full_like(z, -kk), p[1], r[0]), _fma(np.full_like(z, kk), p[0], r[1])
                d.append((_fma(u, ip.real, _fma(-v, ip.imag, u)), _fma(u, ip.imag, _fma(v, ip.real, v))))
            oa, ob = np.zeros_like(a), np.zeros_like(b)
            f = d[n - 1]
            oa[n], ob[n] = f
            for t in range(n - 2, -1, -1):
                c = cp[t]
                f = (d[t][0] - _fma(np.full_like(z, c.real), f[0], -c.imag * f[1]),
                     d[t][1] - _fma(np.full_like(z, c.real), f[1], c.imag * f[0]))
                oa[t + 1], ob[t + 1] = f
            re, im = np.moveaxis(oa, 0, ax), np.moveaxis(ob, 0, ax)
    return re + 1j * im


def test_two_pass_real_time_rounds_as_modelled():
    """The kernel's error is its model's: 5 roundings a node and sweep.  One more is sqrt(6/5) on a sweep's share, 6 % with
    the kick's two; two draws of 107 520 errors agree within 1 %."""
    from paper_1601_04641_gb300.solver import GP
    f = [np.exp((-0.4 * w + 0.1j) * ((np.arange(n) - 0.5 * (n - 1)) * H - 0.2) ** 2) for n, w in zip(SHAPE, OMEGA)]
    for v in f:
        v[0] = v[-1] = 0.0
    psi = f[0][:, None, None] * f[1][None, :, None] * f[2][None, None, :]
    psi = np.ascontiguousarray(psi / np.sqrt((np.abs(psi) ** 2).sum() * H ** 3))
    dt = 0.02 * H * H
    exact = _reference(psi, dt, False)
    gp = GP(SHAPE, (H, H, H), dt, OMEGA, G, "f64", "complex")
    gp.set_window(0)
    gp.set_psi(psi)
    gp.step_real(STEPS)
    rms = [float(np.sqrt((np.abs(f.astype(exact.dtype) - exact) ** 2).mean())) for f in (gp.get_psi(), _modelled_real_time(psi, dt))]
    gp.close()
    assert rms[0] <= 1.03 * rms[1]
