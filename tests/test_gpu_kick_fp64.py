"""The FP64 kick by itself.  On a grid whose spacings are so wide that dt / d^2
vanishes against one, every line solve is the identity to the last bit, and
the buffer after one step (without its renormalisation factor) holds the
kicked values.

A node's kick is a function of its own value: the same whatever its
neighbours hold, however its line is cut into chunks, and in both solves.

Error bounds, u = 2^-53.  Imaginary time at small exponents: the factor's
deviation from one is a sum of four terms, each within 8 relative roundings,
and the value is rounded once: u (1 + 8 sum|dev|) of the result.  At large
exponents: the exponent is within 3 relative roundings, the product within 6:
u (8 + 3 y) of the result, which must not vanish."""
import ctypes

import numpy as np
import pytest

from paper_1601_04641_gb300 import _native as N
from paper_1601_04641_gb300 import build

pytestmark = pytest.mark.gpu

SHAPE, D, DT, U = (20, 12, 40), 1e20, 0.01, 2.0 ** -53
LD = np.longdouble


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


class _Buffer:
    """A device buffer as torch takes one in."""

    def __init__(self, ptr, dtype):
        self.__cuda_array_interface__ = {"shape": SHAPE, "typestr": np.dtype(dtype).str, "data": (ptr, False), "version": 3}


def _kicked(psi, form, g, omega, two_pass):
    """One step's stored values, before the renormalisation factor."""
    import torch
    from paper_1601_04641_gb300.solver import GP
    gp = GP(SHAPE, (D, D, D), DT, (omega,) * 3, g, "f64", "real" if form == "real" else "complex")
    if two_pass:
        gp.set_window(0)
    gp.set_psi(psi)
    (gp.step_real if form == "realtime" else gp.step_imag)(1)
    gp.sync()
    ptr, pending = ctypes.c_void_p(), ctypes.c_int(0)
    assert gp.lib.gp_psi_device_ptr(gp.h, ctypes.byref(ptr), ctypes.byref(pending)) == N.GP_OK
    raw = torch.as_tensor(_Buffer(ptr.value, psi.dtype), device="cuda").cpu().numpy().copy()
    gp.close()
    return raw


def _interior(f):
    return f[1:-1, 1:-1, 1:-1].reshape(-1)


@pytest.mark.parametrize("trap", [False, True])
@pytest.mark.parametrize("form", ["real", "complex", "realtime"])
def test_a_nodes_kick_does_not_depend_on_its_neighbours(form, trap):
    """600 values at random places, exponents and phases from 1e-3 to 3 (both sides of every series' range), half of the x
    lines with small ones alone: without a trap equal values give equal results; with one and without, both solves do (one
    kicks node by node, the other in chunks with a shorter last one)."""
    rng = np.random.default_rng(4)
    amp = np.concatenate([rng.uniform(0.08, 0.0998, 300), np.exp(rng.uniform(np.log(0.02), np.log(1.0), 300))])
    vals = amp if form == "real" else amp * np.exp(1j * rng.uniform(-3.0, 3.0, 600))
    which, small = rng.integers(0, 600, SHAPE), np.flatnonzero(3.0 * amp ** 2 < 0.0299)
    even = np.add.outer(np.arange(SHAPE[1]), np.arange(SHAPE[2])) % 2 == 0
    which = np.where(even[None], small[which % len(small)], which)
    psi = np.zeros(SHAPE, vals.dtype)
    psi[1:-1, 1:-1, 1:-1] = vals[which[1:-1, 1:-1, 1:-1]]
    omega = 0.1 / (20 * D) if trap else 0.0
    outs = [_interior(_kicked(psi, form, 300.0, omega, two_pass)) for two_pass in (False, True)]
    if not trap:
        idx = _interior(which)
        for out in outs:
            assert all(len(np.unique(out[idx == q])) <= 1 for q in range(600))
    assert np.array_equal(outs[0], outs[1])


@pytest.mark.parametrize("two_pass", [False, True])
@pytest.mark.parametrize("form", ["real", "complex"])
@pytest.mark.parametrize("most", [0.015, 60.0])
def test_imaginary_time_kick_against_extended_precision(form, most, two_pass):
    rng = np.random.default_rng(9)
    amp = np.sqrt(rng.uniform(1e-3, 1.0, SHAPE))
    psi = amp if form == "real" else amp * np.exp(1j * rng.uniform(-3.0, 3.0, SHAPE))
    for ax in range(3):
        np.moveaxis(psi, ax, 0)[[0, -1]] = 0.0
    g, omega = most / DT, (0.1 / (20 * D)) if most < 1.0 else 0.0
    out = _kicked(psi, form, g, omega, two_pass)
    x = [(np.arange(n) - 0.5 * (n - 1)) * D for n in SHAPE]
    dv = [LD(DT) * LD(0.5) * LD(omega) ** 2 * a.astype(LD) ** 2 for a in x]
    dv = dv[0][:, None, None] + dv[1][None, :, None] + dv[2][None, None, :]
    y = LD(DT) * LD(g) * (psi.real.astype(LD) ** 2 + psi.imag.astype(LD) ** 2)
    assert most > 1.0 or 1e-5 < float(dv.max()) < 0.02
    exact = psi.astype(LD if form == "real" else np.clongdouble) * np.exp(-(dv + y))
    bound = U * (1.0 + 8.0 * (dv + y) if most < 1.0 else 8.0 + 3.0 * y)
    for part in ("real", "imag"):
        e, o = _interior(getattr(exact, part)), _interior(getattr(out, part))
        assert np.all(np.abs(o - e) <= _interior(bound) * np.abs(e))
