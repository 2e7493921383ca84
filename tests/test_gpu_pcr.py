"""FP64 line solves by truncated cyclic reduction (the automatic choice on
grids with too few lines to fill the GPU one thread each) against the FP64
oracle, at the sizes and steps where they can go wrong: interiors of one node,
lengths at and around the reduction distances, line counts off the lines per
block, long lines, and dt from a few levels of reduction to the most.

Bound: a value passes through at most 3 sweeps a step, each at most 2 levels
+ 6 rounded operations on sums of weights at most 1 + 4c (c = dt / 4 d^2, so
at most 1 + 10 here); 2 steps of 3 sweeps of 26 operations at 2^-53 and an
amplification of at most 11 give 2e-13 of max|psi|."""
import numpy as np
import pytest

import oracle
from paper_1601_04641_gb300 import build, inputs

pytestmark = pytest.mark.gpu

OMEGA = (1.0, 1.4, 2.0)
TOL = 2e-13


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


@pytest.mark.parametrize("shape", [(3, 3, 3), (4, 19, 34), (18, 3, 17), (33, 35, 66), (10, 130, 9), (300, 12, 5), (64, 48, 40)])
@pytest.mark.parametrize("factor", [0.02, 0.1, 1.0, 10.0])
@pytest.mark.parametrize("form", ["real", "complex", "realtime"])
def test_pcr_steps_match_oracle(shape, factor, form):
    from paper_1601_04641_gb300.solver import GP
    d = (0.31, 0.27, 0.29)
    dt, g = factor * min(d) ** 2, 12.0
    psi = inputs.random_field(shape, seed=3, complex_=form != "real").astype(np.complex128)
    gp = GP(shape, d, dt, OMEGA, g, "f64", "real" if form == "real" else "complex")
    gp.set_psi(psi.real.copy() if form == "real" else psi)
    (gp.step_real if form == "realtime" else gp.step_imag)(2)
    got = gp.get_psi().astype(np.complex128)
    gp.close()
    ref = psi.copy()
    oracle.step(ref, d, dt, OMEGA, g, form == "realtime", 2)
    assert np.max(np.abs(got - ref)) <= TOL * np.max(np.abs(ref))


@pytest.mark.parametrize("shape", [(3, 3), (4, 160), (150, 5), (61, 120), (8200, 5)])
@pytest.mark.parametrize("dt", [0.002, 0.2])
@pytest.mark.parametrize("form", ["real", "complex", "realtime"])
def test_axial_pcr_steps_match_oracle(shape, dt, form):
    """The radial lines' varying matrix, the weighted norm of the z sweep, and a radial line too long for a block."""
    from paper_1601_04641_gb300.solver import AxialGP
    nx, nz = shape
    drho, dz, g = 0.2, 0.22, 9.0
    rng = np.random.default_rng(5)
    r, z = (np.arange(nx) - 0.5)[:, None] / min(nx, 40), np.linspace(-1, 1, nz)[None, :]
    psi = np.exp(-3 * r * r - 2 * z * z) * (1 + 0.2 * rng.standard_normal(shape)) + 0j
    if form != "real":
        psi = psi * np.exp(1j * rng.uniform(-3, 3, shape))
    psi[0] = psi[-1] = 0
    psi[:, 0] = psi[:, -1] = 0
    a = AxialGP(nx, nz, drho, dz, dt, 1.2, 1.9, g, "f64", "real" if form == "real" else "complex")
    a.set_psi(psi.real.copy() if form == "real" else psi)
    (a.step_real if form == "realtime" else a.step_imag)(2)
    got = a.get_psi().astype(np.complex128)
    a.close()
    ref = psi.copy()
    oracle.axial_step(ref, drho, dz, dt, 1.2, 1.9, g, form == "realtime", 2)
    assert np.max(np.abs(got - ref)) <= TOL * np.max(np.abs(ref))
