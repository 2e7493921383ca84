"""FP64 handles whose dt changes across the switch between the cyclic
reduction and the two-pass solve: an axis must not go on solving with the
tables of an earlier dt.  Each step after a change equals, bit for bit, the
step of a fresh handle of that dt; real time is held to the FP64 oracle too.

Oracle bound: at most 6 real-time steps (no renormalisation) of 3 sweeps of
26 rounded operations at 2^-53 on values that the solves amplify by at most
1 + 4c (c = dt / 4 d^2, at most 2 here): 6 x 78 x 2^-53 x 2 = 1.1e-13 of
max|psi|."""
import numpy as np
import pytest

import oracle
from paper_1601_04641_gb300 import build, inputs

pytestmark = pytest.mark.gpu

OMEGA, G, D = (1.0, 1.4, 2.0), 12.0, (0.31, 0.27, 0.29)
H2 = min(D) ** 2
TOL = 1.1e-13


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _handle(shape, factor, field, psi):
    from paper_1601_04641_gb300.solver import GP
    gp = GP(shape, D, factor * H2, OMEGA, G, "f64", field)
    gp.set_psi(psi)
    return gp


def _psi(shape, field):
    psi = inputs.random_field(shape, seed=8, complex_=field == "complex")
    return psi.astype(np.complex128) if field == "complex" else np.ascontiguousarray(psi.real.astype(np.float64))


@pytest.mark.parametrize("shape,field,factors", [
    ((96, 96, 96), "real", (0.1, 0.5, 0.1)), ((100, 100, 100), "real", (0.1, 0.5, 0.1)),
    ((96, 96, 96), "real", (1.0, 0.1, 1.0)), ((80, 80, 80), "complex", (0.05, 1.0, 0.05)),
    ((160, 128, 96), "complex", (0.02, 0.1, 1.0))])
def test_steps_after_a_change_of_dt(shape, field, factors):
    psi = _psi(shape, field)
    gp, ref = _handle(shape, factors[0], field, psi), psi.astype(np.complex128)
    for f in factors:
        gp.set_dt(f * H2)
        gp.set_psi(psi)
        fresh = _handle(shape, f, field, psi)
        for h in (gp, fresh):
            (h.step_imag if field == "real" else h.step_real)(2)
        psi = gp.get_psi()
        assert np.array_equal(psi, fresh.get_psi())
        fresh.close()
        if field == "complex":
            oracle.step(ref, D, f * H2, OMEGA, G, True, 2)
            assert np.max(np.abs(psi - ref)) <= TOL * np.max(np.abs(ref))
    gp.close()


def test_schedule_across_the_switch():
    shape, psi = (96, 96, 96), _psi((96, 96, 96), "real")
    gp = _handle(shape, 0.1, "real", psi)
    gp.run_imag_schedule([(5.0, 1e-30), (1.0, 1e-30)], 2, 4)
    got = gp.get_psi()
    gp.close()
    for f in (0.5, 0.1):
        h = _handle(shape, f, "real", psi)
        for _ in range(2):  # as the schedule goes, from check to check
            h.step_imag(2)
            h.observables()
        psi = h.get_psi()
        h.close()
    # the schedule carries its renormalisation factor across the change, the handles fold it into psi: one rounding a step
    assert np.max(np.abs(got - psi)) <= 1e-14 * np.max(np.abs(psi))
