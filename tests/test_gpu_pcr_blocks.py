"""The cyclic reduction at every number of (node, line) pairs a thread, up to
its most shared memory and levels, and past its last level (where the
two-pass solve takes over), against the two-pass solve.

Bound: two steps of 3 sweeps, in each form at most 2 x 10 + 6 + 20 (kick)
rounded operations a sweep at 2^-53 on sums of weights at most 1 + 4c
(c = dt / 4 d^2); a wide smooth field keeps the renormalisation below two;
both solves: 2 x 2 x 3 x 46 x 2 x 2^-53 (1 + 4c) = 1.3e-13 (1 + 4c), and the
norms' sums 2e-14."""
import numpy as np
import pytest

from paper_1601_04641_gb300 import build

pytestmark = pytest.mark.gpu

OMEGA, G = (1.0, 1.4, 2.0), 12.0
# pairs a thread (real; complex): 2; 2 | 4; 2 | 8; 4 | long z lines, 2 and 4 | 1
SHAPES = [(80, 64, 48), (96, 80, 64), (100, 90, 80), (30, 31, 300), (33, 35, 66)]
FACTORS = [0.1, 1.0, 100.0, 1000.0, 10000.0]


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("factor", FACTORS)
@pytest.mark.parametrize("form", ["real", "complex", "realtime"])
def test_blocks_match_the_two_pass_solve(shape, factor, form):
    from paper_1601_04641_gb300.solver import GP
    # spacings of one condensate width in all: the trap's and the nonlinear exponents stay small at any factor
    h = min(0.2, 0.2 / factor ** 0.5)
    rng = np.random.default_rng(1)
    f = []
    for n in shape:
        v = np.exp(-1.5 * np.linspace(-1, 1, n) ** 2) * (1.0 if form == "real" else np.exp(1j * np.linspace(0, 2, n)))
        v[0] = v[-1] = 0.0
        f.append(v)
    psi = f[0][:, None, None] * f[1][None, :, None] * f[2][None, None, :] * (1.0 + 0.05 * rng.random(shape))
    psi, dt = np.ascontiguousarray(psi), factor * h * h
    out = []
    for two_pass in (False, True):
        gp = GP(shape, (h, h, h), dt, OMEGA, G, "f64", "real" if form == "real" else "complex")
        if two_pass:
            gp.set_window(0)
        gp.set_psi(psi)
        (gp.step_real if form == "realtime" else gp.step_imag)(2)
        out.append(gp.get_psi())
        gp.close()
    assert np.max(np.abs(out[0] - out[1])) <= (1.3e-13 * (1.0 + factor) + 2e-14) * np.max(np.abs(out[1]))
