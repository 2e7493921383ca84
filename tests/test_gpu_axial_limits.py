"""FP64 axial condensates at the ends of what the cyclic reduction takes."""
import numpy as np
import pytest

import oracle
from paper_1601_04641_gb300 import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


@pytest.mark.parametrize("field", ["real", "complex"])
@pytest.mark.parametrize("drho,dt", [(10.0, 0.5), (3.0, 0.5), (2.4, 0.4)])
def test_trap_factors_below_the_roundoff(field, drho, dt):
    """dt V up to 500 at every site: the factors are far below 2^-53 and the renormalised field is still the oracle's.  The
    exponent is within 4 relative roundings, so a value within (4 dt V + 30) 2^-53 a step, dt V < 60 where the field is
    largest: 2 steps, 6e-14 of max|psi|."""
    from paper_1601_04641_gb300.solver import AxialGP
    nx, nz, dz, gamma, lam, g = 4, 7, 1.0, 3.0, 1.0, 2.0
    rng = np.random.default_rng(3)
    psi = rng.uniform(0.2, 1.0, (nx, nz)) * (np.exp(1j * rng.uniform(-3, 3, (nx, nz))) if field == "complex" else 1.0) + 0j
    psi[0] = psi[-1] = 0
    psi[:, 0] = psi[:, -1] = 0
    a = AxialGP(nx, nz, drho, dz, dt, gamma, lam, g, "f64", field)
    a.set_psi(psi if field == "complex" else psi.real.copy())
    a.step_imag(2)
    got, obs = a.get_psi().astype(np.complex128), a.observables()
    a.close()
    ref = psi.copy()
    oracle.axial_step(ref, drho, dz, dt, gamma, lam, g, False, 2)
    assert abs(obs["norm"] - 1.0) <= 1e-12
    assert np.max(np.abs(got - ref)) <= 6e-14 * np.max(np.abs(ref))


def test_a_long_radial_line_gets_no_reduction_tables():
    """2e6 radial nodes: two fields (96 MB), the radial two-pass tables (128), the Cartesian ones (80) and the nodes' (48);
    the reduction's, for lines that no block can hold, would add at least 144."""
    import torch
    from paper_1601_04641_gb300.solver import AxialGP
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    a = AxialGP(2000000, 3, 0.5, 0.5, 1e-3, 1e-9, 1.0, 1.0, "f64", "real")
    used = free - torch.cuda.mem_get_info()[0]
    a.init_gaussian()
    a.step_imag(1)
    assert abs(a.observables()["norm"] - 1.0) <= 1e-10
    a.close()
    assert used <= 400e6
