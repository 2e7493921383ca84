"""A change of dt that needs larger coefficient tables (FP64: the cyclic
reduction's) and cannot get them: GP_ERR_NOMEM, and the handle goes on at its
old dt with the same results, bit for bit."""
import numpy as np
import pytest

from paper_1601_04641_gb300 import _native as N
from paper_1601_04641_gb300 import build, inputs

pytestmark = pytest.mark.gpu


def test_failed_allocation_keeps_the_old_dt():
    build.build()
    from paper_1601_04641_gb300.solver import GP
    shape, d = (64, 48, 40), (0.2, 0.2, 0.2)
    psi = np.ascontiguousarray(inputs.random_field(shape, seed=2, complex_=False).real.astype(np.float64))
    got = []
    for fail in (False, True):
        gp = GP(shape, d, 0.004, (1.0, 1.4, 2.0), 10.0, "f64", "real")
        gp.set_psi(psi)
        if fail:
            gp.lib.gp_debug_fail_alloc(1)
            try:
                with pytest.raises(N.GPError) as e:
                    gp.set_dt(0.4)  # more reduction levels: larger tables
            finally:
                gp.lib.gp_debug_fail_alloc(0)
            assert e.value.status == N.GP_ERR_NOMEM
        gp.step_imag(3)
        got.append((gp.get_psi(), gp.observables()))
        gp.close()
    assert np.array_equal(got[0][0], got[1][0]) and got[0][1] == got[1][1]
