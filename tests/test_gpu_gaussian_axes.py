"""The Gaussian start on both sides of the node count up to which its per-axis
factors are held in shared memory, against numpy.

Bound: a value is three factors of at most 4 roundings each on exponents
below 13, two products and the normalisation, whose sum has under 64
roundings in a row: 2^-53 (3 (4 + 13 x 2) + 3 + 64) = 1.8e-14 of the largest;
FP32 fields round once more, and their sums are of the rounded values:
2^-24 x 3."""
import numpy as np
import pytest

from paper_1601_04641_gb300 import build

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [4989, 4990])  # 5000 and 5001 nodes on the three axes
@pytest.mark.parametrize("precision,field,tol", [("f64", "real", 1.8e-14), ("f64", "complex", 1.8e-14), ("f32", "real", 1.8e-7)])
def test_gaussian_start(nx, precision, field, tol):
    build.build()
    from paper_1601_04641_gb300.solver import GP
    shape, d, omega = (nx, 3, 8), (0.002, 0.3, 0.4), (1.0, 1.3, 0.7)
    gp = GP(shape, d, 1e-7, omega, 5.0, precision, field)
    gp.init_gaussian()
    got, norm = gp.get_psi(), gp.observables()["norm"]
    gp.close()
    f = []
    for n, h, w in zip(shape, d, omega):
        x = (np.arange(n) - 0.5 * (n - 1)) * h
        v = (w / np.pi) ** 0.25 * np.exp(-0.5 * w * x * x)
        v[0] = v[-1] = 0.0
        f.append(v)
    ref = f[0][:, None, None] * f[1][None, :, None] * f[2][None, None, :]
    ref /= np.sqrt((ref ** 2).sum() * d[0] * d[1] * d[2])
    assert np.max(np.abs(got - ref)) <= tol * ref.max()
    assert abs(norm - 1.0) <= 4 * tol
