"""Launch settings of FP64 handles: what is set is what runs, and what is not
set is the automatic choice."""
import numpy as np
import pytest

from paper_1601_04641_gb300 import build, inputs

pytestmark = pytest.mark.gpu

SHAPE, D, DT, OMEGA, G = (64, 48, 40), (0.2, 0.2, 0.2), 0.004, (1.0, 1.4, 2.0), 10.0


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _gp():
    from paper_1601_04641_gb300.solver import GP
    gp = GP(SHAPE, D, DT, OMEGA, G, "f64", "real")
    gp.set_psi(np.ascontiguousarray(inputs.random_field(SHAPE, seed=6, complex_=False).real.astype(np.float64)))
    return gp


def _after(settings):
    gp = _gp()
    settings(gp)
    lines = gp.lines_per_thread(0)
    gp.step_imag(3)
    psi = gp.get_psi()
    gp.close()
    return lines, psi


def test_lines_per_thread_that_are_set_are_taken():
    """Four adjacent lines are more than FP64 has a form for: the widest group, two.  Any count set keeps the two-pass solve
    (whose arithmetic per line is the same for every count); nothing set leaves one line and the automatic form."""
    two_pass = _after(lambda gp: gp.set_window(0))
    assert two_pass[0] == (1, 1, 1) and _after(lambda gp: None)[0] == (1, 1, 1)
    for set_lines, want in ((lambda gp: gp.set_pair_lines(True), 2), (lambda gp: gp.set_pair_lines(False), 1)):
        lines, psi = _after(lambda gp: (set_lines(gp), gp.set_axis_window(2, 0)))
        assert lines == (want, want, 1) and np.array_equal(psi, two_pass[1])
    for n, want in ((1, 1), (2, 2), (4, 2)):
        lines, psi = _after(lambda gp: ([gp.set_lines_per_thread(ax, n) for ax in (0, 1)], gp.set_axis_window(2, 0)))
        assert lines == (want, want, 1) and np.array_equal(psi, two_pass[1])
    assert not np.array_equal(_after(lambda gp: None)[1], two_pass[1])  # the automatic form rounds differently here


def test_autotune_ignores_entries_that_predate_the_automatic_form(tmp_path):
    """An older cache holds a block size for every FP64 axis; taking it would keep the cyclic reduction from running."""
    cache = tmp_path / "tune.txt"
    cache.write_text("".join("64x48x40/f64/r/it/w0/ax%d/v2 64 0 4\n" % ax for ax in range(3)))
    gp = _gp()
    before = gp.get_psi()
    gp.autotune(False, 3, str(cache))
    assert np.array_equal(gp.get_psi(), before)
    lines = cache.read_text().split("\n")[3:6]
    assert [ln.split()[0] for ln in lines] == ["64x48x40/f64/r/it/w0/ax%d/l4/v3" % ax for ax in range(3)]
    gp.close()
    # another dt with other levels is another entry; the same dt reads its own back
    gp = _gp()
    gp.autotune(False, 3, str(cache))
    assert len(cache.read_text().split("\n")) == 7
    gp.set_dt(20 * DT)
    gp.autotune(False, 3, str(cache))
    assert len(cache.read_text().split("\n")) == 10
    gp.close()


def test_autotuned_steps_match_the_automatic_ones(tmp_path):
    gp = _gp()
    gp.autotune(False, 3, str(tmp_path / "tune.txt"))
    gp.step_imag(3)
    psi = gp.get_psi()
    gp.close()
    ref = _after(lambda gp: None)[1]
    assert np.max(np.abs(psi - ref)) <= 2e-13 * np.max(np.abs(ref))  # two forms of 3 sweeps of 26 operations, 3 steps
