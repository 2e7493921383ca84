"""The host rules that choose kernels and lay out their tables, asked of
libgpcn.so itself through a small C++ client (no GPU)."""
import os
import random
import re
import subprocess

import pytest

from paper_1601_04641_gb300 import _native as N
from paper_1601_04641_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    build.build()
    exe = str(tmp_path_factory.mktemp("probe") / "probe")
    cuda = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
    lib = os.path.dirname(N.LIB_PATH)
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", build.INCLUDE, "-I", build.CSRC, "-I", cuda, os.path.join(HERE, "host_probe.cpp"),
                    "-L", lib, "-lgpcn", "-Wl,-rpath," + lib, "-o", exe], check=True, capture_output=True, text=True)

    def ask(*args):
        out = subprocess.run([exe] + [str(a) for a in args], check=True, capture_output=True, text=True, timeout=120).stdout
        return [[float(v) for v in line.split()] for line in out.splitlines()]

    return ask


@pytest.mark.parametrize("shape,modes,factors", [
    ((96, 96, 96), 1, (0.1, 0.5, 0.1, 1.0, 0.1)), ((100, 100, 100), 1, (0.1, 0.5, 0.1)), ((80, 80, 80), 2, (0.05, 1.0, 0.05)),
    ((64, 48, 40), 1, (0.1, 1.0, 10.0, 0.1)), ((160, 128, 96), 2, (0.02, 0.1, 1.0))])
def test_tables_of_a_new_dt_keep_nothing_of_the_old(probe, shape, modes, factors):
    """A handle's tables are rebuilt in place when dt changes: an axis that takes the cyclic reduction at one dt and not at
    the next must not keep the old levels and offsets."""
    got = probe("tables", *shape, modes, *factors)
    assert [g[0] for g in got] == [1.0] * len(factors)


def test_shared_memory_opt_in_is_kept_per_device(probe):
    """The limit is a property of a kernel on one device: the second device gets its own call, a larger launch raises it, a
    smaller one and one from another thread never lower it, and a failed call is made again."""
    d0, d1, d2, bad, threads = probe("optin")
    assert d0 == [60000, 1] and d1 == [70000, 2] and d2 == [60000, 1]
    assert bad == [3, 0]  # two failed calls and one on a device beyond those kept
    assert threads[0] == 50000 + 999 * 37 + 7 * 911 and threads[1] == 0


def test_no_launcher_keeps_a_process_wide_opt_in():
    for name in sorted(os.listdir(build.CSRC)):
        src = open(os.path.join(build.CSRC, name)).read()
        assert not re.search(r"static\s+(bool|int)\s+attr\b", src), name


@pytest.mark.parametrize("asked", [0, 1, 2, 3, 5, 16])
@pytest.mark.parametrize("kinds", [1, 2, 4, 8])
def test_stream_groups_are_no_more_than_asked_for(probe, asked, kinds):
    """Every instance in one group; at most as many groups as set, where not set two or one per kind; groups of one kind
    wherever there are enough of them; balanced by sites within the largest instance."""
    rng = random.Random(7)
    items = [(rng.randrange(kinds) if q >= kinds else q, rng.randrange(1000, 50000)) for q in range(24)]
    groups = [[int(v) for v in g] for g in probe("streams", asked, *[v for it in items for v in it])]
    assert sorted(i for g in groups for i in g) == list(range(24))
    most = asked or max(2, kinds)
    assert len(groups) == min(most, 24)
    if most >= kinds:
        assert all(len({items[i][0] for i in g}) == 1 for g in groups)
        shared = [[g for g in groups if items[g[0]][0] == k] for k in range(kinds)]
    else:
        shared = [groups]
    for gs in shared:
        load = [sum(items[i][1] for i in g) for g in gs]
        assert max(load) - min(load) <= max(items[i][1] for g in gs for i in g)


# grid, form (0 real, 1 complex, 2 real time), levels, axis, us a step gained by the reduction on that axis (measured)
CROSSOVER = [
    ((64, 48, 40), 0, 4, 0, 41.7), ((80, 80, 80), 0, 4, 1, 10.4), ((80, 80, 80), 2, 4, 0, 45.5), ((96, 96, 96), 0, 4, 1, 6.3),
    ((96, 96, 96), 0, 4, 2, 7.3), ((96, 96, 96), 1, 4, 1, 7.1), ((112, 112, 112), 0, 4, 0, 8.5), ((160, 128, 96), 0, 4, 0, 12.7),
    ((40, 200, 300), 2, 3, 2, 41.7), ((150, 60, 250), 2, 3, 2, 30.8),
    ((160, 128, 96), 0, 4, 2, -5.7), ((160, 128, 96), 1, 4, 2, -19.6), ((60, 120, 180), 1, 4, 0, -7.2),
    ((60, 120, 180), 0, 5, 0, -6.3), ((90, 157, 150), 0, 4, 0, -13.2), ((90, 157, 150), 2, 3, 0, -29.1),
    ((128, 128, 128), 0, 4, 0, -5.9), ((200, 160, 120), 0, 4, 1, -38.4), ((30, 150, 150), 1, 4, 0, -7.3),
]


@pytest.mark.parametrize("shape,form,levels,axis,gain", CROSSOVER)
def test_the_choice_of_the_reduction_follows_the_measurements(probe, shape, form, levels, axis, gain):
    lines = shape[0] * shape[1] * shape[2] // shape[axis]
    (chosen, tl), = probe("choose", lines, shape[axis] - 2, form, axis, levels, 8 if form == 0 else 16)
    assert bool(chosen) == (gain > 0)


@pytest.mark.parametrize("form,elem", [(0, 8), (1, 16), (2, 16)])
def test_a_blocks_lines_fit_its_threads_and_shared_memory(probe, form, elem):
    for shape in ((64, 48, 40), (100, 90, 80), (90, 157, 150), (20, 300, 300), (400, 20, 30), (3, 3, 3)):
        for axis in range(3):
            n, lines = shape[axis] - 2, shape[0] * shape[1] * shape[2] // shape[axis]
            for levels in range(1, 11):
                _, tl = probe("choose", lines, n, form, axis, levels, elem)[0]
                assert tl * n <= (8192 if elem == 8 else 4096)
                assert tl == 0 or tl * (2 * n * elem + 8) + n * (2 * levels + 3) * (16 if form == 2 else 8) <= 100 * 1024


def test_gpu_block_cases_reach_every_form(probe):
    """The grids of test_gpu_pcr_blocks.py take the reduction with 1, 2, 4 and (real fields) 8 pairs a thread, with more than
    48 KB of shared memory, and with 3 to 10 levels."""
    from tests import test_gpu_pcr_blocks as blocks
    seen, big, levels_seen = set(), False, set()
    for form, elem in ((0, 8), (1, 16), (2, 16)):
        for shape in blocks.SHAPES:
            for factor in blocks.FACTORS:
                c = factor / 4.0 * (1j if form == 2 else 1.0)
                b, levels = c / (1.0 + 2.0 * c), 0
                while levels == 0 or 2.0 * abs(b) > 2.0 ** -55:
                    b, levels = b * b / (1.0 - 2.0 * b * b), levels + 1
                if levels > 10:
                    continue
                for axis in range(3):
                    n, lines = shape[axis] - 2, shape[0] * shape[1] * shape[2] // shape[axis]
                    (chosen, tl), = probe("choose", lines, n, form, axis, levels, elem)
                    if chosen:
                        seen.add((form, 1 if tl * n <= 1024 else 2 if tl * n <= 2048 else 4 if tl * n <= 4096 else 8))
                        big |= tl * 2 * n * elem > 48 * 1024
                        levels_seen.add(levels)
    assert seen == {(0, 1), (0, 2), (0, 4), (0, 8), (1, 1), (1, 2), (1, 4), (2, 1), (2, 2), (2, 4)}
    assert big and levels_seen >= set(range(4, 11)) - {6, 7}
