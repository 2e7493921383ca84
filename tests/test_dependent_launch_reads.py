"""A kernel that may be launched as a programmatic dependent lives while its
predecessor still writes: read-only (non-coherent) loads are for tables that
no launch writes, never for the field, the renormalisation factor or partial
sums.  A check of the sources of the sweeps' kernels (no GPU)."""
import os
import re

import pytest

from paper_1601_04641_gb300 import build

WRITTEN = re.compile(r"\b(scale|psi|psi_out|in|out|partials|counter|norm_out|scale_out)\b")


@pytest.mark.parametrize("name", ["gp_sweep.cuh", "gp_pcr.cuh"])
def test_read_only_loads_are_of_tables(name):
    src = open(os.path.join(build.CSRC, name)).read()
    src = re.sub(r"//[^\n]*", "", src)
    loads = re.findall(r"\b(?:__ldg|ldc)\(([^;]*?)\)", src)
    assert loads
    assert not [a for a in loads if WRITTEN.search(a)]
    assert "__restrict__ psi" not in src and "__restrict__ scale" not in src


def test_the_previous_launch_is_waited_for_before_the_field_is_read():
    src = re.sub(r"//[^\n]*", "", open(os.path.join(build.CSRC, "gp_pcr.cuh")).read())
    body = src[src.index("void __launch_bounds__(1024) lines_pcr_kernel"):]
    wait = body.index("pdl_wait()")
    assert wait < body.index("kick_init") and wait < body.index("= in[")
