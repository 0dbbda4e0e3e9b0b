"""The stage kernels run while the kernel before them still writes (programmatic
dependent launch), so what a kernel of the step writes may not be read through
the read-only path.  A stale read cannot be provoked on demand, so this checks
the sources: read-only loads and the qualifiers that allow them appear only on
the run descriptors, the block table and the twiddle tables."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2208_02682_gb300", "csrc")


def _code(name):
    src = open(os.path.join(CSRC, name)).read()
    src = re.sub(r"/\*.*?\*/", " ", src, flags=re.S)
    return re.sub(r"//[^\n]*", "", src)


@pytest.mark.parametrize("name", ["common.cuh", "kernels.cuh", "stage.cuh"])
def test_no_read_only_loads_of_step_memory(name):
    """(fft.cuh holds the twiddle tables' read-only loads.)"""
    code = _code(name)
    if name == "stage.cuh":  # the descriptor copy
        code, n = re.subn(r"dst\[i\] = __ldg\(src \+ i\);", "", code)
        assert n == 1
    assert re.findall(r"[^\n]*(?:__ldg|ld\.global\.nc|__ldlu|__ldcs)[^\n]*", code) == []


def test_no_restrict_on_step_memory():
    code = _code("stage.cuh")
    names = set(re.findall(r"__restrict__\s+(\w+)", code))
    assert names == {"runs", "start"}
    # shared with the kernels around the stepping: the row spectra and the gather
    for f in ("load_rows_ct", "bilinear"):
        (params,) = re.findall(r"%s\(([^)]*\)?[^)]*)\)\s*\{" % f, _code("kernels.cuh"))
        assert "__restrict__" not in params, f
