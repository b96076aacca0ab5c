"""Loads through the read-only path (__ldg, ld.global.nc) are defined only for
memory that nothing writes as long as the kernel runs.  The kernels start
before the ones in front of them have ended, so what a caller passes (keys,
values, masks, gammas, biases) may still be written while they are resident;
only the rotation tables, filled when a cache is made, may be read so."""
import glob
import os
import re

from tests.conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2609_22283_gb300", "csrc")


def _code(path):
    return re.sub(r"//[^\n]*", "", open(path).read())


def test_read_only_loads_are_of_the_tables():
    files = sorted(glob.glob(os.path.join(CSRC, "*.cu*")))
    assert files
    for path in files:
        code = _code(path)
        assert not re.search(r"ld\.global[.\w]*\.nc", code) and "__restrict__" not in code, path
        for arg in re.findall(r"__ldg\(([^;]*)\);", code):
            assert re.match(r"(r?p\.tab_[thw]\b|tab\b)", arg), f"{os.path.basename(path)}: __ldg({arg})"
