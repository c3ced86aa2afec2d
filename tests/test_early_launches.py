"""Kernels that launch_early starts are resident while the kernel before them
still writes what they will read.  Read off the sources (a race cannot be
shown by running it): such a kernel waits before it lets the next one in and
before it reads.  CPU only."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1506_01418_gb300", "csrc")
EARLY = ["psgld_rows.cu", "psgld_step.cu", "psgld_dense.cu"]


def _source(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def _functions(src):
    """Last line of the head, and body, of every function (braces at the margin)."""
    return re.findall(r"\n([^\n]+)\n\{\n(.*?)\n\}", src, flags=re.S)


@pytest.mark.parametrize("name", EARLY)
def test_waits_come_before_the_next_launch_is_let_in(name):
    found = 0
    for head, body in _functions(_source(name)):
        if "let_next" not in body:
            continue
        found += 1
        assert body.count("dev::wait_prior();") == 1 == body.count("dev::let_next();"), head
        assert body.index("dev::wait_prior();") < body.index("dev::let_next();"), head
        assert not re.search(r"if \([^;]*\)\s*dev::wait_prior", body), head
        # nothing is read through a pointer of the parameters before the wait
        before = body[:body.index("dev::wait_prior();")]
        assert not re.search(r"__ldg|bulk_g2s|ld4|load\(", before), head
    assert found

