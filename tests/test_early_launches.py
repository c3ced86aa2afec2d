"""Kernels that launch_early starts are resident while the kernel before them
still writes what they will read.  Read off the sources (a race cannot be
shown by running it): such a kernel waits before it lets the next one in and
before it reads; factors, their copies, gradients and the step-size table are
read by ordinary loads, and the read-only path (__ldg, ld.global.nc) only
reads what no kernel of a sweep writes.  CPU only."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1506_01418_gb300", "csrc")
EARLY = ["psgld_rows.cu", "psgld_step.cu", "psgld_dense.cu"]

# the entries and row offsets of the layout, the lists of its rows, V, and
# the prefix arrays of a batch's tables
READ_ONLY = r"(S\.heavy|S\.mid|S\.idx|S\.val|ptr|vrow|item_start|cta_start|(src\.)?(rows|cols)_start|" \
            r"(src\.)?[wh]start|start|pre)\b"


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


@pytest.mark.parametrize("name", EARLY)
def test_read_only_loads_read_what_a_sweep_does_not_write(name):
    src = _source(name)
    loads = re.findall(r"__ldg\(\s*([^;]*)", src)
    assert loads
    for x in loads:
        assert re.match(READ_ONLY, x), x
    assert not re.search(r"\bldg4\(|__ldc[ags]\(", src)
    for x in re.findall(r"ldg_stream\((?!const)([^;]*)", src):
        assert x.startswith("src_v"), x                     # V's tiles
    # the only other mention of the read-only path: ldg_stream itself
    assert len(re.findall(r"ld\.global\.nc", src)) == ("ldg_stream" in src)


def test_kernels_that_use_read_only_loads_of_factors_are_launched_plainly():
    users = [f for f in sorted(os.listdir(CSRC)) if re.search(r"\bldg4\(", _source(f)) and f != "psgld_update.cuh"]
    for f in users:
        assert "launch_early" not in _source(f) and "let_next" not in _source(f), f
