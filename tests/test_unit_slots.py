"""Where the units of a sparse part keep a row's sums, for parts of any size:
one of several parts may hold every entry (block-diagonal data), so a slot's
offset is not bounded by that of an average part.  The header that both
kernels take the offsets from is compiled for the host and compared with
Python's integers.  CPU only."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1506_01418_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "psgld_slots.cuh"
int main(int argc, char **argv)
{
    const long long n = atoll(argv[1]);
    const int unit = atoi(argv[2]), ldk = atoi(argv[3]);
    const int last = (int)((n - 1) / unit);   // as the kernels hold a unit's number
    printf("%lld %lld %lld\n", (long long)psgld::head_slot(last, ldk), (long long)psgld::tail_slot(last, ldk),
           (long long)psgld::slot_floats(n, unit, ldk));
}
"""


@pytest.fixture(scope="module")
def slots(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("slots")
    src, exe = d / "main.cpp", d / "main"
    src.write_text(MAIN)
    subprocess.run([gxx, "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)

    def run(n, unit, ldk):
        out = subprocess.run([str(exe), str(n), str(unit), str(ldk)], check=True, capture_output=True, text=True)
        return [int(x) for x in out.stdout.split()]
    return run


# entries of the largest part, entries per unit, row length: small ones, 10^6 x
# 10^5 (K = 512) and 6 10^5 x 2 10^5 (K = 388) with everything in one of 64
# parts, and the most entries that data can hold
@pytest.mark.parametrize("n,unit,ldk", [(1, 32, 4), (32, 32, 4), (33, 32, 128), (34_500_000, 8, 512),
                                        (46_000_000, 8, 388), (2 ** 31 - 1, 8, 512), (2 ** 31 - 1, 32, 128)])
def test_slots_of_a_part_with_every_entry(slots, n, unit, ldk):
    last = (n - 1) // unit
    head, tail, floats = slots(n, unit, ldk)
    assert (head, tail) == (2 * last * ldk, (2 * last + 1) * ldk)
    assert tail + ldk <= floats


def test_kernels_take_their_offsets_from_the_header():
    src = open(os.path.join(CSRC, "psgld_units.cu")).read()
    offsets = re.findall(r"(?:partial|hp) \+ ([^;?:)]+)", src)
    assert len(offsets) >= 6
    for o in offsets:
        assert o.startswith(("head_slot(", "tail_slot(", "4u * q")), o
