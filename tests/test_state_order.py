"""psgld_set_state is synchronous: its copies run on the legacy stream, and
the calls after it run on non-blocking ones (read off the source: the race
between a copy's tail and the next call cannot be shown by running it).  CPU
only."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1506_01418_gb300", "csrc")


def test_set_state_waits_for_its_copies():
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "psgld_api.cu")).read())
    body = re.search(r"\npsgld_status psgld_set_state\(.*?\n\{\n(.*?)\n\}", src, flags=re.S).group(1)
    assert "cudaMemcpyHostToDevice" in body
    assert "cudaStreamSynchronize(nullptr)" in body[body.rindex("cudaMemcpyHostToDevice"):]
