"""Device memory is cleared in the order of the plan's stream: a clear on the
legacy default stream is not waited for by a non-blocking stream, whose first
pass could then read an error flag that is not cleared yet."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1910_06409_gb300", "csrc")


def test_clears_name_their_stream():
    sources = glob.glob(os.path.join(CSRC, "*.cu*"))
    assert sources
    for path in sources:
        with open(path) as f:
            assert not re.search(r"\bcudaMemset\s*\(", f.read()), os.path.basename(path)
