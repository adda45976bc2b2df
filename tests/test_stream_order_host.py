"""Device memory is set in the order of the stream that uses it: contexts work on non-blocking streams, which
the legacy stream of a plain cudaMemset does not order itself with."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2111_13072_gb300", "csrc")


def _sources():
    for path in sorted(glob.glob(os.path.join(CSRC, "*"))):
        with open(path) as f:
            yield os.path.basename(path), re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


def test_memory_is_zeroed_on_a_stream():
    found = [name for name, text in _sources() if re.search(r"\bcudaMemset\s*\(", text)]
    assert not found
