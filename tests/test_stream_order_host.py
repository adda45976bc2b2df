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


def test_uploads_are_done_before_kernels_on_other_streams():
    text = dict(_sources())
    # the one other user copies and reads on the legacy stream
    before, own = text["imrp_api.cu"].split("int imrp_admittance(", 1)
    assert not re.search(r"\bcudaMemcpy\s*\(", before + own.split("\n}\n", 1)[1])
    init = text["imrp_inst.cuh"].rpartition("cudaMemcpyToSymbol")[2]
    assert "cudaStreamSynchronize(cudaStreamLegacy)" in init.split("done[dev] = true")[0]
