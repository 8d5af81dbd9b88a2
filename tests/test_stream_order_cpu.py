"""Device memory is written in stream order: the handles' streams are not ordered with the default one."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1812_06765_gb300", "csrc")


def test_no_copy_or_fill_without_a_stream():
    """cudaMemcpy and cudaMemset run on the legacy default stream, and one from pageable memory may return
    before its transfer has finished; kernels on a non-blocking stream would not wait for it."""
    found = []
    for f in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, f)) as src:
            code = re.sub(r"//[^\n]*|/\*.*?\*/", "", src.read(), flags=re.S)
        found += ["%s: %s" % (f, m) for m in re.findall(r"\bcuda(?:Memcpy|Memset)(?:2D|3D)?\s*\(", code)]
    assert not found
