"""Shared-memory limits belong to a device's context: a limit raised once per process leaves the kernels of a
second device without it.  One device cannot show that, so the sources are read: no cudaFuncSetAttribute (nor a
query that depends on one) runs under std::call_once."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1703_01545_gb300", "csrc")


def once_bodies(text):
    """The argument lists of every std::call_once(...) in `text`."""
    for m in re.finditer(r"call_once\s*\(", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        yield text[m.end():i - 1]


def test_no_limit_is_raised_once_per_process():
    files = sorted(glob.glob(os.path.join(CSRC, "*.cu")))
    assert any("cudaFuncSetAttribute" in open(f).read() for f in files)
    for f in files:
        for body in once_bodies(open(f).read()):
            assert not re.search(r"cudaFuncSetAttribute|find_pair_clusters|cudaOccupancy", body), os.path.basename(f)
