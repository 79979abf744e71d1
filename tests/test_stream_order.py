"""A context's device memory is written on its own (non-blocking) stream, which
the legacy default stream is not ordered with: a clear or an upload queued
there can run after, or in the middle of, the work that uses the memory, most
of all in a batch, where it may wait behind another system's graph.  So the
sources hold no clear, upload or launch without a stream."""

import glob
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_25161_gb300", "csrc")


def calls(text, name):
    """Argument texts of the calls of `name`."""
    for m in re.finditer(r"\b%s\(" % name, text):
        depth, k = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[k], 0)
            k += 1
        yield text[m.end():k - 1]


def test_nothing_writes_device_memory_on_the_legacy_stream():
    for path in sorted(glob.glob(os.path.join(SRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        where = os.path.basename(path)
        for name in ("cudaMemset", "cudaMemset2D", "cudaMemcpyToSymbol", "cudaMemcpy2D"):
            assert not list(calls(text, name)), (where, name)
        for args in calls(text, "cudaMemcpy"):  # blocking reads of the caller's arrays only
            assert args.replace(" ", "").endswith("cudaMemcpyDeviceToHost"), (where, args)
        for m in re.finditer(r"<<<(.*?)>>>", text, re.S):
            depth = commas = 0
            for ch in m.group(1):
                depth += {"(": 1, "[": 1, ")": -1, "]": -1}.get(ch, 0)
                commas += ch == "," and depth == 0
            assert commas == 3, (where, m.group(0))
