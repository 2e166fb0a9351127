"""Kernels of a call may start before the one before them in the stream has ended
(launch_next), so what another kernel of the call writes is not read with
non-coherent loads: in the sources, __ldg and ldg2 take a plan's constant tables
only (copied there before any of the call's kernels), never frames, planes,
intermediates or taps."""

import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2003_08960_gb300", "csrc")
TABLES = {"twl", "twx", "twy", "ox", "oy", "cx", "cy", "cx2", "cy2", "wq", "cis", "bmat"}
FILES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))


def _arguments(text):
    """The argument of every __ldg( and ldg2( call, to its closing bracket."""
    for m in re.finditer(r"\b(?:__ldg|ldg2)\(", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        yield text[m.end():i - 1]


@pytest.mark.parametrize("path", FILES, ids=[os.path.basename(f) for f in FILES])
def test_non_coherent_loads_take_tables_only(path):
    text = re.sub(r"//[^\n]*", "", open(path).read())
    # the wrapper itself, and the row and column DFTs' twiddle argument (always p.tw*)
    text = text.replace("float2 ldg2(const float2* p) { return __ldg(p); }", "")
    for call in re.findall(r"\b(?:row_dft|col_dft)<[^;]*?>\(a, ([^,]*),", text):
        assert call in ("p.twx", "p.twy", "p.twl"), call
    for arg in _arguments(text):
        if os.path.basename(path) == "sharpness.cu" and arg == "tw + k2 * N1 + j1":
            continue
        names = set(re.findall(r"\b[pc]\.(\w+)", arg)) - {"z0", "slot0", "nl"}
        assert names and names <= TABLES, f"{os.path.basename(path)}: non-coherent load of {arg}"
