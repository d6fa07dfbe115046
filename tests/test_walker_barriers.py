"""Barriers of the row walkers' emitters, read from the sources.

`walk_rows` instantiates a walker, and the emitter in it, once for inner strips
and once for edge strips, and each warp of a CTA picks its own.  CUDA C++
defines __syncthreads() in conditional code only where the whole block takes
the same side, so an emitter may not call it: a CTA barrier there is PTX's
barrier.sync, which counts threads whatever instruction they arrive from.
"""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1803_00737_gb300", "csrc")


def _bodies():
    """(file, name, text) of every struct handed to the walkers (they define kMode and row_end)."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"^struct (\w+) \{.*?^\};", text, re.S | re.M):
            if "row_end" in m.group(0):
                yield os.path.basename(path), m.group(1), m.group(0)


def test_emitters_hold_no_block_uniform_barrier():
    found = list(_bodies())
    assert {"DirectEmit", "StagedEmit", "MetricEmit"} <= {name for _, name, _ in found}
    for path, name, body in found:
        assert not re.search(r"__syncthreads|bar\.sync|\.aligned\b", body), f"{path}: {name}"
