"""The sweep kernel's loads of what the sweep before it writes.

Sweeps are programmatic dependents: one is resident while the one before still writes the vector it will
gather. ld.global.nc (and __ldg, which compiles to it) is only defined for data that no one writes while
the kernel runs, so the walk vectors need coherent loads. A wrong kind of load shows up only as a rare
wrong count, so the source is checked.
"""
import os
import re

from paper_1910_13874_gb300 import build


def sweep_code():
    text = open(os.path.join(build.CSRC, "sweep.cu")).read()
    return re.sub(r"//[^\n]*", "", text)


def test_walk_vectors_are_loaded_coherently():
    code = sweep_code()
    assert "griddepcontrol.launch_dependents" in code
    # the only non-coherent inline load is that of the column indices
    for m in re.finditer(r"ld\.global\.nc", code):
        fn = code.rfind("__device__ __forceinline__", 0, m.start())
        assert "ld_idx(" in code[fn:m.start()], code[m.start() - 80:m.end() + 40]
    # __ldg only on what no sweep writes: bit masks and vertex scales
    for m in re.finditer(r"__ldg\(([^;]*);", code):
        assert re.match(r"(mask|nz|rs) \+", m.group(1)), m.group(0)
