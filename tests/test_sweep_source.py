"""What the kernels' source must keep to and no small input shows.

The sweep kernel's loads of what the sweep before it writes.

Sweeps are programmatic dependents: one is resident while the one before still writes the vector it will
gather. ld.global.nc (and __ldg, which compiles to it) is only defined for data that no one writes while
the kernel runs, so the walk vectors need coherent loads. A wrong kind of load shows up only as a rare
wrong count, so the source is checked.

Entry positions. A CSR holds up to 2^31 - 1 entries, and a lane adds up to 127 to a position before it compares
with its row's end: in 32 signed bits the sum would wrap, compare as smaller and read far out of range.
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


def test_entry_positions_do_not_wrap():
    for name in ("sweep.cu", "noalloc.cu"):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(build.CSRC, name)).read())
        uses = list(re.finditer(r"\bci \+ (\w+)", text))
        assert len(uses) >= 3
        for use in uses:  # the last declaration of the position before its use: unsigned or 64 bits wide
            decl = re.compile(r"\b(int|int32_t|unsigned|uint32_t|int64_t)\s+(?:\w+ = [^;=]*, )*" + use.group(1) + r"\s*=")
            kinds = [m.group(1) for m in decl.finditer(text, 0, use.start())]
            assert kinds and kinds[-1] in ("unsigned", "uint32_t", "int64_t"), f"{name}: {kinds[-1:]} {use.group(0)}"
