"""The in-tree build: what it recompiles for."""
import os
import re

from paper_1910_13874_gb300 import build


def test_every_included_header_is_a_dependency():
    # an object older than a header it includes is stale: each local include counts, whatever its suffix
    deps = {os.path.basename(p) for p in build._deps()}
    for src in build._sources():
        for name in re.findall(r'#include "([^"]+)"', open(src).read()):
            assert name in deps, f"{os.path.basename(src)} includes {name}"
