"""Kernels launched dependently start beside the kernel before them, so they
must not tell the compiler that what it writes is constant: a non-coherent
load may then be moved above the wait."""
from __future__ import annotations

import glob
import os
import re

from tests import cpp_extract

# arrays that no kernel of a sweep writes: SITES tables and the couplings
_CONSTANT = re.compile(r"__ldg\((p\.cum|lg|J) \+ ")


def test_no_noncoherent_loads_behind_the_wait():
    seen = 0
    for path in sorted(glob.glob(os.path.join(cpp_extract.CSRC, "*.cu"))):
        text = open(path).read()
        for m in re.finditer(r"__global__", text):
            head = text[m.start():text.index("{", m.start())]
            body = cpp_extract.function(os.path.basename(path), head)
            if "pdl_begin()" not in body:
                continue
            seen += 1
            name = re.search(r"(\w+)\(", head[head.index("void"):].replace("__launch_bounds__(", "")).group(1)
            assert "__restrict__" not in head, name
            for use in re.finditer(r"__ldg\(", body):
                assert _CONSTANT.match(body, use.start()), (name, body[use.start():use.start() + 40])
    assert seen >= 10   # the sweep, PT and measurement kernels of the three packings
