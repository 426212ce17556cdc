"""The digest that dates captured traffic figures covers every source of the solver kernels: what solver_inst.cu
includes, directly or through a header of its own folder."""

import os
import re

from paper_1602_03638_gb300 import build


def test_digest_covers_the_included_sources():
    seen, todo = set(), ["solver_inst.cu"]
    while todo:
        name = todo.pop()
        seen.add(name)
        with open(os.path.join(build.CSRC, name)) as f:
            for inc in re.findall(r'#include\s+"([^"]+)"', f.read()):
                if os.path.exists(os.path.join(build.CSRC, inc)) and inc not in seen:
                    todo.append(inc)
    assert seen <= set(build.KERNEL_SOURCES) | {"solver_inst.cu"}
