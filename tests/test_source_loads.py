"""Kernels are launched while their predecessor in the stream still writes (janus_common.cuh: launch_kernel), so none may read global memory
through the read-only path, which asks for memory that nobody writes during the kernel's whole life.  No run shows a breach; the source does."""
import os
import re

from paper_2609_36938_b200 import build


def test_no_read_only_loads():
    shared = {"wchunk"}      # pointers into shared memory
    for name in sorted(os.listdir(build.CSRC)):
        with open(os.path.join(build.CSRC, name)) as f:
            code = re.sub(r"//[^\n]*", "", f.read())
        assert "__ldg" not in code and not re.search(r"ld\.global(\.\w+)*\.nc", code), name
        assert {m.group(1) for m in re.finditer(r"const\s+[\w ]+\*\s*__restrict__\s+(\w+)", code)} <= shared, name
