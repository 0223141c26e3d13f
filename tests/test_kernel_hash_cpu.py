"""The hash that ties the committed traffic record to the kernel source covers
every file the kernels are compiled from."""
import os
import re

import bench

CSRC = os.path.join(bench.ROOT, "paper_0807_4471_gb300", "csrc")


def test_hash_covers_all_included_sources():
    todo, seen = ["lb_kernels.cu"], set()
    while todo:
        f = todo.pop()
        if f in seen or not os.path.exists(os.path.join(CSRC, f)):
            continue
        seen.add(f)
        with open(os.path.join(CSRC, f)) as fh:
            todo += re.findall(r'^\s*#include "([^"/]+)"', fh.read(), flags=re.M)
    assert {os.path.basename(p) for p in bench.KERNEL_SRCS} == seen
