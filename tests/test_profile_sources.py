"""A recorded profile counts only for the sources it was taken from: the hash covers
every file that the plan codec kernels are compiled from."""
import os
import re

import bench


def test_every_included_header_is_hashed():
    csrc = os.path.join(bench.ROOT, "paper_2609_24294_gb300", "csrc")
    seen, todo = set(), ["codec.cu"]
    while todo:
        name = todo.pop()
        if name in seen:
            continue
        seen.add(name)
        with open(os.path.join(csrc, name)) as f:
            todo += [i for i in re.findall(r'#include "([^"/]+)"', f.read())]
    assert seen == set(bench.CODEC_SOURCES)
