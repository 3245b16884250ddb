"""Shared memory of another CTA is touched only once that CTA is known to run: in every kernel a barrier of its cluster stands in
front of the first access through map_shared_rank (a lambda that only returns the address is not an access).  Read from the source,
since a kernel that breaks the rule mostly works."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2405_01067_b200", "csrc")
BARRIER = re.compile(r"cluster\w*(\(\))?\.(sync|barrier_wait)\(")


def kernels():
    for name in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        for part in text.split("__global__")[1:]:
            body = part[:part.index("\n}\n")]
            if "map_shared_rank" in body:
                yield pytest.param(body, id=f"{name}:{re.search(r'(\w+_kernel)', body).group(1)}")


@pytest.mark.parametrize("body", list(kernels()))
def test_barrier_before_first_access(body):
    lines = body.split("\n")
    access = next(i for i, line in enumerate(lines) if "map_shared_rank" in line and not line.strip().startswith("return"))
    assert any(BARRIER.search(line) for line in lines[:access])
