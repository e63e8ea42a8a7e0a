"""A problem's device memory is allocated and freed by one pair of functions."""
import os
import re

from paper_2505_04328_gb300 import _build


def test_problem_memory_is_allocated_as_it_is_freed():
    """free_dev frees with cudaFreeAsync where the problem's allocations are stream-ordered, so no
    member of a problem may come from an allocator of its own."""
    with open(os.path.join(_build.CSRC, "jd_api.cu")) as f:
        code = re.sub(r"//[^\n]*", "", f.read())
    calls = re.findall(r"\bcuda(?:Malloc|MallocAsync|Free|FreeAsync)\(([^;{]*?)[;{]", code)
    assert len(calls) >= 4 and not [c for c in calls if "&p->" in c or re.match(r"p->", c)]
