"""bench.py reports DRAM traffic only while the kernel's sources are those of the capture: the guard covers every file that the
kernel is compiled from."""
import importlib.util
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2511_04002_b200", "csrc")


def reached(name, seen):
    """The file and what it includes, directly or not, from the same folder."""
    if name in seen or not os.path.exists(os.path.join(CSRC, name)):
        return seen
    seen.add(name)
    with open(os.path.join(CSRC, name)) as f:
        for inner in re.findall(r'#include "([^"]+)"', f.read()):
            reached(inner, seen)
    return seen


@pytest.mark.parametrize("kernel", ["encode", "decode"])
def test_every_source_of_the_kernel_is_in_the_guard(kernel):
    spec = importlib.util.spec_from_file_location("bench_for_guard", os.path.join(ROOT, "bench.py"))
    bench = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(bench)
    assert set(bench.KERNEL_SOURCES[kernel]) == reached("tsq_%s.cu" % kernel, set())
    assert len(bench.kernel_sources_sha256(kernel)) == 64
