"""Asynchronous copies are waited for.  `cp.async.wait_group` and `cp.async.bulk.wait_group` wait for committed groups only: a copy that
no commit precedes the wait for is not waited for at all, and the data are there only when other work happens to take longer.
`cp.async.wait_all` waits for every copy of the thread.  Read from the sources, in the order of the text: a race that usually goes well
does not show in a run."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_04002_b200", "csrc")
EFFECTS = [  # instruction -> (kind of copy, what it does)
    (r"cp\.async\.bulk\.commit_group", ("bulk", "commit")), (r"cp\.async\.bulk\.wait_group", ("bulk", "wait for groups")),
    (r"cp\.async\.bulk\.", ("bulk", "copy")),
    (r"cp\.async\.commit_group", ("thread", "commit")), (r"cp\.async\.wait_group", ("thread", "wait for groups")),
    (r"cp\.async\.wait_all", ("thread", "wait for all")), (r"cp\.async\.c[ag]\.", ("thread", "copy")),
]
HELPER = re.compile(r"__forceinline__ void (\w+)\([^)]*\)\s*\{\s*asm volatile\(\"([^\"]+)")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))


def helpers():
    """Name of each one-instruction helper -> its effect."""
    out = {}
    for path in sources():
        for name, text in HELPER.findall(open(path).read()):
            for pattern, effect in EFFECTS:
                if re.match(pattern, text):
                    out[name] = effect
                    break
    return out


def unwaited(text, known):
    """(kind, name of the wait) of every wait for groups that follows a copy that is not in a group."""
    text = re.sub(r"//[^\n]*", "", HELPER.sub("", text))
    pending, bad = {"thread": False, "bulk": False}, []
    for call in re.finditer(r"\b(%s)\(" % "|".join(known), text):
        kind, does = known[call.group(1)]
        if does == "copy":
            pending[kind] = True
        elif does == "wait for groups" and pending[kind]:
            bad.append((kind, call.group(1)))
        else:
            pending[kind] = False
    return bad + [(kind, "end of file") for kind, left in pending.items() if left]


def test_the_helpers_are_recognised():
    does = set(helpers().values())
    assert {("thread", "copy"), ("bulk", "copy"), ("bulk", "commit"), ("bulk", "wait for groups")} <= does
    assert ("thread", "wait for all") in does or ("thread", "wait for groups") in does


@pytest.mark.parametrize("name", [os.path.basename(p) for p in sources()])
def test_every_copy_is_waited_for(name):
    assert unwaited(open(os.path.join(CSRC, name)).read(), helpers()) == []
