"""Kernels read nothing of a metadata buffer but its header before the header has matched the call (no GPU needed).

The attention entry points are given the buffer's address and not its size, so the offsets of its arrays follow from the sizes
the caller names; in a buffer that was built for a smaller batch they may lie past its end.  A read there can fault, so it is
the source that is checked: in every function that tests the header, no element of anything but shared memory is loaded
before the test."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_35750_b200", "csrc")


def _functions_that_test_the_header():
    found = []
    for name in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(os.path.join(CSRC, name)).read(), flags=re.S)
        for at in re.finditer(r"\bif \(!meta_matches\(", text):
            start = max(text.rfind("\n" + kind, 0, at.start()) for kind in ("__global__", "__device__"))
            body = text.index(") {\n", start)
            found.append((name, text[body:at.start()]))
    return found


FOUND = _functions_that_test_the_header()


@pytest.mark.parametrize("name,before", FOUND, ids=[f"{name}-{i}" for i, (name, _) in enumerate(FOUND)])
def test_only_the_header_is_read_before_it_matches(name, before):
    before = re.sub(r"[^;{}]*__shared__[^;]*;", "", before)
    loads = re.findall(r"\w+\s*\[[^\]]+\]|__ld\w+\s*\(|=\s*\*\w+", before)
    assert not loads, (name, loads)


def test_all_main_kernels_and_the_plan_are_covered():
    assert sorted(n for n, _ in FOUND) == ["kvs_bwd.cu", "kvs_bwd.cu", "kvs_bwd_pair.cu", "kvs_fwd.cu"]
