"""Every kernel launched with launch_dep may start before its predecessor has completed, so it waits
(griddepcontrol.wait, in dep_begin) in every thread before it reads anything another kernel wrote."""
import glob
import os
import re

import pytest

from tests.simt import CSRC

SOURCES = {os.path.basename(f): open(f).read() for f in glob.glob(os.path.join(CSRC, "*.cu"))}


def _launched():
    names = set()
    for text in SOURCES.values():
        names |= set(re.findall(r"launch_dep\(\s*(k_\w+)", text))
    return sorted(names)


def _kernel(name):
    for text in SOURCES.values():
        m = re.search(r"__global__[^;{]*?\b%s\s*\(" % name, text)
        if m:
            i = text.index("{", m.end())
            return text[m.end():i], text[i:]
    raise AssertionError(name)


@pytest.mark.parametrize("name", _launched())
def test_waits_before_the_first_read(name):
    params, body = _kernel(name)
    at = body.index("dep_begin();")
    start = re.sub(r"//[^\n]*", "", body[:at])
    assert re.search(r"[;{}]\s*$", start) and start.count("{") == 1, "dep_begin() is conditional"
    for p in re.findall(r"(\w+)\s*(?:,|\)|$)", re.sub(r"\)\s*$", "", params)):
        assert not re.search(r"\b%s\b" % p, start), f"{p} is used before the wait"
