"""Rules that the library's sources keep, checked on their text."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1010_5534_gb300", "csrc")


def _code(name):
    s = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", s)


def test_the_network_entries_allocate_nothing_that_throws():
    """No exception crosses the C interface: the depth network's file uses no
    container that throws when host memory runs out."""
    s = _code("air_mlp.cu")
    assert not re.search(r"\bstd::(vector|string|deque|map)\b", s)
    assert not re.search(r"\bnew\b(?!\s*\(std::nothrow\))", s)
