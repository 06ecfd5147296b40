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


def test_dependent_kernels_read_by_ordinary_loads():
    """A kernel that is launched while the one before it still runs takes no
    pointer as `const __restrict__`: the compiler may read through those with
    read-only loads, which must not be used for what that kernel writes."""
    found = 0
    for name in sorted(os.listdir(CSRC)):
        s = _code(name)
        for m in re.finditer(r"__global__\s+void\b", s):
            body = s.index("{", m.end())
            end = s.find("__global__", m.end())
            if "wait_prior_grid()" not in s[body:end if end > 0 else len(s)]:
                continue
            found += 1
            bad = re.findall(r"const\s+\w+\s*\*\s*__restrict__\s*\w+", s[m.end():body])
            assert not bad, (name, bad)
    assert found >= 8
