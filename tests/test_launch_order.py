"""What programmatic dependents rely on, read from the sources: a kernel waits for the launch in front of it before it
releases the one behind it, and pins the pointers that the compiler may read ahead of a wait."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_27744_b200", "csrc")


def _statements(path):
    text = re.sub(r"//[^\n]*", "", open(path).read())
    return [s.strip() for s in re.split(r"[;{}]", text) if s.strip()]


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu"))), ids=os.path.basename)
def test_a_kernel_waits_before_it_releases(path):
    s = _statements(path)
    for i, statement in enumerate(s):
        if "griddep_launch_dependents()" not in statement:
            continue
        assert statement in ("griddep_launch_dependents()", "ptx::griddep_launch_dependents()"), "released under a condition"
        if s[i - 1].startswith("if (!beside)"):   # the request table, beside the request half: see launch_dependent
            continue
        assert re.match(r"(ptx::)?griddep_wait(_for)?\(", s[i - 1]), f"{s[i - 1]!r} in front of a release"


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu"))), ids=os.path.basename)
def test_a_wait_names_what_may_be_read_ahead_of_it(path):
    # a load through a const __restrict__ pointer may be moved over any fence, so a plain wait does not hold it back
    text = re.sub(r"//[^\n]*", "", open(path).read())
    for k in re.split(r"\b__global__\b", text)[1:]:
        if "griddep_wait" not in k:
            continue
        k = re.sub(r"__launch_bounds__\((?:[^()]|\([^()]*\))*\)", "", k)
        name, params = re.search(r"(\w+)\(([^{]*)\)\s*\{", k).groups()
        read = re.findall(r"\bconst\s+\w+\s*\*\s*__restrict__\s+(\w+)", params)
        named = {n.strip() for group in re.findall(r"griddep_wait_for\(([^)]*)\)", k) for n in group.split(",")}
        missing = [n for n in read if n not in named]
        assert not missing, f"{name} reads {missing} behind a wait that does not name them"
