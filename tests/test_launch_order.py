"""What programmatic dependents rely on, read from the sources: a kernel waits for the launch in front of it before it
releases the one behind it."""
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
