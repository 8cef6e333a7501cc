"""A kernel that is launched early (programmatic dependent launch) is resident while its predecessors still write what it will read, so
the non-coherent load, which is for data that nothing writes during the kernel's whole lifetime, is not for anything a call computes."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_15773_b200", "csrc")


def _code(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


@pytest.mark.parametrize("name", sorted(os.listdir(CSRC)))
def test_no_load_is_written_as_non_coherent(name):
    assert not re.findall(r"ld\.global\S*\.nc\b", _code(name))
