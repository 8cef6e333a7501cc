"""A kernel that is launched early (programmatic dependent launch) is resident while its predecessors still write what it will read, so
the non-coherent load, which is for data that nothing writes during the kernel's whole lifetime, is not for anything a call computes.
Three ways to ask for it: the instruction itself, __ldg, and a pointer to const with __restrict__, of which the compiler may make one."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_15773_b200", "csrc")
FILES = sorted(os.listdir(CSRC))

# set when the weights are loaded: weights and the tables of the timesteps
LOADED = set("""W W_in b_in W_outT b_out pos cpos bias b gam bet g be ln1_g ln1_b ln3_g ln3_b lnf_g lnf_b bo2 mod kv_time pos_row w_row
w.W_o w.W_a w.W_1 P.W_in P.b_in P.pos g.bias""".split()) | {"mrow", "gate_base", "gp", "wp", "wr"}      # (rows of them, by their local names)
# copied to the device before the first kernel of a call
COPIED = {"sched", "seedp", "obs", "progress", "n_items"}


def _code(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def _functions(code):
    """Functions of the device, but for kernels that are launched behind everything before them."""
    for f in re.split(r"(?=__global__|__device__)", code)[1:]:
        if f.startswith("__device__") or "pdl_wait()" in f:
            yield f


@pytest.mark.parametrize("name", FILES)
def test_no_load_is_written_as_non_coherent(name):
    assert not re.findall(r"ld\.global\S*\.nc\b", _code(name))


@pytest.mark.parametrize("name", FILES)
def test_read_only_loads_are_of_data_that_no_call_writes(name):
    for f in _functions(_code(name)):
        for arg in re.findall(r"__ldg\((.*)", f):
            root = re.match(r"(?:reinterpret_cast<[^>]*>\()?\(*([A-Za-z_][\w.]*)", arg).group(1)
            assert root in LOADED, (root, arg)


@pytest.mark.parametrize("name", FILES)
def test_restricted_pointers_to_const_are_to_data_that_no_call_writes(name):
    for f in _functions(_code(name)):
        got = set(re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", f))
        assert got <= LOADED | COPIED, (got - LOADED - COPIED, f[:200])
