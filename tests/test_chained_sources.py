"""A kernel that is launched chained (it waits in chain_wait for the grid
before it) is resident while that grid still writes the data it will read.
The non-coherent load path promises data that does not change for the whole
life of the kernel, so these kernels and the functions that read for them may
not ask for it: no __ldg, no ld.global.nc, no __restrict__ pointer."""
import re
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parents[1] / "paper_2012_11075_gb300" / "csrc"
CHAINED = {"lbm_kernels.cuh": ["strip_pass", "lbm_strip_kernel", "emit_node"],
           "tile.cu": ["lbm_tile_kernel", "lbm_tile_split_kernel"],
           "d3q19.cu": ["d3_density", "d3_chem_pot", "grad3x12", "Node3", "d3_collide",
                        "d3_moments", "d3_step_f32"]}


def source(name):
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", (CSRC / name).read_text(), flags=re.S)


def parameters(text, function):
    """Parameter lists of the definitions of `function` (its name, then a list
    that a body or an initialiser follows)."""
    found = []
    for m in re.finditer(r"\b%s\s*\(" % function, text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        if re.match(r"\s*\{", text[i:]):
            found.append(text[m.end():i - 1])
    return found


@pytest.mark.parametrize("name", sorted(CHAINED))
def test_no_non_coherent_loads_of_chained_data(name):
    text = source(name)
    assert "__ldg" not in text and "global.nc" not in text
    for function in CHAINED[name]:
        lists = parameters(text, function)
        assert lists, function
        assert not any("__restrict__" in p for p in lists), function


def test_every_kernel_that_waits_is_listed():
    for path in CSRC.glob("*.cu*"):
        text = source(path.name)
        kernels = re.split(r"__global__", text)[1:]
        waiting = [k for k in kernels if "chain_wait()" in k.split("__global__")[0]
                   and path.name != "lbm_kernels.cuh"]
        for k in waiting:
            head = k[:k.index("{")]
            assert any(re.search(r"\b%s\s*\(" % f, head) for f in CHAINED.get(path.name, [])), head
