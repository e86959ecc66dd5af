"""Kernels that may begin before the one ahead of them on the stream has ended (programmatic launches) read what that
one writes by ordinary loads: a read-only load promises that nobody writes the word while the kernel lives.  Nothing
can show the difference on a GPU, so the sources are looked at: read-only loads and const __restrict__ parameters only
for the caller's arrays and those of the tiling pass, which are complete before the first such launch."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_05138_b200", "csrc")
FILES = ["screen.cuh", "screen_order.cu", "screen_prep.cu", "sweep_screen.cu", "screen_verify.cu", "screen_dense.cu"]
# weights (p, col, row: pointers into W), the corpus, norms, and the tiling pass's arrays
COMPLETE = {"W", "p", "col", "row", "rowptr", "colidx", "norms", "feat", "rank", "ids", "perm", "key", "tile_len",
            "tile_off", "tile_head"}


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//.*", "", f.read())


@pytest.mark.parametrize("name", FILES)
def test_read_only_loads_are_of_arrays_that_are_complete(name):
    for arg in re.findall(r"__ldg\((?:reinterpret_cast<[^>]*>\()?([\w.]+)", source(name)):
        assert arg.split(".")[-1] in COMPLETE, (name, arg)
    for param in re.findall(r"const [\w]+ \*__restrict__ (\w+)", source(name)):
        # (screen_range_kernel itself is an ordinary launch and writes what it does not read)
        assert param in COMPLETE, (name, param)


def test_every_programmatic_launch_waits():
    """A kernel that is launched so waits before anything else, also where it then has nothing to do."""
    for name in FILES:
        for body in re.split(r"__global__", source(name))[1:]:
            head = body[:body.index("{\n")]
            kernel = re.search(r"(\w+)\(", head.split(")", 1)[1] if "__launch_bounds__" in head else head).group(1)
            if kernel == "screen_range_kernel":
                continue
            wait, leave = body.find("griddepcontrol.wait"), body.find("return")
            assert 0 <= wait < leave or (wait >= 0 and leave < 0), kernel
