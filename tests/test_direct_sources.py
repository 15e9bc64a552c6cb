"""Rules of the direct route's kernels that no run on a GPU would show."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_1108_1320_gb300", "csrc")

# hash tables (complete before a call's first kernel starts) and the batch's
# arguments (copied when the batch is made)
READ_ONLY = re.compile(r"^(h1|h2|hh|a|c)\b|^l\.start|^start")


def body(src, name):
    """The text of kernel `name`, from its parameter list to its last brace."""
    at = re.search(r"\b" + name + r"\(const|\b" + name + r"\([a-zA-Z_]* ", src).start()
    i = src.index("{", src.index(") {", at))
    depth, j = 0, i
    while True:
        depth += {"{": 1, "}": -1}.get(src[j], 0)
        j += 1
        if depth == 0:
            return src[at:j]


@pytest.mark.parametrize("name,path", [("k_direct_tile", "k_direct_tile.cu"), ("k_direct_grid", "k_direct.cu"),
                                       ("k_direct_window", "k_direct.cu"), ("k_direct_finish", "k_direct.cu")])
def test_programmatic_launches_read_results_past_the_read_only_path(name, path):
    # these start while the kernel before them still writes: __ldg (and
    # __restrict__, which lets the compiler use it) only where nothing is written
    with open(os.path.join(CSRC, path)) as f:
        text = body(f.read(), name)
    assert "__restrict__" not in text
    loads = re.findall(r"__ldg\(\s*&?\(?([^;]*)", text)
    for arg in loads:
        assert READ_ONLY.match(arg), arg


def test_superblocks_are_counted_within_a_grid_dimension():
    # a grid's y and z end at 65535: inner indices by the 128 pass that at 8.4 M
    with open(os.path.join(CSRC, "k_direct.cu")) as f:
        src = f.read()
    for dims in re.findall(r"dim3 \w+\(([^;]*)\);|dim3\(([^;]*)\)", src):
        y = (dims[0] or dims[1]).split(",", 1)
        if len(y) == 2 and "nsb" in y[1]:
            assert "65535)" in y[1]
