"""Orderings the kernels rely on, read in their sources: a missing one is a race
that a run may or may not show."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1309_3452_gb300", "csrc")


def source(name):
    """The file's code without comments."""
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"/\*.*?\*/", "", re.sub(r"//[^\n]*", "", f.read()), flags=re.S)


def body(text, head):
    """The braces that follow the first `head`."""
    i = text.index("{", text.index(head))
    depth = 0
    for j in range(i, len(text)):
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return text[i + 1:j]
    raise ValueError(head)


def test_strip_items_end_with_a_warp_barrier():
    """A wave's factors are written by a few lanes and read by all: between the last read of one item
    and the first write of the warp's next item all lanes meet."""
    march = body(source("fused2d.cuh"), "void march2d(")
    tail = march[march.rindex("cp_async_wait<0>()"):]
    assert re.search(r"if \(LINK == LINK_PLANE\) __syncwarp\(\);", tail)


# what a fused step may read through the read-only path: tables made with the simulation, and the
# argument tables of a batched call, uploaded before its first launch
FIXED = ("sc_sq", "b_map", "class_z", "sc_corr", "t + 2 *", "first + mid", "s + i")


@pytest.mark.parametrize("name", ["quad.cuh", "fused2d.cuh", "fused3d.cuh", "fused_common.cuh"])
def test_evolving_data_is_read_by_ordinary_loads(name):
    """A dependent launch is resident while the one before it writes the state and a wave's factors."""
    text = source(name)
    for m in re.finditer(r"__ldg\(", text):
        arg = text[m.end():m.end() + 60]
        assert any(f in arg for f in FIXED), arg
    # "t" in quad.cuh is the static link table or the coefficient table
    assert set(re.findall(r"const float4\* t = ([\w.]+)", text)) <= {"h.lq", "h.bq"}


def test_no_copies_on_the_legacy_stream():
    """Kernels on a non-blocking stream are not ordered after what goes through the legacy one."""
    for name in sorted(os.listdir(CSRC)):
        assert not re.search(r"\bcuda(Memcpy|Memset)\(", source(name)), name


def test_grid_rules_ask_for_the_device_size():
    assert "152" not in source("step_split.cu")
    assert "sm_count()" in body(source("observables.cu"), "int observables_blocks(")
