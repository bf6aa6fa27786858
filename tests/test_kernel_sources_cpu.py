"""Rules that every kernel keeps because each is launched while the one before it still runs, checked on the sources: no GPU
shows reliably what breaks when one is forgotten."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_00523_b200", "csrc")
WAIT = "after_previous_kernel();"


def kernels():
    """(name, body without comments) of every __global__ function."""
    found = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^)]*\)\s*)?(\w+)\s*\(", text):
            at = text.index("{", m.end())
            depth, end = 1, at + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
            found.append((m.group(1), text[at:end]))
    return found


KERNELS = kernels()


def test_all_kernels_are_found():
    assert len(KERNELS) == 13 and {"attention_merge_kernel", "expand_topk_kernel", "tree_attention_rows_kernel"} <= {n for n, _ in KERNELS}


@pytest.mark.parametrize("name,body", KERNELS, ids=[n for n, _ in KERNELS])
def test_no_thread_leaves_before_the_wait(name, body):
    """A kernel waits for its direct predecessor only, so stream order holds as long as no kernel can finish without
    having waited for its own."""
    assert body.count(WAIT) == 1
    assert not re.search(r"\breturn\b", body[:body.index(WAIT)])


@pytest.mark.parametrize("name,body", KERNELS, ids=[n for n, _ in KERNELS])
def test_nothing_in_global_memory_is_touched_before_the_wait(name, body):
    """Node offsets, lengths and page tables are written on the device every round, and only the wait makes the writes of
    earlier kernels visible."""
    ahead = body[:body.index(WAIT)]
    assert not re.search(r"p\.\w+\s*\[|node_offsets|seq_len|page_table|parent|part_|load_item|make_plan|locate|atomic|report_status", ahead)


@pytest.mark.parametrize("name,body", KERNELS, ids=[n for n, _ in KERNELS])
def test_no_tensor_memory_is_held_while_waiting(name, body):
    """A block that holds it while it waits for the kernel in front can keep a block of that kernel on the same SM from ever
    getting its own."""
    ahead = body[:body.index(WAIT)]
    assert "tcgen05" not in ahead and "set_up" not in ahead
