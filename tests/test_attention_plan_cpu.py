"""Which schedule sage_tree_attention gives a launch: host arithmetic, for 148 multiprocessors where there is no GPU to ask."""
import pytest

import paper_2602_00523_b200 as sage

STREAMING, SPLIT = 1, 2


def schedule(layers, batch, nodes, heads, pages):
    return sage.sage_debug_attention_plan(layers, batch, batch * nodes, heads[0], heads[1], pages)["schedule"]


@pytest.mark.parametrize("layers,batch,nodes,heads,pages", [
    (3, 27, 42, (8, 1), 21), (1, 12, 64, (64, 8), 21), (2, 10, 42, (64, 8), 21), (1, 8, 24, (64, 8), 33), (1, 13, 36, (64, 8), 33),
    (1, 39, 64, (8, 1), 40), (1, 11, 60, (64, 8), 40)])
def test_short_launches_are_split_whatever_table_and_arrays_could_hold(layers, batch, nodes, heads, pages):
    """Fewer than twelve steps of 128 keys per multiprocessor even if every table is full: how little there is may not show in the
    sizes, and a streaming launch costs its twenty microseconds all the same."""
    assert layers * batch * heads[1] * -(-pages // 2) < 12 * 148
    assert schedule(layers, batch, nodes, heads, pages) == SPLIT


@pytest.mark.parametrize("heads,narrow,batch", [((64, 8), 33, 18), ((32, 8), 33, 18), ((16, 8), 24, 36), ((8, 8), 24, 36)])
def test_only_narrow_tables_are_split_for_several_long_sequences(heads, narrow, batch):
    """One sequence may fill the table while the others are short: the split launch then takes what that one takes a block of its own,
    the streaming one next to nothing."""
    for pages in (narrow - 1, narrow, narrow + 1, narrow + 4, 40, 41, 129):
        assert schedule(1, batch, 12, heads, pages) == (SPLIT if pages <= narrow else STREAMING), pages


@pytest.mark.parametrize("layers,batch,sum_nodes,heads,pages,overlaps", [
    (1, 1, 10, (32, 8), 33, True),          # 88 split blocks, 40 merge blocks on the 60 multiprocessors left
    (1, 4, 168, (8, 8), 8, False),          # 128, 168 on 20
    (1, 5, 210, (8, 8), 9, False),          # 120, 212 on 28
    (1, 2, 24, (8, 8), 8, True),            # 64, 24 on 84
    (1, 1, 60, (64, 8), 257, False),        # 144, 480 on 4
    (2, 3, 72, (64, 8), 42, True),          # 288: more than one wave
    (1, 1, 60, (64, 8), 1, False)])         # one slice: no merge
def test_a_merge_waits_on_free_multiprocessors_only_if_its_blocks_are_few(layers, batch, sum_nodes, heads, pages, overlaps):
    plan = sage.sage_debug_attention_plan(layers, batch, sum_nodes, heads[0], heads[1], pages)
    assert plan["schedule"] == SPLIT and plan["merge_overlaps"] == overlaps, plan


def test_long_launches():
    assert schedule(80, 1, 60, (64, 8), 257) == STREAMING
    assert schedule(1, 1, 60, (64, 8), 257) == SPLIT
    assert schedule(1, 16, 42, (64, 8), 129) == STREAMING
    assert schedule(1, 70000, 1, (8, 1), 20) == STREAMING           # more items than the split grid takes
    assert schedule(1, 36, 12, (64, 8), 17) == SPLIT                # a wave and most of another, short items


@pytest.mark.parametrize("nodes", [26, 44, 54])
def test_the_long_launches_of_the_parity_tests_are_streamed(nodes):
    """26 layers of three sequences of 33 pages, one row tile to more than two: those tests leave the choice to the library and are about the
    streaming kernels, of which the trees on the device decide."""
    assert sage.sage_debug_attention_plan(26, 3, nodes, 16, 2, 33)["schedule"] == STREAMING


def test_sizes_that_no_call_takes_are_refused():
    with pytest.raises(sage.SageError):
        sage.sage_debug_attention_plan(1, 1, 8, 60, 8, 4)
    with pytest.raises(sage.SageError):
        sage.sage_debug_attention_plan(1, 0, 8, 64, 8, 4)
