"""The marshalling of calls rejects what the kernels could not take, before anything is enqueued (no GPU needed)."""
import pytest
import torch

import paper_2602_00523_b200 as sage


def test_host_tensors_and_wrong_types_are_rejected():
    x, i = torch.zeros(2, 8), torch.zeros(2, dtype=torch.int32)
    with pytest.raises(ValueError, match="device tensors only"):
        sage.sage_expand_topk(x, 2, 2)
    with pytest.raises(AssertionError):
        sage.sage_expand_topk(x.half(), 2, 2)
    with pytest.raises(TypeError):                       # a tree policy where the history policy belongs
        sage.sage_update_history(i, sage.make_policy([]), i, i, x)
    with pytest.raises(ValueError, match="device tensors only"):
        sage.sage_accept(i, i, i, i, 4)
    with pytest.raises(AssertionError):
        sage.sage_tree_attention(torch.zeros(1, 2, 8, 128), x, x, i, i, i, i, 1.0, out=x, ws=x)


def test_static_variant_allocates_nothing():
    with pytest.raises(KeyError, match="topk_idx"):
        sage.sage_expand_topk_static(torch.zeros(2, 8), 2, 2, out={})
