"""The marshalling of calls rejects what the kernels could not take, before anything is enqueued (no GPU needed)."""
from collections import UserDict, defaultdict

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


@pytest.mark.parametrize("kind", [dict, UserDict, lambda d: defaultdict(lambda: torch.zeros(4), d)])
def test_outputs_and_trees_may_be_any_mapping(kind):
    """Anything with items by name serves: the calls below get as far as the check of where the tensors are."""
    x, i = torch.zeros(2, 8), torch.zeros(2, dtype=torch.int32)
    names = ["topk_idx", "topk_logprob", "entropy_full", "entropy_topk", "alpha", "lse"]
    with pytest.raises(ValueError, match="device tensors only"):
        sage.sage_expand_topk_static(x, 2, 2, out=kind({n: x for n in names}))
    tree = {n: i for n in ("parent", "rank", "depth", "token", "n_nodes", "frontier_begin")}
    with pytest.raises(ValueError, match="device tensors only"):
        sage.sage_grow_tree(torch.zeros(128, 4, dtype=torch.int32), x, x, sage.make_policy([]), kind({**tree, "cum_logprob": x}))
    with pytest.raises(ValueError, match="device tensors only"):
        sage.sage_accept(i, i, i, i, 4, out=kind({"path": i, "path_len": i, "bonus_token": i}))
    with pytest.raises(KeyError):
        sage.sage_grow_tree(torch.zeros(128, 4, dtype=torch.int32), x, x, sage.make_policy([]), UserDict(parent=i))
    with pytest.raises(TypeError):
        sage.sage_accept(i, i, i, i, 4, out=3)
