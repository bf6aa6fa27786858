"""sage_tree_attention where its schedules have edges: launches cut into 1 to 32 context slices (some of them empty) or
into ranges that end inside a sequence; batches that mix trees of one to four row tiles, so that two small trees share a
gang of thread blocks, with an odd number of KV heads; the last row of a tile; node arrays with spare capacity behind the
last tree; and scores that grow along the context until a row's softmax reference has to move, several times."""
import numpy as np
import pytest
import torch

import oracle
import paper_2602_00523_b200 as sage
from helpers import check_attention, dev_bf16, dev_i32, host_bits, widen
from workloads import bf16_bits, make_kv_cache, make_q, random_tree

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("schedule", [1, 2], ids=["streaming", "split"])
@pytest.mark.parametrize("layers,heads,G,Ls,Ns,ramp,spare", [
    (1, 1, 8, [4100], [17], 0, 0),                                     # most slices (row tile 1 holds 8 rows)
    (1, 8, 8, [1090], [60], 0, 2),                                     # nine slices
    (3, 8, 8, [600], [60], 0, 0), (2, 8, 8, [700, 90], [33, 16], 0, 4),    # few; a sequence that leaves slices empty
    (2, 7, 8, [300, 1300, 64, 129], [60, 9, 33, 32], 0, 0),            # trees of all sizes, an odd head without a partner
    (1, 2, 8, [2000], [16], 5, 0), (2, 2, 8, [1500, 900], [60, 20], 5, 1),  # growing scores
    (2, 1, 1, [511], [64], 5, 0), (2, 3, 2, [127, 129, 1500], [64, 63, 1], 0, 3)])
def test_attention_edges(schedule, layers, heads, G, Ls, Ns, ramp, spare):
    r = np.random.Generator(np.random.Philox(sum(Ls) + sum(Ns) + heads))
    kv = make_kv_cache(r, Ls, Ns, [l // 2 for l in Ls], heads, n_layers=layers, shuffle=True, spare_frac=0.2)
    if ramp:
        # page i of a sequence times 2^(-2 .. ramp), exactly: the scores' range grows along the context
        for b in range(len(Ls)):
            n = (Ls[b] + Ns[b] + 63) // 64
            for i, page in enumerate(kv["page_table"][b, :n]):
                f = 2.0 ** round(-2 + (ramp + 2) * i / n)
                kv["k_pool"][:, page] = bf16_bits((widen(kv["k_pool"][:, page]) * f).astype(np.float32))
    nodes = sum(Ns)
    q = make_q(r, nodes + spare, heads * G, n_layers=layers)
    parent = np.concatenate([random_tree(r, n)["parent"] for n in Ns] + [np.full(spare, -1)]).astype(np.int32)
    off = np.concatenate([[0], np.cumsum(Ns)]).astype(np.int32)
    st = sage.new_status()
    out = torch.zeros(layers, nodes + spare, heads * G, 128, dtype=torch.bfloat16, device="cuda")
    sage.sage_debug_attention_schedule(schedule)
    try:
        sage.sage_tree_attention(dev_bf16(q), dev_bf16(kv["k_pool"]), dev_bf16(kv["v_pool"]), dev_i32(kv["page_table"]),
                                 dev_i32(kv["seq_len"]), dev_i32(parent), dev_i32(off), 128 ** -0.5, out=out, status=st)
        torch.cuda.synchronize()
    finally:
        sage.sage_debug_attention_schedule(0)
    assert int(st.item()) == 0
    got = host_bits(out)
    assert not got[:, nodes:].any()                                    # spare rows are not written
    for layer in range(layers):
        want = oracle.tree_attention(q[layer, :nodes], kv["k_pool"][layer], kv["v_pool"][layer], kv["page_table"], kv["seq_len"],
                                     parent[:nodes], off, heads * G, heads, 128, 64, 128 ** -0.5)
        # Probabilities are rounded to bf16: at most 2^-9 of the largest value in play (below 5) = 0.0098 per output
        # before its own rounding, for which the half unit is added.
        check_attention(got[layer, :nodes], want, bf16_slack=True)
