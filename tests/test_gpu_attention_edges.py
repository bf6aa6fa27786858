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


@pytest.mark.parametrize("layers,heads,G,L,N,batch,width", [
    (80, 8, 8, 100, 12, 1, 19),             # items of one step
    (80, 8, 8, 90, 36, 1, 19),              # the same with trees of two row pairs
    (1, 8, 8, 200, 12, 16, 28),             # two steps, a thread block for each item
    (1, 8, 8, 200, 30, 37, 6)])             # two whole items per thread block
def test_launches_in_which_no_range_cuts_an_item(layers, heads, G, L, N, batch, width):
    """Nothing to merge: every block of the merge leaves at once, and what follows in the stream must find the attention
    finished all the same.  Rounds of attention, then compaction of the very rows that it reads, without a pause."""
    r = np.random.Generator(np.random.Philox(layers * 1000 + batch + N))
    tree = random_tree(r, N)
    used = (L + N + 63) // 64
    kv = make_kv_cache(r, [L] * batch, [N] * batch, [L // 2] * batch, heads, n_layers=layers, shuffle=True, spare_frac=0.1)
    table = np.full((batch, width), -1, np.int32)
    table[:, :used] = kv["page_table"][:, :used]
    path = np.full((batch, 9), -1, np.int32)         # the last node's root path: its rows have the furthest to go
    chain = [N - 1]
    while chain[-1]:
        chain.append(int(tree["parent"][chain[-1]]))
    path[:, :len(chain)] = chain[::-1][:9]
    length = np.full(batch, min(9, len(chain)), np.int32)
    q = make_q(r, batch * N, heads * G, n_layers=layers)
    parent, off = np.tile(tree["parent"], batch).astype(np.int32), (np.arange(batch + 1) * N).astype(np.int32)
    st, dev = sage.new_status(), dict(q=dev_bf16(q), table=dev_i32(table), parent=dev_i32(parent), off=dev_i32(off),
                                      path=dev_i32(path), length=dev_i32(length), L=dev_i32(kv["seq_len"]))
    k0, v0 = dev_bf16(kv["k_pool"]), dev_bf16(kv["v_pool"])
    outs = [torch.zeros_like(dev["q"]) for _ in range(4)]
    sage.sage_debug_attention_schedule(1)
    try:
        for out in outs:
            k, v, seq = k0.clone(), v0.clone(), dev["L"].clone()
            sage.sage_tree_attention(dev["q"], k, v, dev["table"], seq, dev["parent"], dev["off"], 128 ** -0.5, out=out, status=st)
            sage.sage_compact_kv(k, v, dev["table"], seq, dev["path"], dev["length"], status=st)
        torch.cuda.synchronize()
    finally:
        sage.sage_debug_attention_schedule(0)
    assert int(st.item()) == 0
    assert np.array_equal(seq.cpu().numpy(), kv["seq_len"] + length)
    for out in outs[1:]:
        assert torch.equal(out.view(torch.int16), outs[0].view(torch.int16))
    got = host_bits(outs[0])
    for layer in sorted({0, layers // 2, layers - 1}):
        want = oracle.tree_attention(q[layer], kv["k_pool"][layer], kv["v_pool"][layer], table, kv["seq_len"], parent, off,
                                     heads * G, heads, 128, 64, 128 ** -0.5)
        check_attention(got[layer], want, bf16_slack=True)       # (bound: see test_attention_edges)


@pytest.mark.parametrize("schedule", [1, 2], ids=["streaming", "split"])
@pytest.mark.parametrize("N", [5, 21, 37])
@pytest.mark.parametrize("behind", ["spare", "sequence"])
def test_rows_behind_a_tree_do_not_change_a_bit_of_it(schedule, N, behind):
    """The last warp of a tree's rows also holds rows that are not the tree's: spare capacity, or the next sequence's.  Rows
    beside it that have to move their softmax reference must not make a row of the tree go another way."""
    r = np.random.Generator(np.random.Philox(N))
    heads, G, L = 2, 8, 1500
    Ns = [N] if behind == "spare" else [N, 8]
    kv = make_kv_cache(r, [L] * len(Ns), Ns, [0] * len(Ns), heads, shuffle=True)
    for i, page in enumerate(kv["page_table"][0, :(L + N + 63) // 64]):      # scores that grow and fall along the context
        kv["k_pool"][:, page] = bf16_bits((widen(kv["k_pool"][:, page]) * (1 + i // 2 % 12 / 2)).astype(np.float32))
    parent = np.concatenate([random_tree(r, n)["parent"] for n in (N, 8)]).astype(np.int32)
    off = np.concatenate([[0], np.cumsum(Ns)]).astype(np.int32)
    q = make_q(r, N + 8, heads * G)
    got = []
    sage.sage_debug_attention_schedule(schedule)
    try:
        for f in (0.0, 30.0):
            q_f = q.copy()
            q_f[:, N:] = bf16_bits((widen(q[:, N:]) * f).astype(np.float32))
            st = sage.new_status()
            out = sage.sage_tree_attention(dev_bf16(q_f), dev_bf16(kv["k_pool"]), dev_bf16(kv["v_pool"]), dev_i32(kv["page_table"]),
                                           dev_i32(kv["seq_len"]), dev_i32(parent), dev_i32(off), 128 ** -0.5, status=st)
            torch.cuda.synchronize()
            assert int(st.item()) == 0
            got.append(host_bits(out)[0, :N])
    finally:
        sage.sage_debug_attention_schedule(0)
    np.testing.assert_array_equal(got[0], got[1])


@pytest.mark.parametrize("schedule", [1, 2], ids=["streaming", "split"])
@pytest.mark.parametrize("N", [12, 30])
def test_the_reference_stays_close_enough_for_the_largest_probability(schedule, N):
    """Scores that grow by 2^8 to 2^30 within a thread block's range.  A row's largest probability is exact where the softmax
    reference is its score and rounded to bf16 (2^-9) where the reference lags; rows dominated by a few keys show that.  Rounding
    the outputs costs 1.66e-3 of their 2-norm (uniform within a unit, over spread mantissas); a dominant probability that is
    rounded as well brings that to 1.66e-3 * 2^0.5 = 2.3e-3 at most.  The bound lies between: references that may lag by 2^8
    or 2^12 gave 1.71e-3 to 1.87e-3, by 2^30 2.08e-3 to 2.16e-3."""
    r = np.random.Generator(np.random.Philox(100 + N))
    layers, heads, G, L = 4, 8, 8, 3000
    kv = make_kv_cache(r, [L], [N], [0], heads, n_layers=layers, shuffle=True)
    for i, page in enumerate(kv["page_table"][0, :(L + N + 63) // 64]):
        kv["k_pool"][:, page] = bf16_bits((widen(kv["k_pool"][:, page]) * (1 + i % 12 / 2)).astype(np.float32))
    parent, off = random_tree(r, N)["parent"], np.array([0, N], np.int32)
    q = make_q(r, N, heads * G, n_layers=layers)
    st = sage.new_status()
    sage.sage_debug_attention_schedule(schedule)
    try:
        out = sage.sage_tree_attention(dev_bf16(q), dev_bf16(kv["k_pool"]), dev_bf16(kv["v_pool"]), dev_i32(kv["page_table"]),
                                       dev_i32(kv["seq_len"]), dev_i32(parent), dev_i32(off), 128 ** -0.5, status=st)
        torch.cuda.synchronize()
    finally:
        sage.sage_debug_attention_schedule(0)
    assert int(st.item()) == 0
    got, err, ref = host_bits(out), 0.0, 0.0
    for layer in (0, layers - 1):
        want = oracle.tree_attention(q[layer], kv["k_pool"][layer], kv["v_pool"][layer], kv["page_table"], kv["seq_len"], parent, off,
                                     heads * G, heads, 128, 64, 128 ** -0.5)
        err, ref = err + ((widen(got[layer]) - want) ** 2).sum(), ref + (want ** 2).sum()
    assert (err / ref) ** 0.5 <= 2.0e-3, (err / ref) ** 0.5


def test_widely_spread_scores_take_little_longer():
    """Steps in which a row outgrows its softmax reference are computed twice.  Scores of three times the usual spread took 1.35
    times as long as usual ones where the reference followed a row's maximum at a distance of 2^8, 1.1 times with 2^12."""
    L, N, heads, G = 16384, 60, 8, 8
    pages = (L + N + 63) // 64
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    k, v = (torch.randn(1, pages, heads, 64, 128, generator=gen, device="cuda").bfloat16() for _ in range(2))
    q = torch.randn(1, N, heads * G, 128, generator=gen, device="cuda").bfloat16()
    table, off = torch.randperm(pages, generator=gen, device="cuda").to(torch.int32)[None], dev_i32([0, N])
    parent = dev_i32(random_tree(np.random.Generator(np.random.Philox(1)), N)["parent"])
    out, L = torch.empty_like(q), dev_i32([L])
    ws = torch.empty(sage.sage_tree_attention_workspace_size(1, 1, N, heads * G, heads, 128, pages), dtype=torch.uint8, device="cuda")

    def us(keys):
        times = []
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                sage.sage_tree_attention(q, keys, v, table, L, parent, off, 128 ** -0.5, out=out, ws=ws)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return min(times)

    k[:, table[0, :2 * pages // 5].long()] *= 1.5        # (the visual part of a context)
    usual = us(k)
    assert us(k * 3) <= 1.25 * usual


@pytest.mark.parametrize("heads,Ns", [(8, [12]), (8, [40, 12, 20, 9]), (7, [36, 5]), (3, [24])], ids=["one_tile", "mixed", "odd_heads", "two_tiles"])
def test_ranges_that_end_at_the_end_of_an_item(heads, Ns):
    """Items of one to nine steps, ranges of about as many: boundaries fall on every step of an item, and into the extra that stands for
    its end, where the range ends with the item and the next one starts with the next item."""
    r = np.random.Generator(np.random.Philox(heads * 100 + len(Ns)))
    batch, G = 24, 8
    Ns = [Ns[b % len(Ns)] for b in range(batch)]
    Ls = [int(v) for v in r.integers(1, 1100, batch)]
    kv = make_kv_cache(r, Ls, Ns, [0] * batch, heads, shuffle=True)
    q = make_q(r, sum(Ns), heads * G)
    parent = np.concatenate([random_tree(r, n)["parent"] for n in Ns]).astype(np.int32)
    off = np.concatenate([[0], np.cumsum(Ns)]).astype(np.int32)
    st = sage.new_status()
    sage.sage_debug_attention_schedule(1)
    try:
        out = sage.sage_tree_attention(dev_bf16(q), dev_bf16(kv["k_pool"]), dev_bf16(kv["v_pool"]), dev_i32(kv["page_table"]),
                                       dev_i32(kv["seq_len"]), dev_i32(parent), dev_i32(off), 128 ** -0.5, status=st)
        torch.cuda.synchronize()
    finally:
        sage.sage_debug_attention_schedule(0)
    assert int(st.item()) == 0
    want = oracle.tree_attention(q[0], kv["k_pool"][0], kv["v_pool"][0], kv["page_table"], kv["seq_len"], parent, off, heads * G, heads,
                                 128, 64, 128 ** -0.5)
    check_attention(host_bits(out)[0], want, bf16_slack=True)       # (bound: see test_attention_edges)


@pytest.mark.parametrize("G,N,batch,heads", [(4, 24, 21, 7), (8, 60, 9, 8), (1, 12, 16, 8)], ids=["147_items", "72_pairs", "128_items"])
def test_items_of_two_steps_are_not_cut_while_there_is_a_gang_for_each(G, N, batch, heads):
    """Nearly as many items as thread blocks (or pairs of them): equal ranges would cut every one.  An item that is not cut has the bits that
    it has in a launch of its own."""
    r = np.random.Generator(np.random.Philox(batch))
    L = 250 - N
    kv = make_kv_cache(r, [L] * batch, [N] * batch, [0] * batch, heads, shuffle=True)
    q, parent = make_q(r, batch * N, heads * G), random_tree(r, N)["parent"].astype(np.int32)
    k, v, qd = dev_bf16(kv["k_pool"]), dev_bf16(kv["v_pool"]), dev_bf16(q)
    st = sage.new_status()

    def attention(b0, b1):
        return sage.sage_tree_attention(qd[:, b0 * N:b1 * N].contiguous(), k, v, dev_i32(kv["page_table"][b0:b1]), dev_i32(kv["seq_len"][b0:b1]),
                                        dev_i32(np.tile(parent, b1 - b0)), dev_i32(np.arange(b1 - b0 + 1) * N), 128 ** -0.5, status=st)
    sage.sage_debug_attention_schedule(1)
    try:
        together, alone = attention(0, batch), torch.cat([attention(b, b + 1) for b in range(batch)], dim=1)
        torch.cuda.synchronize()
    finally:
        sage.sage_debug_attention_schedule(0)
    assert int(st.item()) == 0
    np.testing.assert_array_equal(host_bits(together), host_bits(alone))


def test_a_nearly_empty_row_tile_costs_no_more_than_a_half_empty_one():
    """Seventeen nodes of eight queries leave the second row tile eight rows, in one warp; twenty-four leave it two warps of rows.  While
    warps without rows polled beside the working ones, the smaller trees took 1.03 times as long as the larger, now 0.96 times."""
    L, batch, heads, G = 24 * 64 - 64, 9, 8, 8
    gen = torch.Generator(device="cuda")
    gen.manual_seed(4)
    k, v = (torch.randn(4, batch * 24, heads, 64, 128, generator=gen, device="cuda").bfloat16() for _ in range(2))     # (beyond L2)
    table = torch.randperm(batch * 24, generator=gen, device="cuda").to(torch.int32).reshape(batch, 24)
    seq, times = dev_i32([L] * batch), {}
    st = sage.new_status()
    sage.sage_debug_attention_schedule(2)
    try:
        calls = {}
        for N in (17, 24):
            q = torch.randn(1, batch * N, heads * G, 128, generator=gen, device="cuda").bfloat16()
            parent = dev_i32(np.tile(random_tree(np.random.Generator(np.random.Philox(1)), N)["parent"], batch))
            off, out = dev_i32(np.arange(batch + 1) * N), torch.empty_like(q)
            ws = torch.empty(max(16, sage.sage_tree_attention_workspace_size(1, batch, batch * N, heads * G, heads, 128, 24)),
                             dtype=torch.uint8, device="cuda")
            calls[N] = (q, parent, off, out, ws)
        for _ in range(8):                               # in turn
            for N, (q, parent, off, out, ws) in calls.items():
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                for i in range(40):
                    sage.sage_tree_attention(q, k[i % 4:i % 4 + 1], v[i % 4:i % 4 + 1], table, seq, parent, off, 128 ** -0.5, out=out, ws=ws, status=st)
                b.record()
                torch.cuda.synchronize()
                times[N] = min(times.get(N, 1e9), a.elapsed_time(b))
    finally:
        sage.sage_debug_attention_schedule(0)
    assert int(st.item()) == 0
    assert times[17] <= times[24], times


@pytest.mark.parametrize("N", [1, 4, 5, 9, 13, 17, 20, 21, 25, 29, 33, 49, 53, 57])
def test_row_tiles_of_one_to_four_warps(N):
    """The split schedule with one to four warps of rows in the first to the fourth row tile; warps without rows take no part."""
    r = np.random.Generator(np.random.Philox(300 + N))
    heads, G, Ls = 2, 8, [300, 700]
    kv = make_kv_cache(r, Ls, [N, N], [0, 0], heads, shuffle=True)
    q = make_q(r, 2 * N, heads * G)
    parent, off = np.concatenate([random_tree(r, N)["parent"] for _ in Ls]).astype(np.int32), np.array([0, N, 2 * N], np.int32)
    st = sage.new_status()
    sage.sage_debug_attention_schedule(2)
    try:
        out = sage.sage_tree_attention(dev_bf16(q), dev_bf16(kv["k_pool"]), dev_bf16(kv["v_pool"]), dev_i32(kv["page_table"]),
                                       dev_i32(kv["seq_len"]), dev_i32(parent), dev_i32(off), 128 ** -0.5, status=st)
        torch.cuda.synchronize()
    finally:
        sage.sage_debug_attention_schedule(0)
    assert int(st.item()) == 0
    want = oracle.tree_attention(q[0], kv["k_pool"][0], kv["v_pool"][0], kv["page_table"], kv["seq_len"], parent, off, heads * G, heads,
                                 128, 64, 128 ** -0.5)
    check_attention(host_bits(out)[0], want, bf16_slack=True)       # (bound: see test_attention_edges)


@pytest.mark.parametrize("pages", [1, 31, 32, 33, 224, 225, 255, 256, 257])
def test_page_tables_that_are_read_ahead_and_wider_ones(pages):
    """The split schedule reads rows of up to 256 page ids whole, 32 at a time, wider ones where it needs them.  Two sequences, the second
    of which uses its row to the last slot of the last page."""
    r = np.random.Generator(np.random.Philox(400 + pages))
    heads, G, N = 1, 8, 6
    Ls = [max(0, pages * 32 - 5), pages * 64 - N]
    kv = make_kv_cache(r, Ls, [N, N], [0, 0], heads, shuffle=True)
    assert kv["page_table"].shape[1] == pages and (kv["page_table"][1] >= 0).all()
    q = make_q(r, 2 * N, heads * G)
    parent, off = np.concatenate([random_tree(r, N)["parent"] for _ in Ls]).astype(np.int32), np.array([0, N, 2 * N], np.int32)
    st = sage.new_status()
    sage.sage_debug_attention_schedule(2)
    try:
        out = sage.sage_tree_attention(dev_bf16(q), dev_bf16(kv["k_pool"]), dev_bf16(kv["v_pool"]), dev_i32(kv["page_table"]),
                                       dev_i32(kv["seq_len"]), dev_i32(parent), dev_i32(off), 128 ** -0.5, status=st)
        torch.cuda.synchronize()
    finally:
        sage.sage_debug_attention_schedule(0)
    assert int(st.item()) == 0
    want = oracle.tree_attention(q[0], kv["k_pool"][0], kv["v_pool"][0], kv["page_table"], kv["seq_len"], parent, off, heads * G, heads,
                                 128, 64, 128 ** -0.5)
    check_attention(host_bits(out)[0], want, bf16_slack=True)       # (bound: see test_attention_edges)
